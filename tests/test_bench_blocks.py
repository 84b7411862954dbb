"""The bench's work models of the trailing updates: units are counted by their chunk's largest order (one large
matrix turns its own chunk into a blocked one, not all), the constants are the library's, and the updates of
a block add up to those of an unblocked factorization's columns."""
import os
import re
import sys

import pytest

from ._util import ROOT

sys.path.insert(0, ROOT)
import bench  # noqa: E402


def _models(ns, chunks=1):
    return bench.kernel_models(16, ns, (0 * bench.np.array(ns, float),) * 4, 1, 2, 1e13, 1.1, 340.0, 6800.0, "mixed",
                               bf16_peak=1900.0, chunks=chunks)


def test_constants_are_the_librarys():
    src = ""
    for name in ("lu.cu", "common.cuh"):
        with open(os.path.join(ROOT, "paper_2311_12134_gb300", "csrc", name)) as f:
            src += f.read()
    assert int(re.search(r"kTwoLevelRows = (\d+)", src).group(1)) == bench.BLOCK_N
    assert int(re.search(r"kBlkK = (\d+)", src).group(1)) == bench.BLOCK_COLS


def test_units_are_counted_by_their_chunk():
    ns = [688] * 50 + [944] + [720] * 49
    assert bench.split_by_chunks(ns, 1) == ([944] + [720] * 49 + [688] * 50, [])
    assert bench.split_by_chunks(ns, 2) == ([944] + [720] * 49, [688] * 50)
    assert bench.split_by_chunks([688] * 3, 5) == ([], [688] * 3)
    both, a, b = _models(ns, 2), _models([944] + [720] * 49), _models([688] * 50)
    assert "k_gemm_tc96" not in b and both["k_gemm_tc96"][0] == pytest.approx(a["k_gemm_tc96"][0])
    for i in (0, 3):
        assert both["k_gemm_tc"][i] == pytest.approx(a["k_gemm_tc"][i] + b["k_gemm_tc"][i])


@pytest.mark.parametrize("n", [800, 928, 944, 2192])
def test_block_updates_against_a_count_by_columns(n):
    fl, _, inner, _ = bench.block_update_work([n])
    want = tri = 0.0
    for k in range(0, n, 32):
        k1 = k // 96 * 96 + 96
        for c in range(k + 32, n):
            if c < k1:
                want += 8.0 * 32 * (n - k - 32)        # within the block, at once
            else:
                tri += 8.0 * 32 * max(0, n - k1)        # later, rows below the block
    assert inner == pytest.approx(want) and fl == pytest.approx(tri)
