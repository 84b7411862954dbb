"""The bench's work models of the trailing updates: units are counted by their own order (a few large ones do
not turn all into blocked ones), the constants are the library's, and the updates of a block add up to those
of an unblocked factorization's columns."""
import os
import re
import sys

import pytest

from ._util import ROOT

sys.path.insert(0, ROOT)
import bench  # noqa: E402


def _models(ns, precision="mixed"):
    return bench.kernel_models(16, ns, (0 * bench.np.array(ns, float),) * 4, 1, 2, 1e13, 1.1, 340.0, 6800.0, precision,
                               bf16_peak=1900.0)


def test_constants_are_the_librarys():
    src = ""
    for name in ("lu.cu", "common.cuh"):
        with open(os.path.join(ROOT, "paper_2311_12134_gb300", "csrc", name)) as f:
            src += f.read()
    assert int(re.search(r"kTwoLevelRows = (\d+)", src).group(1)) == bench.BLOCK_N
    assert int(re.search(r"kBlkK = (\d+)", src).group(1)) == bench.BLOCK_COLS


def test_units_are_counted_by_their_own_order():
    small, large = [688] * 50, [944]
    both = _models(small + large)
    assert both["k_gemm_tc96"][0] == _models(large)["k_gemm_tc96"][0]
    assert both["k_gemm_tc"][0] == pytest.approx(_models(small)["k_gemm_tc"][0] + _models(large)["k_gemm_tc"][0])
    assert both["k_gemm_tc"][3] == pytest.approx(_models(small)["k_gemm_tc"][3] + _models(large)["k_gemm_tc"][3])
    assert "k_gemm_tc96" not in _models(small)


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
