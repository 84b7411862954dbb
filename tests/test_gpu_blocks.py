"""The mixed form's factorization in blocks of 96 columns (matrices from n = 800: k_swap_left,
k_swap_trsm_blk in csrc/lu.cu, k_gemm_tc96 in csrc/tc_gemm96.cu, the row-order pass by blocks): orders
whose last block is partial (800, 1200, 1264), a multiple of 96 (1248), one with a
partial block of whole channels (1296, lmax 2), and a chunk that mixes orders.  tau matches the FP64
form to the mixed form's bound (1e-8) with no unit flagged or re-solved."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_12134_gb300 import workload as wl

from ._util import ensure_built, unit_rel_errors


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2311_12134_gb300 import binding
    return binding


def _tau(B, w, lz, precision):
    tau, st = B.tau_blocks(lz, w.lmax, torch.as_tensor(w.species).cuda(), torch.as_tensor(w.tinv).cuda(), w.z, precision)
    return tau.cpu().numpy(), st.cpu().numpy()


@pytest.mark.parametrize("lmax,n_atoms,r_liz", [(3, 50, 1e3), (3, 75, 1e3), (3, 78, 1e3), (3, 79, 1e3), (2, 144, 1e3), (3, 90, 22.0)])
def test_blocked_factorization_against_fp64(B, lmax, n_atoms, r_liz):
    w = wl.cluster(n_atoms, lmax, seed=80 + n_atoms, spread=2.4 * n_atoms ** (1 / 3) + 4.0, r_liz=r_liz)
    lz = B.build_liz(w.pos, w.lattice, w.r_liz)
    K = (lmax + 1) ** 2
    assert K * lz.max_sites >= 800 if r_liz > 100 else K * lz.max_sites > K * lz.min_sites
    tau, st = _tau(B, w, lz, "mixed")
    ref, _ = _tau(B, w, lz, "fp64")
    assert not np.any(st & 0xff)
    assert unit_rel_errors(tau, ref, lz.export()["offsets"]).max() < 1e-8
