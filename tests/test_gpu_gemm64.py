"""The complex128 LU whose trailing update runs as exact digit products on the tensor cores
(csrc/tc_gemm64.cu), against NumPy's LAPACK solve on the same matrices: sizes around its tiles (one
and two 128-row blocks, 16-column tiles with remainders, the column split of few units) and matrices
whose rows differ by many orders of magnitude (the row and column scales).

Tolerance: both solves are backward stable, so each differs from the exact solution by at most a
modest multiple of n eps cond(M); the test allows n eps cond(M) with the 2-norm condition number of
the matrix computed here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import kkr as okkr
from oracle import liz as oliz
from paper_2311_12134_gb300 import workload as wl

from ._util import ensure_built


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2311_12134_gb300 import binding
    return binding


# (lmax, atoms): n = 33 (one trailing row), 64, 160, 161, 176, 207, 297, 320
@pytest.mark.parametrize("lmax,n_atoms", [(0, 33), (1, 16), (3, 10), (0, 161), (3, 11), (2, 23), (2, 33), (3, 20)])
@pytest.mark.parametrize("grade", [0, 6])
def test_fp64_tau_against_lapack(B, lmax, n_atoms, grade):
    w = wl.cluster(n_atoms, lmax, seed=40 + n_atoms, spread=2.4 * n_atoms ** (1 / 3) + 4.0)
    rng = np.random.default_rng(n_atoms)
    # one species per atom, its t^-1 scaled by 10^(-grade .. grade): rows of very different size
    w.species = np.arange(n_atoms, dtype=np.int32)
    scale = 10.0 ** rng.uniform(-grade, grade, n_atoms)
    w.tinv = np.ascontiguousarray(w.tinv[np.arange(n_atoms) % 2] * scale[:, None, None, None])
    lz = B.build_liz(w.pos, w.lattice, w.r_liz)
    tau, st = B.tau_blocks(lz, lmax, torch.as_tensor(w.species).cuda(), torch.as_tensor(w.tinv).cuda(), w.z, "fp64")
    assert not np.any(st.cpu().numpy() & 0xff)
    tau = tau.cpu().numpy()
    L = oliz.build_liz(w.pos, w.lattice, w.r_liz)
    off, K = L["offsets"], (lmax + 1) ** 2
    for m in (0, n_atoms - 1):
        s = slice(off[m], off[m + 1])
        for e in range(2):
            M = okkr.kkr_matrix(lmax, L["disp"][s], w.tinv[w.species[L["site_atom"][s]], e], w.z[e])
            ref, _ = okkr.tau_col_row(M, K)
            err = np.linalg.norm(tau[e, s] - ref) / np.linalg.norm(ref)
            assert err < M.shape[0] * np.finfo(float).eps * np.linalg.cond(M), (m, e, err)
