"""The adjoint's workspace: without a cap all units run in one chunk, with the smallest one in chunks of
one atom; the gradients agree to the refinement's tolerance (the mixed form's solves may take another
path when a chunk holds few units; 1e-9 of the largest entry, ten times its stopping tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_12134_gb300 import workload as wl

from ._util import ensure_built


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_adjoint_in_one_chunk_matches_one_atom_chunks(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2311_12134_gb300 import binding as B
    from paper_2311_12134_gb300.conductivity import Problem
    w = wl.make_supercell(name="chunks", kind="fcc", n_cells=2, a=7.65, counts=[20, 12], sigma_disp=0.1,
                          r_liz=0.85 * 7.65, phases=[wl.PHASE_A, wl.PHASE_B], e_fermi=0.6, deltas=[0.002], seed=11)
    J = B.dipole_current(w.lmax, w.r_ll)
    got, size = {}, {}
    for cap in (None, 1):
        p = Problem(w.pos, w.lattice, w.r_liz, w.lmax, w.species, w.tinv, w.z, J, w.volume, precision=precision,
                    workspace_bytes=cap)
        gs = torch.zeros((1, 3, 3), dtype=torch.complex128, device="cuda")
        gs[0, 0, 0] = 1
        _, (g, _) = p.step(gs)
        p.check()
        got[cap], size[cap] = g.cpu().numpy(), p._bw_ws.numel()
    mn, al = B.backward_workspace_bytes(p.liz, p.lmax, 2, B._prec(precision) | B.LSMS_WS_STORE)
    assert size[None] == al and size[1] < al
    assert np.abs(got[None] - got[1]).max() <= 1e-9 * np.abs(got[1]).max()
