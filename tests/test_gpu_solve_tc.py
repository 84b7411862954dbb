"""The mixed form's tensor-core chain solves (csrc/tc_solve.cu) at the sizes where their groups of 128
rows, blocks of 32 and column counts end: one partial block (n = 27), one group less or more a block
(n = 126, 128, 135, 144), two groups (256, 261, 272), with 9 and 16 columns forward and 18 and 32 in the
adjoint; and the block-step path chosen for few large matrices against the chains.  The tau blocks and
the gradient match the FP64 form to the mixed form's bound (1e-8), every unit converges in the sweep
that the refinement takes on these matrices anyway (at most 2), and no unit needs the FP64 fallback."""
import contextlib

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_12134_gb300 import workload as wl

from ._util import ensure_built


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2311_12134_gb300 import binding
    return binding


def _run(B, w, precision):
    lz = B.build_liz(w.pos, w.lattice, w.r_liz)
    sp, t = torch.as_tensor(w.species).cuda(), torch.as_tensor(w.tinv).cuda()
    J = torch.as_tensor(B.dipole_current(w.lmax, w.r_ll)).cuda()
    gs = torch.eye(3, dtype=torch.complex128, device="cuda")[None].contiguous()
    store = torch.empty(B.lu_store_bytes(lz, w.lmax, 2, B._prec(precision)), dtype=torch.uint8, device="cuda")
    tau, st = B.tau_blocks(lz, w.lmax, sp, t, w.z, precision, lu_store=store)
    g, _ = B.kubo_sigma_backward(lz, w.lmax, sp, t, w.z, J, tau, w.volume, gs, precision, lu_store=store)
    torch.cuda.synchronize()
    return tau.cpu().numpy(), g.cpu().numpy(), st.cpu().numpy()


@pytest.mark.parametrize("lmax,n_atoms", [(2, 3), (2, 14), (2, 15), (2, 29), (3, 8), (3, 9), (3, 16), (3, 17)])
def test_chain_solves_at_group_edges(B, lmax, n_atoms):
    w = wl.cluster(n_atoms, lmax, seed=60 + n_atoms, spread=2.4 * n_atoms ** (1 / 3) + 4.0)
    tau, g, st = _run(B, w, "mixed")
    ref, gref, _ = _run(B, w, "fp64")
    assert not np.any(st & 0xff) and ((st >> 8) & 0xff).max() <= 2
    assert np.linalg.norm(tau - ref) < 1e-8 * np.linalg.norm(ref)
    assert np.linalg.norm(g - gref) < 1e-8 * np.linalg.norm(gref)


def test_block_steps_chosen_for_few_large_matrices(B):
    """n = 4144, 4 units: the default path (block steps) and the chains give the same tau to the
    refinement's tolerance."""
    w = wl.make_supercell(name="bcc2_liz259", kind="bcc", n_cells=1, a=5.42, counts=[1, 1], r_liz=3.1 * 5.42,
                          phases=[wl.PHASE_A, wl.PHASE_B], e_fermi=0.62, deltas=[0.002], seed=3)
    lz = B.build_liz(w.pos, w.lattice, w.r_liz)
    assert 16 * lz.max_sites >= 3000
    out = {}
    for steps in (0, 1):
        with contextlib.ExitStack() as s:
            saved = B.get_option("solve_steps")
            s.callback(B.set_option, "solve_steps", saved)
            B.set_option("solve_steps", steps)
            tau, st = B.tau_blocks(lz, w.lmax, torch.as_tensor(w.species).cuda(), torch.as_tensor(w.tinv).cuda(), w.z,
                                   "mixed")
            assert not np.any(st.cpu().numpy() & 0xff)
            out[steps] = tau.cpu().numpy()
    assert np.abs(out[0] - out[1]).max() <= 1e-9 * np.abs(out[1]).max()
