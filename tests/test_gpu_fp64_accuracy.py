"""The FP64 form on matrices whose t^-1 spans many orders of magnitude (weakly scattering high l, atoms or
channels scaled at random): tau as accurate as LAPACK's solution of the same matrix.

Tolerance: 8 times the error of numpy.linalg.solve (FP64, partial pivoting), both against a solution refined
in long double: two backward stable eliminations differ in their roundings, by a factor of two to three on
these matrices (test_digit_products.py restates both).  Added are 16 times the change of the solution when
the entries of g change by one eps at random: the kernel's and the reference's g are rounded on their own,
each to a few eps, the phase kappa R (up to 16) included.  The energies are such that kappa has no
cancellation: kappa = (1 + i / 256) / sqrt 2 comes from exact sums.  A complex64 solution, or row scales that
lose the small entries, exceed the tolerance by orders of magnitude; that the former does is asserted."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_12134_gb300 import workload as wl

from ._accuracy import err, grade, refined, unit_matrix
from ._util import ensure_built


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2311_12134_gb300 import binding
    return binding


Z = ((256 ** 2 - 1) + 512j) / (2 * 256 ** 2)  # |z| = (256^2 + 1) / (2 256^2)


def _cluster(lmax, n_atoms):
    return wl.cluster(n_atoms, lmax, seed=40 + n_atoms, spread=2.4 * n_atoms ** (1 / 3) + 4.0)


def _fcc43():  # 43-site LIZ, n = 688: five 128-row tiles and a remainder
    return wl.make_supercell(name="fcc", kind="fcc", n_cells=2, a=7.65, counts=[16, 16], r_liz=1.30 * 7.65,
                             phases=[wl.PHASE_A, wl.PHASE_B], e_fermi=0.6, deltas=[0.002], seed=5)


@pytest.mark.parametrize("make,kind,size", [
    (lambda: _cluster(3, 20), "f", 5e-3), (lambda: _cluster(3, 20), "f", 1e-6), (lambda: _cluster(3, 20), "f", 1e-8),
    (_fcc43, "f", 1e-4), (_fcc43, "f", 1e-6),
    (lambda: _cluster(3, 11), "atom", 6), (lambda: _cluster(2, 33), "atom", 6), (lambda: _cluster(1, 40), "atom", 12),
    (lambda: _cluster(3, 20), "channel", 6), (lambda: _cluster(3, 20), "channel", 12),
    (lambda: _cluster(0, 161), "atom", 6), (lambda: _cluster(3, 20), "dense", 3)])
def test_fp64_tau_is_as_accurate_as_lapack(B, make, kind, size):
    w = make()
    w.z = np.array([Z, np.conj(Z)])
    w.tinv = wl.tinv_from_phase_shifts([wl.PHASE_A[:w.lmax + 1], wl.PHASE_B[:w.lmax + 1]], w.z, w.lmax)
    grade(w, kind, size)
    lz = B.build_liz(w.pos, w.lattice, w.r_liz)
    tau, st = B.tau_blocks(lz, w.lmax, torch.as_tensor(w.species).cuda(), torch.as_tensor(w.tinv).cuda(), w.z, "fp64")
    assert not np.any(st.cpu().numpy() & 0xff)
    M, s = unit_matrix(w)
    n, K = len(M), w.K
    ref, E0 = refined(M, K), np.eye(len(M), K, dtype=complex)
    lapack = err(np.linalg.solve(M, E0), ref)
    g = np.kron(np.eye(n // K), np.ones((K, K))) == 0  # the blocks off the diagonal
    noise = np.random.default_rng(1).normal(size=M.shape) * np.finfo(float).eps
    change = err(refined(M * (1 + g * noise), K), ref)
    tol = 8 * lapack + 16 * change
    assert err(np.linalg.solve(M.astype(np.complex64), E0.astype(np.complex64)), ref) > 100 * tol
    got = err(tau[0, s].cpu().numpy().reshape(n, K), ref)
    assert got <= tol, (got, lapack, change)
