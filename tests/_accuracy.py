"""Matrices with t^-1 of very different sizes, and solutions to compare with (no package code)."""
import numpy as np
import scipy.linalg

from oracle import kkr as okkr
from oracle import liz as oliz
from paper_2311_12134_gb300 import workload as wl


def grade(w, kind, size):
    """Replace w's t^-1: kind "f" (lmax 3), the package's phase shifts with f phases of size and 4 size; "atom"
    and "channel", one species per atom, each atom's or channel's t^-1 times 10^(-size .. size); "dense",
    random full symmetric t^-1 matrices with such factors on both sides."""
    if kind == "f":
        w.tinv = wl.tinv_from_phase_shifts([wl.PHASE_A[:3] + (size,), wl.PHASE_B[:3] + (4 * size,)], w.z, w.lmax)
        return w
    n, K = len(w.species), w.K
    rng = np.random.default_rng(n)
    t = w.tinv[np.arange(n) % 2]
    w.species = np.arange(n, dtype=np.int32)
    if kind == "atom":
        t = t * 10.0 ** rng.uniform(-size, size, n)[:, None, None, None]
    else:
        s = 10.0 ** rng.uniform(-size, size, (n, 1, K, 1))
        if kind == "dense":
            t = rng.normal(size=(n, 1, K, K)) + 1j * rng.normal(size=(n, 1, K, K))
            t = np.broadcast_to((t + np.swapaxes(t, 2, 3)) * np.swapaxes(s, 2, 3), (n, len(w.z), K, K))
        t = t * s
    w.tinv = np.ascontiguousarray(t)
    return w


def unit_matrix(w, atom=0, energy=0):
    L = oliz.build_liz(w.pos, w.lattice, w.r_liz)
    s = slice(L["offsets"][atom], L["offsets"][atom + 1])
    M = okkr.kkr_matrix(w.lmax, L["disp"][s], w.tinv[w.species[L["site_atom"][s]], energy], w.z[energy])
    return M, s


def graded_matrix(w, kind, size):
    return unit_matrix(grade(w, kind, size))[0]


def refined(M, K):
    """The first K columns of M^-1, refined with long double residuals (M equilibrated by powers of two)."""
    d = np.exp2(np.round(-0.5 * np.log2(np.abs(M).max(1))))
    Ms = d[:, None] * M * d
    E0 = np.eye(len(M), K, dtype=complex) * d[:, None]
    f = scipy.linalg.lu_factor(Ms)
    X = scipy.linalg.lu_solve(f, E0).astype(np.clongdouble)
    Ml = Ms.astype(np.clongdouble)
    for _ in range(8):
        D = scipy.linalg.lu_solve(f, (E0 - Ml @ X).astype(complex))
        X = X + D
        if np.linalg.norm(D) < 1e-18 * np.linalg.norm(X.astype(complex)):
            break
    return X * d[:, None]


def err(X, ref):
    return np.linalg.norm((X - ref).astype(complex)) / np.linalg.norm(ref.astype(complex))
