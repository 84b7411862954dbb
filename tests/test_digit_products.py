"""The arithmetic of the complex128 digit products (csrc/tc_gemm64.cu) restated in NumPy: operands balanced
along K, seven base-256 digits relative to the largest entry of each row and column, eight classes.  An LU
and solve by it in panels of 32 is as accurate as one with FP64 row updates, on matrices whose t^-1 spans
up to 24 orders of magnitude too, where it is not without the balance.

Tolerance: both solutions come from the same pivoted elimination and differ in their roundings only, so
the digits' error is held to 4 times that of the FP64 updates (with both measured against a solution
refined in long double)."""
import numpy as np
import pytest
import scipy.linalg

from paper_2311_12134_gb300 import workload as wl

from ._accuracy import err, graded_matrix, refined

NB, ND, NG, TOP = 32, 7, 8, 7


def _exponent(v):
    e = np.frexp(np.maximum(np.abs(v.real), np.abs(v.imag)))[1]
    return np.where(v == 0, -4096, e)


def _digits(v, shift):
    q = np.rint(np.ldexp(v, shift)).astype(np.int64)
    out = []
    for _ in range(ND - 1):
        d = ((q + 128) & 255) - 128
        out.append(d.astype(float))
        q = (q - d) >> 8
    assert np.abs(q).max(initial=0) <= 128
    return [q.astype(float)] + out[::-1]


def _product(A, B, balance):
    """A @ B as the kernels form it; balance: "A" (largest entries of A's columns, per 128 rows), "B" (of
    B's rows) or None."""
    out = np.empty((len(A), B.shape[1]), dtype=complex)
    eB = _exponent(B)
    for r0 in range(0, len(A), 128):
        a = A[r0:r0 + 128]
        eA = _exponent(a)
        s = -eA.max(0) if balance == "A" else eB.max(1) if balance == "B" else np.zeros(len(B), int)
        s = np.where(np.abs(s) == 4096, 0, s)
        er, ec = (eA + s).max(1), (eB - s[:, None]).max(0)
        sa = np.clip(8 * (ND - 1) + TOP - er[:, None] + s, -1000, 1000)
        sb = np.clip(8 * (ND - 1) + TOP - ec - s[:, None], -1000, 1000)
        ar, ai, br, bi = _digits(a.real, sa), _digits(a.imag, sa), _digits(B.real, sb), _digits(B.imag, sb)
        parts = []
        for p, q, x, y, sign in ((ar, br, ai, bi, -1.0), (ar, bi, ai, br, 1.0)):
            c = [sum(p[i] @ q[g - i] + sign * (x[i] @ y[g - i]) for i in range(max(0, g - ND + 1), min(g, ND - 1) + 1))
                 for g in range(NG)]
            assert max(np.abs(v).max(initial=0) for v in c) < 1 << 24  # exact in FP32
            c = [v.astype(np.int64) for v in c]
            whole = ((c[0] * 256 + c[1]) << 34) + ((c[2] * 256 + c[3]) << 18) + (c[4] * 256 + c[5]) * 4
            whole += (c[6] * 256 + c[7] + (1 << 13)) >> 14
            parts.append(np.ldexp(whole.astype(float), np.clip(er[:, None] + ec - 2 * TOP - 42, -2000, 2000)))
        out[r0:r0 + 128] = parts[0] + 1j * parts[1]
    return out


def _solve(M, B, update):
    """X = M^-1 B; update(A, B, side) is the product of the row updates, side "A" in the LU, "B" in the solves."""
    A, n, X = M.copy(), len(M), B.copy()
    for k in range(0, n, NB):
        e = min(n, k + NB)
        for j in range(k, e):
            p = j + np.argmax(np.abs(A[j:, j].real) + np.abs(A[j:, j].imag))
            A[[j, p]], X[[j, p]] = A[[p, j]], X[[p, j]]
            A[j + 1:, j] *= 1 / A[j, j]
            A[j + 1:, j + 1:e] -= np.outer(A[j + 1:, j], A[j, j + 1:e])
        A[k:e, e:] = scipy.linalg.solve_triangular(A[k:e, k:e], A[k:e, e:], lower=True, unit_diagonal=True)
        A[e:, e:] -= update(A[e:, k:e], A[k:e, e:], "A")
    for k in range(0, n, NB):
        e = min(n, k + NB)
        X[k:e] = scipy.linalg.solve_triangular(A[k:e, k:e], X[k:e], lower=True, unit_diagonal=True)
        X[e:] -= update(A[e:, k:e], X[k:e], "B")
    for k in range((n - 1) // NB * NB, -1, -NB):
        e = min(n, k + NB)
        X[k:e] = scipy.linalg.solve_triangular(A[k:e, k:e], X[k:e])
        X[:k] -= update(A[:k, k:e], X[k:e], "B")
    return X


@pytest.mark.parametrize("lmax,n_atoms,kind,size", [
    (3, 20, "f", 5e-3), (3, 20, "f", 1e-4), (3, 20, "f", 1e-8)] + [
    (lmax, n_atoms, kind, size) for lmax, n_atoms in ((3, 20), (2, 33))
    for kind, size in (("atom", 6), ("atom", 12), ("channel", 6), ("channel", 12), ("dense", 3))])
def test_digit_products_are_as_accurate_as_fp64(lmax, n_atoms, kind, size):
    M = graded_matrix(wl.cluster(n_atoms, lmax, seed=40 + n_atoms, spread=2.4 * n_atoms ** (1 / 3) + 4.0), kind, size)
    K = (lmax + 1) ** 2
    ref = refined(M, K)
    E0 = np.eye(len(M), K, dtype=complex)
    plain = err(_solve(M, E0, lambda a, b, side: a @ b), ref)
    got = err(_solve(M, E0, _product), ref)
    assert got <= 4 * plain, (got, plain)
    if (kind, size) in (("f", 1e-8), ("atom", 12), ("channel", 12)):
        assert err(_solve(M, E0, lambda a, b, side: _product(a, b, None)), ref) > 100 * plain


def test_non_rank_one_scales_and_zeros():
    """Zero rows, columns and K lines, and products whose scales no balance evens out, keep the normwise bound."""
    rng = np.random.default_rng(3)
    A = rng.normal(size=(200, 32)) * 10.0 ** rng.uniform(-8, 8, (200, 32)) + 0j
    B = (rng.normal(size=(32, 17)) + 1j * rng.normal(size=(32, 17))) * 10.0 ** rng.uniform(-8, 8, (32, 17))
    A[5] = 0
    A[:, 3] = 0
    B[7] = 0
    B[:, 2] = 0
    for side in ("A", "B", None):
        e = np.abs(_product(A, B, side) - A @ B)
        s = np.exp2(np.where(_exponent(A).max(0) > -4096, _exponent(A).max(0), 0)) if side == "A" else np.exp2(
            -np.where(_exponent(B).max(1) > -4096, _exponent(B).max(1), 0.0)) if side == "B" else np.ones(32)
        bound = np.abs(A / s).max(1)[:, None] * np.abs(B * s[:, None]).max(0)
        assert (e <= 64 * 2.0 ** -50 * bound).all()
        assert not e[5].any() and not e[:, 2].any()
