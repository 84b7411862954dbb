"""Workloads that stand for what a user of this package computes, with the plain 64-bit values they should give.

A case is a dict of plain values.  ``call`` names what the user's program calls:

* ``forward``  ``Problem.forward``: the tau blocks of every (atom, energy) unit, sigma and rho (a conductivity run);
* ``step``     ``Problem.step``: the forward and the gradient of sigma (fitting or inverting t-matrices);
* ``graph``    the same step captured once and replayed (``StepGraph``), as an optimisation loop runs it;
* ``host``     ``conductivity``: NumPy in, NumPy out (one structure of a sweep over many);
* ``traces``   ``binding.kubo_sigma`` on given tau blocks (new current matrices for a solved structure).

The other keys are the structure (``lattice`` fcc or bcc with ``cells``^3 conventional cells and a LIZ ``radius`` in
lattice constants, or a finite ``cluster`` of ``cells`` atoms), ``minority`` (share of the second species),
``vacancies`` (share of removed sites), ``disp`` (Gaussian displacement in lattice constants), ``deltas`` (number of
broadenings), ``lmax``, ``precision`` and ``conj`` (conjugate energy pairs).  The sizes are those of the package's
seeded workloads, tests and benchmark, in cells that fit a GPU several times over.
"""
import functools
import math

import numpy as np
import torch

from paper_2311_12134_gb300 import binding, workload
from paper_2311_12134_gb300.conductivity import Problem, StepGraph, conductivity

A = {"fcc": 7.65, "bcc": 5.42}          # lattice constants (bohr) of the package's workloads
E_FERMI = {"fcc": 0.60, "bcc": 0.62, "cluster": 0.55}
DELTAS = {1: [0.002], 2: [0.001, 0.002], 3: [0.001, 0.002, 0.004]}
DEVICE = "cuda"


def _case(name, call, lattice, cells, radius, **more):
    c = dict(call=call, lattice=lattice, cells=cells, radius=radius, minority=0.0, vacancies=0.0, disp=0.0, deltas=1,
             lmax=3, precision="mixed", conj=False)
    c.update(more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest calls: a ten-atom cluster through the host call with its default precision
        _case("cluster10_host_fp64", "host", "cluster", 10, 20.0, minority=0.5, precision="fp64"),
        # the 32-atom pure crystal with a one-shell LIZ (n = 208): gradient in both forms, launched call by call
        _case("fcc32_step_fp64", "step", "fcc", 2, 0.85, precision="fp64"),
        _case("fcc32_step", "step", "fcc", 2, 0.85),
        # an optimisation loop on a small disordered cell with d states (lmax = 2, odd n = 243), replayed from a graph
        _case("bcc54_lmax2_graph", "graph", "bcc", 3, 1.45, minority=0.25, lmax=2),
        # an alloy at three shells with d states and two broadenings (n = 387)
        _case("fcc256_lmax2_step", "step", "fcc", 4, 1.30, minority=0.5, lmax=2, deltas=2),
        # the plain FP64 form at the three-shell LIZ (n = 688): the reference run of an alloy
        _case("fcc108_forward_fp64", "forward", "fcc", 3, 1.30, minority=0.5, precision="fp64"),
        # the random alloy at three shells (n = 688), conductivity and gradient
        _case("fcc256_step", "step", "fcc", 4, 1.30, minority=0.5),
        # the four-shell alloy (n = 880) with conjugate energy pairs, so half the matrices are factored
        _case("fcc108_conj_step", "step", "fcc", 3, 1.50, minority=0.3, conj=True),
        # the benchmark's recipe (vacancies, displacements, uneven LIZ, three broadenings; n about 850) on 5^3 cells
        _case("bcc250_uneven_step", "step", "bcc", 5, 1.75, minority=0.165, vacancies=0.01, disp=0.05, deltas=3),
        # a converged LIZ of 137 sites (n = 2192)
        _case("bcc54_liz137_forward", "forward", "bcc", 3, 2.5, minority=0.02),
        # the paper's LIZ of about 1000 sites (965 sites through periodic images, n = 15,440)
        _case("bcc2_liz965_forward", "forward", "bcc", 1, 4.9, minority=0.5),
        # new current matrices on the tau blocks of the 2000-site structure at three broadenings
        _case("bcc2000_traces", "traces", "bcc", 10, 1.75, minority=0.165, deltas=3),
    ]


_SHELLS = {"fcc": (0.85, 1.05, 1.30, 1.50), "bcc": (1.05, 1.45, 1.75, 1.85, 2.2, 2.5)}


def draw(rng):
    while True:
        lattice = rng.choice(("fcc", "fcc", "bcc", "bcc", "bcc", "cluster"))
        precision = rng.choice(("mixed", "mixed", "fp64"))
        if lattice == "cluster":
            call, cells, radius = rng.choice(("host", "forward", "step")), rng.randint(3, 40), 60.0
            disp = vac = 0.0
        else:
            call = rng.choice(("forward", "step", "step", "graph", "host", "traces"))
            cells, radius = rng.randint(1, 4 if lattice == "fcc" else 6), rng.choice(_SHELLS[lattice])
            disp, vac = rng.choice((0.0, 0.0, 0.05)), rng.choice((0.0, 0.0, 0.01))
        conj = call not in ("host", "traces") and rng.random() < 0.2
        c = _case(None, call, lattice, cells, radius, minority=rng.choice((0.02, 0.1, 0.165, 0.3, 0.5)), vacancies=vac,
                  disp=disp, deltas=rng.choice((1, 1, 2, 3)), lmax=rng.choice((1, 2, 3, 3)), precision=precision,
                  conj=conj)
        if work(c)["flops"] <= (0.3e12 if precision == "fp64" else 2.5e12) and _sites(c)[0] * c["deltas"] <= 1000:
            return c


# ------------------------------------------------------------------ what the user's program has in hand


def _phases(case, rng):
    """Two species' phase shifts, a little off the package's (another iteration of the potentials)."""
    out = []
    for ph in (workload.PHASE_A, workload.PHASE_B):
        out.append(tuple(float(x) for x in np.array(ph[:case["lmax"] + 1]) * (1 + 0.05 * rng.uniform(-1, 1))))
    return out


def _inputs(case, seed):
    rng = np.random.default_rng(1000003 * seed + 17)
    phases = _phases(case, rng)
    lat, lmax = case["lattice"], case["lmax"]
    deltas = DELTAS[case["deltas"]]
    sub = int(rng.integers(1 << 31))
    if lat == "cluster":
        w = workload.cluster(case["cells"], lmax, seed=sub, spread=2.4 * case["cells"] ** (1 / 3) + 4.0,
                             r_liz=5.0 * case["radius"])
        w.z = workload.energies(E_FERMI[lat], deltas)
        w.n_delta = len(deltas)
        w.tinv = workload.tinv_from_phase_shifts(phases, w.z, lmax)
        return w
    n = (4 if lat == "fcc" else 2) * case["cells"] ** 3
    b = int(round(case["minority"] * n))
    return workload.make_supercell(name="case", kind=lat, n_cells=case["cells"], a=A[lat], counts=[n - b, b],
                                   n_vacancies=int(round(case["vacancies"] * n)), sigma_disp=case["disp"] * A[lat],
                                   r_liz=case["radius"] * A[lat], phases=phases, e_fermi=E_FERMI[lat], deltas=deltas,
                                   lmax=lmax, seed=sub)


def _weights(case, n_delta):
    """The loss is the mean of the diagonal of Re sigma over the broadenings."""
    return np.repeat(np.eye(3, dtype=np.complex128)[None] / (3 * n_delta), n_delta, axis=0)


def _random_tau(case, w, disp, seed):
    """tau blocks with the decay of a solved structure: of the order of t on the centre, 1/(kappa d) away from it."""
    K = w.K
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    d = torch.as_tensor(np.linalg.norm(disp, axis=1), device=DEVICE)
    size = 0.5 / (1.0 + math.sqrt(E_FERMI[case["lattice"]]) * d)
    tau = torch.randn((2 * w.n_delta, len(d), K, K), dtype=torch.complex128, device=DEVICE, generator=g)
    return tau.mul_(size[None, :, None, None])


def prepare(case, seed):
    w = _inputs(case, seed)
    J = binding.dipole_current(w.lmax, w.r_ll)
    s = {"case": case, "w": w, "J": J}
    if case["call"] == "host":
        return s
    if case["call"] == "traces":
        s["liz"] = binding.build_liz(w.pos, w.lattice, w.r_liz)
        s["species"] = torch.as_tensor(w.species, device=DEVICE)
        s["J"] = torch.as_tensor(J, device=DEVICE)
        s["tau"] = _random_tau(case, w, s["liz"].export()["disp"], seed)
        return s
    step = case["call"] != "forward"
    s["problem"] = Problem(w.pos, w.lattice, w.r_liz, w.lmax, w.species, w.tinv, w.z, J, w.volume,
                           precision=case["precision"], keep_factors=step, conj_pairs=case["conj"])
    if step:
        s["weights"] = torch.as_tensor(_weights(case, w.n_delta), device=DEVICE)
    if case["call"] == "graph":
        s["graph"] = StepGraph(s["problem"], s["weights"])
    return s


# ------------------------------------------------------------------ one pass


def _tau_has_one_shape(case):
    """With displacements or vacancies the number of sites, so tau's shape, depends on the seed."""
    return case["lattice"] != "cluster" and not case["disp"] and not case["vacancies"]


def run(s):
    case, w = s["case"], s["w"]
    if case["call"] == "host":
        sigma, rho = conductivity(w.pos, w.lattice, w.r_liz, w.lmax, w.species, w.tinv, w.z, s["J"], w.volume,
                                  precision=case["precision"])
        return {"sigma": sigma, "rho": rho}
    if case["call"] == "traces":
        sigma, sigma_tilde, rho = binding.kubo_sigma(s["liz"], w.lmax, s["species"], s["J"], s["tau"], w.n_delta,
                                                     w.volume, precision=case["precision"])
        return {"sigma": sigma, "sigma_tilde": sigma_tilde, "rho": rho}
    p = s["problem"]
    out = {}
    if case["call"] == "forward":
        p.forward()
    elif case["call"] == "step":
        _, (out["grad"], out["grad_species"]) = p.step(s["weights"])
    else:
        s["graph"].replay()
        out["grad"], out["grad_species"] = s["graph"].grads
    out.update(sigma=p.sigma_out, sigma_tilde=p.sigma_tilde, rho=p.rho)
    if _tau_has_one_shape(case) or case["lattice"] == "cluster":
        out["tau"] = p.tau
    return out


# ------------------------------------------------------------------ the work of a pass


@functools.lru_cache(maxsize=None)
def _liz_sites(lattice, radius):
    """Sites within the radius of the perfect lattice."""
    r = int(radius) + 2
    cells = np.stack(np.meshgrid(*[np.arange(-r, r + 1)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)
    basis = workload.FCC_BASIS if lattice == "fcc" else workload.BCC_BASIS
    d = np.linalg.norm((cells[:, None, :] + basis[None, :, :]).reshape(-1, 3), axis=1)
    return int((d <= radius + 1e-8).sum())


def _sites(case):
    """(atoms, sites of one LIZ, about)"""
    if case["lattice"] == "cluster":
        return case["cells"], case["cells"]
    n = (4 if case["lattice"] == "fcc" else 2) * case["cells"] ** 3
    S = _liz_sites(case["lattice"], case["radius"])
    if case["disp"]:
        S *= 0.9  # displaced sites leave the outermost shell
    return n - int(round(case["vacancies"] * n)), max(1, int(round(S * (1 - case["vacancies"]))))


def work(case):
    """Factor each unit's matrix, solve for K columns (and 2K in the adjoint), take the traces; read the inputs and
    write the results once."""
    N, S = _sites(case)
    K = (case["lmax"] + 1) ** 2
    n, units = K * S, N * 2 * case["deltas"]
    factored = units // 2 if case["conj"] else units
    nz = 3  # nonzeros in a row of a dipole current matrix
    traces = 8.0 * N * case["deltas"] * 4 * S * 3 * (nz * K * K + nz * K * K)
    small = 16.0 * 2 * (2 * case["deltas"] + 12) * K * K + 36.0 * N + 16 * 9 * 6 * case["deltas"]
    tau = 16.0 * units * S * K * K
    if case["call"] == "traces":
        return {"bytes": tau + small, "flops": traces}
    grad = case["call"] in ("step", "graph")
    flops = factored * (8.0 / 3.0 * n ** 3 + 8.0 * n * n * K) + traces
    if grad:
        flops += units * (8.0 * n * n * 2 * K + 8.0 * S * (2 * K ** 3 + 12 * nz * K * K))
    return {"bytes": tau + small + (16.0 * units * K * K if grad else 0.0), "flops": flops}


# ------------------------------------------------------------------ the same in plain torch, 64 bits


def _harmonics(lmax, v):
    """Real harmonics (no Condon-Shortley phase, L = l l + l + m) at the directions of v [..., 3]."""
    r = v.norm(dim=-1, keepdim=True)
    x, y, z = (v / r).unbind(-1)
    out = [None] * (lmax + 1) ** 2
    c, s = torch.ones_like(x), torch.zeros_like(x)   # sin^m cos(m phi), sin^m sin(m phi)
    top = 1.0                                        # (2m - 1)!!
    for m in range(lmax + 1):
        if m:
            c, s = c * x - s * y, c * y + s * x
            top *= 2 * m - 1
        before, p = torch.zeros_like(z), torch.full_like(z, top)
        for l in range(m, lmax + 1):
            if l > m:
                before, p = p, ((2 * l - 1) * z * p - (l + m - 1) * before) / (l - m)
            f = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            if m == 0:
                out[l * l + l] = f * p
            else:
                out[l * l + l + m] = math.sqrt(2) * f * p * c
                out[l * l + l - m] = math.sqrt(2) * f * p * s
    return torch.stack(out, dim=-1)


@functools.lru_cache(maxsize=None)
def _gaunt(l1, l3):
    """int Y_L1 Y_L2 Y_L3 by Gauss-Legendre times a uniform grid in phi (exact for these degrees)."""
    deg = 2 * l1 + l3
    ct, wt = np.polynomial.legendre.leggauss(deg // 2 + 2)
    n_phi = deg + 2
    ph = 2 * math.pi * np.arange(n_phi) / n_phi
    st = np.sqrt(1 - ct ** 2)
    nodes = np.stack(np.broadcast_arrays(st[:, None] * np.cos(ph), st[:, None] * np.sin(ph), ct[:, None]), -1)
    Y = _harmonics(max(l1, l3), torch.as_tensor(nodes.reshape(-1, 3)))
    wq = torch.as_tensor(np.repeat(wt, n_phi) * 2 * math.pi / n_phi)
    Ya, Yc = Y[:, :(l1 + 1) ** 2], Y[:, :(l3 + 1) ** 2]
    C = torch.einsum("q,qa,qb,qc->abc", wq, Ya, Ya, Yc)
    la = torch.tensor([math.isqrt(L) for L in range((l1 + 1) ** 2)])
    lc = torch.tensor([math.isqrt(L) for L in range((l3 + 1) ** 2)])
    even = (la[:, None, None] + la[None, :, None] + lc[None, None, :]) % 2 == 0
    fits = (lc <= la[:, None, None] + la[None, :, None]) & (lc >= (la[:, None, None] - la[None, :, None]).abs())
    return torch.where(even & fits, C, 0.0)


def _propagator(lmax, R, z):
    """g_{LL'}(z) for separations R [..., 3] (nonzero): the outgoing form for Im z >= 0, its conjugate below."""
    l3 = 2 * lmax
    C = _gaunt(lmax, l3)
    l1 = [math.isqrt(L) for L in range((lmax + 1) ** 2)]
    lc = [math.isqrt(L) for L in range((l3 + 1) ** 2)]
    phase = torch.tensor([[[1j ** ((a - b - c) % 4) for c in lc] for b in l1] for a in l1], dtype=torch.complex128)
    P = (phase * C).to(R.device)
    k = np.sqrt(np.complex128(z if z.imag >= 0 else np.conj(z)))
    x = complex(k) * R.norm(dim=-1).to(torch.complex128)
    h = []
    for l in range(l3 + 1):
        poly = sum(math.factorial(l + j) / (math.factorial(j) * math.factorial(l - j)) * (1j / (2 * x)) ** j
                   for j in range(l + 1))
        h.append((-1j) ** (l + 1) * torch.exp(1j * x) / x * poly)
    v = torch.stack([h[l] for l in lc], dim=-1) * _harmonics(l3, R)
    K, K3 = len(l1), len(lc)
    g = -4j * math.pi * complex(k) * (v.reshape(-1, K3) @ P.reshape(K * K, K3).T).reshape(*R.shape[:-1], K, K)
    return g if z.imag >= 0 else g.conj()


def _zone(pos, lattice, r, m):
    """Atoms and displacements of the sites within r of atom m: the centre first, then by (atom, image)."""
    if lattice is None:
        images = np.zeros((1, 3))
    else:
        reach = [int((r + 1.0) / lattice[i, i]) + 1 for i in range(3)]  # cubic cells, displacements below 1 bohr
        g = np.meshgrid(*[np.arange(-k, k + 1) for k in reach], indexing="ij")
        images = np.stack(g, axis=-1).reshape(-1, 3) @ lattice
    d = pos[:, None, :] - pos[m] + images[None, :, :]
    atom, img = np.nonzero(np.linalg.norm(d, axis=-1) <= r + 1e-8)
    disp = d[atom, img]
    centre = np.flatnonzero((atom == m) & (np.abs(disp).max(axis=1) < 1e-9))
    order = np.concatenate([centre, np.delete(np.arange(len(atom)), centre)])
    return atom[order], disp[order]


def _current(lmax, r_ll):
    """The dipole current matrices r_{ll'} C_{LL'(1 m)}, x, y, z <-> m = 1, -1, 0."""
    C = _gaunt(lmax, 1)[:, :, [3, 1, 2]].permute(2, 0, 1)
    l = torch.tensor([math.isqrt(L) for L in range((lmax + 1) ** 2)])
    r = torch.as_tensor(r_ll)[:, :, l[:, None], l[None, :]]
    return (r[:, :, None] * C.to(torch.complex128)).to(DEVICE)


def _atom_sigma(Jm, Jn, tau_row, tau_col, n_delta):
    """S_c[mu][nu] of one centre, [n_delta, 4, 3, 3]; tau_row[e][n] = tau^{0n}, tau_col[e][n] = tau^{n0}."""
    out = []
    for d in range(n_delta):
        for c in range(4):
            a, b, back = c >> 1, c & 1, ((c & 1) << 1) | (c >> 1)
            P = Jn[:, c] @ tau_col[2 * d + b][:, None]                       # [S, 3, K, K]
            Y = torch.einsum("sij,svjk->vik", tau_row[2 * d + a], P)
            out.append(torch.einsum("uki,vik->uv", Jm[back], Y))
    return torch.stack(out).reshape(n_delta, 4, 3, 3)


def exact(case, seed):
    if work(case)["flops"] > 5e12:
        return None
    w = _inputs(case, seed)
    K, N, nE, nd = w.K, w.n_atoms, len(w.z), w.n_delta
    J = _current(w.lmax, w.r_ll)
    grad = case["call"] in ("step", "graph")
    zones = [_zone(w.pos, w.lattice, w.r_liz, m) for m in range(N)]
    if case["call"] == "traces":
        disp = np.concatenate([z[1] for z in zones])
        tau = _random_tau(case, w, disp, seed)
    tinv = torch.as_tensor(w.tinv, device=DEVICE)
    species = torch.as_tensor(w.species.astype(np.int64), device=DEVICE)
    total = torch.zeros((nd, 4, 3, 3), dtype=torch.complex128, device=DEVICE)
    g_out = torch.zeros((nE, N, K, K), dtype=torch.complex128, device=DEVICE)
    taus = []
    signs = torch.tensor([1.0, -1.0, -1.0, 1.0], dtype=torch.complex128, device=DEVICE)
    weights = torch.as_tensor(_weights(case, nd), device=DEVICE)
    at = 0
    for m in range(N):
        atoms, disp = zones[m]
        S = len(atoms)
        atoms = torch.as_tensor(np.asarray(atoms, dtype=np.int64), device=DEVICE)
        Jm, Jn = J[species[m]], J[species[atoms]]
        if case["call"] == "traces":
            X = tau[:, at:at + S]
            at += S
            total += _atom_sigma(Jm, Jn, X.transpose(-1, -2), X, nd)
            continue
        d = torch.as_tensor(disp, device=DEVICE)
        eye = torch.eye(S, dtype=torch.bool, device=DEVICE)
        R = torch.where(eye[..., None], torch.ones(3, dtype=torch.float64, device=DEVICE), d[None, :] - d[:, None])
        E0 = torch.eye(K * S, K, dtype=torch.complex128, device=DEVICE)
        lus, X = [], []
        for e in range(nE):
            if e % 2 and w.z[e] == np.conj(w.z[e - 1]):
                blocks = off_diagonal.conj()
            else:
                off_diagonal = blocks = -_propagator(w.lmax, R, w.z[e])
            M = torch.where(eye[..., None, None], tinv[species[atoms], e][:, None], blocks)
            lu = torch.linalg.lu_factor(M.transpose(1, 2).reshape(K * S, K * S))
            lus.append(lu if grad else None)
            X.append(torch.linalg.lu_solve(*lu, E0).reshape(S, K, K))
        col = torch.stack(X).requires_grad_(grad)
        row = torch.stack(X).transpose(-1, -2).detach().requires_grad_(grad)  # M is symmetric: tau^{0n} = tau^{n0}^T
        st = _atom_sigma(Jm, Jn, row, col, nd)
        total += st.detach()
        if _tau_has_one_shape(case) or case["lattice"] == "cluster":
            taus.append(col.detach())
        if grad:
            sigma = -(signs[None, :, None, None] * st).sum(1) / (4 * math.pi * w.volume)
            gc, gr = torch.autograd.grad((weights.conj() * sigma).sum().real, (col, row))
            for e in range(nE):
                # X = M^-1 E0 gives -(M^-H G) X^H; the row block is X of the transposed matrix
                G = torch.cat([gc[e].reshape(K * S, K), gr[e].transpose(-1, -2).reshape(K * S, K)], dim=1)
                W = torch.linalg.lu_solve(*lus[e], G, adjoint=True).reshape(S, K, 2 * K)
                Xh = X[e].conj().transpose(-1, -2)
                D = -(W[..., :K] @ Xh) - (W[..., K:] @ Xh).transpose(-1, -2)
                g_out[e].index_add_(0, atoms, D)
    total = -total / (math.pi * w.volume)
    sigma = (signs[None, :, None, None] * total).sum(1) / 4
    out = {"sigma": sigma, "rho": torch.linalg.inv(sigma.real)}
    if case["call"] == "host":
        return {k: v.cpu().numpy() for k, v in out.items()}
    out["sigma_tilde"] = total
    if taus:
        out["tau"] = torch.cat(taus, dim=1)
    if grad:
        out["grad"] = g_out
        out["grad_species"] = torch.stack([g_out[:, species == s].sum(1) for s in range(w.n_species)])
    return out
