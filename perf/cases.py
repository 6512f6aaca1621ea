"""Performance cases of the library: what its users have it do, through the Python binding.

``listed()`` names the cases, ``draw`` takes another one from the same ranges, ``prepare``
builds what a program holds before the call (structures on the device, a configured model, a
captured graph), ``run`` is one pass and ``work`` the bytes and operations that no
implementation of that pass can avoid.  ``exact`` evaluates the same pass in 64 bits with
plain torch operations and none of the library's code: radial coefficients by Gauss-Legendre
quadrature of the orthonormal functions (built at 120 decimal digits, so that the
orthonormalisation amplifies no rounding), harmonics from solid-harmonic recurrences,
analytic gradients.  The sparse sets of the models are descriptors of a separate random box,
evaluated by the same plain code.

Structures are random periodic boxes with a minimum distance between atoms, the stand-in
for the amorphous-carbon and two-species training data of such models.
"""
from __future__ import annotations

import functools
import math
from decimal import Decimal, localcontext

import numpy as np
import torch

from paper_1905_02142_gb300.api import CapturedEvaluation, SoapGap, SoapGapEnergy, Structures, VelocityVerlet

F64 = torch.float64
EV_PER_AMU_A2_FS2 = 1.0 / 103.642697
MD_STEPS = 8
MD_DT = 0.5          # fs
MD_MASS = 12.011     # amu


# ------------------------------------------------------------------------------- cases
def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, precision="mixed", structures=1, atoms=64, atoms_hi=0, density=0.15,
             density_hi=0.0, dmin=1.2, shear=0.0, species=1, r_cut=5.0, buffer=0.5, sigma_r=0.5,
             sigma_p=0.5, alpha_r=0.0, alpha_p=0.0, amp_a=1.0, n_max=8, l_max=8, sparse=0, zeta=4.0)
    c.update(kw)
    return c


def listed():
    return [
        # descriptors of one small cell, in 64 bits: the plain method, as a reference for a
        # fit or a check; the smallest call
        _case("desc_box64_fp64", "desc", precision="fp64", atoms=64, density=0.125, r_cut=3.7,
              n_max=6, l_max=6),
        # one energy-and-forces call on a small cell, as a relaxation or a phonon calculation
        # makes by the thousand: launches, synchronisations and host work count
        _case("ef_box64", "compute", atoms=64, density=0.125, r_cut=3.7, n_max=6, l_max=6, sparse=32),
        # the energy as a node of an autograd graph, forward and backward
        _case("autograd_box1000", "autograd", atoms=1000, sparse=500),
        # energies and forces in 64 bits, as a fit's validation or a phonon calculation wants
        _case("ef_box1000_fp64", "compute", precision="fp64", atoms=1000, sparse=500),
        # a stretch of molecular dynamics with a Verlet skin, each step replayed from a graph
        _case("md_box1000", "md", atoms=1000, sparse=500),
        # descriptors alone (clustering, selection of environments, the paper's timing box);
        # an odd basis size
        _case("desc_box10000_n7l5", "desc", atoms=10000, density=0.10029, dmin=0.7, n_max=7, l_max=5),
        # NumPy in, NumPy out: an external code calls with a few uneven triclinic structures
        # of two species and a basis and widths of its own
        _case("host_triclinic_n5l9", "host", structures=5, atoms=37, atoms_hi=1200, density=0.08,
              density_hi=0.12, dmin=1.0, shear=0.17, species=2, r_cut=4.3, sigma_r=0.4, sigma_p=0.55,
              alpha_r=0.08, alpha_p=0.06, amp_a=1.6, n_max=5, l_max=9, sparse=777, zeta=3.0),
        # energies and forces of a two-species box with a wide descriptor
        _case("ef_twospecies4096", "compute", atoms=4096, density=0.10, dmin=1.0, species=2, sparse=2000),
        # a batch of uneven structures (a training set, a replica ensemble) from one graph
        _case("graph_batch256", "graph", structures=256, atoms=16, atoms_hi=2000, density=0.08,
              density_hi=0.18, r_cut=4.5, sparse=1000, zeta=2.0),
        # one evaluation of a large box for molecular dynamics: energies, forces, virial
        _case("efv_box100k", "compute_virial", atoms=100000, n_max=10, l_max=10, sparse=4000),
        # rows of the fitting matrices of a set of training structures: energy and force rows
        _case("design_batch24", "design", structures=24, atoms=16, atoms_hi=2000, density=0.08,
              density_hi=0.18, r_cut=4.5, sparse=1000, zeta=2.0),
        # the kernel matrix of the sparse set with itself, once per fit
        _case("kernel_rows_4000", "kernel_rows", atoms=8000, n_max=10, l_max=10, sparse=4000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["desc", "desc", "compute", "compute", "compute", "compute_virial", "autograd", "md",
                       "host", "graph", "design", "kernel_rows"])
    precision = "fp64" if kind in ("desc", "compute") and rng.random() < 0.25 else "mixed"
    species = 2 if rng.random() < 0.25 else 1
    hi = 8 if species == 2 else 10
    kw = dict(precision=precision, species=species, n_max=rng.randint(3, hi), l_max=rng.randint(3, hi),
              r_cut=round(rng.uniform(3.7, 5.0), 2), density=round(rng.uniform(0.08, 0.15), 3),
              dmin=1.0 if species == 2 else 1.2, zeta=float(rng.choice([2, 3, 4])),
              sparse=_log_int(rng, 32, 2000), shear=rng.choice([0.0, 0.0, 0.15]))
    if kind == "desc":
        kw["atoms"] = _log_int(rng, 64, 1000 if precision == "fp64" else 40000)
        if species == 1 and precision == "mixed":
            kw["n_max"], kw["l_max"] = rng.randint(3, 12), rng.randint(3, 12)
    elif kind in ("compute", "compute_virial"):
        kw["atoms"] = _log_int(rng, 64, 1000 if precision == "fp64" else (10000 if species == 2 else 60000))
        if precision == "fp64":
            kw["sparse"] = min(kw["sparse"], 500)
    elif kind in ("autograd", "md"):
        kw["atoms"] = _log_int(rng, 64, 4000)
    elif kind == "host":
        kw.update(structures=rng.randint(1, 9), atoms=_log_int(rng, 16, 64), atoms_hi=_log_int(rng, 100, 3000),
                  density_hi=kw["density"] + 0.02)
    elif kind == "graph":
        kw.update(structures=_log_int(rng, 8, 200), atoms=16, atoms_hi=_log_int(rng, 200, 2000),
                  density_hi=kw["density"] + 0.03, shear=0.0)
        if species == 2:
            kw["structures"] = min(kw["structures"], 32)
    elif kind == "design":
        kw.update(species=1, structures=_log_int(rng, 2, 16), atoms=16, atoms_hi=_log_int(rng, 100, 1000),
                  density_hi=kw["density"] + 0.03, sparse=_log_int(rng, 32, 1000), shear=0.0)
    elif kind == "kernel_rows":
        kw.update(atoms=4000, shear=0.0, sparse=_log_int(rng, 100, 3000))
    c = _case("", kind, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------------------- inputs
def _box(counts, sides, dmin, rng):
    """Random positions in periodic cubes, no two atoms of a cube closer than dmin: rounds of
    candidates; one is kept if no kept atom and no earlier candidate lies within dmin.
    Fractional coordinates [N, 3], structure by structure."""
    dev = "cuda"
    S = len(counts)
    g = np.maximum(np.ceil(sides * math.sqrt(3.0) / dmin).astype(np.int64), 1)   # at most one atom per cell
    reach = int(np.max(np.ceil(dmin / (sides / g))))
    offs = torch.as_tensor(np.concatenate([[0], np.cumsum(g ** 3)]), device=dev)
    gd, sd = torch.as_tensor(g, device=dev), torch.as_tensor(sides, device=dev)
    grid = torch.full((int(offs[-1]),), -1, dtype=torch.int64, device=dev)
    kept_x = torch.zeros((0, 3), dtype=F64, device=dev)
    kept_s = torch.zeros((0,), dtype=torch.int64, device=dev)
    need = np.asarray(counts, dtype=np.int64).copy()
    rr = range(-reach, reach + 1)
    nb = torch.as_tensor([(a, b, c) for a in rr for b in rr for c in rr], device=dev)

    def clash(x, s, cell, table, tx, before=None):
        if not len(tx):
            return torch.zeros(len(x), dtype=torch.bool, device=dev)
        gs = gd[s, None]
        cc = torch.remainder(cell[:, None, :] + nb, gs[:, :, None])
        k = table[offs[s, None] + (cc[:, :, 0] * gs + cc[:, :, 1]) * gs + cc[:, :, 2]]
        hit = k >= 0 if before is None else (k >= 0) & (k < before[:, None])
        dx = tx[k.clamp(min=0)] - x[:, None, :]
        dx = (dx - torch.round(dx)) * sd[s, None, None]
        return (hit & ((dx * dx).sum(2) < dmin * dmin)).any(1)

    for _ in range(200):
        if need.sum() == 0:
            break
        cs = np.repeat(np.arange(S), np.where(need > 0, (1.5 * need).astype(np.int64) + 4, 0))
        x = torch.as_tensor(rng.random((len(cs), 3)), device=dev)
        s = torch.as_tensor(cs, device=dev)
        cell = torch.minimum((x * gd[s, None]).long(), gd[s, None] - 1)
        ok = ~clash(x, s, cell, grid, kept_x)
        x, s, cell = x[ok], s[ok], cell[ok]
        flat = offs[s] + (cell[:, 0] * gd[s] + cell[:, 1]) * gd[s] + cell[:, 2]
        order = torch.arange(len(x), device=dev)
        first = torch.full_like(grid, len(x)).scatter_reduce(0, flat, order, "amin")
        own = first[flat] == order                      # the earliest candidate of its cell
        first = torch.where(first == len(x), -1, first)
        ok = own & ~clash(x, s, cell, first, x, before=order)
        x, s, flat = x[ok], s[ok], flat[ok]
        sn = s.cpu().numpy()
        rank = np.arange(len(sn)) - np.searchsorted(sn, sn, side="left")
        take = torch.as_tensor(rank < need[sn], device=dev)
        x, s, flat = x[take], s[take], flat[take]
        grid[flat] = torch.arange(len(x), device=dev) + len(kept_x)
        kept_x, kept_s = torch.cat([kept_x, x]), torch.cat([kept_s, s])
        need -= np.bincount(s.cpu().numpy(), minlength=S)
    if need.sum() != 0:
        raise RuntimeError("could not place all atoms")
    return kept_x[torch.sort(kept_s, stable=True).indices].cpu().numpy()


def _structures(case, rng, counts, rho):
    counts, rho = np.asarray(counts, dtype=np.int64), np.asarray(rho, dtype=np.float64)
    sides = np.cbrt(counts / rho)
    frac = _box(counts, sides, case["dmin"], rng)
    t = case["shear"]
    shape = np.array([[1.0, 0.0, 0.0], [t, 1.0, 0.0], [t, 0.0, 1.0]])
    cell = sides[:, None, None] * shape[None]
    offs = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    pos = np.einsum("ia,iab->ib", frac, np.repeat(cell, counts, axis=0))
    spec = (rng.random(len(pos)) >= 0.7).astype(np.int32) if case["species"] == 2 else \
        np.zeros(len(pos), np.int32)
    return dict(pos=np.ascontiguousarray(pos), cell=np.ascontiguousarray(cell), species=spec, offs=offs)


def _counts(case):
    """Atoms of each structure: the quantiles of a log-uniform distribution, in mixed order."""
    lo, hi, S = case["atoms"], case["atoms_hi"], case["structures"]
    u = (np.arange(S) * 0.6180339887498949 + 0.5 / S) % 1.0
    return np.rint(lo * (hi / lo) ** u).astype(int)


def _inputs(case, seed):
    """Structures and model of a case: NumPy arrays made from the seed alone."""
    rng = np.random.default_rng([seed, 1905])
    S = case["structures"]
    if case["atoms_hi"]:
        counts = _counts(case)
        rho = rng.uniform(case["density"], max(case["density"], case["density_hi"]), S)
    else:
        counts, rho = [case["atoms"]] * S, [case["density"]] * S
    s = _structures(case, rng, counts, rho)
    m = case["sparse"]
    if m:
        box_atoms = max(200, m if case["kind"] != "kernel_rows" else case["atoms"])
        mid = 0.5 * (case["density"] + max(case["density"], case["density_hi"]))
        sb = _structures(dict(case, shear=0.0), rng, [box_atoms], [mid])
        pick = np.sort(rng.choice(box_atoms, size=m, replace=False))
        s["q_sparse"] = _Reference(case).descriptors(sb, pick)[0].cpu().numpy()
        s["alpha"] = rng.normal(0.0, 0.1, size=m)
    if case["kind"] == "autograd":
        s["weight"] = rng.uniform(0.5, 1.5, S)
    if case["kind"] == "md":
        s["vel"] = rng.normal(0.0, math.sqrt(0.025852 / MD_MASS * EV_PER_AMU_A2_FS2), (len(s["pos"]), 3))
    return s


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    model = SoapGap(r_cut=case["r_cut"], r_soft=case["r_cut"] - case["buffer"], sigma_r0=case["sigma_r"],
                    sigma_p0=case["sigma_p"], alpha_r=case["alpha_r"], alpha_p=case["alpha_p"],
                    amp_a=case["amp_a"], n_max=case["n_max"], l_max=case["l_max"], n_species=case["species"],
                    precision=case["precision"])
    if case["sparse"] and kind != "desc":
        model.set_model(x["q_sparse"], x["alpha"], case["zeta"])
    st = dict(kind=kind, model=model)
    if kind == "host":
        st["x"] = x
        return st
    if kind == "kernel_rows":
        st["q"] = torch.as_tensor(x["q_sparse"], dtype=model.dtype, device="cuda")
        return st
    s = Structures(x["pos"], x["cell"], x["species"], x["offs"])
    st["s"] = s
    if kind == "autograd":
        st["weight"] = torch.as_tensor(x["weight"], device="cuda")
    elif kind == "md":
        model.set_skin(0.4)
        st["pos"], st["vel"] = s.pos.clone(), torch.as_tensor(x["vel"], device="cuda")
        st["md"] = VelocityVerlet(model, s, MD_MASS, MD_DT, vel=st["vel"], capture=True)
        st["f"] = st["md"].f.clone()
    elif kind == "graph":
        # a long-running program tunes its batch class once and captures the evaluation
        model.autotune(s)
        st["pos"] = s.pos.clone()
        st["graph"] = CapturedEvaluation(model, s, energy=True, forces=True)
    elif kind == "compute_virial":
        model.autotune(s)
    return st


def run(state):
    kind, model = state["kind"], state["model"]
    if kind == "desc":
        o = model.compute(state["s"], desc=True)
        return [o["q"], o["pnorm"]]
    if kind == "compute":
        o = model.compute(state["s"], energy=True, forces=True)
        return [o["e_atom"], o["e_struct"], o["forces"]]
    if kind == "compute_virial":
        o = model.compute(state["s"], energy=True, forces=True, virial=True)
        return [o["e_atom"], o["e_struct"], o["forces"], o["virial"]]
    if kind == "autograd":
        s = state["s"]
        pos = s.pos.detach().requires_grad_(True)
        e = SoapGapEnergy.apply(pos, model, s)
        (e * state["weight"]).sum().backward()
        return [e.detach(), pos.grad]
    if kind == "md":
        md, s = state["md"], state["s"]
        s.pos.copy_(state["pos"])
        md.vel.copy_(state["vel"])
        md.f.copy_(state["f"])
        md.step(MD_STEPS)
        return [s.pos, md.vel, md.f, md.out["e_struct"]]
    if kind == "host":
        x = state["x"]
        o = model.compute_host(x["pos"], x["cell"], x["species"], x["offs"], energy=True, forces=True, virial=True)
        return [o["e_atom"], o["e_struct"], o["forces"], o["virial"]]
    if kind == "graph":
        state["s"].pos.copy_(state["pos"])
        o = state["graph"].replay()
        return [o["e_atom"], o["e_struct"], o["forces"]]
    if kind == "design":
        o = model.design(state["s"], k_struct=True, dk=True)
        return [o["k_struct"], o["dk"]]
    if kind == "kernel_rows":
        return [model.kernel_rows(state["q"])]
    raise ValueError(kind)


def work(case):
    kind = case["kind"]
    es = 8 if case["precision"] == "fp64" else 4
    S = case["structures"]
    rho = 0.5 * (case["density"] + max(case["density"], case["density_hi"]))
    N = float(_counts(case).sum()) if case["atoms_hi"] else float(S * case["atoms"])
    P = N * rho * 4.0 / 3.0 * math.pi * case["r_cut"] ** 3
    nch, n, lm = case["species"] * case["n_max"], case["n_max"], case["l_max"] + 1
    L = lm * lm
    D, M = nch * (nch + 1) // 2 * lm, case["sparse"]
    if kind == "kernel_rows":
        return {"bytes": es * (2.0 * M * D + M * M), "flops": 2.0 * M * M * D}
    ins = N * 28.0 + S * 80.0
    fwd = P * 2.0 * n * L + N * nch * (nch + 1) * L
    if kind == "desc":
        return {"bytes": ins + es * N * (D + 1), "flops": fwd}
    model = es * M * (D + 1.0)
    grad = P * 4.0 * n * L + N * 2.0 * nch * nch * L
    if kind == "design":
        return {"bytes": ins + model + es * 3.0 * N * M + 8.0 * S * M,
                "flops": fwd + 2.0 * N * M * D + P * 6.0 * n * L * nch + 6.0 * (P + N) * D * M}
    out = es * N + 8.0 * S + 24.0 * N + (72.0 * S if kind in ("compute_virial", "host") else 0.0)
    w = {"bytes": ins + model + out, "flops": fwd + 4.0 * N * M * D + grad}
    if kind == "md":
        return {"bytes": MD_STEPS * (w["bytes"] + 72.0 * N), "flops": MD_STEPS * w["flops"]}
    return w


# -------------------------------------------------------------------- the same in 64 bits
DIGITS = 120


def _dec_pi():
    def atan_inv(k):
        k2, term, total, i = Decimal(k * k), Decimal(1) / k, Decimal(0), 0
        while abs(term) > Decimal(10) ** -(DIGITS + 5):
            total += term / (2 * i + 1) * (1 if i % 2 == 0 else -1)
            term /= k2
            i += 1
        return total
    return 4 * (4 * atan_inv(5) - atan_inv(239))


def _dec_erf(x, pi):
    term, total, i = x, x, 0
    while abs(term) > Decimal(10) ** -(DIGITS - 20):
        i += 1
        term = -term * x * x / i
        total += term / (2 * i + 1)
    return 2 * total / pi.sqrt()


def _dec_inverse(a):
    n = len(a)
    a = [row[:] + [Decimal(int(i == j)) for j in range(n)] for i, row in enumerate(a)]
    for k in range(n):
        p = max(range(k, n), key=lambda i: abs(a[i][k]))
        a[k], a[p] = a[p], a[k]
        inv = 1 / a[k][k]
        a[k] = [v * inv for v in a[k]]
        for i in range(n):
            if i != k and a[i][k] != 0:
                f = a[i][k]
                a[i] = [v - f * u for v, u in zip(a[i], a[k])]
    return [row[n:] for row in a]


@functools.lru_cache(maxsize=64)
def _radial_basis(n_max, r_cut, sigma, r_soft, n_f, sigma_min):
    """Quadrature nodes x and the matrix F [n_max, nodes] with
    b_n(r) = A(r) sum_k F[n, k] exp(-(x_k - r)^2 / (2 sigma_r(r)^2)): the orthonormalised
    functions sum_a W_na phi_a, W = S^-1/2, with the smoothing of the density on the
    polynomials and, beyond r_cut, the tail of the auxiliary Gaussian; weights included."""
    with localcontext() as ctx:
        ctx.prec = DIGITS
        pi = _dec_pi()
        rc, s0 = Decimal(r_cut), Decimal(sigma)
        norm = [(rc / (2 * a + 5)).sqrt() for a in range(1, n_max)]
        gn = Decimal(2).sqrt() / (s0.sqrt() * pi.sqrt().sqrt())
        e_rc = (-rc * rc / (2 * s0 * s0)).exp()
        j = [s0 * (pi / 2).sqrt() * _dec_erf(rc / (Decimal(2).sqrt() * s0), pi)]
        j.append(j[0] + s0 * s0 / rc * (e_rc - 1))
        for k in range(n_max):
            j.append((k + 1) * (s0 / rc) ** 2 * j[k] + j[k + 1] - s0 * s0 / rc)
        S = [[Decimal(0)] * n_max for _ in range(n_max)]
        for a in range(1, n_max):
            for b in range(1, n_max):
                S[a - 1][b - 1] = rc / (a + b + 5) / (norm[a - 1] * norm[b - 1])
            S[a - 1][n_max - 1] = S[n_max - 1][a - 1] = gn * j[a + 2] / norm[a - 1]
        S[-1][-1] = gn * gn * s0 * pi.sqrt() / 2 * _dec_erf(rc / s0, pi)
        # W = S^-1/2 by the Denman-Beavers iteration
        Y, Z = S, [[Decimal(int(p == q)) for q in range(n_max)] for p in range(n_max)]
        for _ in range(200):
            iy, iz = _dec_inverse(Y), _dec_inverse(Z)
            Yn = [[(Y[p][q] + iz[p][q]) / 2 for q in range(n_max)] for p in range(n_max)]
            Zn = [[(Z[p][q] + iy[p][q]) / 2 for q in range(n_max)] for p in range(n_max)]
            step = max(abs(Zn[p][q] - Z[p][q]) for p in range(n_max) for q in range(n_max))
            size = max(abs(v) for row in Zn for v in row)
            Y, Z = Yn, Zn
            if step < size * Decimal(10) ** -40:
                break
        W = Z
        gx, gw = np.polynomial.legendre.leggauss(20)
        tau = (r_cut - r_soft) / n_f if r_soft < r_cut else sigma_min
        edges = []
        for lo, hi, scale in ((0.0, r_soft, sigma_min), (r_soft, r_cut, min(sigma_min, tau)),
                              (r_cut, r_cut + 10.0 * max(sigma, sigma_min), sigma_min)):
            if hi > lo:
                e = np.linspace(lo, hi, int(math.ceil((hi - lo) / scale)) + 1)
                edges += list(zip(e[:-1], e[1:]))
        x = np.concatenate([0.5 * (b - a) * gx + 0.5 * (a + b) for a, b in edges])
        w = np.concatenate([0.5 * (b - a) * gw for a, b in edges])
        F = np.zeros((n_max, len(x)))
        for k, (xk, wk) in enumerate(zip(x, w)):
            r = Decimal(float(xk))
            gauss = gn * (-r * r / (2 * s0 * s0)).exp()
            poly = []
            if xk < r_cut:
                f = Decimal(1)
                if xk > r_soft:
                    f = (-(Decimal(n_f) * (r - Decimal(r_soft)) / (rc - Decimal(r_soft))) ** 2 / 2).exp()
                t = 1 - r / rc
                poly = [f * t ** (a + 2) / norm[a - 1] for a in range(1, n_max)]
            for n in range(n_max):
                v = W[n][n_max - 1] * gauss
                for a, pv in enumerate(poly):
                    v += W[n][a] * pv
                F[n, k] = float(v) * wk
    return x, F


class _Reference:
    """The separable-density descriptor and the GAP model on it, 64-bit torch operations."""

    N_F = 4.0

    def __init__(self, case, device="cuda"):
        self.c, self.dev = case, device
        self.n, self.lmax, self.nsp = case["n_max"], case["l_max"], case["species"]
        self.nch, self.L = self.nsp * self.n, (self.lmax + 1) ** 2
        smin = min(case["sigma_r"], case["sigma_r"] + case["alpha_r"] * case["r_cut"])
        x, F = _radial_basis(self.n, case["r_cut"], case["sigma_r"], case["r_cut"] - case["buffer"], self.N_F, smin)
        self.x, self.F = self._t(x), self._t(F)
        iu = np.triu_indices(self.nch)
        self.iu = (torch.as_tensor(iu[0], device=device), torch.as_tensor(iu[1], device=device))
        self.pack = self._t(np.where(iu[0] == iu[1], 1.0, math.sqrt(2.0)))

    def _t(self, a):
        return torch.as_tensor(np.asarray(a), dtype=F64, device=self.dev)

    # --- one pair: radial and angular coefficients and their gradients
    def radial(self, r):
        c = self.c
        sr, sp = c["sigma_r"] + c["alpha_r"] * r, c["sigma_p"] + c["alpha_p"] * r
        u = r / c["r_cut"]
        y = (1.0 + 2.0 * u ** 3 - 3.0 * u ** 2).clamp(min=0.0)
        a, dy = c["amp_a"], (6.0 * u ** 2 - 6.0 * u) / c["r_cut"]
        amp = y ** a / (sr * sp * sp)
        if a == 0.0:
            damp = torch.zeros_like(r)
        else:
            damp = a * y ** (a - 1.0) * dy / (sr * sp * sp)
        damp = damp - amp * (c["alpha_r"] / sr + 2.0 * c["alpha_p"] / sp)
        d = self.x[None, :] - r[:, None]
        t = d / sr[:, None]
        e = torch.exp(-0.5 * t * t)
        s0 = e @ self.F.T
        s1 = (e * (t / sr[:, None]) * (1.0 + c["alpha_r"] * t)) @ self.F.T
        return amp[:, None] * s0, damp[:, None] * s0 + amp[:, None] * s1

    def ilexp(self, z):
        """e^-z i_l(z) and its derivative, l = 0..l_max: ratios i_l / i_(l-1) by their
        continued fraction, downwards."""
        ratio, q = [None] * (self.lmax + 2), torch.zeros_like(z)
        for l in range(self.lmax + 160, 0, -1):
            q = 1.0 / ((2 * l + 1) / z + q)
            if l <= self.lmax + 1:
                ratio[l] = q
        il = [-torch.expm1(-2.0 * z) / (2.0 * z)]
        for l in range(1, self.lmax + 2):
            il.append(il[-1] * ratio[l])
        dil = [il[l + 1] + l / z * il[l] - il[l] for l in range(self.lmax + 1)]
        return torch.stack(il[:-1], 1), torch.stack(dil, 1)

    def harmonics(self, u, grad=True):
        """Real orthonormal Y_lm(u), index l^2 + l + m, and the gradient of the extension
        Q_lm(z) C_m(x, y) (S_m for m < 0) at the unit vectors u: [P, L] and, with grad,
        [P, 3, L]."""
        x, y, z = u[:, 0], u[:, 1], u[:, 2]
        one, zero = torch.ones_like(x), torch.zeros_like(x)
        C, S = [one], [zero]
        for m in range(1, self.lmax + 1):
            C.append(x * C[-1] - y * S[-1])
            S.append(x * S[-1] + y * C[m - 1])
        Y = [None] * self.L
        G = [None] * self.L
        for m in range(self.lmax + 1):
            q = {m: one * math.sqrt(math.prod((2 * k - 1) / (2 * k) for k in range(1, m + 1)) * (2 * m + 1))}
            dq = {m: zero}
            for l in range(m + 1, self.lmax + 1):
                a = math.sqrt((4.0 * l * l - 1.0) / (l * l - m * m))
                b = math.sqrt(((l - 1.0) ** 2 - m * m) * (2 * l + 1) / ((2 * l - 3) * (l * l - m * m))) \
                    if l > m + 1 else 0.0
                q[l] = a * z * q[l - 1] - (b * q[l - 2] if b else 0.0)
                dq[l] = a * (q[l - 1] + z * dq[l - 1]) - (b * dq[l - 2] if b else 0.0)
            w = math.sqrt((1.0 if m == 0 else 2.0) / (4.0 * math.pi))
            for l in range(m, self.lmax + 1):
                k = l * l + l
                Y[k + m] = w * q[l] * C[m]
                if not grad:
                    Y[k - m] = w * q[l] * S[m] if m else Y[k]
                    continue
                G[k + m] = torch.stack([w * q[l] * m * C[m - 1], -w * q[l] * m * S[m - 1], w * dq[l] * C[m]], 1) \
                    if m else torch.stack([zero, zero, w * dq[l]], 1)
                if m:
                    Y[k - m] = w * q[l] * S[m]
                    G[k - m] = torch.stack([w * q[l] * m * S[m - 1], w * q[l] * m * C[m - 1], w * dq[l] * S[m]], 1)
        return torch.stack(Y, 1), torch.stack(G, 2) if grad else None

    def angular(self, rv, grad):
        r = rv.norm(dim=1)
        u = rv / r[:, None]
        c = self.c
        sp = c["sigma_p"] + c["alpha_p"] * r
        il, dil = self.ilexp((r / sp) ** 2)
        reps = torch.as_tensor([2 * l + 1 for l in range(self.lmax + 1)], device=self.dev)
        il = 4.0 * math.pi * torch.repeat_interleave(il, reps, 1)
        Y, G = self.harmonics(u, grad)
        if not grad:
            return il * Y, None
        dz = 2.0 * (r / sp) * (1.0 / sp - r * c["alpha_p"] / sp ** 2)
        dil = 4.0 * math.pi * torch.repeat_interleave(dil, reps, 1) * dz[:, None]
        G = (G - u[:, :, None] * torch.einsum("pa,pal->pl", u, G)[:, None, :]) / r[:, None, None]
        return il * Y, u[:, :, None] * (dil * Y)[:, None, :] + il[:, None, :] * G

    # --- neighbours
    def pairs(self, s, centres=None):
        """(i, j, r_ij) of every neighbour of the centres, i nondecreasing."""
        rc = self.c["r_cut"]
        oi, oj, orv = [], [], []
        for t in range(len(s["cell"])):
            a, b = int(s["offs"][t]), int(s["offs"][t + 1])
            ci = np.arange(a, b) if centres is None else centres[(centres >= a) & (centres < b)]
            if not len(ci):
                continue
            h = s["cell"][t]
            hinv = np.linalg.inv(h)
            width = 1.0 / np.linalg.norm(hinv, axis=0)
            frac = s["pos"][a:b] @ hinv
            base = np.floor(frac)
            fr = self._t(frac - base)
            pos, pw = self._t(s["pos"][a:b]), self._t(s["pos"][a:b] - base @ h)
            m = np.ceil(rc / width).astype(int)
            sh = self._t([(p, q, r) for p in range(-m[0], m[0] + 1) for q in range(-m[1], m[1] + 1)
                          for r in range(-m[2], m[2] + 1)])
            near = self._t(rc / width * (1.0 + 1e-9))
            gj, gx = [], []
            for v in sh:
                f = fr + v
                k = torch.nonzero(((f >= -near) & (f <= 1.0 + near)).all(1))[:, 0]
                gj.append(k)
                gx.append(pw[k] + v @ self._t(h))
            gj, gx = torch.cat(gj), torch.cat(gx)
            order = torch.argsort(gx[:, 0])
            gj, gx = gj[order], gx[order]
            gx0 = gx[:, 0].contiguous()
            loc = torch.as_tensor(ci - a, device=self.dev)
            loc = loc[torch.argsort(pw[loc, 0])]
            block = 2048
            for k0 in range(0, len(loc), block):
                c = loc[k0:k0 + block]
                xc = pw[c]
                lo = int(torch.searchsorted(gx0, xc[0, 0] - rc))
                hi = int(torch.searchsorted(gx0, xc[-1, 0] + rc, right=True))
                d2 = torch.zeros((len(c), hi - lo), dtype=F64, device=self.dev)
                for ax in range(3):
                    d2 += (gx[None, lo:hi, ax] - xc[:, None, ax]) ** 2
                bi, bj = torch.nonzero((d2 < rc * rc) & (d2 > 1e-8), as_tuple=True)
                oi.append(c[bi] + a)
                oj.append(gj[lo + bj] + a)
                orv.append(gx[lo + bj] - xc[bi])
        if not oi:
            z = torch.zeros(0, dtype=torch.int64, device=self.dev)
            return z, z, torch.zeros((0, 3), dtype=F64, device=self.dev)
        i, j, rv = torch.cat(oi), torch.cat(oj), torch.cat(orv)
        order = torch.argsort(i, stable=True)
        return i[order], j[order], rv[order]

    # --- descriptors and their adjoint, in blocks of centres
    def blocks(self, s, centres=None, limit=120000):
        cen = np.arange(len(s["pos"])) if centres is None else centres
        i, j, rv = self.pairs(s, centres)
        ct = torch.as_tensor(cen, device=self.dev)
        starts = torch.searchsorted(i, ct).cpu().numpy()
        ends = torch.searchsorted(i, ct, right=True).cpu().numpy()
        k = 0
        while k < len(cen):
            e = int(np.searchsorted(ends, starts[k] + limit, side="right"))
            e = min(max(e, k + 1), k + 20000, len(cen))
            sl = slice(int(starts[k]), int(ends[e - 1]))
            yield ct[k:e], torch.searchsorted(ct[k:e], i[sl]), j[sl], rv[sl]
            k = e

    def coefficients(self, spec, cc, li, j, b, a):
        n_c = len(cc)
        order = torch.argsort(li * self.nsp + spec[j], stable=True)
        key = (li * self.nsp + spec[j])[order]
        c = torch.zeros((n_c * self.nsp, self.n, self.L), dtype=F64, device=self.dev)
        step = max(1, 40_000_000 // (self.n * self.L))
        for p in range(0, len(key), step):
            o = order[p:p + step]
            c.index_add_(0, key[p:p + step], b[o][:, :, None] * a[o][:, None, :])
        b0 = self.radial(torch.zeros(1, dtype=F64, device=self.dev))[0][0]
        c[torch.arange(n_c, device=self.dev) * self.nsp + spec[cc], :, 0] += math.sqrt(4.0 * math.pi) * b0
        return c.reshape(n_c, self.nch, self.L)

    def spectrum(self, c):
        p = []
        for l in range(self.lmax + 1):
            cl = c[:, :, l * l:(l + 1) ** 2]
            p.append((cl @ cl.transpose(1, 2))[:, self.iu[0], self.iu[1]] * self.pack)
        p = torch.stack(p, 2).reshape(len(c), -1)
        pn = p.norm(dim=1)
        return p / pn[:, None], pn

    def descriptors(self, s, centres=None):
        spec = torch.as_tensor(s["species"], dtype=torch.int64, device=self.dev)
        q, pn = [], []
        for cc, li, j, rv in self.blocks(s, centres):
            b, _ = self.radial(rv.norm(dim=1))
            a, _ = self.angular(rv, False)
            out = self.spectrum(self.coefficients(spec, cc, li, j, b, a))
            q.append(out[0])
            pn.append(out[1])
        return torch.cat(q), torch.cat(pn)

    def evaluate(self, s, weight=None):
        """e_atom, e_struct, forces (of the weighted energy sum) and virial."""
        N, S = len(s["pos"]), len(s["cell"])
        spec = torch.as_tensor(s["species"], dtype=torch.int64, device=self.dev)
        own = torch.as_tensor(np.repeat(np.arange(S), np.diff(s["offs"])), device=self.dev)
        w = torch.ones(S, dtype=F64, device=self.dev) if weight is None else self._t(weight)
        qs, al, zeta = self._t(s["q_sparse"]), self._t(s["alpha"]), self.c["zeta"]
        e = torch.zeros(N, dtype=F64, device=self.dev)
        f = torch.zeros((N, 3), dtype=F64, device=self.dev)
        vir = torch.zeros((S, 3, 3), dtype=F64, device=self.dev)
        for cc, li, j, rv in self.blocks(s):
            r = rv.norm(dim=1)
            b, db = self.radial(r)
            a, da = self.angular(rv, True)
            c = self.coefficients(spec, cc, li, j, b, a)
            q, pn = self.spectrum(c)
            k = q @ qs.T
            e[cc] = (k ** zeta) @ al
            g = (k ** (zeta - 1.0) * (zeta * al)) @ qs * w[own[cc]][:, None]
            g = (g - q * (g * q).sum(1, keepdim=True)) / pn[:, None]
            g = g.reshape(len(cc), len(self.pack), self.lmax + 1) * self.pack[None, :, None]
            G = torch.empty_like(c)
            for l in range(self.lmax + 1):
                H = torch.zeros((len(cc), self.nch, self.nch), dtype=F64, device=self.dev)
                H[:, self.iu[0], self.iu[1]] = g[:, :, l]
                cl = slice(l * l, (l + 1) ** 2)
                G[:, :, cl] = (H + H.transpose(1, 2)) @ c[:, :, cl]
            G = G.reshape(len(cc) * self.nsp, self.n, self.L)
            key = li * self.nsp + spec[j]
            dr = torch.empty_like(rv)
            step = max(1, 40_000_000 // (self.n * self.L))
            for p in range(0, len(r), step):
                x = slice(p, p + step)
                Gp = G[key[x]]
                ub = torch.einsum("pnl,pn->pl", Gp, b[x])
                ur = (torch.einsum("pnl,pn->pl", Gp, db[x]) * a[x]).sum(1)
                dr[x] = torch.einsum("pal,pl->pa", da[x], ub) + ur[:, None] * rv[x] / r[x, None]
            f.index_add_(0, cc[li], dr)
            f.index_add_(0, j, -dr)
            vir.index_add_(0, own[j], -dr[:, :, None] * rv[:, None, :])
        es = torch.zeros(S, dtype=F64, device=self.dev).index_add_(0, own, e)
        return e, es, f, vir

    def design(self, s):
        """Energy rows [S, M] and force rows [N, 3, M] of the fitting matrices."""
        N, S = len(s["pos"]), len(s["cell"])
        spec = torch.as_tensor(s["species"], dtype=torch.int64, device=self.dev)
        own = torch.as_tensor(np.repeat(np.arange(S), np.diff(s["offs"])), device=self.dev)
        qs, zeta = self._t(s["q_sparse"]), self.c["zeta"]
        M = len(qs)
        ks = torch.zeros((S, M), dtype=F64, device=self.dev)
        dk = torch.zeros((N, 3, M), dtype=F64, device=self.dev)
        for cc, li, j, rv in self.blocks(s, limit=20000):
            r = rv.norm(dim=1)
            b, db = self.radial(r)
            a, da = self.angular(rv, True)
            c = self.coefficients(spec, cc, li, j, b, a)
            q, pn = self.spectrum(c)
            k = q @ qs.T
            ks.index_add_(0, own[cc], k ** zeta)
            X = torch.empty((len(r), 3, self.nch, self.nch, self.lmax + 1), dtype=F64, device=self.dev).zero_()
            ch = spec[j][:, None] * self.n + torch.arange(self.n, device=self.dev)
            pi = torch.arange(len(r), device=self.dev)[:, None]
            for l in range(self.lmax + 1):
                cl = slice(l * l, (l + 1) ** 2)
                cm = c[li][:, :, cl].transpose(1, 2)
                A = a[:, None, cl] @ cm                             # [P, 1, nch]
                dA = da[:, :, cl] @ cm                              # [P, 3, nch]
                t = b[:, None, :, None] * dA[:, :, None, :] \
                    + (rv / r[:, None])[:, :, None, None] * db[:, None, :, None] * A[:, :, None, :]
                X[pi, :, ch, :, l] = t.transpose(1, 2)
            X = X + X.transpose(2, 3)
            dp = (X[:, :, self.iu[0], self.iu[1]] * self.pack[None, None, :, None]).reshape(len(r), 3, -1)
            dq = (dp - q[li][:, None, :] * (dp * q[li][:, None, :]).sum(2, keepdim=True)) / pn[li][:, None, None]
            row = (dq @ qs.T) * (zeta * k ** (zeta - 1.0))[li][:, None, :]
            dk.index_add_(0, j, row)
            dk.index_add_(0, cc[li], -row)
        return ks, dk


def exact(case, seed):
    x = _inputs(case, seed)
    ref, kind = _Reference(case), case["kind"]
    if kind == "desc":
        return list(ref.descriptors(x))
    if kind in ("compute", "graph"):
        return list(ref.evaluate(x)[:3])
    if kind == "compute_virial":
        return list(ref.evaluate(x))
    if kind == "host":
        return [t.cpu().numpy() for t in ref.evaluate(x)]
    if kind == "autograd":
        _, es, f, _ = ref.evaluate(x, weight=x["weight"])
        return [es, -f]
    if kind == "md":
        pos, vel = torch.as_tensor(x["pos"]), torch.as_tensor(x["vel"])
        _, _, f, _ = ref.evaluate(x)
        kick = 0.5 * MD_DT * EV_PER_AMU_A2_FS2 / MD_MASS
        for _ in range(MD_STEPS):
            vel = vel + kick * f.cpu()
            pos = pos + MD_DT * vel
            _, es, f, _ = ref.evaluate(dict(x, pos=pos.numpy()))
            vel = vel + kick * f.cpu()
        return [pos.cuda(), vel.cuda(), f, es]
    if kind == "design":
        return list(ref.design(x))
    if kind == "kernel_rows":
        q = torch.as_tensor(x["q_sparse"], dtype=F64, device="cuda")
        if case["precision"] != "fp64":
            q = q.float().double()          # the rows as the call gets them
        return [(q @ torch.as_tensor(x["q_sparse"], dtype=F64, device="cuda").T) ** case["zeta"]]
    return None
