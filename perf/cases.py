"""Performance cases of the library: the calls a user's program makes, at the sizes it makes them.

A case names a system, its grid and one call of the public binding:

* systems: a water molecule; a heavy/light cluster (half Pb/I with 2s2p1d1f, half C/H with 2s1p); a set of independent
  small molecules in one grid; a periodic slab (heavy layer of 64-function atoms, light atoms around it);
* calls: the integration, the density and its gradient form, the differentiable integration with its backward pass,
  the whole one-pass SCF step, the per-column operator, the scalar <-> spinor transformation and the k-phase fold;
* precisions: "fp64" (the default of every call) and "split" (the tensor-core path).

The case fixes the geometry (and with it the points, the batches and the block pattern, which a program keeps over many
steps); exponents, effective nuclear charges, potential and matrices come from the seed.  exact() evaluates the definitions in plain FP64 torch
on the points and weights of the case's grid.
"""
import math

import numpy as np
import torch

import paper_2608_00773_gb300 as q4c

R_CUT, R_ON, R_MIN, N_LOG, R_NB = 6.0, 5.0, 1e-4, 200, 12.0


# ------------------------------------------------------------------ the cases
def _case(name, system, n, op, prec, n_rad, n_theta, n_phi, batch_max, tuned=False, n_k=0):
    """tuned: the program calls q4c_autotune once after building the grid (as one that reuses it for many steps does)."""
    c = dict(system=system, n=n, op=op, prec=prec, n_rad=n_rad, n_theta=n_theta, n_phi=n_phi, batch_max=batch_max,
             tuned=tuned, n_k=n_k)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one small molecule, one call: latency and launches are what a geometry scan or a test waits for
        _case("water_integrate_split", "water", 3, "integrate", "split", 30, 8, 16, 128),
        # the same molecule through the default precision, a whole SCF step
        _case("water_scf_fp64", "water", 3, "scf", "fp64", 30, 8, 16, 128),
        # a small cluster in the training direction at the default precision (autograd forward and backward)
        _case("cluster8_autograd_fp64", "cluster", 8, "autograd", "fp64", 24, 8, 16, 200),
        # the throughput workload, 64 atoms with 392 angular points per shell: a whole SCF step ...
        _case("cluster64_scf_split", "cluster", 64, "scf", "split", 60, 14, 28, 300, tuned=True),
        # ... the integration with its spinor blocks alone (setup of a Hamiltonian) at both precisions ...
        _case("cluster64_integrate_split", "cluster", 64, "integrate", "split", 60, 14, 28, 300),
        _case("cluster64_integrate_fp64", "cluster", 64, "integrate", "fp64", 60, 14, 28, 300),
        # ... the density update alone ...
        _case("cluster64_density_split", "cluster", 64, "density", "split", 60, 14, 28, 300),
        # ... and the per-column operator of the large-component matrix
        _case("cluster64_columns_split", "cluster", 64, "columns", "split", 60, 14, 28, 300),
        # many independent molecules in one call, forward and backward (a training step over a batch of structures)
        _case("molecules24_autograd_split", "molecules", 24, "autograd", "split", 40, 10, 20, 128),
        # a periodic cell whose batches hold hundreds of functions: a whole SCF step
        _case("slab304_scf_split", "slab", 304, "scf", "split", 12, 6, 12, 300, tuned=True),
        # what follows the integration: spinor blocks and their reverse map, and H(k) at a few k-points
        _case("cluster64_spinor", "cluster", 64, "spinor", "fp64", 8, 5, 10, 300),
        _case("slab304_kfold", "slab", 304, "kfold", "fp64", 4, 4, 8, 300, n_k=4),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    """A case of the same ranges: any system, call and precision that go together, odd sizes and ragged batches."""
    system = rng.choice(["water", "cluster", "cluster", "cluster", "molecules", "slab"])
    op = rng.choice(["integrate", "density", "density_full", "autograd", "scf", "scf", "columns", "spinor", "kfold"])
    prec = rng.choice(["split", "split", "fp64"])
    batch_max = rng.choice([64, 97, 128, 200, 256, 300, 333])
    n_theta = rng.randint(5, 14)
    n_phi = rng.randint(10, 28)
    n_k = 0
    if op == "kfold":
        system, n_k = "slab", rng.randint(1, 6)
    if system == "water":
        n, n_rad = 3, rng.randint(20, 60)
        op = "integrate" if op == "spinor" else op
    elif system == "cluster":
        n, n_rad = _log(rng, 4, 64 if prec == "split" else 32), rng.randint(20, 60 if prec == "split" else 40)
    elif system == "molecules":
        n, n_rad = _log(rng, 2, 24 if prec == "split" else 5), rng.randint(20, 40 if prec == "split" else 30)
        n_theta, n_phi = min(n_theta, 10), min(n_phi, 20)
    else:
        n, n_rad, n_theta, n_phi = rng.randint(200, 304), rng.randint(6, 12), rng.randint(4, 6), rng.randint(8, 12)
        prec = "split"
        batch_max = max(batch_max, 128)
    if op in ("spinor", "kfold"):
        prec, n_rad, n_theta, n_phi = "fp64", rng.randint(4, 8), 4, 8
    return _case(None, system, n, op, prec, n_rad, n_theta, n_phi, batch_max,
                 tuned=prec == "split" and rng.random() < 0.5, n_k=n_k)


# ------------------------------------------------------------------ structures
def _exponents(rng, ls):
    return [(l, float(10.0 ** rng.uniform(-1.0, 1.0))) for l in ls]


def _place(rng, n, box, sep, placed=(), placed_sep=(), period=None):
    """n points uniform in the box ((lo, hi) per axis), at least sep apart and placed_sep from the placed ones."""
    box = np.asarray(box, float)
    pts, seps = list(placed), list(placed_sep)
    n0 = len(pts)
    while len(pts) < n0 + n:
        c = rng.uniform(box[:, 0], box[:, 1])
        if pts:
            d = np.asarray(pts) - c
            if period is not None:
                d -= period * np.round(d / period)
            if np.any((d * d).sum(1) < np.square(seps)):
                continue
        pts.append(c)
        seps.append(sep)
    return np.asarray(pts[n0:]).reshape(-1, 3)


def _structure(case, seed):
    """dict: xyz, species (index per atom), Z and basis [(l, alpha)] per species, effective charge per atom, lattice,
    molecule ranges."""
    geo, rng = np.random.default_rng([1002, case["n"]]), np.random.default_rng([seed & 0x7FFFFFFF, case["n"]])
    light = [0, 0, 1]
    S = dict(lattice=None, n_shell=0, mol=None)
    if case["system"] in ("water", "molecules"):
        S["Z"], S["basis"] = [8.0, 1.0], [_exponents(rng, [0, 0, 0, 1, 1, 2]), _exponents(rng, light)]
        if case["system"] == "water":
            S["xyz"] = np.array([[0.0, 0.0, 0.0], [1.43, 1.11, 0.0], [-1.43, 1.11, 0.0]]) + geo.normal(0, 0.02, (3, 3))
            S["species"] = np.array([0, 1, 1], np.int32)
        else:
            xyz, kinds, ptr = [], [], [0]
            for _ in range(case["n"]):
                n = int(geo.integers(3, 41))
                side = 3.0 * n ** (1.0 / 3.0) + 2.0
                xyz.append(_place(geo, n, [(0.0, side)] * 3, 1.8))
                kinds.append((geo.uniform(size=n) >= 1.0 / 3.0).astype(np.int32))
                ptr.append(ptr[-1] + n)
            S["xyz"], S["species"], S["mol"] = np.vstack(xyz), np.concatenate(kinds), np.array(ptr, np.int32)
    elif case["system"] == "cluster":
        heavy = [0, 0, 1, 1, 2, 3]
        S["Z"] = [82.0, 53.0, 6.0, 1.0]
        S["basis"] = [_exponents(rng, heavy), _exponents(rng, heavy), _exponents(rng, light), _exponents(rng, light)]
        S["species"] = geo.permutation(np.arange(case["n"]) % 4).astype(np.int32)
        S["xyz"] = _place(geo, case["n"], [(0.0, 24.0 * (case["n"] / 64.0) ** (1.0 / 3.0) + 1.0)] * 3, 4.0)
    else:
        heavy, mid = [0] * 4 + [1] * 4 + [2] * 4 + [3] * 4, [0, 0, 0, 1, 1, 2]
        S["Z"] = [82.0, 53.0, 1.0, 6.0, 7.0]
        S["basis"] = [_exponents(rng, ls) for ls in (heavy, heavy, light, mid, mid)]
        side = 30.0 * math.sqrt(case["n"] / 304.0)
        L = np.array([side, side, 25.0])
        nh = int(round(0.3 * case["n"]))
        hv = _place(geo, nh, [(0, side), (0, side), (4.5, 20.5)], 4.0, period=L)
        lt = _place(geo, case["n"] - nh, [(0, side), (0, side), (20.5, 29.5)], 1.8, list(hv), [1.8] * nh, period=L)
        lt[:, 2] %= L[2]
        u = geo.uniform(size=case["n"] - nh) * 3024
        S["xyz"] = np.vstack([hv, lt])
        S["species"] = np.concatenate([(geo.uniform(size=nh) >= 1 / 3).astype(np.int32),
                                       np.where(u < 1728, 2, np.where(u < 2880, 3, 4)).astype(np.int32)])
        S["lattice"], S["n_shell"] = np.diag(L), 1
    S["charge"] = np.array(S["Z"])[S["species"]] * rng.uniform(0.6, 1.0, len(S["xyz"]))
    S["nf"] = np.array([sum(2 * l + 1 for l, _ in b) for b in S["basis"]])
    return S


def _handles(case, S):
    t = q4c.Tables([len(b) for b in S["basis"]], [l for b in S["basis"] for l, _ in b],
                   [a for b in S["basis"] for _, a in b], R_CUT, R_ON, R_MIN, N_LOG)
    g = q4c.Grid(t, S["xyz"], S["species"], case["n_rad"], 1.0, case["n_theta"], case["n_phi"], R_NB, case["batch_max"],
                 S["lattice"], S["n_shell"], S["mol"])
    return t, g


# ------------------------------------------------------------------ inputs on the grid
def _cells(S):
    k = S["n_shell"]
    T = np.array([(a, b, c) for a in range(-k, k + 1) for b in range(-k, k + 1) for c in range(-k, k + 1)])
    return T, (T @ S["lattice"] if S["lattice"] is not None else np.zeros((1, 3)))


def _point_molecules(case, S, ex):
    """Ranges [a, z) of consecutive points and the atoms they see: whole system, or each run of one molecule's points."""
    n = len(ex["xyz"])
    if S["mol"] is None:
        return [(0, n, np.arange(len(S["xyz"])))]
    atom = ex["point_id"] // (case["n_rad"] * case["n_theta"] * case["n_phi"])
    mol = np.searchsorted(S["mol"], atom, side="right") - 1
    cut = np.concatenate([[0], np.nonzero(np.diff(mol))[0] + 1, [n]])
    return [(int(a), int(z), np.arange(S["mol"][mol[a]], S["mol"][mol[a] + 1])) for a, z in zip(cut[:-1], cut[1:])]


def _potential(case, S, ex, dev):
    """v(r) = sum_A -Z_A erf(d)/d; for a cell the images within 12 Bohr, switched off smoothly."""
    Z = S["charge"]
    _, sh = _cells(S)
    v = torch.empty(len(ex["xyz"]), dtype=torch.float64, device=dev)
    for a, z, atoms in _point_molecules(case, S, ex):
        for s in range(a, z, 16384):
            e = min(z, s + 16384)
            P = ex["xyz"][s:e]
            C = (S["xyz"][atoms][None] + sh[:, None]).reshape(-1, 3)
            Zc = np.tile(Z[atoms], len(sh))
            if S["lattice"] is not None:
                gap = np.maximum(0.0, np.maximum(P.min(0) - C, C - P.max(0)))
                near = (gap * gap).sum(1) < 144.0
                C, Zc = C[near], Zc[near]
            d = torch.cdist(torch.tensor(P, device=dev), torch.tensor(C, device=dev),
                            compute_mode="donot_use_mm_for_euclid_dist")
            f = torch.special.erf(d) / d.clamp_min(1e-12)
            if S["lattice"] is not None:
                t = (d - 11.0).clamp(0.0, 1.0)
                f = f * (1.0 - t ** 3 * (10.0 - 15.0 * t + 6.0 * t * t))
            v[s:e] = -(f @ torch.tensor(Zc, device=dev))
    return v


def _pattern(S, ex, dev):
    """Block rows, columns, first values and transposed partners, and per value its transposed value, on the device."""
    ptr, col, T = ex["blk_ptr"], ex["blk_col"].astype(np.int64), ex["blk_T"].astype(np.int64)
    row = np.repeat(np.arange(len(ptr) - 1), np.diff(ptr))
    nf = S["nf"][S["species"]]
    key = lambda A, B, T: ((A * len(nf) + B) * 32 + T[:, 0] + 16) * 1024 + (T[:, 1] + 16) * 32 + T[:, 2] + 16  # noqa: E731
    k = key(row, col, T)
    order = np.argsort(k, kind="stable")
    partner = order[np.searchsorted(k[order], key(col, row, -T))]
    up = lambda x: torch.tensor(np.ascontiguousarray(x), device=dev)  # noqa: E731
    off = up(ex["blk_off"])
    blk = torch.repeat_interleave(torch.arange(len(col), device=dev), off[1:] - off[:-1])
    e = torch.arange(int(ex["blk_off"][-1]), device=dev) - off[blk]
    nB, nA = up(nf[col])[blk], up(nf[row])[blk]
    i, j = e // nB, e % nB
    R = S["xyz"][row] - S["xyz"][col] - (T @ S["lattice"] if S["lattice"] is not None else 0.0)
    return dict(row=row, col=col, T=T, blk=blk, trans=off[up(partner)[blk]] + j * nA + i,
                decay=torch.exp(-up(np.sqrt((R * R).sum(1))) / 4.0)[blk])


def _matrix(pat, gen, antisym=False):
    """A random (anti)symmetric matrix on the pattern, decaying with the distance of the atoms."""
    r = torch.randn(len(pat["blk"]), dtype=torch.float64, device=gen.device, generator=gen) * pat["decay"]
    return 0.5 * (r - r[pat["trans"]]) if antisym else 0.5 * (r + r[pat["trans"]])


def _columns(S, seed):
    """eps and defining potential at the knots per radial function."""
    rng = np.random.default_rng([seed & 0x7FFFFFFF, 77])
    n = sum(len(b) for b in S["basis"])
    Z = np.array([z for z, b in zip(S["Z"], S["basis"]) for _ in b])
    r = R_MIN * (R_CUT / R_MIN) ** (np.arange(N_LOG) / (N_LOG - 1))
    a = rng.uniform(0.8, 1.5, n)
    return rng.uniform(-3.0, -0.1, n), -Z[:, None] * np.array([[math.erf(x * y) / y for y in r] for x in a])


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    S = _structure(case, seed)
    t, g = _handles(case, S)
    ex = g.export()
    st = dict(case=case, S=S, tables=t, grid=g, ex=ex)
    op = case["op"]
    if op in ("integrate", "autograd", "scf", "columns") or case["tuned"]:
        st["v"] = _potential(case, S, ex, dev)
    if op == "columns":
        st["columns"] = _columns(S, seed)
        q4c.q4c_tables_set_columns(t, *st["columns"])
    if op not in ("integrate", "columns"):
        pat = _pattern(S, ex, dev)
        if op in ("density", "density_full", "scf"):
            st["P"] = [_matrix(pat, gen)]
            if op == "density_full":
                st["P"] += [_matrix(pat, gen)] + [_matrix(pat, gen, True) for _ in range(3)]
        if op in ("autograd", "scf", "spinor", "kfold"):
            st["G"] = [_matrix(pat, gen) for _ in range(2)] + [_matrix(pat, gen, True) for _ in range(3)]
        if op == "spinor":
            st["D"] = torch.randn(4 * g.nnz, 2, dtype=torch.float64, device=dev, generator=gen)
            st["D"] = torch.view_as_complex(st["D"])
        if op == "kfold":
            st["k"] = np.random.default_rng(seed & 0x7FFFFFFF).uniform(-0.5, 0.5, (case["n_k"], 3))
    if case["tuned"]:
        q4c.q4c_autotune(t, g, st["v"])
    torch.cuda.synchronize()
    return st


def run(st):
    t, g, prec, op = st["tables"], st["grid"], st["case"]["prec"], st["case"]["op"]
    if op == "integrate":
        return q4c.q4c_integrate(t, g, st["v"], prec, spinor=True)
    if op == "density":
        return q4c.q4c_density(t, g, st["P"][0], prec)
    if op == "density_full":
        return q4c.q4c_density_full(t, g, st["P"], prec)
    if op == "autograd":
        v = st["v"].detach().requires_grad_(True)
        M = q4c.integrate(v, t, g, prec)
        (dv,) = torch.autograd.grad(M, v, st["G"])
        return [m.detach() for m in M] + [dv]
    if op == "scf":
        H, n, dv = q4c.q4c_scf_pass(t, g, v=st["v"], P=st["P"] + [None] * 4, G=st["G"], prec=prec, spinor=True)
        return H + [n, dv]
    if op == "columns":
        return q4c.q4c_integrate_columns(t, g, st["v"], prec)
    if op == "spinor":
        HL, HS = q4c.q4c_spinor_transform(t, g, st["G"])
        return [HL, HS] + q4c.q4c_spinor_density_matrices(t, g, st["D"])
    return [q4c.q4c_kfold(g, H, st["k"]) for H in st["G"]]


_work = {}


def work(case):
    """Algorithmic operations (14 n_p n_b^2 per batch for the seven products of the integration or of the adjoint, 2 for
    the density and the per-column operator), inputs and outputs once; of the structure of seed 0."""
    key = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _work:
        _, g = _handles(case, _structure(case, 0))
        i = g.info
        n, nnz, f, op = float(i.n_points), float(i.nnz), float(i.flops_alg), case["op"]
        b, w = {"integrate": (8 * n + 104 * nnz, f), "density": (8 * nnz + 8 * n, f / 7), "columns": (8 * n + 8 * nnz, f / 7),
                "density_full": (40 * nnz + 8 * n, f), "autograd": (16 * n + 80 * nnz, 2 * f),
                "scf": (24 * n + 152 * nnz, f * 15 / 7), "spinor": (40 * nnz + 128 * nnz + 64 * nnz + 40 * nnz, 600 * nnz),
                "kfold": (40 * nnz + 80 * case["n_k"] * float(g.kpattern()[2][-1]), 20 * case["n_k"] * nnz)}[op]
        _work[key] = {"bytes": b, "flops": w}
    return dict(_work[key])


# ------------------------------------------------------------------ the definitions in plain FP64
def _spline(u):
    """Natural cubic spline in the index: coefficients [n - 1][4] of c0 + c1 s + c2 s^2 + c3 s^3."""
    n = len(u)
    A = np.diag(np.full(n - 2, 4.0)) + np.diag(np.ones(n - 3), 1) + np.diag(np.ones(n - 3), -1)
    M = np.zeros(n)
    M[1:-1] = np.linalg.solve(A, 6.0 * (u[:-2] - 2.0 * u[1:-1] + u[2:]))
    return np.stack([u[:-1], np.diff(u) - (2.0 * M[:-1] + M[1:]) / 6.0, M[:-1] / 2.0, np.diff(M) / 6.0], 1)


def _harmonics():
    """Per l and m = -l..l the solid harmonic as {(a, b, c): coefficient} of x^a y^b z^c, (-1)^m times the phase-free one."""
    p = math.pi
    c1, c2, c20, c22 = math.sqrt(3 / (4 * p)), math.sqrt(15 / p) / 2, math.sqrt(5 / p) / 4, math.sqrt(15 / p) / 4
    c33, c32, c31 = math.sqrt(35 / (2 * p)) / 4, math.sqrt(105 / p) / 2, math.sqrt(21 / (2 * p)) / 4
    c30 = math.sqrt(7 / p) / 4
    X, Y, Z = (1, 0, 0), (0, 1, 0), (0, 0, 1)
    return [
        [{(0, 0, 0): 0.5 / math.sqrt(p)}],
        [{Y: -c1}, {Z: c1}, {X: -c1}],
        [{(1, 1, 0): c2}, {(0, 1, 1): -c2}, {(0, 0, 2): 2 * c20, (2, 0, 0): -c20, (0, 2, 0): -c20}, {(1, 0, 1): -c2},
         {(2, 0, 0): c22, (0, 2, 0): -c22}],
        [{(2, 1, 0): -3 * c33, (0, 3, 0): c33}, {(1, 1, 1): c32}, {(0, 1, 2): -4 * c31, (2, 1, 0): c31, (0, 3, 0): c31},
         {(0, 0, 3): 2 * c30, (2, 0, 1): -3 * c30, (0, 2, 1): -3 * c30},
         {(1, 0, 2): -4 * c31, (3, 0, 0): c31, (1, 2, 0): c31}, {(2, 0, 1): c32 / 2, (0, 2, 1): -c32 / 2},
         {(3, 0, 0): -c33, (1, 2, 0): 3 * c33}],
    ]


class _Basis:
    """phi and grad phi of the functions of a set of centres at a set of points."""

    def __init__(self, S, columns, dev):
        r = R_MIN * (R_CUT / R_MIN) ** (np.arange(N_LOG) / (N_LOG - 1))
        r[-1] = R_CUT
        s = np.clip((r - R_ON) / (R_CUT - R_ON), 0, 1)
        taper = 1 - s ** 3 * (10 - 15 * s + 6 * s * s)
        self.S, self.dev, self.h = S, dev, math.log(R_CUT / R_MIN) / (N_LOG - 1)
        up = lambda x: torch.tensor(x, dtype=torch.float64, device=dev)  # noqa: E731
        u = [[r ** (l + 1) * np.exp(-a * r * r) * taper for l, a in b] for b in S["basis"]]
        self.g0 = [[x[0] / R_MIN ** (l + 1) for x, (l, _) in zip(us, b)] for us, b in zip(u, S["basis"])]
        self.coef = [[up(_spline(x)) for x in us] for us in u]
        self.H = _harmonics()
        if columns is not None:
            self.eps, self.vcoef = columns[0], [up(_spline(x)) for x in columns[1]]
            self.rad0 = np.concatenate([[0], np.cumsum([len(b) for b in S["basis"]])])

    @staticmethod
    def _poly(P, mono):
        y = torch.zeros_like(P[0][0])
        for (a, b, c), w in mono.items():
            y = y + w * P[0][a] * P[1][b] * P[2][c]
        return y

    @staticmethod
    def _d(mono, c):
        """The derivative of a polynomial along axis c."""
        return {tuple(y - (z == c) for z, y in enumerate(e)): w * e[c] for e, w in mono.items() if e[c]}

    def __call__(self, pts, cxyz, csp, v=None):
        """phi [np, nb], grad [3, np, nb] (v given: psi = (v + eps_j - V_j) phi instead of the gradient)."""
        nf = self.S["nf"][csp]
        f0 = np.concatenate([[0], np.cumsum(nf)])
        out = torch.zeros((4 if v is None else 2, len(pts), int(f0[-1])), dtype=torch.float64, device=self.dev)
        for sp in np.unique(csp):
            at = np.nonzero(csp == sp)[0]
            d = pts[:, None, :] - torch.tensor(cxyz[at], device=self.dev)[None]
            d2 = d * d
            r = torch.sqrt((d2[..., 0] + d2[..., 1]) + d2[..., 2])
            ir = 1.0 / r
            t = torch.log(r / R_MIN) / self.h
            k = t.long().clamp(0, N_LOG - 2)
            s = t - k
            inside, below = r < R_CUT, r < R_MIN
            x = [[torch.ones_like(r)] for _ in range(3)]
            for c in range(3):
                for _ in range(3):
                    x[c].append(x[c][-1] * d[..., c])
            sh, dsh, unit = {}, {}, d * ir[..., None]
            for l in {l for l, _ in self.S["basis"][sp]}:  # harmonics and their gradients, [np, nc, 2l + 1]
                sh[l] = torch.stack([self._poly(x, mono) for mono in self.H[l]], -1)
                if v is None:
                    dsh[l] = [torch.stack([self._poly(x, self._d(mono, c)) for mono in self.H[l]], -1) for c in range(3)]
            fn = 0
            for q, (l, _) in enumerate(self.S["basis"][sp]):
                C = self.coef[sp][q][k]
                u = C[..., 0] + s * (C[..., 1] + s * (C[..., 2] + s * C[..., 3]))
                du = C[..., 1] + s * (2 * C[..., 2] + 3 * s * C[..., 3])
                irl = ir ** (l + 1)
                g = (torch.where(below, self.g0[sp][q], u * irl) * inside)[..., None]
                cols = torch.tensor(f0[at][:, None] + fn + np.arange(2 * l + 1), device=self.dev).reshape(-1)
                fn += 2 * l + 1
                phi = g * sh[l]
                out[0][:, cols] = phi.reshape(len(pts), -1)
                if v is not None:
                    W = self.vcoef[self.rad0[sp] + q]
                    V = W[k][..., 0] + s * (W[k][..., 1] + s * (W[k][..., 2] + s * W[k][..., 3]))
                    V = torch.where(below, W[0, 0], V)
                    psi = (v[:, None] + self.eps[self.rad0[sp] + q] - V)[..., None] * phi
                    out[1][:, cols] = psi.reshape(len(pts), -1)
                    continue
                gp = torch.where(below, 0.0, (du / self.h - (l + 1) * u) * ir * irl) * inside
                for c in range(3):
                    out[1 + c][:, cols] = ((gp * unit[..., c])[..., None] * sh[l] + g * dsh[l][c]).reshape(len(pts), -1)
        return out


def _chunks(case, S, ex, basis, dev, column_v=None):
    """(points slice, basis values, value index [nb, nb] into the pattern or -1) over the whole grid."""
    T, sh = _cells(S)
    nA = len(S["xyz"])
    k2, step = 4 * S["n_shell"] + 1, 4800 if S["lattice"] is None else 600
    table = np.full((nA, nA, k2, k2, k2), -1, np.int64)
    row = np.repeat(np.arange(nA), np.diff(ex["blk_ptr"]))
    sT = ex["blk_T"] + 2 * S["n_shell"]
    table[row, ex["blk_col"], sT[:, 0], sT[:, 1], sT[:, 2]] = ex["blk_off"][:-1]
    for a, z, atoms in _point_molecules(case, S, ex):
        C = (S["xyz"][atoms][None] + sh[:, None]).reshape(-1, 3)
        cA, cT = np.tile(atoms, len(sh)), np.repeat(np.arange(len(sh)), len(atoms))
        for s in range(a, z, step):
            e = min(z, s + step)
            P = torch.tensor(ex["xyz"][s:e], device=dev)
            gap = np.maximum(0.0, np.maximum(ex["xyz"][s:e].min(0) - C, C - ex["xyz"][s:e].max(0)))
            near = np.nonzero((gap * gap).sum(1) < R_CUT ** 2)[0]
            dist = torch.cdist(P, torch.tensor(C[near], device=dev), compute_mode="donot_use_mm_for_euclid_dist")
            near = near[(dist.min(0).values < R_CUT + 1e-6).cpu().numpy()]
            sp = S["species"][cA[near]]
            dT = T[cT[near]][None, :] - T[cT[near]][:, None] + 2 * S["n_shell"]
            off = table[cA[near][:, None], cA[near][None, :], dT[..., 0], dT[..., 1], dT[..., 2]]
            nf = S["nf"][sp]
            slot = torch.tensor(np.repeat(np.arange(len(near)), nf), device=dev)
            idx = torch.tensor(np.concatenate([np.arange(n) for n in nf]), device=dev)
            o = torch.tensor(off, device=dev)[slot][:, slot]
            val = torch.where(o < 0, -1, o + idx[:, None] * torch.tensor(nf, device=dev)[slot][None] + idx[None])
            yield slice(s, e), basis(P, C[near], sp, None if column_v is None else column_v[s:e]), val


def _spinor_G(ls):
    """[2 nf, ns] Clebsch-Gordan matrix of one species: rows 2t + s, columns per radial j = l - 1/2, l + 1/2 and m_j."""
    cols, t0, nf = [], 0, sum(2 * l + 1 for l in ls)
    for l in ls:
        for j2 in ([2 * l - 1] if l else []) + [2 * l + 1]:
            a = 1 if j2 > 2 * l else -1
            for m2 in range(-j2, j2 + 1, 2):
                c = np.zeros(2 * nf, complex)
                for s, cg in ((0, a * math.sqrt((2 * l + a * m2 + 1) / (4 * l + 2))),
                              (1, math.sqrt((2 * l - a * m2 + 1) / (4 * l + 2)))):
                    m = (m2 + (-1 if s == 0 else 1)) // 2
                    if abs(m) > l:
                        continue
                    r2 = math.sqrt(0.5)
                    for mr, w in ([(0, 1.0)] if m == 0 else [(m, r2), (-m, 1j * r2)] if m > 0 else
                                  [(-m, (-1) ** m * r2), (m, -1j * (-1) ** m * r2)]):
                        c[2 * (t0 + mr + l) + s] += cg * w
                cols.append(c)
        t0 += 2 * l + 1
    return np.array(cols).T


def _exact_spinor(st, dev):
    S, ex, nnz = st["S"], st["ex"], st["grid"].nnz
    pat = _pattern(S, ex, dev)
    cplx = dict(dtype=torch.complex128, device=dev)
    G = [torch.tensor(_spinor_G([l for l, _ in b]), **cplx) for b in S["basis"]]
    HL, HS = torch.empty(4 * nnz, **cplx), torch.empty(4 * nnz, **cplx)
    Pm = [torch.empty(nnz, dtype=torch.float64, device=dev) for _ in range(5)]
    W = [x for x in st["G"]]
    rs, cs = S["species"][pat["row"]], S["species"][pat["col"]]
    pauli = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], **cplx)
    one = torch.eye(2, **cplx)
    for a in range(len(G)):
        for b in range(len(G)):
            q = np.nonzero((rs == a) & (cs == b))[0]
            if not len(q):
                continue
            nA, nB = int(S["nf"][a]), int(S["nf"][b])
            o = torch.tensor(ex["blk_off"][q], device=dev)
            e = o[:, None] + torch.arange(nA * nB, device=dev)
            M = [x[e].reshape(-1, nA, nB).to(torch.complex128) for x in W]
            kron = lambda x, s: torch.einsum("qij,st->qisjt", x, s).reshape(-1, 2 * nA, 2 * nB)  # noqa: E731
            e4 = 4 * o[:, None] + torch.arange(4 * nA * nB, device=dev)
            HL[e4] = (G[a].conj().T @ kron(M[0], one) @ G[b]).reshape(len(q), -1)
            F = kron(M[1], one) + sum(1j * kron(M[2 + k], pauli[k]) for k in range(3))
            HS[e4] = (G[a].conj().T @ F @ G[b]).reshape(len(q), -1)
            D = (G[a].conj() @ st["D"][e4].reshape(-1, 2 * nA, 2 * nB) @ G[b].T).reshape(-1, nA, 2, nB, 2)
            tr = torch.einsum("qisjs->qij", D).real.reshape(len(q), -1)
            Pm[0][e] = Pm[1][e] = tr
            for k in range(3):
                Pm[2 + k][e] = (1j * torch.einsum("st,qisjt->qij", pauli[k], D)).real.reshape(len(q), -1)
    return [HL, HS] + Pm


def _exact_kfold(st, dev):
    S, ex = st["S"], st["ex"]
    pat = _pattern(S, ex, dev)
    pair = pat["row"] * len(S["xyz"]) + pat["col"]
    _, first, which = np.unique(pair, return_index=True, return_inverse=True)
    nf = S["nf"][S["species"]]
    size = nf[pat["row"][first]] * nf[pat["col"][first]]
    koff = torch.tensor(np.concatenate([[0], np.cumsum(size)]), device=dev)
    blk, off = pat["blk"], torch.tensor(ex["blk_off"], device=dev)
    to = koff[torch.tensor(which, device=dev)[blk]] + torch.arange(len(blk), device=dev) - off[blk]
    out = []
    for H in st["G"]:
        R = torch.zeros((len(st["k"]), int(koff[-1])), dtype=torch.complex128, device=dev)
        for i, k in enumerate(st["k"]):
            ph = torch.tensor(np.exp(2j * np.pi * (pat["T"] @ k)), device=dev)
            R[i].index_add_(0, to, H * ph[blk])
        out.append(R)
    return out


def exact(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    st = prepare(dict(case, tuned=False), seed)
    S, ex, g, op = st["S"], st["ex"], st["grid"], case["op"]
    if op == "spinor":
        return _exact_spinor(st, dev)
    if op == "kfold":
        return _exact_kfold(st, dev)
    if case["system"] == "slab" and work(case)["flops"] > 5e11:
        return None
    new = lambda n, k: [torch.zeros(n, dtype=torch.float64, device=dev) for _ in range(k)]  # noqa: E731
    w = torch.tensor(ex["w"], device=dev)
    basis = _Basis(S, st.get("columns"), dev)
    if op == "columns":
        (F,) = new(g.nnz, 1)
        for sl, B, idx in _chunks(case, S, ex, basis, dev, st["v"]):
            F.index_add_(0, idx[idx >= 0], ((B[0] * w[sl, None]).T @ B[1])[idx >= 0])
        return F
    M, (n, dv) = new(g.nnz, 5), new(g.n_points, 2)
    G = st.get("G") if op in ("autograd", "scf") else st.get("P")
    for sl, B, idx in _chunks(case, S, ex, basis, dev):
        ok = idx >= 0
        if "v" in st:
            D = B * (w[sl] * st["v"][sl])[None, :, None]
            c = lambda a, b: D[a].T @ B[b]  # noqa: E731
            for m, x in zip(M, (c(0, 0), c(1, 1) + c(2, 2) + c(3, 3), c(2, 3) - c(3, 2), c(3, 1) - c(1, 3),
                                c(1, 2) - c(2, 1))):
                m.index_add_(0, idx[ok], x[ok])
        if op == "integrate":
            continue
        dense = lambda x: torch.where(ok, x[idx.clamp_min(0)], 0.0)  # noqa: E731
        if op in ("scf", "density"):
            n[sl] = ((B[0] @ dense(st["P"][0])) * B[0]).sum(1)
        if op != "density":
            g5 = [dense(x) for x in G]
            y = ((B[0] @ g5[0]) * B[0]).sum(1)
            for k in range(3):
                a, b = (k + 1) % 3 + 1, (k + 2) % 3 + 1
                y += ((B[1 + k] @ g5[1]) * B[1 + k]).sum(1)
                y += ((B[a] @ g5[2 + k]) * B[b]).sum(1) - ((B[b] @ g5[2 + k]) * B[a]).sum(1)
            dv[sl] = y
    if op == "density":
        return n
    if op == "density_full":
        return dv
    dv *= w
    if op == "autograd":
        return M + [dv]
    SS = torch.empty(4 * g.nnz, dtype=torch.complex128, device=dev)
    pat = _pattern(S, ex, dev)
    off = torch.tensor(ex["blk_off"], device=dev)[pat["blk"]]
    nB = torch.tensor(S["nf"][S["species"]][pat["col"]], device=dev)[pat["blk"]]
    e = torch.arange(g.nnz, device=dev) - off
    r0 = 4 * off + 2 * (e // nB) * 2 * nB + 2 * (e % nB)
    SS[r0], SS[r0 + 1] = torch.complex(M[1], M[4]), torch.complex(M[3], M[2])
    SS[r0 + 2 * nB], SS[r0 + 2 * nB + 1] = torch.complex(-M[3], M[2]), torch.complex(M[1], -M[4])
    H = M + [torch.view_as_real(SS).reshape(-1)]
    return H if op == "integrate" else H + [n, dv]
