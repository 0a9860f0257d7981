"""Performance cases: the calls that a program built on this library spends its time in.

A case names one public entry point (``op``), a mesh, a polynomial degree and the options a user
sets.  Solves are whole calls (CG preconditioned by one V-cycle per iteration); the operator, the
smoother and the transfers between levels are what a program calls that runs its own Krylov method
or its own cycle on the handle's levels.

``exact`` restates the discretisation from the mesh cells in plain fp64 PyTorch (dense element
matrices, index maps, hanging nodes as interpolation from the parent's nodes).  It reads the
handle's numbering (cells, support points) and the Chebyshev intervals as data and uses none of its
arithmetic.
"""
import math
import random

import numpy as np
import torch

import paper_2203_12292_gb300 as g

ALL, OCTANT, SPHERE, SHELL = 0, 1, 2, 3  # refinement predicates
MOST = 1.9e7  # degrees of freedom of the largest case
DTYPES = {"f32": torch.float32, "f64": torch.float64}


def listed():
    return [
        # smallest call: the operator on 6 thousand DoFs, launches and latency
        dict(name="vmult_q2_small_f64", op="vmult", mesh="cube", depth=3, extra=1, at=0.5, k=2, dtype="f64"),
        # low order on the deepest octant hierarchy: more cells than DoFs, metadata instead of arithmetic
        dict(name="vmult_q1_octant_f32", op="vmult", mesh="octant", depth=7, extra=0, at=0.0, k=1, dtype="f32"),
        # the fine-level operator of the V-cycle and of CG on the headline mesh (18.7 M DoFs)
        dict(name="vmult_q4_octant_f32", op="vmult", mesh="cube", depth=5, extra=2, at=0.5, k=4, dtype="f32"),
        dict(name="vmult_q4_octant_f64", op="vmult", mesh="cube", depth=5, extra=2, at=0.5, k=4, dtype="f64"),
        # Chebyshev postsmoothing where many cells have hanging faces and edges
        dict(name="smooth_q4_sphere_f32", op="smooth", mesh="sphere", depth=7, extra=0, at=0.3, k=4, dtype="f32",
             zero_init=False),
        # residual down, correction up between the two finest levels
        dict(name="restrict_q4_octant_f32", op="restrict", mesh="cube", depth=5, extra=2, at=0.5, k=4, dtype="f32"),
        dict(name="prolong_q4_octant_f32", op="prolong", mesh="cube", depth=5, extra=2, at=0.5, k=4, dtype="f32"),
        # a solve small enough to live in the caches
        dict(name="solve_q2_small_f64", op="solve", mesh="cube", depth=3, extra=1, at=0.5, k=2, p=False, mg32=False,
             coef=0.0),
        # the headline solve, its all-fp64 variant, and the polynomial hierarchy 4 -> 2 -> 1 on the sphere mesh
        dict(name="solve_q4_octant_mixed", op="solve", mesh="cube", depth=5, extra=2, at=0.5, k=4, p=False, mg32=True,
             coef=0.0),
        dict(name="solve_q4_octant_f64", op="solve", mesh="cube", depth=5, extra=2, at=0.5, k=4, p=False, mg32=False,
             coef=0.0),
        dict(name="solve_q4_sphere_mixed", op="solve", mesh="sphere", depth=7, extra=0, at=0.3, k=4, p=True, mg32=True,
             coef=0.0),
        # independent problems of uneven degree and size in one graph launch
        dict(name="batch_16", op="batch", problems=16, mesh_seed=5),
    ]


def draw(rng):
    while True:
        op = rng.choice(["vmult", "vmult", "smooth", "restrict", "prolong", "solve", "solve", "batch"])
        if op == "batch":
            return dict(op="batch", problems=rng.randint(3, 20), mesh_seed=rng.randint(0, 1 << 20))
        c = dict(op=op, mesh=rng.choice(["cube", "cube", "octant", "sphere", "shell"]), k=rng.randint(1, 4))
        # refinement depth, extra local steps and the position of the refined region
        c["depth"] = {"cube": rng.randint(2, 5), "octant": rng.randint(4, 7), "sphere": rng.randint(4, 7),
                      "shell": rng.randint(5, 7)}[c["mesh"]]
        c["extra"] = rng.randint(0, 2) if c["mesh"] == "cube" else 0
        c["at"] = {"cube": rng.choice([0.2, 0.3, 0.5, 0.6]), "octant": 0.0,
                   "sphere": round(rng.uniform(0.15, 0.45), 3), "shell": 0.0}[c["mesh"]]
        if op == "solve":
            c.update(p=rng.random() < 0.3, mg32=rng.random() < 0.6, coef=rng.choice([0.0, 0.0, 10.0]))
        else:
            c["dtype"] = rng.choice(["f32", "f64"])
        if op == "smooth":
            c["zero_init"] = rng.random() < 0.5
        if 2000 <= _cells(c) * c["k"] ** 3 <= MOST:
            return c


# ---- meshes -------------------------------------------------------------------------------------

def _mesh(c):
    d = c["depth"]
    if c["mesh"] == "cube":  # uniform, then local steps in the corner box
        return g.Mesh(0.0, 1.0, [(ALL,)] * d + [(OCTANT, 0.0, c["at"])] * c["extra"])
    if c["mesh"] == "octant":
        return g.Mesh(-1.0, 1.0, [(OCTANT, -1.0, 0.0)] * d)
    if c["mesh"] == "sphere":
        return g.Mesh(0.0, 1.0, [(SPHERE, 0.5, c["at"])] * d)
    return g.Mesh(-1.0, 1.0, [(ALL,)] * (d - 3) + [(SHELL, 0.0, 0.55), (SHELL, 0.3, 0.43), (SHELL, 0.335, 0.39)])


def _cells(c):
    m = _mesh(c)
    return m.level_cells(m.num_levels - 1)


def _problems(c):
    """(degree, depth, local steps) of a batch: uneven, the total bounded by the largest case"""
    r = random.Random(c["mesh_seed"])
    out, total = [], 0.0
    while len(out) < c["problems"]:
        p = dict(mesh="cube", k=r.randint(1, 4), depth=r.randint(2, 5), extra=r.randint(0, 2), at=0.5)
        n = _cells(p) * p["k"] ** 3
        if n <= 4e6 and total + n <= MOST:
            out.append(p)
            total += n
    return out


# ---- inputs, calls ------------------------------------------------------------------------------

def _field(seed, i=0):
    """right-hand side f: eight random Fourier modes of unit variance"""
    r = np.random.RandomState((seed * 131 + i) % (1 << 31))
    kappa = r.randint(-4, 5, size=(8, 3))
    kappa[(kappa == 0).all(1)] = 1
    return kappa, r.uniform(0, 2 * math.pi, 8), 0.5


def _vec(mg, level, dtype, gen):
    return torch.randn(mg.n_free(level), dtype=DTYPES[dtype], device="cuda", generator=gen)


def prepare(c, seed):
    if c["op"] == "batch":
        ps = _problems(c)
        B = g.Batch([_mesh(p) for p in ps], [g.make_config(p["k"], mg_fp32=True) for p in ps])
        bs = [m.rhs(_field(seed, i)) for i, m in enumerate(B.problems)]
        return dict(case=c, batch=B, b=bs, x=[torch.zeros_like(b) for b in bs])
    mg = g.Multigrid(_mesh(c), c["k"], p_coarsening=bool(c.get("p")), mg_fp32=bool(c.get("mg32", True)))
    s = dict(case=c, mg=mg)
    L = mg.finest
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if c["op"] == "solve":
        if c["coef"]:  # cell-wise coefficient of that contrast, smooth in space
            ijk = torch.tensor(mg.level_cells(L), device="cuda").double()
            xc = (ijk[:, 1:] + 0.5) * 0.5 ** ijk[:, :1]
            s["nu"] = c["coef"] ** torch.sin(6.0 * xc).prod(1).contiguous()
            mg.set_coefficient(s["nu"])
        s["b"] = mg.rhs(_field(seed))
        s["x"] = torch.zeros_like(s["b"])
    elif c["op"] in ("restrict", "prolong"):
        s["fine"], s["coarse"] = _vec(mg, L, c["dtype"], gen), _vec(mg, L - 1, c["dtype"], gen)
    else:
        s["b"] = _vec(mg, L, c["dtype"], gen)
        s["x"] = _vec(mg, L, c["dtype"], gen)
    return s


def run(s):
    c = s["case"]
    if c["op"] == "batch":
        st = s["batch"].cg_solve(s["b"], s["x"], 1e-8, 100)
        return {"x": s["x"], "iterations": [int(t.iterations) for t in st]}
    mg = s["mg"]
    L = mg.finest
    if c["op"] == "solve":
        st = mg.cg_solve(s["b"], s["x"], 1e-8, 100)
        return {"x": s["x"], "iterations": int(st.iterations)}
    if c["op"] == "vmult":
        mg.vmult(L, s["b"], s["x"])
        return s["x"]
    if c["op"] == "smooth":
        mg.smooth(L, s["x"], s["b"], c["zero_init"])
        return s["x"]
    if c["op"] == "restrict":
        mg.restrict_add(L, s["fine"], s["coarse"])
        return s["coarse"]
    mg.prolongate_add(L, s["coarse"], s["fine"])
    return s["fine"]


# ---- what a pass cannot do without ----------------------------------------------------------------

ITERATIONS = 7  # CG iterations to 1e-8, about the same for every mesh and degree


def _flops_cell(k):
    """fast diagonalisation: six sweeps of (k+1)^2 even-odd 1D transforms and one scaling"""
    n = k + 1
    nh, ne = n // 2, (n + 1) // 2
    return 6 * n * n * (2 * nh + ne * (2 * ne - 1) + nh * (2 * nh - 1)) + n ** 3


def work(c):
    if c["op"] == "batch":
        ws = [work(dict(p, op="solve", mg32=True)) for p in _problems(c)]
        return {m: sum(w[m] for w in ws) for m in ("bytes", "flops")}
    cells, k = _cells(c), c["k"]
    n, op_flops = cells * k ** 3, cells * _flops_cell(k)
    if c["op"] == "solve":
        v = 4 if c["mg32"] else 8
        cycle = 8 / 7 * (6 * 2 * v + 5 * 2 * v + 3 * v)  # operators, smoother updates, transfers of every level
        cg = 16 + 8 * 8  # the fp64 operator; x, r, p read and written, q and z read
        return {"bytes": ITERATIONS * n * (cycle + cg), "flops": ITERATIONS * op_flops * (1 + 6 * 8 / 7)}
    v = 4 if c["dtype"] == "f32" else 8
    if c["op"] == "vmult":
        return {"bytes": 2 * v * n, "flops": op_flops}
    if c["op"] == "smooth":
        applications = 2 if c["zero_init"] else 3
        return {"bytes": (3 if c["zero_init"] else 4) * v * n, "flops": applications * op_flops}  # x, b, D^-1
    sweep = 2 * (2 * k + 1) * (k + 1) * ((2 * k + 1) ** 2 + (2 * k + 1) * (k + 1) + (k + 1) ** 2)
    both = n * (1 + 1 / 8)
    written = n if c["op"] == "prolong" else n / 8
    return {"bytes": v * (both + written), "flops": cells / 8 * sweep}


# ---- the same in plain fp64 PyTorch ---------------------------------------------------------------

def _nodes(k):
    return 0.5 + 0.5 * np.array({1: [-1, 1], 2: [-1, 0, 1], 3: [-1, -(1 / 5) ** 0.5, (1 / 5) ** 0.5, 1],
                                 4: [-1, -(3 / 7) ** 0.5, 0, (3 / 7) ** 0.5, 1]}[k], dtype=np.float64)


def _basis(k, t, derivative=False):
    """Lagrange basis of the Gauss-Lobatto points at the points t: (len(t), k + 1)"""
    x = _nodes(k)
    out = np.empty((len(t), k + 1))
    for a in range(k + 1):
        p = np.poly1d(np.delete(x, a), r=True)
        p = p / p(x[a])
        out[:, a] = (p.deriv() if derivative else p)(t)
    return out


def _kron(z, y, x):
    """rows and columns in x-fastest order"""
    return torch.tensor(np.kron(z, np.kron(y, x)), dtype=torch.float64, device="cuda")


def _reference(k):
    t, w = np.polynomial.legendre.leggauss(k + 1)
    t, w = 0.5 + 0.5 * t, 0.5 * w
    v, d = _basis(k, t), _basis(k, t, True)
    M, K = v.T @ (w[:, None] * v), d.T @ (w[:, None] * d)
    return _kron(M, M, K) + _kron(M, K, M) + _kron(K, M, M)


def _cell_key(l, i, j, k):
    return (l << 57) | (i << 38) | (j << 19) | k


def _find(sorted_keys, keys):
    at = torch.searchsorted(sorted_keys, keys).clamp(max=len(sorted_keys) - 1)
    return at, sorted_keys[at] == keys


class _Level:
    """one level: per cell the indices of its (parent's, where hanging) nodes and its constraint"""

    def __init__(self, mg, l, lo, hi):
        self.k = k = int(mg.info[l].degree)
        self.n, n1 = int(mg.n_free(l)), k + 1
        self.N = n1 ** 3
        cells = torch.tensor(mg.level_cells(l), device="cuda").long()
        self.lev, self.ijk = cells[:, 0], cells[:, 1:]
        self.h = (hi - lo) * 0.5 ** self.lev.double()
        self.keys, self.order = _cell_key(self.lev, *self.ijk.T).sort()
        pos, parent = self.ijk & 1, self.ijk >> 1
        out = 2 * pos - 1

        def coarse(move):  # is the parent's neighbour there a leaf?
            q = parent + out * torch.tensor(move, device="cuda")
            inside = ((q >= 0) & (q < (1 << (self.lev - 1).clamp(min=0))[:, None])).all(1) & (self.lev > 0)
            return inside & _find(self.keys, _cell_key(self.lev - 1, *q.clamp(min=0).T))[1]

        face = [coarse([int(d == e) for e in range(3)]) for d in range(3)]
        mask = pos[:, 0] + 2 * pos[:, 1] + 4 * pos[:, 2]
        for d in range(3):
            mask = mask + (8 << d) * face[d]
            edge = coarse([int(e != d) for e in range(3)])
            for e in range(3):
                edge = edge | (face[e] if e != d else False)
            mask = mask + (64 << d) * edge
        self.masks, cat = torch.where(mask < 8, 0, mask).unique(return_inverse=True)
        local = torch.arange(self.N, device="cuda")
        a = torch.stack([local % n1, local // n1 % n1, local // (n1 * n1)], 1)
        hang, self.C = [], []
        interp = [_basis(k, (p + _nodes(k)) / 2) for p in (0, 1)]
        for m in self.masks.tolist():
            p = [m >> d & 1 for d in range(3)]
            on = [a[:, d] == k * p[d] for d in range(3)]
            hn = torch.zeros(self.N, dtype=torch.bool, device="cuda")
            for d in range(3):
                if m >> (3 + d) & 1:
                    hn |= on[d]
                if m >> (6 + d) & 1:
                    hn |= on[(d + 1) % 3] & on[(d + 2) % 3]
            full = _kron(interp[p[2]], interp[p[1]], interp[p[0]])
            self.C.append(torch.where(hn[:, None], full, torch.eye(self.N, device="cuda", dtype=torch.float64)))
            hang.append(hn)
        self.hang = torch.stack(hang)[cat]
        self.groups = [(cat == i).nonzero()[:, 0] for i in range(len(self.masks))]
        xi = torch.tensor(_nodes(k), device="cuda")[a]
        unit = 0.5 ** self.lev.double()
        own = (self.ijk[:, None] + xi[None]) * unit[:, None, None]
        up = (parent[:, None] + xi[None]) * (2 * unit)[:, None, None]
        xyz = (torch.tensor(mg.dof_coords(l), device="cuda") - lo) / (hi - lo)
        dkeys, dorder = self._point(xyz).sort()
        self.idx = torch.full((len(cells), self.N), self.n, device="cuda")  # n: not a free DoF
        if self.n:
            at, ok = _find(dkeys, self._point(torch.where(self.hang[:, :, None], up, own)))
            self.idx = torch.where(ok, dorder[at], self.n)
        self.scale = self.h
        ref = _reference(k)
        self.A = [C.T @ ref @ C for C in self.C]

    @staticmethod
    def _point(x):
        q = (x * (1 << 20)).round().long()
        return (q[..., 0] << 42) | (q[..., 1] << 21) | q[..., 2]

    def gather(self, x):
        return torch.cat([x.double(), x.new_zeros(1, dtype=torch.float64)])[self.idx]

    def scatter(self, e):
        y = torch.zeros(self.n + 1, dtype=torch.float64, device="cuda")
        return y.index_add_(0, self.idx.reshape(-1), e.reshape(-1))[:-1]

    def per_cell(self, mats, e, transposed=False):
        out = torch.empty_like(e)
        for M, grp in zip(mats, self.groups):
            out[grp] = e[grp] @ (M if transposed else M.T)
        return out

    def apply(self, x):
        return self.scatter(self.per_cell(self.A, self.gather(x)) * self.scale[:, None])

    def diagonal(self):
        d = torch.stack([A.diagonal() for A in self.A])
        e = torch.empty(self.idx.shape, dtype=torch.float64, device="cuda")
        for i, grp in enumerate(self.groups):
            e[grp] = d[i]
        return self.scatter(e * self.scale[:, None])

    def owners(self):
        """for every DoF one (cell, node) that holds it unconstrained"""
        flat = torch.where(self.hang, self.n, self.idx).reshape(-1)
        own = torch.empty(self.n + 1, dtype=torch.long, device="cuda")
        own[flat] = torch.arange(len(flat), device="cuda")
        return own[:-1]


class _Transfer:
    def __init__(self, fine, coarse):
        self.f, self.c, self.own = fine, coarse, fine.owners()
        kf, kc = fine.k, coarse.k
        if kf != kc:  # same cells in the same order
            P = _basis(kc, _nodes(kf))
            self.cats = [(_kron(P, P, P), torch.arange(len(fine.lev), device="cuda"),
                          torch.arange(len(fine.lev), device="cuda"))]
            return
        at, same = _find(coarse.keys, _cell_key(fine.lev, *fine.ijk.T))
        up = _find(coarse.keys, _cell_key((fine.lev - 1).clamp(min=0), *(fine.ijk >> 1).T))[0]
        cell = coarse.order[torch.where(same, at, up)]
        child = ((fine.ijk & 1) * torch.tensor([1, 2, 4], device="cuda")).sum(1)
        interp = [_basis(kf, (p + _nodes(kf)) / 2) for p in (0, 1)]
        self.cats = [(torch.eye(fine.N, dtype=torch.float64, device="cuda"), same.nonzero()[:, 0])]
        self.cats += [(_kron(interp[q >> 2], interp[q >> 1 & 1], interp[q & 1]), (~same & (child == q)).nonzero()[:, 0])
                      for q in range(8)]
        self.cats = [(P, fi, cell[fi]) for P, fi in self.cats]

    def prolong(self, xc):
        u = self.c.per_cell(self.c.C, self.c.gather(xc))
        e = torch.empty((len(self.f.lev), self.f.N), dtype=torch.float64, device="cuda")
        for P, fi, ci in self.cats:
            e[fi] = u[ci] @ P.T
        return e.reshape(-1)[self.own]

    def restrict(self, r):
        e = torch.zeros(len(self.f.lev) * self.f.N, dtype=torch.float64, device="cuda")
        e[self.own] = r.double()
        e = e.reshape(-1, self.f.N)
        u = torch.zeros((len(self.c.lev), self.c.N), dtype=torch.float64, device="cuda")
        for P, fi, ci in self.cats:
            u.index_add_(0, ci, e[fi] @ P)
        return self.c.scatter(self.c.per_cell(self.c.C, u, True))


def _chebyshev(level, lam, dinv, x, b, zero_init):
    """degree 3, eigenvalues [lam / 20, lam] of D^-1 A (three-term recurrence)"""
    theta, delta = 0.525 * lam, 0.475 * lam
    rho, d = delta / theta, None
    for it in range(3):
        r = b if zero_init and it == 0 else b - level.apply(x)
        if it == 0:
            d = dinv * r / theta
        else:
            new = 1 / (2 * theta / delta - rho)
            d = new * rho * d + 2 * new / delta * dinv * r
            rho = new
        x = d if zero_init and it == 0 else x + d
    return x


class _Solver:
    def __init__(self, mg, lo, hi, nu=None):
        self.lev = [_Level(mg, l, lo, hi) for l in range(mg.num_levels)]
        self.tr = [None] + [_Transfer(self.lev[l], self.lev[l - 1]) for l in range(1, mg.num_levels)]
        self.lam = [mg.get_lambda(l) for l in range(mg.num_levels)]
        if nu is not None:  # a coarse cell takes its fine cell's value or the mean of its children
            for l in range(mg.num_levels - 1, -1, -1):
                self.lev[l].scale = self.lev[l].h * nu
                if l:
                    s = torch.zeros(len(self.lev[l - 1].lev), 2, dtype=torch.float64, device="cuda")
                    for _, fi, ci in self.tr[l].cats:
                        s.index_add_(0, ci, torch.stack([nu[fi], torch.ones_like(nu[fi])], 1))
                    nu = s[:, 0] / s[:, 1]
        self.dinv = [1 / L.diagonal() for L in self.lev]
        n0 = self.lev[0].n
        eye = torch.eye(n0, dtype=torch.float64, device="cuda")
        self.A0 = torch.stack([self.lev[0].apply(e) for e in eye]) if n0 else None

    def cycle(self, l, b):
        L = self.lev[l]
        if l == 0:
            return torch.linalg.solve(self.A0, b) if L.n else b
        x = _chebyshev(L, self.lam[l], self.dinv[l], None, b, True)
        if self.lev[l - 1].n:
            x = x + self.tr[l].prolong(self.cycle(l - 1, self.tr[l].restrict(b - L.apply(x))))
        return _chebyshev(L, self.lam[l], self.dinv[l], x, b, False)

    def solve(self, b, rtol, most):
        top, x, r = len(self.lev) - 1, torch.zeros_like(b), b
        z = p = self.cycle(top, r)
        rz = r @ z
        for it in range(1, most + 1):
            q = self.lev[top].apply(p)
            alpha = rz / (p @ q)
            x, r = x + alpha * p, r - alpha * q
            if r.norm() <= rtol * b.norm():
                break
            z = self.cycle(top, r)
            rz, old = r @ z, rz
            p = z + rz / old * p
        return x


def exact(c, seed):
    if c["op"] == "batch":
        s = prepare(c, seed)
        return {"x": [_Solver(m, 0.0, 1.0).solve(b, 1e-8, 100) for m, b in zip(s["batch"].problems, s["b"])],
                "iterations": None}
    s = prepare(c, seed)
    mg = s["mg"]
    lo, hi = (-1.0, 1.0) if c["mesh"] in ("octant", "shell") else (0.0, 1.0)
    L = mg.finest
    if c["op"] == "solve":
        return {"x": _Solver(mg, lo, hi, s.get("nu")).solve(s["b"], 1e-8, 100), "iterations": None}
    fine = _Level(mg, L, lo, hi)
    if c["op"] == "vmult":
        return fine.apply(s["b"])
    if c["op"] == "smooth":
        dinv = 1 / fine.diagonal()
        return _chebyshev(fine, mg.get_lambda(L), dinv, s["x"].double(), s["b"].double(), c["zero_init"])
    t = _Transfer(fine, _Level(mg, L - 1, lo, hi))
    if c["op"] == "restrict":
        return s["coarse"].double() + t.restrict(s["fine"])
    return s["fine"].double() + t.prolong(s["coarse"])
