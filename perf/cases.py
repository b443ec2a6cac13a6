"""Performance cases of the FOSB library: the calls its users make, over the sizes they make them at.

Every case runs through the public Python entry points.  Inputs are drawn from a seed: the
shape (a seeded ellipsoid or torus of a given resolution), the wave and, where a handle is
part of the input, the assembled and factored system a program would keep.

``exact`` restates the discrete problem (RWG elements, the 6-point triangle rule on
vertex-disjoint pairs, Sauter-Schwab with 5 points per coordinate on touching ones) in
64-bit torch, without the library.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2308_01457_gb300 as F
from paper_2308_01457_gb300.autograd import FosbRCS
from paper_2308_01457_gb300.batched import BatchedProblem
from paper_2308_01457_gb300.ct import FOSBProblem

DEV = "cuda:0"
C128 = torch.complex128


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # one small scatterer assembled on its own: launch and latency bound (the plain
        # k = 1 sphere of 320 triangles)
        dict(name="assemble-ff-N480", op="assemble", shape="ellipsoid", size=2, k=1.0, n_inc=1, arith="ff"),
        # a ragged surface and a fan of 16 incident directions: the ordinary assembly
        dict(name="assemble-ff-torus-N7503", op="assemble", shape="torus", nu=61, nv=41, k=5.0, n_inc=16, arith="ff"),
        # the finest level of the mixed sphere workload: the largest assembly
        dict(name="assemble-ff-N30720", op="assemble", shape="ellipsoid", size=5, k=4.0, n_inc=1, arith="ff"),
        # the plain method: everything in FP64, assembly to far field
        dict(name="direct-fp64-N1920", op="direct", shape="ellipsoid", size=3, k=1.0, n_inc=1, prec="fp64"),
        # a small system with 16 directions, factored once and solved: one scatterer of a batch
        dict(name="lu-mixed-N1920-rhs16", op="lu", shape="ellipsoid", size=3, k=3.0, n_rhs=16),
        # one large system and one wave: the nominal solve of a fine level
        dict(name="lu-mixed-N15360-rhs1", op="lu", shape="torus", nu=80, nv=64, k=4.0, n_rhs=1),
        # many right-hand sides on a factorisation in hand: the covariance solves
        dict(name="solve-mixed-N7503-rhs163", op="solve", shape="torus", nu=61, nv=41, k=4.0, n_rhs=163),
        # one off-diagonal block of the combination technique with its far-field moments
        dict(name="covariance-3-over-2", op="covariance", level1=4, level2=3, k=4.0, n_dir=181),
        # monostatic RCS at 8 angles with its vertex gradient: forward and backward
        dict(name="rcs-gradient-N7680", op="gradient", shape="ellipsoid", size=4, k=3.0, n_inc=8),
        # the dielectric sphere's 2N x 2N system
        dict(name="pmchwt-N7680", op="pmchwt", shape="ellipsoid", size=4, k=3.0, n_inc=1, eps_r=2.1),
        # scatterers of uneven size, 16 directions each, assembled and solved together
        dict(name="batched-24", op="batched", count=24, max_level=4, n_inc=16),
        # the whole first-order step: means and covariance over levels 0..3
        dict(name="step-ct-L3", op="step", levels=4, k=4.0, n_dir=181),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """A torus of lo .. hi quads (N = 3 quads), odd counts among them."""
    quads = rng.uniform(math.log(lo), math.log(hi))
    nv = max(4, round(math.sqrt(math.exp(quads) / rng.uniform(1.5, 3.0))))
    return dict(shape="torus", nu=max(5, int(math.exp(quads) / nv)), nv=nv)


def draw(rng):
    op = rng.choice(["assemble", "assemble", "direct", "lu", "lu", "solve", "covariance", "gradient", "pmchwt",
                     "batched", "step"])
    k = round(rng.uniform(1.0, 6.0), 3)
    if op == "assemble":
        return dict(op=op, k=k, **_grid(rng, 40, 5120), n_inc=rng.randint(1, 16),
                    arith=rng.choice(["ff", "ff", "ff", "fp64", "fp32"]) if rng.random() < 0.5 else "ff")
    if op == "direct":
        prec = rng.choice(["fp64", "fp32"])
        return dict(op=op, k=k, **_grid(rng, 40, 640 if prec == "fp64" else 2560),
                    n_inc=rng.randint(1, 8), prec=prec)
    if op == "lu":
        return dict(op=op, k=k, **_grid(rng, 40, 5120), n_rhs=rng.randint(1, 20))
    if op == "solve":
        return dict(op=op, k=k, **_grid(rng, 100, 2560), n_rhs=_loguniform(rng, 1, 642))
    if op == "covariance":
        l2 = rng.choice([1, 2, 3])
        return dict(op=op, level1=rng.randint(l2, 4), level2=l2, k=k, n_dir=rng.randint(9, 181))
    if op == "gradient":
        return dict(op=op, k=k, **_grid(rng, 40, 700), n_inc=rng.randint(1, 8))
    if op == "pmchwt":
        return dict(op=op, k=round(rng.uniform(1.0, 4.0), 3), **_grid(rng, 40, 2560),
                    n_inc=rng.randint(1, 4), eps_r=round(rng.uniform(1.5, 4.0), 3))
    if op == "batched":
        return dict(op=op, count=rng.randint(3, 24), max_level=rng.choice([3, 4]), n_inc=rng.randint(1, 16))
    return dict(op=op, levels=rng.randint(2, 4), k=k, n_dir=rng.randint(19, 181))


# --------------------------------------------------------------------------- shapes and waves
def _outward(v, t, out):
    n = np.cross(v[t[:, 1]] - v[t[:, 0]], v[t[:, 2]] - v[t[:, 0]])
    flip = (n * out[t].mean(axis=1)).sum(axis=1) < 0
    t = t.copy()
    t[flip, 1], t[flip, 2] = t[flip, 2].copy(), t[flip, 1].copy()
    return t.astype(np.int32)


def _sphere(level):
    g = (1 + math.sqrt(5)) / 2
    v = np.array([[s * a, u * b, 0] for a, b in ((1, g),) for s in (-1, 1) for u in (-1, 1)], np.float64)
    v = np.concatenate([v, v[:, [2, 0, 1]], v[:, [1, 2, 0]]])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    d = np.linalg.norm(v[:, None] - v[None], axis=2)
    near = (d > 0) & (d < 1.1)
    f = np.array([(i, j, m) for i in range(12) for j in range(i + 1, 12) for m in range(j + 1, 12)
                  if near[i, j] and near[j, m] and near[i, m]])
    for _ in range(level):
        e = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), axis=1)
        u, inv = np.unique(e, axis=0, return_inverse=True)
        mid = v[u].sum(axis=1)
        mid /= np.linalg.norm(mid, axis=1, keepdims=True)
        ab, bc, ca = (len(v) + inv.reshape(-1)).reshape(3, -1)
        v = np.concatenate([v, mid])
        a, b, c = f.T
        f = np.stack([np.stack([a, ab, ca], 1), np.stack([b, bc, ab], 1), np.stack([c, ca, bc], 1),
                      np.stack([ab, bc, ca], 1)], axis=1).reshape(-1, 3)
    return v, _outward(v, f, v)


def _ellipsoid(level, axes):
    v, t = _sphere(level)
    n = v / axes
    return SimpleNamespace(verts=v * axes, tris=t, vnormals=n / np.linalg.norm(n, axis=1, keepdims=True))


def _torus(nu, nv, r):
    """The nu x nv grid of quads, N = 3 nu nv edges."""
    iu, iv = (x.ravel() for x in np.meshgrid(np.arange(nu), np.arange(nv), indexing="ij"))
    a, b = 2 * np.pi * iu / nu, 2 * np.pi * iv / nv
    n = np.stack([np.cos(b) * np.cos(a), np.cos(b) * np.sin(a), np.sin(b)], axis=1)
    v = np.stack([np.cos(a), np.sin(a), 0 * a], axis=1) + r * n
    at = lambda i, j: (i % nu) * nv + j % nv  # noqa: E731
    p, q, s, w = at(iu, iv), at(iu + 1, iv), at(iu + 1, iv + 1), at(iu, iv + 1)
    t = np.stack([np.stack([p, q, s], 1), np.stack([p, s, w], 1)], axis=1).reshape(-1, 3)
    return SimpleNamespace(verts=v, tris=_outward(v, t, n), vnormals=n)


def _shape(case, g):
    if case["shape"] == "torus":
        return _torus(case["nu"], case["nv"], g.uniform(0.32, 0.38))
    return _ellipsoid(case["size"], g.uniform(0.9, 1.1, 3))


def _waves(g, n):
    """n unit directions and orthogonal unit polarisations."""
    d = g.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    p = np.cross(d, g.standard_normal((n, 3)))
    return d, p / np.linalg.norm(p, axis=1, keepdims=True)


def _hplane(n):
    t = np.linspace(0.0, np.pi, n)
    return np.stack([0 * t, np.sin(t), np.cos(t)], axis=1)


def _batch(case, g):
    """Semi-axes U[0.5, 1.5], k U[1, 6], sizes N = 480 .. 7680 as the batched workload has them."""
    rows = []
    for i in range(case["count"]):
        lvl = 2 + i % (case["max_level"] - 1) if i % 8 else 2
        rows.append((_ellipsoid(lvl, g.uniform(0.5, 1.5, 3)), float(g.uniform(1.0, 6.0))))
    return rows


def _case_rng(case, seed):
    return np.random.Generator(np.random.PCG64([seed, 230801457]))


def _problem(case, seed):
    """The shapes and waves of a case, as host arrays."""
    g = _case_rng(case, seed)
    op = case["op"]
    P = SimpleNamespace()
    if op == "covariance":
        ax = g.uniform(0.9, 1.1, 3)
        P.meshes = [_ellipsoid(case["level1"], ax), _ellipsoid(case["level2"], ax)]
        P.d, P.p = _waves(g, 1)
    elif op == "step":
        ax = g.uniform(0.9, 1.1, 3)
        P.meshes = [_ellipsoid(l + 1, ax) for l in range(case["levels"])]
        P.d, P.p = _waves(g, 1)
    elif op == "batched":
        P.batch = _batch(case, g)
        P.d, P.p = _waves(g, case["n_inc"])
    else:
        P.mesh = _shape(case, g)
        P.d, P.p = _waves(g, case.get("n_inc", case.get("n_rhs", 1)))
        if op == "solve":
            n = P.mesh.tris.shape[0] * 3 // 2
            P.B = g.standard_normal((n, case["n_rhs"])) + 1j * g.standard_normal((n, case["n_rhs"]))
        if op == "gradient":
            P.w = g.uniform(0.5, 1.5, case["n_inc"])
    return P


def _mesh(sm):
    return F.mesh_create(sm.verts, sm.tris, sm.vnormals)


def _assembled(sm, k, d, p):
    """What a program has before the factorisation: the mesh handle, Z and b."""
    m = _mesh(sm)
    n = m.n_edges
    Z = torch.empty((n, n), dtype=C128, device=DEV)
    b = torch.empty((n, d.shape[0]), dtype=C128, device=DEV)
    F.assemble_efie(m, k, Z, inc=F.incidence(d, p), b=b, arith=F.ASM_FF)
    return m, Z, b


# --------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    P = _problem(case, seed)
    s = SimpleNamespace(case=case)
    op = case["op"]
    if op in ("assemble", "direct"):
        s.mesh = _mesh(P.mesh)
        n = s.mesh.n_edges
        s.c64 = case.get("arith") == "fp32" or case.get("prec") == "fp32"
        dt = torch.complex64 if s.c64 else C128
        s.Z = torch.empty((n, n), dtype=dt, device=DEV)
        s.b = torch.empty((n, case["n_inc"]), dtype=dt, device=DEV)
        s.inc = F.incidence(P.d, P.p)
        if op == "direct":
            s.dirs = _hplane(181)
            s.X = torch.empty_like(s.b)
            s.F = torch.empty((543, case["n_inc"]), dtype=dt, device=DEV)
    elif op == "lu":
        s.mesh, s.Z, s.b = _assembled(P.mesh, case["k"], P.d, P.p)
        s.X = torch.empty_like(s.b)
    elif op == "solve":
        s.mesh, s.Z, _ = _assembled(P.mesh, case["k"], P.d[:1], P.p[:1])
        s.B = torch.from_numpy(P.B).to(DEV)
        s.X = torch.empty_like(s.B)
        s.lu = F.factor(s.Z, prec=F.MIXED)
    elif op == "covariance":
        s.sides = []
        for sm in P.meshes:
            m, Z, b = _assembled(sm, case["k"], P.d, P.p)
            lu = F.factor(Z, prec=F.MIXED)
            F.solve(lu, b)
            s.sides.append((m, lu, b))
        s.Sigma = torch.empty((s.sides[0][0].n_edges, s.sides[1][0].n_edges), dtype=C128, device=DEV)
        s.out = torch.empty((3 * case["n_dir"], 3 * case["n_dir"]), dtype=C128, device=DEV)
        s.dirs = _hplane(case["n_dir"])
    elif op == "gradient":
        s.verts = torch.from_numpy(P.mesh.verts).to(DEV)
        s.tris, s.d, s.p, s.w = P.mesh.tris, P.d, P.p, torch.from_numpy(P.w).to(DEV)
    elif op == "pmchwt":
        s.mesh = _mesh(P.mesh)
        n2 = 2 * s.mesh.n_edges
        s.Z = torch.empty((n2, n2), dtype=C128, device=DEV)
        s.b = torch.empty((n2, case["n_inc"]), dtype=C128, device=DEV)
        s.inc = F.incidence(P.d, P.p)
    elif op == "batched":
        s.prob = BatchedProblem([sm for sm, _ in P.batch], [k for _, k in P.batch], P.d, P.p).setup(DEV)
    elif op == "step":
        s.prob = FOSBProblem(P.meshes, case["k"], P.d[0], P.p[0], _hplane(case["n_dir"]), 0, case["levels"] - 1,
                             kernel=F.COV_GAUSS, sigma=0.005, ell=0.3, arith=F.ASM_FF).setup(DEV)
    return s


ARITH = {"ff": F.ASM_FF, "fp64": F.ASM_FP64, "fp32": F.ASM_FP32}


def run(s):
    case = s.case
    op, k = case["op"], case.get("k")
    if op == "assemble":
        F.assemble_efie(s.mesh, k, s.Z, inc=s.inc, b=s.b, arith=ARITH[case["arith"]])
        return {"Z": s.Z, "b": s.b}
    if op == "direct":
        prec = F.FP32 if s.c64 else F.FP64
        F.assemble_efie(s.mesh, k, s.Z, inc=s.inc, b=s.b, arith=F.ASM_FP32 if s.c64 else F.ASM_FP64, prec=prec)
        F.solve(F.factor(s.Z, prec=prec), s.b, s.X)
        F.farfield_moments(s.mesh, k, s.dirs, s.X, s.F, prec=prec)
        return {"Z": s.Z, "X": s.X, "F": s.F}
    if op == "lu":
        F.solve(F.factor(s.Z, prec=F.MIXED), s.b, s.X)
        return {"X": s.X}
    if op == "solve":
        F.solve(s.lu, s.B, s.X)
        return {"X": s.X}
    if op == "covariance":
        (m1, lu1, u1), (m2, lu2, u2) = s.sides
        F.covariance(m1, lu1, u1, m2, lu2, u2, k, s.Sigma, F.COV_GAUSS, 0.005, 0.3)
        F.farfield_moments(m1, k, s.dirs, s.Sigma, s.out, m2=m2, mirror=True, prec=F.MIXED)
        return {"Sigma": s.Sigma, "cov": s.out}
    if op == "gradient":
        v = s.verts.clone().requires_grad_(True)
        sigma = FosbRCS.apply(v, s.tris, k, s.d, s.p)
        sigma.backward(s.w)
        return {"sigma": sigma, "grad": v.grad}
    if op == "pmchwt":
        F.assemble_pmchwt(s.mesh, k, case["eps_r"], 1.0, s.Z, inc=s.inc, b=s.b, arith=F.ASM_FF)
        return {"Z": s.Z, "b": s.b}
    if op == "batched":
        return {"X": s.prob.run()}
    Fm, cov = s.prob.run()
    return {"F": Fm, "cov": cov, "rcs_db": s.prob.rcs_db, "var_f": s.prob.var_f}


# --------------------------------------------------------------------------- work
def _n_of(case):
    if case["shape"] == "torus":
        return 3 * case["nu"] * case["nv"]
    return 30 * 4 ** case["size"]


def _w_assemble(n, elem=16, n_inc=1, ops=27):
    """Z and b written once; `ops` FP64-class operations per point pair of the unordered
    triangle pairs (the kernel is symmetric), 36 point pairs each."""
    t = 2 * n / 3
    return elem * (n * n + n * n_inc), 36 * t * (t + 1) / 2 * ops


def _w_lu(n):
    return 16 * n * n, 8 * n ** 3 / 3


def _w_solve(n, r):
    return 16 * n * r * 2, 8 * n * n * r


def work(case):
    op = case["op"]
    if op == "assemble":
        parts = [_w_assemble(_n_of(case), 8 if case["arith"] == "fp32" else 16, case["n_inc"])]
    elif op == "direct":
        n, e = _n_of(case), 8 if case["prec"] == "fp32" else 16
        parts = [_w_assemble(n, e, case["n_inc"]), _w_lu(n), _w_solve(n, case["n_inc"]), (0, 8 * 543 * n * case["n_inc"])]
    elif op == "lu":
        n = _n_of(case)
        parts = [_w_lu(n), _w_solve(n, case["n_rhs"])]
    elif op == "solve":
        n = _n_of(case)
        parts = [_w_solve(n, case["n_rhs"]), (8 * n * n, 0)]
    elif op == "covariance":
        n1, n2 = 30 * 4 ** case["level1"], 30 * 4 ** case["level2"]
        r, f = n2 // 3 + 2, 3 * case["n_dir"]
        parts = [_w_solve(n1, r), _w_solve(n2, r), (16 * n1 * n2 + 8 * n1 * n1 + 8 * n2 * n2, 8 * n1 * n2 * r),
                 (16 * f * f, 8 * f * min(n1 * n2 + f * n1, n1 * n2 + f * n2))]
    elif op == "gradient":
        n = _n_of(case)
        parts = [_w_assemble(n), _w_lu(n), _w_solve(n, 2 * case["n_inc"]), (0, 3 * _w_assemble(n)[1])]
    elif op == "pmchwt":
        n = _n_of(case)
        b, f = _w_assemble(n, ops=51)
        parts = [(4 * b, 2 * f)]
    elif op == "batched":
        parts = []
        for i in range(case["count"]):
            n = 30 * 4 ** (2 + i % (case["max_level"] - 1) if i % 8 else 2)
            parts += [_w_assemble(n, n_inc=case["n_inc"]), _w_lu(n), _w_solve(n, case["n_inc"])]
    else:
        parts, L = [], case["levels"] - 1
        ns = [30 * 4 ** (l + 1) for l in range(L + 1)]
        for n in ns:
            parts += [_w_assemble(n), _w_lu(n), _w_solve(n, 1)]
        f = 3 * case["n_dir"]
        for tot in (L, L - 1):
            for a in range(tot + 1):
                if a >= tot - a >= 0:
                    n1, n2 = ns[a], ns[tot - a]
                    r = n2 // 3 + 2
                    parts += [_w_solve(n1, r), _w_solve(n2, r), (0, 8 * f * r * (n1 + n2 + f))]
    return {"bytes": float(sum(p[0] for p in parts)), "flops": float(sum(p[1] for p in parts))}


# --------------------------------------------------------------------------- 64-bit restatement
def _rule6():
    s, r = math.sqrt(10.0), math.sqrt(38.0 - 44.0 * math.sqrt(0.4))
    q = math.sqrt(213125.0 - 53320.0 * s)
    bary, w = [], []
    for a, wt in (((8 - s + r) / 18, (620 + q) / 3720), ((8 - s - r) / 18, (620 - q) / 3720)):
        for j in range(3):
            bary.append([1 - 2 * a if c == j else a for c in range(3)])
            w.append(wt)
    t = lambda x: torch.tensor(x, dtype=torch.float64, device=DEV)  # noqa: E731
    return t(bary), t(w)


class _Rwg:
    """RWG tables: edges in lexicographic vertex order, local edge i opposite local vertex i,
    sign + where the edge runs from its lower to its higher vertex.  Differentiable in verts."""

    def __init__(self, sm, verts=None):
        tr = np.asarray(sm.tris, np.int64)
        lo, hi = tr[:, [1, 2, 0]], tr[:, [2, 0, 1]]
        e = np.stack([np.minimum(lo, hi), np.maximum(lo, hi)], axis=2).reshape(-1, 2)
        self.edges, inv = np.unique(e, axis=0, return_inverse=True)
        self.tris_np = tr
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
        self.te = dev(inv.reshape(-1, 3))
        sign = dev(np.where(lo < hi, 1.0, -1.0))
        self.tris = dev(tr)
        self.nt, self.n, self.nv = tr.shape[0], self.edges.shape[0], sm.verts.shape[0]
        self.v = dev(np.asarray(sm.verts, np.float64)) if verts is None else verts
        self.vn = dev(np.asarray(sm.vnormals, np.float64))
        self.P = self.v[self.tris]  # T x 3 x 3
        self.E = torch.stack([self.P[:, 1] - self.P[:, 0], self.P[:, 2] - self.P[:, 1], self.P[:, 0] - self.P[:, 2]], 1)
        ends = self.v[dev(self.edges)]
        self.sl = sign * torch.linalg.norm(ends[:, 1] - ends[:, 0], dim=1)[self.te]
        nrm = torch.linalg.cross(self.E[:, 0], self.P[:, 2] - self.P[:, 0])
        self.area = 0.5 * torch.linalg.norm(nrm, dim=1)
        self.nrm = nrm / (2 * self.area)[:, None]
        self.bary, self.w = _rule6()
        self.qp = torch.einsum("qa,tac->tqc", self.bary, self.P)
        # f_i at the quadrature points, and its divergence
        self.f = (self.qp[:, :, None] - self.P[:, None]) * (self.sl / (2 * self.area[:, None]))[:, None, :, None]
        self.div = self.sl / self.area[:, None]

    def touching(self):
        """Unordered touching pairs t1 <= t2 with their Sauter-Schwab vertex orders, by kind."""
        tr = self.tris_np
        order = np.argsort(tr.ravel(), kind="stable")
        vert, tri = tr.ravel()[order], order // 3
        pairs = [np.stack([np.arange(self.nt)] * 2, 1)] * 3
        for d in range(1, int(np.bincount(vert).max())):
            same = vert[d:] == vert[:-d]
            a, b = tri[:-d][same], tri[d:][same]
            pairs.append(np.stack([np.minimum(a, b), np.maximum(a, b)], 1))
        pairs, shared = np.unique(np.concatenate(pairs), axis=0, return_counts=True)
        out = []
        for kind in (1, 2, 3):
            pr = pairs[shared == kind]
            A, B = tr[pr[:, 0]], tr[pr[:, 1]]
            eq = A[:, :, None] == B[:, None, :]
            rows = np.arange(len(pr))
            if kind == 3:
                p, q = A, A
            elif kind == 1:
                i, j = eq.any(2).argmax(1), eq.any(1).argmax(1)
                cyc = lambda X, s: np.stack([X[rows, (s + c) % 3] for c in range(3)], 1)  # noqa: E731
                p, q = cyc(A, i), cyc(B, j)
            else:
                i0 = ((~eq.any(2)).argmax(1) + 1) % 3  # the shared edge runs i0 -> i0 + 1
                c2 = B[rows, (~eq.any(1)).argmax(1)]
                p = np.stack([A[rows, (i0 + c) % 3] for c in range(3)], 1)
                q = np.stack([p[:, 0], p[:, 1], c2], 1)
            dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
            out.append((kind, dev(pr), dev(p), dev(q)))
        return out


def _ss_rule(kind, n=5):
    """(u1, u2, v1, v2, w) of the regularised 4-cube for x = P0 + u1 (P1 - P0) + u2 (P2 - P1)."""
    gx, gw = np.polynomial.legendre.leggauss(n)
    gx, gw = 0.5 * (gx + 1), 0.5 * gw
    xi, e1, e2, e3 = (a.ravel() for a in np.meshgrid(gx, gx, gx, gx, indexing="ij"))
    w = np.prod([a.ravel() for a in np.meshgrid(gw, gw, gw, gw, indexing="ij")], axis=0) * xi ** 3
    if kind == 3:
        w = w * e1 ** 2 * e2
        S = [(1, 1 - e1 + e1 * e2, 1 - e1 * e2 * e3, 1 - e1), (1 - e1 * e2 * e3, 1 - e1, 1, 1 - e1 + e1 * e2),
             (1, e1 * (1 - e2 + e2 * e3), 1 - e1 * e2, e1 * (1 - e2)),
             (1 - e1 * e2, e1 * (1 - e2), 1, e1 * (1 - e2 + e2 * e3)),
             (1 - e1 * e2 * e3, e1 * (1 - e2 * e3), 1, e1 * (1 - e2)),
             (1, e1 * (1 - e2), 1 - e1 * e2 * e3, e1 * (1 - e2 * e3))]
        ws = [w] * 6
    elif kind == 2:
        w = w * e1 ** 2
        S = [(1, e1 * e3, 1 - e1 * e2, e1 * (1 - e2)), (1, e1, 1 - e1 * e2 * e3, e1 * e2 * (1 - e3)),
             (1 - e1 * e2, e1 * (1 - e2), 1, e1 * e2 * e3), (1 - e1 * e2 * e3, e1 * e2 * (1 - e3), 1, e1),
             (1 - e1 * e2 * e3, e1 * (1 - e2 * e3), 1, e1 * e2)]
        ws = [w] + [w * e2] * 4
    else:
        w = w * e2
        S = [(1, e1, e2, e2 * e3), (e2, e2 * e3, 1, e1)]
        ws = [w] * 2
    u = [np.concatenate([xi * s[c] for s in S]) for c in range(4)]
    return [torch.tensor(a, dtype=torch.float64, device=DEV) for a in u + [np.concatenate(ws)]]


def _phase(r, k):
    """exp(ikr) as a complex tensor."""
    return torch.complex(torch.cos(k * r), torch.sin(k * r))


def _regular_blocks(m, k, t1, mfio=False):
    """The EFIO (and MFIO) 3 x 3 blocks of triangles t1 (a slice) against all triangles,
    C x T x 3 x 3, zero for touching pairs."""
    touch = (m.tris[t1][:, None, :, None] == m.tris[None, :, None, :]).flatten(2).any(2)
    diff = m.qp[t1][:, :, None, None] - m.qp[None, None]
    r = torch.sqrt((diff * diff).sum(-1) + touch[:, None, :, None])  # C x 6 x T x 6
    del diff
    G = _phase(r, k) / r
    wb = (m.bary * m.w[:, None]).to(C128)
    mom = lambda g: torch.einsum("cptq,pa,qb->ctab", g, wb, wb)  # noqa: E731
    mu = mom(G) * (~touch)[:, :, None, None]
    P1, P2 = m.P[t1], m.P
    D1 = P1[:, None] - P1[:, :, None]  # C x i x a: P_a - P_i
    D2 = P2[:, None] - P2[:, :, None]
    s = m.sl[t1][:, None, :, None] * m.sl[None, :, None, :] / (4 * math.pi)
    V = 0
    for c in range(3):
        W = torch.einsum("ctab,cia->ctib", mu, D1[..., c].to(C128))
        V = V + torch.einsum("ctib,tjb->ctij", W, D2[..., c].to(C128))
    Z = s * (-0.25j * k * V + (1j / k) * mu.sum((2, 3))[:, :, None, None])
    if not mfio:
        return Z, None
    nu = mom(G * torch.complex(-torch.ones_like(r), k * r) / (r * r)) * (~touch)[:, :, None, None]
    X = 0
    for c in range(3):  # (p_i - q_j) . ((Q_b - q_j) x (P_a - p_i))
        c1, c2 = (c + 1) % 3, (c + 2) % 3
        d = (P1[:, None, :, None, c] - P2[None, :, None, :, c]).to(C128)
        for x, y, sg in ((c1, c2, 1.0), (c2, c1, -1.0)):
            W = torch.einsum("ctab,cia->ctib", nu, D1[..., y].to(C128))
            X = X + sg * d * torch.einsum("ctib,tjb->ctij", W, D2[..., x].to(C128))
    return Z, -0.25 * s * X


def _touching_blocks(m, k, kind, pr, p, q, mfio=False):
    """The blocks of the touching pairs `pr` (C x 3 x 3), local edges in stored order."""
    u1, u2, v1, v2, w = _ss_rule(kind)
    P, Q = m.v[p], m.v[q]
    x = u1[:, None] * (P[:, 1] - P[:, 0])[:, None] + u2[:, None] * (P[:, 2] - P[:, 1])[:, None]  # C x S x 3, from P0 = Q0
    y = v1[:, None] * (Q[:, 1] - Q[:, 0])[:, None] + v2[:, None] * (Q[:, 2] - Q[:, 1])[:, None]
    d = x - y
    r = torch.sqrt((d * d).sum(2))
    G = w * _phase(r, k) / r
    a, b = pr[:, 0], pr[:, 1]
    pa = m.P[a] - P[:, :1]  # C x i x 3
    qb = m.P[b] - P[:, :1]
    xc, yc, pc, qc = (t.to(C128) for t in (x, y, pa, qb))
    I0 = G.sum(1)
    X, Y = torch.einsum("cs,csd->cd", G, xc), torch.einsum("cs,csd->cd", G, yc)
    XY = torch.einsum("cs,cs->c", G, (x * y).sum(2).to(C128))
    V = (XY[:, None, None] - torch.einsum("cd,cjd->cj", X, qc)[:, None] - torch.einsum("cd,cid->ci", Y, pc)[:, :, None]
         + torch.einsum("cid,cjd->cij", pc, qc) * I0[:, None, None])
    s = m.sl[a][:, :, None] * m.sl[b][:, None] / (4 * math.pi)
    Z = s * (-1j * k * V + (4j / k) * I0[:, None, None])
    if not mfio:
        return Z, None
    if kind == 3:
        return Z, torch.zeros_like(Z)
    g = G * torch.complex(-torch.ones_like(r), k * r) / (r * r)
    K = torch.zeros_like(Z)
    for i in range(3):
        f = x - pa[:, i:i + 1]
        for j in range(3):
            K[:, i, j] = -(g * (d * torch.linalg.cross(y - qb[:, j:j + 1], f)).sum(2)).sum(1)
    return Z, s * K


def _chunks(n, per, budget):
    c = max(1, int(budget // per))
    return [slice(i, min(n, i + c)) for i in range(0, n, c)]


def _matrix(m, k, mfio=False):
    """Z (and the MFIO matrix) as dense N x N complex128."""
    out = [torch.zeros((m.n, m.n), dtype=C128, device=DEV) for _ in range(2 if mfio else 1)]
    for t1 in _chunks(m.nt, m.nt, 1 << 20):
        for M, blk in zip(out, _regular_blocks(m, k, t1, mfio)):
            for i in range(3):
                rows = torch.zeros((blk.shape[0], m.n), dtype=C128, device=DEV)
                for j in range(3):
                    rows.index_add_(1, m.te[:, j], blk[:, :, i, j])
                M.index_add_(0, m.te[t1, i], rows)
    for kind, pr, p, q in m.touching():
        for c in _chunks(pr.shape[0], 4000, 3e7):
            a, b = pr[c, 0], pr[c, 1]
            at = m.te[a][:, :, None] * m.n + m.te[b][:, None]
            mirrored = m.te[b][:, None] * m.n + m.te[a][:, :, None]
            for M, blk in zip(out, _touching_blocks(m, k, kind, pr[c], p[c], q[c], mfio)):
                M.view(-1).index_add_(0, at.reshape(-1), blk.reshape(-1))
                if kind < 3:
                    M.view(-1).index_add_(0, mirrored.reshape(-1), blk.reshape(-1))
    return out if mfio else out[0]


def _to(a, dtype=torch.float64):
    return torch.as_tensor(a, dtype=dtype, device=DEV)


def _plane(m, k, d, p):
    """b[m, s] = -int p_s exp(ik d_s.x) . f_m."""
    d, p = _to(d), _to(p)
    ph = _phase(torch.einsum("tqc,sc->tqs", m.qp, d), k) * (m.w[:, None] * m.area[:, None, None])
    v = -torch.einsum("tqs,tqic,sc->tis", ph, m.f.to(C128), p.to(C128))
    return torch.zeros((m.n, d.shape[0]), dtype=C128, device=DEV).index_add(0, m.te.reshape(-1), v.reshape(-1, d.shape[0]))


def _far(m, k, dirs):
    """A (3 n_dir x N)."""
    u = _to(dirs)
    out = torch.zeros((m.n, 3 * u.shape[0]), dtype=C128, device=DEV)
    for c in _chunks(m.nt, 6 * 3 * u.shape[0], 2e7):
        ph = _phase(-torch.einsum("tqc,sc->tqs", m.qp[c], u), k) * (m.w[:, None] * m.area[c][:, None, None])
        J = torch.einsum("tqs,tqic->tisc", ph, m.f[c].to(C128))
        J = -1j * k * (J - torch.einsum("tisc,sc->tis", J, u.to(C128))[..., None] * u.to(C128))
        out = out.index_add(0, m.te[c].reshape(-1), J.reshape(-1, 3 * u.shape[0]))
    return out.T


def _shape_rhs(m, k, u):
    """B (N x V) of the shape derivative at the nominal current u."""
    ul = u[m.te]  # T x 3
    nu = torch.einsum("tac,tc->ta", m.vn[m.tris], m.nrm)
    ff = torch.einsum("tqic,tqjc->tqij", m.f, m.f)
    c = k * ff - (m.div[:, :, None] * m.div[:, None] / k)[:, None]
    w = m.w[:, None] * m.area[:, None, None] * m.bary * nu[:, None]  # T x 6 x a
    v = -1j * torch.einsum("tqa,tqij,tj->tia", w.to(C128), c.to(C128), ul)
    B = torch.zeros(m.n * m.nv, dtype=C128, device=DEV)
    B.index_add_(0, (m.te[:, :, None] * m.nv + m.tris[:, None]).reshape(-1), v.reshape(-1))
    return B.view(m.n, m.nv)


def _gauss(x, y, sigma, ell):
    return (sigma ** 2 * torch.exp(-((x[:, None] - y[None]) ** 2).sum(2) / (2 * ell ** 2))).to(C128)


class _Level:
    def __init__(self, sm, k, d, p):
        self.m, self.k = _Rwg(sm), k
        self.Z = _matrix(self.m, k)
        self.u = torch.linalg.solve(self.Z, _plane(self.m, k, d, p))
        self.Y = torch.linalg.solve(self.Z, _shape_rhs(self.m, k, self.u[:, 0]))  # Z^-1 B


def exact(case, seed):
    P = _problem(case, seed)
    op, k = case["op"], case.get("k")
    if op in ("assemble", "direct"):
        m = _Rwg(P.mesh)
        Z, b = _matrix(m, k), _plane(m, k, P.d, P.p)
        if op == "assemble":
            return {"Z": Z, "b": b}
        X = torch.linalg.solve(Z, b)
        return {"Z": Z, "X": X, "F": _far(m, k, _hplane(181)) @ X}
    if op in ("lu", "solve"):
        m = _Rwg(P.mesh)
        return {"X": torch.linalg.solve(_matrix(m, k), _plane(m, k, P.d, P.p) if op == "lu" else _to(P.B, C128))}
    if op == "covariance":
        a, c = (_Level(sm, k, P.d, P.p) for sm in P.meshes)
        K = _gauss(a.m.v, c.m.v, 0.005, 0.3)
        A1, A2 = (_far(x.m, k, _hplane(case["n_dir"])) for x in (a, c))
        M = (A1 @ a.Y) @ K @ (A2 @ c.Y).mH
        return {"Sigma": (a.Y @ K) @ c.Y.mH, "cov": M + M.mH}
    if op == "gradient":
        return _exact_gradient(P, k)
    if op == "pmchwt":
        m = _Rwg(P.mesh)
        k1, eta = k * math.sqrt(case["eps_r"]), math.sqrt(1 / case["eps_r"])
        T0, K0 = _matrix(m, k, mfio=True)
        T1, K1 = _matrix(m, k1, mfio=True)
        K0 += K1
        Z = torch.cat([torch.cat([K0, T0 + eta * T1], 1), torch.cat([-T0 - T1 / eta, K0], 1)], 0)
        return {"Z": Z, "b": torch.cat([_plane(m, k, P.d, P.p), _plane(m, k, P.d, np.cross(P.d, P.p))], 0)}
    if op == "batched":
        X = []
        for sm, kk in P.batch:
            m = _Rwg(sm)
            X.append(torch.linalg.solve(_matrix(m, kk), _plane(m, kk, P.d, P.p)))
        return {"X": X}
    lv = [_Level(sm, k, P.d, P.p) for sm in P.meshes]
    L, dirs = len(lv) - 1, _hplane(case["n_dir"])
    A = [_far(x.m, k, dirs) for x in lv]
    S = [a @ x.Y for a, x in zip(A, lv)]
    cov = 0
    for tot, sign in ((L, 1.0), (L - 1, -1.0)):
        for i in range(tot + 1):
            cov = cov + sign * S[i] @ _gauss(lv[i].m.v, lv[tot - i].m.v, 0.005, 0.3) @ S[tot - i].mH
    Fm = A[L] @ lv[L].u
    power = (Fm.abs() ** 2).view(-1, 3).sum(1) / (4 * math.pi)
    return {"F": Fm, "cov": cov, "rcs_db": 10 * torch.log10(power), "var_f": cov.diagonal().real}


def _exact_gradient(P, k):
    """sigma_i = |A(-d_i) u_i|^2 / (4 pi) and the gradient of sum w_i sigma_i in the vertices: the
    adjoint identity d sigma = Re[c.dA u + lambda.(db - dZ u)], c = w conj(F)/(2 pi),
    Z lambda = A^T c, with dA, db and dZ by reverse-mode differentiation of the forms above."""
    m = _Rwg(P.mesh)
    Z = _matrix(m, k)
    n = P.d.shape[0]
    U = torch.linalg.solve(Z, _plane(m, k, P.d, P.p))
    A = _far(m, k, -P.d).reshape(n, 3, m.n)
    Fi = torch.einsum("icn,ni->ic", A, U)
    c = _to(P.w)[:, None] * Fi.conj() / (2 * math.pi)
    lam = torch.linalg.solve(Z, torch.einsum("icn,ic->ni", A, c))
    del Z, A
    base = _to(P.mesh.verts)
    grad = torch.zeros_like(base)

    def add(part):
        v = base.clone().requires_grad_(True)
        grad.add_(torch.autograd.grad(part(_Rwg(P.mesh, v)), v)[0])

    add(lambda q: (torch.einsum("icn,ni,ic->", _far(q, k, -P.d).reshape(n, 3, -1), U, c)
                   + (lam * _plane(q, k, P.d, P.p)).sum()).real)
    for t1 in _chunks(m.nt, m.nt, 1 << 18):
        W = torch.einsum("cis,tjs->ctij", lam[m.te[t1]], U[m.te])
        add(lambda q: -(W * _regular_blocks(q, k, t1)[0]).sum().real)
    for kind, pr, p, q_ in m.touching():
        for s in _chunks(pr.shape[0], 4000, 8e6):
            a, b = m.te[pr[s, 0]], m.te[pr[s, 1]]
            W = torch.einsum("cis,cjs->cij", lam[a], U[b])
            if kind < 3:
                W = W + torch.einsum("cjs,cis->cij", lam[b], U[a])
            add(lambda q: -(W * _touching_blocks(q, k, kind, pr[s], p[s], q_[s])[0]).sum().real)
    return {"sigma": (Fi.abs() ** 2).sum(1) / (4 * math.pi), "grad": grad}
