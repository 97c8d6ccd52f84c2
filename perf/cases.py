"""The workloads whose speed and accuracy this library is held to, each run through the public API.

``listed()`` names them, ``draw(rng)`` gives others of the same ranges, ``prepare`` builds what a user's
program holds before the call (meshes, operators, input vectors, output buffers), ``run`` is one pass,
``work`` the bytes and operations a pass cannot do without, and ``exact`` the result in plain FP64 torch,
which shares no code with the library.
"""
import math

import numpy as np
import torch

import paper_2607_03413_gb300 as cw

KINDS = {"laplace": cw.CW_LAPLACE, "mass": cw.CW_MASS, "laplace+mass": cw.CW_LAPLACE_MASS}
GEOMS = {"affine": cw.CW_GEOM_AFFINE, "metric": cw.CW_GEOM_METRIC, "recompute": cw.CW_GEOM_RECOMPUTE}
PRECS = {"f64": cw.CW_PREC_F64, "f64_native": cw.CW_PREC_F64_NATIVE, "f32": cw.CW_PREC_F32,
         "f32_bf16g": cw.CW_PREC_F32_BF16G, "bf16": cw.CW_PREC_BF16}
MODES = {"f64": cw.CW_CG_F64, "ir_f32": cw.CW_CG_IR_F32, "ir_bf16": cw.CW_CG_IR_BF16}
VEC_BYTES = {"f64": 8, "f64_native": 8, "f32": 4, "f32_bf16g": 4, "bf16": 2}
MET_BYTES = {"f64": 8, "f64_native": 8, "f32": 4, "f32_bf16g": 2, "bf16": 2}
AMP = 0.1  # vertex displacement in units of the cell size, as in the benchmark's curved meshes
MOST = 33_000_000  # cell-wise values of the largest single apply (the benchmark step has 32.8 million)


# ------------------------------------------------------------------------------ the cases ----
def listed():
    return [
        # a small uniform Cartesian problem: every launch counts
        apply_case("affine_q2_8_assembled", 2, (8, 8, 8), "laplace", "affine", "f64", True),
        # the benchmark's step: one operator evaluation of a 64^3 curved mesh, coupled across cells
        apply_case("f64_q4_64_assembled", 4, (64, 64, 64), "laplace+mass", "metric", "f64", True),
        # low and high order FP64 operators on meshes of odd sizes, as a residual evaluation uses them
        apply_case("f64_q2_local", 2, (101, 97, 95), "laplace", "metric", "f64", False),
        apply_case("f64_q7_local", 7, (37, 35, 33), "laplace", "metric", "f64", False),
        # the operator of an FP32 Krylov level
        apply_case("f32_q3_assembled", 3, (79, 77, 75), "laplace", "metric", "f32", True),
        # the half-storage operator of a preconditioner
        apply_case("bf16_q5_local", 5, (53, 51, 49), "laplace+mass", "metric", "bf16", False),
        # a mesh whose metric is recomputed because it would not be worth its memory
        apply_case("f64_q4_recompute", 4, (41, 40, 39), "laplace+mass", "recompute", "f64", True),
        # many right-hand sides and many uneven problems in one launch (a serving batch)
        {"name": "batch_f32", "what": "batch", "prec": "f32", "nrhs": 8, "n_rhs_cells": 24, "problems": 12, "lo": 8,
         "hi": 28},
        # Poisson solves to 1e-10: plain FP64, and FP32 with FP64 refinement
        {"name": "cg_f64_q3_32", "what": "cg", "p": 3, "nx": 32, "ny": 32, "nz": 32, "mode": "f64"},
        {"name": "cg_ir_f32_q3_48", "what": "cg", "p": 3, "nx": 48, "ny": 48, "nz": 48, "mode": "ir_f32"},
        # one multigrid cycle, the preconditioner of the multigrid solves
        {"name": "vcycle_f32_q3_64", "what": "vcycle", "p": 3, "n0": 4, "levels": 5, "prec": "f32"},
        # an unstructured block mesh: seven blocks glued in seeded orientations
        {"name": "mblock_f64_q3_16", "what": "mblock", "p": 3, "n": 16, "prec": "f64"},
    ]


def apply_case(name, p, dims, kind, geom, prec, assemble):
    c = {"what": "apply", "p": p, "nx": dims[0], "ny": dims[1], "nz": dims[2], "kind": kind, "geom": geom,
         "prec": prec, "assemble": assemble}
    return dict(c, name=name) if name else c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["apply"] * 8 + ["batch", "cg", "cg", "vcycle", "mblock"])
    if what == "apply":
        p = rng.randint(1, 7)
        geom = rng.choice(["metric"] * 4 + ["recompute", "affine"])
        prec = rng.choice(["f64"] * 4 + ["f64_native", "f32", "f32", "f32_bf16g", "bf16"])
        most = MOST / 4 if geom == "recompute" or prec == "f64_native" else MOST  # dearer per value
        side = (math.exp(rng.uniform(math.log(1e4), math.log(most * 0.9))) / (p + 1) ** 3) ** (1 / 3)
        dims = [max(2, int(side * rng.uniform(0.9, 1.02))) for _ in range(3)]
        return apply_case(None, p, dims, rng.choice(["laplace", "laplace", "laplace+mass", "mass"]), geom, prec,
                          rng.random() < 0.5)
    if what == "batch":
        return {"what": "batch", "prec": rng.choice(["f32", "f64"]), "nrhs": rng.randint(1, 8),
                "n_rhs_cells": rng.randint(6, 20), "problems": rng.randint(2, 12), "lo": 4, "hi": rng.randint(8, 24)}
    if what == "cg":
        p = rng.randint(1, 5)
        n = [_log_int(rng, 6, 96 / p) for _ in range(1)][0]
        return {"what": "cg", "p": p, "nx": n, "ny": max(2, n - rng.randint(0, 2)), "nz": max(2, n - rng.randint(0, 3)),
                "mode": rng.choice(["f64", "ir_f32", "ir_f32", "ir_bf16"])}
    if what == "vcycle":
        p = rng.randint(1, 4)
        return {"what": "vcycle", "p": p, "n0": rng.randint(2, 4), "levels": rng.randint(2, 4 if p > 1 else 5),
                "prec": rng.choice(["f32", "f64"])}
    return {"what": "mblock", "p": rng.randint(1, 4), "n": rng.randint(3, 16), "prec": rng.choice(["f64", "f32"])}


# ------------------------------------------------------------------------- meshes and inputs ----
def box_verts(nx, ny, nz, perturb, freq=(1, 1, 1), direction=(1.0, 1.0, 1.0)):
    """Vertices of the unit cube's nx*ny*nz cells, displaced smoothly inside it."""
    Z, Y, X = np.meshgrid(np.arange(nz + 1) / nz, np.arange(ny + 1) / ny, np.arange(nx + 1) / nx, indexing="ij")
    v = np.stack([X, Y, Z], axis=-1)
    if perturb:
        d = np.asarray(direction) / np.linalg.norm(direction)
        tp = 2 * np.pi
        s = np.sin(tp * freq[0] * X) * np.sin(tp * freq[1] * Y) * np.sin(tp * freq[2] * Z)
        w = v + perturb / max(nx, ny, nz) * s[..., None] * d
        w[:, :, (0, -1), 0], w[:, (0, -1), :, 1], w[(0, -1), :, :, 2] = (v[:, :, (0, -1), 0], v[:, (0, -1), :, 1],
                                                                         v[(0, -1), :, :, 2])
        v = w
    return np.ascontiguousarray(v)


def refine_verts(v):
    for ax in (2, 1, 0):
        lo, hi = np.delete(v, -1, ax), np.delete(v, 0, ax)
        w = np.empty([2 * n - 1 if a == ax else n for a, n in enumerate(v.shape)])
        at = [slice(None)] * 4
        at[ax] = slice(0, None, 2)
        w[tuple(at)] = v
        at[ax] = slice(1, None, 2)
        w[tuple(at)] = 0.5 * (lo + hi)
        v = w
    return np.ascontiguousarray(v)


def cube_in_cube_verts(n, seed):
    """Seven blocks of n^3 cells filling [-1, 1]^3 (an inner cube and six frustum shells around it), the
    local axes of each block turned by a seeded proper rotation."""
    s, t = np.linspace(-1, 1, n + 1), np.linspace(0, 1, n + 1)
    K, J, I = np.meshgrid(s, s, s, indexing="ij")
    blocks = [0.5 * np.stack([I, J, K], axis=-1)]
    for axis in range(3):
        for sign in (1.0, -1.0):
            T, V, U = np.meshgrid(t, s, s, indexing="ij")
            if sign < 0:
                U, V = V, U
            F = np.zeros(T.shape + (3,))
            F[..., axis], F[..., (axis + 1) % 3], F[..., (axis + 2) % 3] = sign, U, V
            blocks.append(((1 - T) * 0.5 + T)[..., None] * F)
    rng = np.random.default_rng(seed)
    out = []
    for v in blocks:
        for _ in range(int(rng.integers(3))):  # cyclic permutations of the axes
            v = np.transpose(v, (1, 2, 0, 3))
        if rng.integers(2):  # a half turn
            v = v[::-1, ::-1]
        out.append(np.ascontiguousarray(v))
    return out


def rand_global(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * 2 - 1


def mesh_of(v):
    return cw.Mesh(v.shape[2] - 1, v.shape[1] - 1, v.shape[0] - 1, v)


def batch_problems(case):
    """The batch's (degree, vertices, right-hand sides): one mesh with many, then single uneven problems."""
    n = case["n_rhs_cells"]
    out = [(5, box_verts(n, n, n, AMP), case["nrhs"])]
    rng = np.random.default_rng(7)
    for i in range(case["problems"]):
        n = int(rng.integers(case["lo"], case["hi"] + 1))
        out.append(((2, 3, 5, 7)[i % 4], box_verts(n, n, n, AMP, rng.integers(1, 4, 3), rng.normal(size=3)), 1))
    return out


def rhs_weights(seed):
    return np.random.default_rng(seed).uniform(0.5, 1.5, 2)


def coarse_verts(case):
    return box_verts(case["n0"], case["n0"], case["n0"], AMP)


# ---------------------------------------------------------------------------- prepare and run ----
def prepare(case, seed):
    s = {"what": case["what"]}
    if case["what"] == "apply":
        s["assemble"] = case["assemble"]
        s["mesh"] = mesh_of(box_verts(case["nx"], case["ny"], case["nz"], 0.0 if case["geom"] == "affine" else AMP))
        s["op"] = cw.Operator(s["mesh"], case["p"], KINDS[case["kind"]], GEOMS[case["geom"]], PRECS[case["prec"]])
        s["x"], s["y"] = s["op"].gather(rand_global(s["op"].NG, seed)), s["op"].empty()
    elif case["what"] == "batch":
        probs = batch_problems(case)
        s["mesh"] = [mesh_of(v) for _, v, _ in probs]
        s["ops"] = [cw.Operator(m, p, prec=PRECS[case["prec"]]) for m, (p, _, _) in zip(s["mesh"], probs)]
        nrhs = [r for _, _, r in probs]
        xs = []
        for i, (o, r) in enumerate(zip(s["ops"], nrhs)):
            xs.append(torch.cat([o.gather(rand_global(o.NG, seed * 1000 + 20 * i + k)) for k in range(r)]))
        s["batch"] = cw.Batch(s["ops"], nrhs, xs, [torch.empty_like(x) for x in xs])
    elif case["what"] == "cg":
        s["mesh"] = mesh_of(box_verts(case["nx"], case["ny"], case["nz"], AMP))
        s["op"] = cw.Operator(s["mesh"], case["p"], bc=cw.CW_BC_DIRICHLET0)
        w = rhs_weights(seed)
        s["b"] = w[0] * s["op"].load_vector(0) + w[1] * s["op"].load_vector(1)
        s["u"], s["mode"] = torch.empty_like(s["b"]), MODES[case["mode"]]
    elif case["what"] == "vcycle":
        v = [coarse_verts(case)]
        while len(v) < case["levels"]:
            v.append(refine_verts(v[-1]))
        s["mesh"] = [mesh_of(x) for x in v]
        s["ops"] = [cw.Operator(m, case["p"], prec=PRECS[case["prec"]], bc=cw.CW_BC_DIRICHLET0) for m in s["mesh"]]
        s["mg"] = cw.Multigrid(s["ops"])
        f64 = cw.Operator(s["mesh"][-1], case["p"], bc=cw.CW_BC_DIRICHLET0)
        w = rhs_weights(seed)  # the averaged residual, which a solver feeds the cycle
        s["b"] = f64.dss(w[0] * f64.load_vector(0) + w[1] * f64.load_vector(1), average=True).to(s["ops"][-1].vec_dtype)
        s["u"] = torch.empty_like(s["b"])
    else:
        s["mesh"] = [mesh_of(v) for v in cube_in_cube_verts(case["n"], 3)]
        s["ops"] = [cw.Operator(m, case["p"], prec=PRECS[case["prec"]]) for m in s["mesh"]]
        s["mb"] = cw.MultiBlock(s["ops"])
        idx = torch.from_numpy(s["mb"].global_index()).cuda()
        s["x"] = mblock_values(case, seed, s["mb"].NG, idx).to(s["mb"].vec_dtype)
        s["y"] = s["mb"].empty()
    return s


def mblock_values(case, seed, ng, idx):
    """A continuous vector that does not depend on the numbering: a seeded sum of plane waves at the nodes."""
    x, w = mblock_nodes(case), np.random.default_rng(seed).uniform(-9, 9, (4, 4))
    u = sum(torch.sin(x @ torch.from_numpy(w[m, :3]).cuda() + float(w[m, 3])) for m in range(4))
    first = torch.full((ng,), u.numel(), device="cuda").scatter_reduce(0, idx, torch.arange(u.numel(), device="cuda"), "amin")
    return u[first[idx]]  # copies of a node bit-identical


def run(s):
    if s["what"] == "apply":
        return s["op"].apply(s["x"], s["y"], assemble=s["assemble"])
    if s["what"] == "batch":
        s["batch"].launch(graph=True)
        return s["batch"].ys
    if s["what"] == "cg":
        return s["op"].cg_solve(s["b"], s["u"], rtol=1e-10, mode=s["mode"])[0]
    if s["what"] == "vcycle":
        return s["mg"].vcycle(s["b"], s["u"])
    return s["mb"].apply(s["x"], s["y"], assemble=True)


def _apply_work(p, cells, kind, geom, prec, nrhs=1):
    n, vb, gb = p + 1, VEC_BYTES[prec], MET_BYTES[prec]
    comps = {"laplace": 6, "mass": 1, "laplace+mass": 7}[kind]
    geo = {"affine": 32, "metric": comps * gb * n ** 3, "recompute": 21 * (8 if vb == 8 else 4)}[geom]
    per = {"laplace": 24 * n + 20, "mass": 12 * n + 2, "laplace+mass": 24 * n + 23}[kind]
    if geom == "affine":
        per = 14 * n + 6
    if geom == "recompute":
        per += 120
    return cells * (nrhs * 2 * vb * n ** 3 + geo), cells * nrhs * n ** 3 * per


def work(case):
    if case["what"] == "apply":
        b, f = _apply_work(case["p"], case["nx"] * case["ny"] * case["nz"], case["kind"], case["geom"], case["prec"])
    elif case["what"] == "batch":
        parts = [_apply_work(p, (v.shape[0] - 1) ** 3, "laplace", "metric", case["prec"], r) for p, v, r in batch_problems(case)]
        b, f = (sum(x) for x in zip(*parts))
    elif case["what"] == "cg":  # Jacobi-CG needs about 2.7 p n iterations, each one operator evaluation
        prec = {"f64": "f64", "ir_f32": "f32", "ir_bf16": "f32_bf16g"}[case["mode"]]
        b, f = _apply_work(case["p"], case["nx"] * case["ny"] * case["nz"], "laplace", "metric", prec)
        it = 2.7 * case["p"] * max(case["nx"], case["ny"], case["nz"])
        b, f = b * it, f * it
    elif case["what"] == "vcycle":  # four sweeps and a residual on each level but the coarsest
        b = f = 0
        for l in range(1, case["levels"]):
            x, y = _apply_work(case["p"], (case["n0"] << l) ** 3, "laplace", "metric", case["prec"])
            b, f = b + 4 * x, f + 4 * y
    else:
        b, f = _apply_work(case["p"], 7 * case["n"] ** 3, "laplace", "metric", case["prec"])
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------- the same in plain FP64 torch ----
def _lagrange(nodes, x):
    """l_m(x_q) and l_m'(x_q) of the Lagrange basis on `nodes`."""
    n = len(nodes)
    B, D = np.ones((len(x), n)), np.zeros((len(x), n))
    for m in range(n):
        others = [k for k in range(n) if k != m]
        for k in others:
            B[:, m] *= (x - nodes[k]) / (nodes[m] - nodes[k])
            term = np.full(len(x), 1.0 / (nodes[m] - nodes[k]))
            for j in others:
                if j != k:
                    term *= (x - nodes[j]) / (nodes[m] - nodes[j])
            D[:, m] += term
    return B, D


def _rules(p):
    gx, gw = np.polynomial.legendre.leggauss(p + 1)
    inner = np.sort(np.polynomial.legendre.Legendre.basis(p).deriv().roots().real) if p > 1 else np.zeros(0)
    return (np.concatenate([[-1], inner, [1]]) + 1) / 2, (gx + 1) / 2, gw / 2


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _c3(t, Mz, My, Mx):
    """(Mz x My x Mx) t for t [cells, k, j, i]."""
    t = torch.matmul(My, torch.matmul(t, Mx.T))
    e, k, b, a = t.shape
    return torch.matmul(Mz, t.reshape(e, k, b * a)).reshape(e, Mz.shape[0], b, a)


class Exact:
    """One block's operator in FP64: vectors are [nz*ny*nx, k, j, i]."""

    def __init__(self, verts, p, kind):
        self.dims, self.p, self.kind = tuple(s - 1 for s in verts.shape[:3]), p, kind
        self.n = p + 1
        self.gll, xq, wq = _rules(p)
        B, Bd = _lagrange(self.gll, xq)
        self.B, self.Bd = _t(B), _t(Bd)
        self.L, self.dL = _t(np.stack([1 - xq, xq], 1)), _t(np.stack([-np.ones_like(xq), np.ones_like(xq)], 1))
        v = _t(verts)
        c = [torch.stack([v[a or None:None if a else -1, b or None:None if b else -1, d or None:None if d else -1]
                          for a in (0, 1) for b in (0, 1) for d in (0, 1)], -2)]
        self.corners = c[0].reshape(-1, 2, 2, 2, 3)
        self.w = _t(wq[:, None, None] * wq[None, :, None] * wq[None, None, :])
        self.cache = None

    def interp(self, cells, M):
        return [_c3(self.corners[cells][..., d], M, M, M) for d in range(3)]

    def metric(self, cells):
        X = self.corners[cells]
        J = [[_c3(X[..., d], *[self.dL if s == 2 - a else self.L for a in range(3)]) for s in range(3)] for d in range(3)]

        def cross(a, b):
            return [a[(i + 1) % 3] * b[(i + 2) % 3] - a[(i + 2) % 3] * b[(i + 1) % 3] for i in range(3)]
        col = [[J[d][s] for d in range(3)] for s in range(3)]
        c = [cross(col[1], col[2]), cross(col[2], col[0]), cross(col[0], col[1])]  # det J times the rows of J^-1
        det = sum(col[0][i] * c[0][i] for i in range(3))
        G = [[None if b < a else self.w / det * sum(c[a][i] * c[b][i] for i in range(3)) for b in range(3)] for a in range(3)]
        return G, self.w * det

    def chunks(self, most=1 << 22):
        E, step = self.corners.shape[0], max(1, most // self.n ** 3)
        return [slice(a, min(E, a + step)) for a in range(0, E, step)]

    def apply(self, x, keep=False):
        y = torch.empty_like(x)
        if keep and self.cache is None:
            self.cache = [self.metric(c) for c in self.chunks()]
        for i, c in enumerate(self.chunks()):
            G, m = self.cache[i] if keep else self.metric(c)
            u, B, D = x[c], self.B, self.Bd
            out = 0
            if self.kind != "mass":
                g = [_c3(u, B, B, D), _c3(u, B, D, B), _c3(u, D, B, B)]
                h = [sum(G[min(a, b)][max(a, b)] * g[b] for b in range(3)) for a in range(3)]
                out = _c3(h[0], B.T, B.T, D.T) + _c3(h[1], B.T, D.T, B.T) + _c3(h[2], D.T, B.T, B.T)
            if self.kind != "laplace":
                out = out + _c3(m * _c3(u, B, B, B), B.T, B.T, B.T)
            y[c] = out
        return y

    def diag(self):
        d = []
        for c in self.chunks():
            G, m = self.metric(c)
            out = 0
            for a in range(3):
                for b in range(a, 3):
                    f = [(self.Bd if 2 - k == a else self.B) * (self.Bd if 2 - k == b else self.B) for k in range(3)]
                    out = out + (1 if a == b else 2) * _c3(G[a][b], f[0].T, f[1].T, f[2].T)
            d.append(out)
        return torch.cat(d)

    def grid(self, x):
        return x.reshape(self.dims + (self.n,) * 3)

    def dss(self, x):
        v = self.grid(x.clone())
        for ax in range(3):
            if self.dims[ax] < 2:
                continue
            l, r = v.narrow(ax, 0, self.dims[ax] - 1).select(3 + ax, self.p), v.narrow(ax, 1, self.dims[ax] - 1).select(3 + ax, 0)
            s = l + r
            l.copy_(s), r.copy_(s)
        return v.reshape(x.shape)

    def valence(self):
        return self.dss(torch.ones((self.corners.shape[0],) + (self.n,) * 3, dtype=torch.float64, device="cuda"))

    def mask(self):
        m = torch.ones(self.dims + (self.n,) * 3, dtype=torch.float64, device="cuda")
        for ax in range(3):
            m.select(ax, 0).select(2 + ax, 0).zero_()
            m.select(ax, self.dims[ax] - 1).select(2 + ax, self.p).zero_()
        return m.reshape((-1,) + (self.n,) * 3)

    def load(self, w):
        out = []
        for c in self.chunks():
            x = self.interp(c, self.L)
            f0 = 3 * math.pi ** 2 * torch.sin(math.pi * x[0]) * torch.sin(math.pi * x[1]) * torch.sin(math.pi * x[2])
            q = [t * (1 - t) for t in x]
            f1 = 2 * (q[1] * q[2] + q[0] * q[2] + q[0] * q[1])
            out.append(_c3(self.metric(c)[1] * (w[0] * f0 + w[1] * f1), self.B.T, self.B.T, self.B.T))
        return torch.cat(out)

    def solve(self, b, most=4000):
        """u with A_CG u = G^T b, zero on the boundary: assembled Jacobi-CG down to rounding."""
        dinv, ik = self.mask() / self.dss(self.diag()), 1 / self.valence()
        r = self.dss(b) * self.mask()
        u, p, rho = torch.zeros_like(r), 0, None
        z = dinv * r
        first = best = float((r * r * ik).sum())
        for it in range(most):
            new = (r * z * ik).sum()
            p = z if rho is None else z + (new / rho) * p
            rho = new
            q = self.dss(self.apply(p, keep=True)) * self.mask()
            a = rho / (p * q * ik).sum()
            u += a * p
            r -= a * q
            z = dinv * r
            if it % 10 == 9:
                best = float((r * r * ik).sum())
                if best < 1e-28 * first:
                    break
        self.cache = None
        return u


def _children(p):
    gll = _rules(p)[0]
    return [_t(_lagrange(gll, (gll + b) / 2)[0]) for b in (0, 1)]


def _exact_cycle(levels, l, b, nu=2, omega=0.7):
    L = levels[l]
    if l == 0:
        return L.solve(b)
    C, n = levels[l - 1], L.n
    dinv, P = omega * L.mask() / L.dss(L.diag()), _children(L.p)

    def smooth(u):
        return u + dinv * L.dss(b - L.apply(u, keep=True))

    def child(v, bz, by, bx):  # the children with the same bits, one per coarse cell
        return L.grid(v)[bz::2, by::2, bx::2]
    u = torch.zeros_like(b)
    for _ in range(nu):
        u = smooth(u)
    r = b - L.apply(u, keep=True)
    bits = [(z, y, x) for z in (0, 1) for y in (0, 1) for x in (0, 1)]
    rc = sum(_c3(child(r, *c).reshape((-1,) + (n,) * 3), P[c[0]].T, P[c[1]].T, P[c[2]].T) for c in bits)
    e = _exact_cycle(levels, l - 1, rc, nu, omega)
    for c in bits:
        child(u, *c).add_(_c3(e, P[c[0]], P[c[1]], P[c[2]]).reshape(C.dims + (n,) * 3))
    for _ in range(nu):
        u = smooth(u)
    L.cache = None
    return u


def mblock_nodes(case):
    """Coordinates of every cell-wise entry of the block mesh."""
    xs = []
    for v in cube_in_cube_verts(case["n"], 3):
        o = Exact(v, case["p"], "laplace")
        M = _t(np.stack([1 - o.gll, o.gll], 1))
        xs.append(torch.stack(o.interp(slice(None), M), -1).reshape(-1, 3))
    return torch.cat(xs)


def exact(case, seed):
    """What run() returns for prepare(case, seed), from the same inputs, in FP64 torch."""
    if case["what"] == "apply":
        s = prepare(case, seed)
        o = Exact(box_verts(case["nx"], case["ny"], case["nz"], 0.0 if case["geom"] == "affine" else AMP), case["p"], case["kind"])
        y = o.apply(s["x"].double().reshape((-1,) + (o.n,) * 3))
        return (o.dss(y) if case["assemble"] else y).reshape(-1)
    if case["what"] == "batch":
        s, out = prepare(case, seed), []
        for (p, v, r), x in zip(batch_problems(case), s["batch"].xs):
            o = Exact(v, p, "laplace")
            out.append(torch.cat([o.apply(t.reshape((-1,) + (o.n,) * 3)).reshape(-1) for t in x.double().reshape(r, -1)]))
        return out
    if case["what"] == "cg":
        o = Exact(box_verts(case["nx"], case["ny"], case["nz"], AMP), case["p"], "laplace")
        return o.solve(o.load(rhs_weights(seed))).reshape(-1)
    if case["what"] == "vcycle":
        b, v = prepare(case, seed)["b"], [coarse_verts(case)]
        while len(v) < case["levels"]:
            v.append(refine_verts(v[-1]))
        levels = [Exact(x, case["p"], "laplace") for x in v]
        return _exact_cycle(levels, len(v) - 1, b.double().reshape((-1,) + (case["p"] + 1,) * 3)).reshape(-1)
    s = prepare(case, seed)
    idx, at, ys = torch.from_numpy(s["mb"].global_index()).cuda(), 0, []
    nodes = torch.round(mblock_nodes(case) * 1e7).long() + (1 << 20) * 16
    idx = torch.unique(nodes[:, 0] * (1 << 50) + nodes[:, 1] * (1 << 25) + nodes[:, 2], return_inverse=True)[1]
    for v in cube_in_cube_verts(case["n"], 3):
        o = Exact(v, case["p"], "laplace")
        x = s["x"][at:at + o.corners.shape[0] * o.n ** 3].double()
        at += x.numel()
        ys.append(o.apply(x.reshape((-1,) + (o.n,) * 3)).reshape(-1))
    y = torch.cat(ys)
    return torch.zeros(int(idx.max()) + 1, dtype=torch.float64, device="cuda").index_add(0, idx, y)[idx]
