"""The work that users of the library have it do, as cases that can be timed.

A case is one public operation on one geometry: a product with an assembled
operator, the assembly itself, a solve, a gradient through a solve, or the
whole path for many small geometries.  The geometries are bumped geodesic
spheres of 20 f^2 panels (every edge of the icosahedron cut into f parts), so
sizes between and beyond the powers of four of the midpoint-subdivided spheres
occur, and leaf clusters of every width.  Their shapes, the point sources, the
vectors and the coefficients come from the seed.

exact() gives what the dense Galerkin matrix of the same panels and quadrature
gives in 64 bits (the 7 x 7 rule; the regularised rule for touching panels), in
torch operations of its own, for sizes where that takes seconds.
"""
import functools
import math

import numpy as np
import torch

import paper_1806_11558_gb300 as hm
from paper_1806_11558_gb300.autograd import DensitySolve, Potential

DTYPES = {"f64": hm.HM_F64, "f32": hm.HM_F32, "bf16": hm.HM_BF16}


def listed():
    return [
        # one product with the operator of the small workload (5,120 panels): tens of microseconds of launches;
        # an explicit time step or an outer iteration of the user's own
        dict(name="matvec_small", op="matvec", f=16, leaf=64, eps=1e-6, dtype="f64", nrhs=1, trans=0),
        # the FP64 product of the precision workload (327,680 panels, 25 GB): what an FP64 Krylov solver repeats
        dict(name="matvec_large", op="matvec", f=128, leaf=64, eps=1e-7, dtype="f64", nrhs=1, trans=0),
        # the transposed product on the FP32 copies (adjoint methods), 200,000 panels, leaves of 48-49 rows
        dict(name="matvec_transposed_f32", op="matvec", f=100, leaf=64, eps=1e-6, dtype="f32", nrhs=1, trans=1),
        # 16 right-hand sides on the tensor cores: the step of a block Krylov method
        dict(name="product16_f32", op="block", f=128, leaf=128, eps=1e-6, dtype="f32", nrhs=16),
        # 20 right-hand sides (a full and a ragged pass) of the FP64 master: residuals of many systems
        dict(name="product20_f64", op="block", f=57, leaf=64, eps=1e-6, dtype="f64", nrhs=20),
        # tree, assembly and load vector of the small workload: the latency of a whole set-up
        dict(name="setup_small", op="setup", f=16, leaf=64, eps=1e-6, dtype="f64", nrhs=1),
        # an ordinary geometry (40,500 panels) with FP32 copies for a refined solve
        dict(name="setup_medium", op="setup", f=45, leaf=64, eps=1e-6, dtype="f32", nrhs=4),
        # a large geometry (655,220 panels) with the parameters of the large workload
        dict(name="setup_large", op="setup", f=181, leaf=128, eps=1e-6, dtype="f32", nrhs=16),
        # GMRES(30) in FP64 on the small workload: hundreds of short dependent launches
        dict(name="solve_small", op="solve", f=16, leaf=64, eps=1e-6, dtype="f64", nrhs=1, restart=30, precond=0),
        # 16 systems in lockstep, FP32 inner solves and FP64 refinement (the large workload's solver, 81,920 panels)
        dict(name="solve16_refined", op="solve", f=64, leaf=128, eps=1e-6, dtype="f32", nrhs=16, restart=128, precond=1),
        # loss and gradients through a solve (21,780 panels, 1,024 evaluation points): forward and adjoint solve
        dict(name="gradient", op="gradient", f=33, leaf=64, eps=1e-6, points=1024),
        # the whole path for 24 small geometries at once, 4 sources each (the batching workload's options)
        dict(name="forest", op="forest", f=32, leaf=64, eps=1e-5, count=24, nrhs=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["matvec", "matvec", "block", "block", "setup", "setup", "solve", "solve", "gradient", "forest"])
    leaf, eps = rng.choice([32, 48, 64, 100, 128]), rng.choice([1e-5, 1e-6, 1e-7])
    if op == "matvec":
        return dict(op=op, f=_log(rng, 8, 120), leaf=leaf, eps=eps, dtype=rng.choice(["f64", "f64", "f32", "bf16"]),
                    nrhs=rng.choice([1, 1, 2, 3]), trans=rng.choice([0, 0, 1]))
    if op == "block":
        return dict(op=op, f=_log(rng, 8, 110), leaf=leaf, eps=eps, dtype=rng.choice(["f64", "f32", "bf16"]),
                    nrhs=rng.randint(2, 24))
    if op == "setup":
        return dict(op=op, f=_log(rng, 8, 140), leaf=leaf, eps=eps, dtype=rng.choice(["f64", "f32"]),
                    nrhs=rng.randint(1, 16))
    if op == "solve":
        dtype, nrhs = rng.choice([("f64", 1), ("f64", 3), ("f32", 1), ("f32", 5), ("f32", 16), ("f32", 17)])
        return dict(op=op, f=_log(rng, 8, 64), leaf=rng.choice([64, 100, 128]), eps=eps, dtype=dtype, nrhs=nrhs,
                    restart=128, precond=1)
    if op == "gradient":
        return dict(op=op, f=_log(rng, 8, 60), leaf=64, eps=rng.choice([1e-6, 1e-7]), points=rng.randint(100, 2000))
    return dict(op=op, f=_log(rng, 10, 40), leaf=rng.choice([48, 64, 100]), eps=1e-5, count=rng.randint(3, 24),
                nrhs=rng.randint(1, 5))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _geodesic(f):
    """Vertices (unit sphere) and triangles of the icosahedron with every edge cut into f parts."""
    phi = (1.0 + math.sqrt(5.0)) / 2.0
    C = np.array([p for a in (-1.0, 1.0) for b in (-phi, phi) for p in ((0, a, b), (a, b, 0), (b, 0, a))])
    D = np.linalg.norm(C[:, None] - C[None], axis=2)
    near = np.abs(D - 2.0) < 1e-9
    faces = [(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
             if near[a, b] and near[b, c] and near[a, c]]
    ij = [(i, j) for i in range(f + 1) for j in range(f + 1 - i)]
    at = {p: k for k, p in enumerate(ij)}
    i, j = np.array(ij).T
    up = [(at[a, b], at[a + 1, b], at[a, b + 1]) for a, b in ij if a + b < f]
    down = [(at[a + 1, b], at[a + 1, b + 1], at[a, b + 1]) for a, b in ij if a + b < f - 1]
    local = np.array(up + down)
    odd = np.random.RandomState(7).randint(1, 1 << 62, 12).astype(np.uint64)  # a point's key: its weights, hashed
    pts, keys, tris = [], [], []
    for k, (a, b, c) in enumerate(faces):
        if np.dot(np.cross(C[b] - C[a], C[c] - C[a]), C[a]) < 0:
            b, c = c, b
        w = np.stack([f - i - j, i, j])
        pts.append((w[0][:, None] * C[a] + w[1][:, None] * C[b] + w[2][:, None] * C[c]) / f)
        wu = w.astype(np.uint64)
        keys.append(wu[0] * odd[a] + wu[1] * odd[b] + wu[2] * odd[c])
        tris.append(local + k * len(ij))
    _, first, inv = np.unique(np.concatenate(keys), return_index=True, return_inverse=True)
    V = np.concatenate(pts)[first]
    V /= np.linalg.norm(V, axis=1)[:, None]
    return V, inv.reshape(-1)[np.concatenate(tris)].astype(np.int32)


def _mesh(f, rng, bump=0.1):
    """A geodesic sphere whose radius varies smoothly, in ways drawn from rng."""
    V, T = _geodesic(f)
    V = torch.from_numpy(V).cuda()
    a, p = rng.uniform(-1.0, 1.0, 6), rng.uniform(0.0, 2.0 * math.pi, 6)
    k = torch.from_numpy(2.0 * rng.standard_normal((3, 6))).cuda()
    r = 1.0 + bump * (torch.cos(V @ k + torch.from_numpy(p).cuda()) @ torch.from_numpy(a).cuda())
    return (V * r[:, None]).contiguous(), torch.from_numpy(T).cuda()


def _sources(rng, n, lo=2.5, hi=4.0):
    d = rng.standard_normal((n, 3))
    return torch.from_numpy(d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(lo, hi, (n, 1))).cuda()


def _forest_sizes(c):
    return [max(3, int(c["f"] * (0.25 + 0.75 * ((7 * g) % c["count"] + 1) / c["count"]))) for g in range(c["count"])]


def _inputs(c, seed):
    """The tensors a user has before any call, from the seed alone."""
    rng = np.random.Generator(np.random.PCG64(seed))
    s = {}
    if c["op"] == "forest":
        Vs, Ts, off, src, nv = [], [], [0], [], 0
        for f in _forest_sizes(c):
            V, T = _mesh(f, rng, 0.05)
            V = V * torch.from_numpy(np.exp(rng.uniform(math.log(0.5), math.log(2.0), 3))).cuda()
            Vs.append(V)
            Ts.append(T + nv)
            nv += V.shape[0]
            off.append(off[-1] + T.shape[0])
            src.append(_sources(rng, c["nrhs"], 3.5, 5.0))
        s.update(V=torch.cat(Vs).contiguous(), T=torch.cat(Ts).contiguous(), off=off, src=torch.stack(src).contiguous())
        return s
    s["V"], s["T"] = _mesh(c["f"], rng)
    n = s["T"].shape[0]
    if c["op"] in ("matvec", "block"):
        s["x"] = torch.from_numpy(rng.standard_normal((c["nrhs"], n))).cuda()
    elif c["op"] == "setup":
        s["src"] = _sources(rng, c["nrhs"])
        s["x"] = torch.from_numpy(rng.standard_normal(n)).cuda()
    elif c["op"] == "solve":
        s["src"] = _sources(rng, c["nrhs"])
    else:
        s["src"] = _sources(rng, 1)
        s["c"] = torch.from_numpy(rng.uniform(0.8, 1.25, n)).cuda()
        s["points"] = _sources(rng, c["points"], 2.4, 2.6).contiguous()
        p = np.array([0.0, 0.0, 3.0])
        s["target"] = 1.0 / (4.0 * math.pi * torch.linalg.norm(s["points"] - torch.from_numpy(p).cuda(), dim=1))
    return s


class _Operator:
    """A tree and a matrix, freed with the object."""

    def __init__(self, tree, matrix=None):
        self.tree, self.matrix = tree, matrix

    def __del__(self):
        for h in (self.matrix, self.tree):
            hm.hm_free(h)


def _assemble(c, tree):
    # FP32 and BF16 factors go with the FP32 copy of the near field; the FP64 master is always there
    low = DTYPES[c.get("dtype", "f64")]
    return hm.hm_assemble(tree, aca_eps=c["eps"], aca_kmax=64, ss_order=8, factor_dtype=low,
                          dense_dtype=hm.HM_F64 if low == hm.HM_F64 else hm.HM_F32)


def prepare(c, seed):
    s = _inputs(c, seed)
    s["case"] = c
    if c["op"] in ("setup", "forest"):
        return s
    op = _Operator(hm.hm_build_tree(s["V"], s["T"], eta=1.5, leaf_size=c["leaf"]))
    op.matrix = _assemble(c, op.tree)
    s["op"], n = op, s["T"].shape[0]
    if c["op"] == "solve":
        s["b"] = hm.hm_load_vector(op.tree, s["src"], torch.empty((c["nrhs"], n), dtype=torch.float64, device="cuda"))
    if c["op"] == "gradient":
        s["f"] = hm.hm_load_vector(op.tree, s["src"], torch.empty((1, n), dtype=torch.float64, device="cuda"))[0]
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    c, n = s["case"], s["T"].shape[0]
    new = functools.partial(torch.empty, dtype=torch.float64, device="cuda")
    if c["op"] == "matvec":
        return hm.hm_matvec(s["op"].matrix, s["x"], new(s["x"].shape), trans=c["trans"], prec=DTYPES[c["dtype"]])
    if c["op"] == "block":
        return hm.hm_matvec_block(s["op"].matrix, s["x"], new(s["x"].shape), prec=DTYPES[c["dtype"]])
    if c["op"] == "setup":
        op = _Operator(hm.hm_build_tree(s["V"], s["T"], eta=1.5, leaf_size=c["leaf"]))
        op.matrix = _assemble(c, op.tree)
        f = hm.hm_load_vector(op.tree, s["src"], new((c["nrhs"], n)))
        y = hm.hm_matvec(op.matrix, s["x"], new(n))
        return {"perm": hm.hm_tree_get_perm(op.tree, n), "f": f, "y": y}
    if c["op"] == "solve":
        x = torch.zeros_like(s["b"])
        opts = dict(rel_tol=1e-12, restart=c["restart"], max_iter=5000, precond=c["precond"], batched=int(c["nrhs"] > 1))
        if c["dtype"] != "f64":
            opts.update(refine=1, inner_dtype=DTYPES[c["dtype"]], inner_tol=1e-4, max_refine=40, resid_df=int(c["nrhs"] > 1))
        hm.hm_solve(s["op"].matrix, s["b"], x, **opts)
        return x
    if c["op"] == "gradient":
        f, k = s["f"].detach().requires_grad_(True), s["c"].detach().requires_grad_(True)
        alpha = DensitySolve.apply(s["op"].matrix, f, k, dict(rel_tol=1e-13, restart=128, max_iter=5000, precond=1))
        loss = torch.mean((Potential.apply(s["op"].tree, s["points"], alpha) - s["target"]) ** 2)
        df, dc = torch.autograd.grad(loss, (f, k))
        return {"alpha": alpha.detach(), "loss": loss.detach(), "df": df, "dc": dc}
    op = _Operator(hm.hm_build_forest(s["V"], s["T"], s["off"], eta=1.5, leaf_size=c["leaf"]))
    op.matrix = _assemble(dict(c, dtype="f32"), op.tree)
    b = hm.hm_load_vector_geom(op.tree, s["src"], new((c["nrhs"], n)))
    x = torch.zeros_like(b)
    # converged well past the workload's 1e-6, so that the solutions are the systems' own and not the stopping test's
    hm.hm_solve(op.matrix, b, x, rel_tol=1e-11, restart=60, max_iter=5000, precond=1, batched=1, refine=1,
                inner_dtype=hm.HM_F32, inner_tol=1e-4, max_refine=40)
    return {"perm": hm.hm_tree_get_perm(op.tree, n), "b": b, "x": x}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _entries(n, leaf, eps):
    """Stored near-field and factor entries of an operator of n panels (fits to operators of 1,280 to 655,220 panels,
    within a few per cent)."""
    depth = max(0, math.ceil(math.log2(n / leaf)))
    near = min(float(n) * n, 38.0 * n * n / 2.0 ** depth)
    far = n * max(60.0, 850.0 * (depth - 5.5) * (1.0 + 0.21 * (-math.log10(eps) - 6.0)))
    return near, far


def work(c):
    if c["op"] == "forest":
        sizes = [20 * f * f for f in _forest_sizes(c)]
        e = [_entries(n, c["leaf"], c["eps"]) for n in sizes]
        near, far, n = sum(v[0] for v in e), sum(v[1] for v in e), sum(sizes)
    else:
        n = 20 * c["f"] ** 2
        near, far = _entries(n, c["leaf"], c["eps"])
    size = {"f64": 8, "f32": 4}
    if c["op"] in ("matvec", "block"):
        both = near * (8 if c["dtype"] == "f64" else 4) + far * {"f64": 8, "f32": 4, "bf16": 2}[c["dtype"]]
        return {"bytes": both + 16.0 * n * c["nrhs"], "flops": 2.0 * c["nrhs"] * (near + far)}
    # an entry of the near field, or of a cross of the approximation, is 49 kernel values of about 12 operations;
    # half of them are mirrored
    entries = 0.5 * (near + far)
    make = {"bytes": 8.0 * (near + far) + 60.0 * n, "flops": 49 * 12.0 * entries}
    if c["op"] == "setup":
        if c["dtype"] != "f64":
            make["bytes"] += 4.0 * (near + far)
        return {"bytes": make["bytes"] + 8.0 * n * (c["nrhs"] + 2), "flops": make["flops"] + 84.0 * n * c["nrhs"]}
    its = 16.0 * math.log10(n)  # products of a solve to 1e-12 (60 to 120)
    if c["op"] == "solve":
        passes = its * (math.ceil(c["nrhs"] / 16) if c["nrhs"] > 1 else 1)
        return {"bytes": passes * (near + far) * size[c["dtype"]] + its * 16.0 * n * c["nrhs"],
                "flops": 2.0 * its * c["nrhs"] * (near + far)}
    if c["op"] == "gradient":
        return {"bytes": 2.0 * its * 8 * (near + far) + 100.0 * n, "flops": 4.0 * its * (near + far) + 168.0 * n * c["points"]}
    return {"bytes": make["bytes"] + 0.5 * its * 4 * (near + far) + 16.0 * n * c["nrhs"],
            "flops": make["flops"] + its * c["nrhs"] * (near + far)}


# ---------------------------------------------------------------------------
# the dense Galerkin matrix in 64 bits
# ---------------------------------------------------------------------------
def _rule():
    """The 7-point rule of degree 5 on a triangle: barycentric points and weights."""
    q = math.sqrt(15.0)
    pts, w = [(1 / 3, 1 / 3, 1 / 3)], [9 / 40]
    for a, v in (((6 - q) / 21, (155 - q) / 1200), ((6 + q) / 21, (155 + q) / 1200)):
        for k in range(3):
            pts.append(tuple(1 - 2 * a if d == k else a for d in range(3)))
            w.append(v)
    return torch.tensor(pts, dtype=torch.float64, device="cuda"), torch.tensor(w, dtype=torch.float64, device="cuda")


def _touching_rule(kind, order=8):
    """Points (u, v) and weights of the regularised rule for panels that share `kind` vertices (the xi integral of
    xi^2 done: 1/3), as coefficients of the two edge vectors of each panel."""
    x, w = np.polynomial.legendre.leggauss(order)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    a, b, e = (t.reshape(-1) for t in np.meshgrid(x, x, x, indexing="ij"))
    W = (w[:, None, None] * w[None, :, None] * w[None, None, :]).reshape(-1)
    one = np.ones_like(a)
    ab, abe = a * b, a * b * e
    if kind == 1:
        at = [((one, a), (b, b * e), b), ((b, b * e), (one, a), b)]
    elif kind == 2:
        J = a * ab
        at = [((one, a * e), (1 - ab, a - ab), a * a), ((one, a), (1 - abe, ab - abe), J),
              ((1 - ab, a - ab), (one, abe), J), ((1 - abe, ab - abe), (one, a), J), ((1 - abe, a - abe), (one, ab), J)]
    else:
        J = a * ab
        half = [((one, 1 - a + ab), (1 - abe, 1 - a)), ((one, a - ab + abe), (1 - ab, a - ab)),
                ((1 - abe, a - abe), (one, a - ab))]
        at = [(u, v, J) for u, v in half] + [(v, u, J) for u, v in half]
    coef = np.concatenate([np.stack([u[0], u[1], v[0], v[1]]) for u, v, _ in at], axis=1)
    wt = np.concatenate([W * J for _, _, J in at]) / 3.0
    return torch.from_numpy(coef).cuda(), torch.from_numpy(wt).cuda()


def _touching(V, T):
    """Pairs (i, j) of panels that share vertices, and their entries of the matrix."""
    n = T.shape[0]
    T = T.long()
    v, order = torch.sort(T.reshape(-1))
    tri, nv = order // 3, V.shape[0]
    count = torch.bincount(v, minlength=nv)
    start = torch.cumsum(count, 0) - count
    slot = torch.arange(3 * n, device="cuda") - start[v]
    star = torch.full((nv, int(count.max())), -1, dtype=torch.long, device="cuda")
    star[v, slot] = tri
    key = (torch.arange(n, device="cuda")[:, None, None] * n + star[T]).reshape(-1)
    key, kinds = torch.unique(key[(star[T] >= 0).reshape(-1)], return_counts=True)
    I, Jt = key // n, key % n
    area = 0.5 * torch.linalg.norm(torch.linalg.cross(V[T[:, 1]] - V[T[:, 0]], V[T[:, 2]] - V[T[:, 0]]), dim=1)
    val = torch.empty(key.shape[0], dtype=torch.float64, device="cuda")
    for kind in (1, 2, 3):
        sel = (kinds == kind).nonzero()[:, 0]
        coef, w = _touching_rule(kind)
        for part in torch.split(sel, max(1, 40_000_000 // w.shape[0])):
            P, Q = T[I[part]], T[Jt[part]]
            same = P[:, :, None] == Q[:, None, :]
            if kind == 1:  # both rotated to start at the shared vertex
                k, l = same.any(2).long().argmax(1), same.any(1).long().argmax(1)
                turn = torch.arange(3, device="cuda")
                P, Q = P.gather(1, (k[:, None] + turn) % 3), Q.gather(1, (l[:, None] + turn) % 3)
            elif kind == 2:  # the shared pair first, in the order of the first panel
                p = torch.sort((~same.any(2)).long(), dim=1, stable=True)[1]
                P, last = P.gather(1, p), Q.gather(1, (~same.any(1)).long().argmax(1)[:, None])
                Q = torch.cat([P[:, :2], last], 1)
            else:
                Q = P
            D = 0.0
            for d in range(3):
                p, q = V[P, d], V[Q, d]
                t = ((p[:, 1] - p[:, 0])[:, None] * coef[0] + (p[:, 2] - p[:, 1])[:, None] * coef[1]
                     - (q[:, 1] - q[:, 0])[:, None] * coef[2] - (q[:, 2] - q[:, 1])[:, None] * coef[3])
                D = D + t * t
            val[part] = 4.0 * area[I[part]] * area[Jt[part]] * (D.rsqrt() @ w) / (4.0 * math.pi)
    return I, Jt, val, area


class _Dense:
    """The Galerkin matrix by blocks of rows (original panel order)."""

    def __init__(self, V, T):
        self.I, self.J, self.val, self.area = _touching(V, T)
        bary, self.w = _rule()
        self.X = torch.einsum("qk,nkd->dqn", bary, V[T.long()]).contiguous()  # [3][7][n]
        self.n = T.shape[0]

    def blocks(self):
        n, step = self.n, max(1, 6_000_000 // self.n)
        for a in range(0, n, step):
            b = min(n, a + step)
            acc = torch.zeros((b - a, n), dtype=torch.float64, device="cuda")
            for p in range(7):
                for q in range(7):
                    d = self.X[0, p, a:b, None] - self.X[0, q]
                    r = d * d
                    for k in (1, 2):
                        torch.sub(self.X[k, p, a:b, None], self.X[k, q], out=d)
                        r.addcmul_(d, d)
                    acc.add_(r.rsqrt_(), alpha=float(self.w[p] * self.w[q]))
            acc *= self.area[a:b, None] * self.area / (4.0 * math.pi)
            at = ((self.I >= a) & (self.I < b)).nonzero()[:, 0]
            acc[self.I[at] - a, self.J[at]] = self.val[at]
            yield a, b, acc

    def times(self, X, trans):
        """[r][n] times the matrix (or its transpose)."""
        Y = torch.zeros_like(X)
        for a, b, A in self.blocks():
            if trans:
                Y += X[:, a:b] @ A
            else:
                Y[:, a:b] = X @ A.T
        return Y

    def whole(self):
        A = torch.empty((self.n, self.n), dtype=torch.float64, device="cuda")
        for a, b, part in self.blocks():
            A[a:b] = part
        return A

    def potential(self, points):
        """[points][n]: the single-layer potential of each panel at the points."""
        E = torch.zeros((points.shape[0], self.n), dtype=torch.float64, device="cuda")
        for q in range(7):
            r = sum((points[:, d, None] - self.X[d, q]) ** 2 for d in range(3))
            E.add_(r.rsqrt(), alpha=float(self.w[q]))
        return E * self.area / (4.0 * math.pi)


def exact(c, seed):
    if c["op"] == "forest":
        s = _inputs(c, seed)
        if max(_forest_sizes(c)) > 32:
            return None
        x, b = [], []
        for g in range(c["count"]):
            t0, t1 = s["off"][g], s["off"][g + 1]
            M = _Dense(s["V"], s["T"][t0:t1])
            b.append(M.potential(s["src"][g]))
            x.append(torch.linalg.solve(M.whole(), b[-1].T).T)
        return {"perm": None, "b": torch.cat(b, 1), "x": torch.cat(x, 1)}
    n = 20 * c["f"] ** 2
    if n > (45000 if c["op"] in ("matvec", "block", "setup") else 24000):
        return None
    s = _inputs(c, seed)
    M = _Dense(s["V"], s["T"])
    if c["op"] in ("matvec", "block"):
        return M.times(s["x"], c.get("trans", 0))
    if c["op"] == "setup":
        return {"perm": None, "f": M.potential(s["src"]), "y": M.times(s["x"][None], 0)[0]}
    LU, piv = torch.linalg.lu_factor(M.whole())
    f = M.potential(s["src"])
    if c["op"] == "solve":
        return torch.linalg.lu_solve(LU, piv, f.T).T.contiguous()
    alpha = torch.linalg.lu_solve(LU, piv, f.T)[:, 0] / s["c"]
    E = M.potential(s["points"])
    r = E @ alpha - s["target"]
    g = 2.0 / r.shape[0] * (r @ E)
    lam = torch.linalg.lu_solve(LU, piv, (g / s["c"])[:, None], adjoint=True)[:, 0]
    return {"alpha": alpha, "loss": torch.mean(r * r), "df": lam, "dc": -alpha * g / s["c"]}
