"""The work a user of the coarsener has it do, as timed cases.

Each case is one call (or the two calls of a training step) through the public API: whole
coarsenings of one graph, the batched training step, the single steps that a program calls on
its own (scores, contraction by a lift it already has), and the differentiable layers on a fixed
lift (coarse weights, node-feature pooling).  Graphs are the constructions of the package's own
workloads -- jittered triangle and tetrahedral meshes with inverse-length weights, random
geometric graphs with Gaussian weights in random node order, batches of meshes -- built here
with torch on the GPU so that new inputs are quick to make.

Programs keep one context for all their calls, so the cases share one: a call on a new graph
runs host-driven.  `repeat` cases stand for the program that coarsens the same graph again and
again (its captured schedule is replayed), and hold a context of their own.
"""
from __future__ import annotations

import math

import torch

from paper_2204_11757_gb300 import api

DTYPES = {"int32": torch.int32, "float32": torch.float32, "float64": torch.float64}
DEV = "cuda"


def listed():
    return [
        # the smallest call: one level of a 4,096-node unit-weight mesh, all launches and latency
        dict(name="coarsen_tri64_i32", op="coarsen", graph="tri", nx=64, ny=64, dtype="int32",
             levels=1, ratio=2, reorder=False, repeat=False),
        # an ordinary small mesh, ragged sides, six halving levels: a mesh hierarchy per request
        dict(name="coarsen_tri257x250_f64", op="coarsen", graph="tri", nx=257, ny=250,
             dtype="float64", levels=6, ratio=64, reorder=False, repeat=False),
        # the 2048^2 mesh coarsened again and again by one program (replayed schedule)
        dict(name="coarsen_tri2048_f64_repeat", op="coarsen", graph="tri", nx=2048, ny=2048,
             dtype="float64", levels=6, ratio=64, reorder=False, repeat=True),
        # the 3D mesh hierarchy, binary64, seven levels (hub rows from the third level on)
        dict(name="coarsen_tet129_f64", op="coarsen", graph="tet", k=129, dtype="float64",
             levels=7, ratio=128, reorder=False, repeat=False),
        # the largest graph: 2^23 points in random order, eight halving levels
        dict(name="coarsen_rgg8m_f32", op="coarsen", graph="rgg", n=1 << 23, dtype="float32",
             levels=8, ratio=256, reorder=False, repeat=False),
        # the adjacency-reordering option on a graph in random order
        dict(name="coarsen_rgg2m_f32_reordered", op="coarsen", graph="rgg", n=1 << 21,
             dtype="float32", levels=8, ratio=256, reorder=True, repeat=False),
        # one pass of the paper's loop straight to n/256, at an odd size
        dict(name="coarsen_rgg1m_f32_one", op="coarsen", graph="rgg", n=1_000_003,
             dtype="float32", levels=1, ratio=256, reorder=False, repeat=False),
        # a training step on a batch of meshes: coarsening, coarse weights, their gradient (a
        # quarter of the 10,000-mesh batch: one of four shards)
        dict(name="train_batch2500_f32", op="batch", B=2500, dtype="float32"),
        # the paper's fitness step alone: every edge's score
        dict(name="score_rgg2m_f32", op="score", graph="rgg", n=1 << 21, dtype="float32"),
        # contraction by a lift the program has (2x2x2 blocks of a 3D mesh)
        dict(name="contract_tet97_f64", op="contract", k=97, dtype="float64", shuffle=False),
        # the differentiable contraction on a fixed lift, forward and backward, on a mesh whose
        # nodes come in random order (as unstructured mesh generators number them)
        dict(name="weights_tet129_f32", op="weights", k=129, dtype="float32", shuffle=True),
        # node-feature pooling onto the super-nodes, forward and backward
        dict(name="pool_4m_f32_64", op="pool", n=1 << 22, ratio=8, F=64, dtype="float32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges; sizes over their logarithm, mostly odd ones."""
    op = rng.choice(["coarsen", "coarsen", "coarsen", "coarsen", "batch", "score", "contract",
                     "weights", "pool"])
    if op == "batch":
        return dict(op=op, B=_log_int(rng, 8, 2500), dtype=rng.choice(["float32", "float32",
                                                                       "float64"]))
    if op == "pool":
        F = _log_int(rng, 3, 128)
        n = _log_int(rng, 1000, min(1 << 22, (1 << 28) // F))
        return dict(op=op, n=n, ratio=rng.choice([2, 8, 64, 256]), F=F,
                    dtype=rng.choice(["float32", "float32", "float64"]))
    if op in ("contract", "weights"):
        return dict(op=op, k=_log_int(rng, 8, 129), dtype=rng.choice(["float32", "float64"]),
                    shuffle=rng.random() < 0.5)
    kind = rng.choice(["tri", "tet", "rgg"])
    if kind == "tri":
        nodes = _log_int(rng, 1024, 1 << 22)
        nx = max(2, int(math.sqrt(nodes) * rng.uniform(0.5, 2.0)))
        size = dict(nx=nx, ny=max(2, nodes // nx))
    elif kind == "tet":
        size = dict(k=_log_int(rng, 9, 129))
    else:
        size = dict(n=_log_int(rng, 4096, 1 << (22 if op == "coarsen" else 21)))
    dtype = rng.choice({"tri": ["int32", "float32", "float64", "float64"],
                        "tet": ["float32", "float64", "float64"],
                        "rgg": ["float32", "float32", "float64"]}[kind])
    case = dict(op=op, graph=kind, dtype=dtype, **size)
    if op == "coarsen":
        case["levels"] = rng.choice([1, 3, 5, 6, 8])
        case["ratio"] = 1 << (case["levels"] if case["levels"] > 1 else rng.choice([1, 2, 6, 8]))
        case["reorder"] = kind == "rgg" and rng.random() < 0.3
        case["repeat"] = rng.random() < 0.25
    return case


# ---- inputs -----------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _rand(gen, *shape):
    return torch.rand(*shape, generator=gen, device=DEV, dtype=torch.float64)


def _csr(n, u, v, w):
    """Symmetric CSR (int64 rowptr, int32 col, w) and the edges in (u, v) order, u < v."""
    lo, hi = torch.minimum(u, v), torch.maximum(u, v)
    key, order = torch.sort(lo * n + hi)
    lo, hi = torch.div(key, n, rounding_mode="floor"), key % n
    w = w[order]
    del key, order
    _, order = torch.sort(torch.cat([lo * n + hi, hi * n + lo]))
    m = lo.shape[0]
    und = torch.where(order < m, order, order - m)
    col = torch.where(order < m, hi[und], lo[und]).to(torch.int32)
    deg = torch.bincount(lo, minlength=n) + torch.bincount(hi, minlength=n)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(deg, 0, out=rowptr[1:])
    return dict(n=n, m=m, rowptr=rowptr, col=col, w=w[und].contiguous(), eu=lo, ev=hi, w_und=w)


def _inv_len(pts, u, v, dtype):
    d = pts[u] - pts[v]
    return (1.0 / (d * d).sum(1).sqrt()).to(dtype)


def _meshes(gen, kx, ky, kz, is3, dtype):
    """Jittered grid meshes, one per entry of kx (int64 tensors): 2D triangulated grids (one
    coin-flip diagonal per cell) where is3 is False, Kuhn-split tetrahedral meshes elsewhere.
    Returns (n, u, v, w, graph_ptr)."""
    B = kx.shape[0]
    size = kx * ky * kz
    ptr = torch.zeros(B + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(size, 0, out=ptr[1:])
    n = int(ptr[-1])
    g = torch.repeat_interleave(torch.arange(B, device=DEV), size)
    loc = torch.arange(n, device=DEV) - ptr[g]
    X, Y, Z, three = kx[g], ky[g], kz[g], is3[g]
    x, y = loc % X, torch.div(loc, X, rounding_mode="floor") % Y
    z = torch.div(loc, X * Y, rounding_mode="floor")
    pts = torch.stack([x, y, z], 1).to(torch.float64)
    jit = torch.where(three, 0.25, 0.3)[:, None] * (2.0 * _rand(gen, n, 3) - 1.0)
    jit[:, 2] = torch.where(three, jit[:, 2], torch.zeros((), dtype=torch.float64, device=DEV))
    pts += jit
    coin = _rand(gen, n) < 0.5
    ids = torch.arange(n, device=DEV)
    us, vs = [], []
    for ox, oy, oz in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1),
                       (1, 1, 1)):
        ok = (x + ox < X) & (y + oy < Y) & (z + oz < Z)
        if (ox, oy, oz) == (1, 1, 0):  # the 2D cell's diagonal goes either way
            anti = ok & ~three & coin
            u = ids[anti]
            us.append(u + 1)
            vs.append(u + X[u])
            ok = ok & ~anti
        u = ids[ok]
        us.append(u)
        vs.append(u + (oz * Y[u] + oy) * X[u] + ox)
    u, v = torch.cat(us), torch.cat(vs)
    return n, u, v, (torch.ones(u.shape[0], dtype=dtype, device=DEV) if dtype == torch.int32
                     else _inv_len(pts, u, v, dtype)), ptr


EDGES_PER_NODE = 5.9  # of the random geometric graphs: mean degree about 12


def _rgg(gen, n, dtype):
    """Random geometric graph: the 5.9 n closest pairs of n random points in the unit cube, ids
    in random order, weight exp(-d^2 / r^2) with r the longest pair's distance.  Candidates come
    from a grid of cells of side >= 1.15 times the radius of mean degree 12."""
    pts = _rand(gen, n, 3)
    r = 1.15 * (36.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    G = max(1, int(1.0 / r))
    c = (pts * G).long().clamp_(max=G - 1)
    cid, order = torch.sort((c[:, 2] * G + c[:, 1]) * G + c[:, 0])
    start = torch.zeros(G ** 3 + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(cid, minlength=G ** 3), 0, out=start[1:])
    pts, c = pts[order], c[order]
    idx = torch.arange(n, device=DEV)
    us, vs, ds = [], [], []
    for dz, dy in ((0, 0), (0, 1), (1, -1), (1, 0), (1, 1)):  # rows of cells ahead of a point's
        z, y = c[:, 2] + dz, c[:, 1] + dy
        ok = (z < G) & (y >= 0) & (y < G)
        row = (z * G + y).clamp_(0, G * G - 1) * G
        first = start[row + (c[:, 0] - 1).clamp_(min=0)] if (dz, dy) != (0, 0) else idx + 1
        cnt = (start[row + (c[:, 0] + 1).clamp_(max=G - 1) + 1] - first) * ok
        i = torch.repeat_interleave(idx, cnt)
        j = torch.arange(i.shape[0], device=DEV) - (torch.cumsum(cnt, 0) - cnt - first)[i]
        d = pts[i] - pts[j]
        d2 = (d * d).sum(1)
        near = d2 < r * r
        us.append(order[i[near]])
        vs.append(order[j[near]])
        ds.append(d2[near])
        del i, j, d, d2, near
    m = int(EDGES_PER_NODE * n)
    d2, by = torch.sort(torch.cat(ds))
    d2, by = d2[:m], by[:m]
    return n, torch.cat(us)[by], torch.cat(vs)[by], torch.exp(-d2 / d2[-1]).to(dtype)


def _one_mesh(gen, kx, ky, kz, is3, dtype):
    one = lambda k: torch.tensor([k], device=DEV)  # noqa: E731
    return _meshes(gen, one(kx), one(ky), one(kz), one(is3), dtype)[:4]


def _graph(case, gen):
    dtype = DTYPES[case["dtype"]]
    if case["graph"] == "rgg":
        return _csr(*_rgg(gen, case["n"], dtype))
    if case["graph"] == "tri":
        return _csr(*_one_mesh(gen, case["nx"], case["ny"], 1, False, dtype))
    return _csr(*_one_mesh(gen, case["k"], case["k"], case["k"], True, dtype))


def _batch(case, gen):
    """B meshes of sizes evenly spread over the logarithm from 200 to 20000, every other one 3D,
    in random order, as one block-diagonal CSR."""
    B = case["B"]
    i = torch.randperm(B, generator=gen, device=DEV)
    N = torch.exp(math.log(200.0) + math.log(100.0) * (i.double() + 0.5) / B)
    is3 = i % 2 == 1
    k = torch.where(is3, N.pow(1.0 / 3.0), N.sqrt()).round().long()
    n, u, v, w, ptr = _meshes(gen, k, k, torch.where(is3, k, torch.ones_like(k)), is3,
                              DTYPES[case["dtype"]])
    return _csr(n, u, v, w), ptr


def _mesh_and_lift(case, seed):
    """A tetrahedral mesh, its nodes in grid or random order, and the lift that a program brings
    along: blocks of 2x2x2 nodes, numbered row by row.  Returns (graph, int32 lift, n_c)."""
    gen, k = _gen(seed), case["k"]
    n, u, v, w = _one_mesh(gen, k, k, k, True, DTYPES[case["dtype"]])
    ids, h = torch.arange(n, device=DEV), (k + 1) // 2
    half = lambda t: torch.div(t, 2, rounding_mode="floor")  # noqa: E731
    x, y, z = ids % k, torch.div(ids, k, rounding_mode="floor") % k, \
        torch.div(ids, k * k, rounding_mode="floor")
    lift = ((half(z) * h + half(y)) * h + half(x)).to(torch.int32)
    if case["shuffle"]:
        p = torch.randperm(n, generator=gen, device=DEV)
        u, v, lift = p[u], p[v], torch.empty_like(lift).index_copy_(0, p, lift)
    return _csr(n, u, v, w), lift, h ** 3


def _pool_inputs(case, gen):
    """Points in random order pooled by neighbourhood, super-nodes of random size around `ratio`:
    (lift, n_c, x, gradient of the means)."""
    n, dtype = case["n"], DTYPES[case["dtype"]]
    n_c = max(1, n // case["ratio"])
    head = torch.zeros(n, dtype=torch.int64, device=DEV)
    head[torch.randperm(n - 1, generator=gen, device=DEV)[:n_c - 1] + 1] = 1
    rank = torch.randperm(n, generator=gen, device=DEV)  # a node's place along the points' order
    lift = torch.cumsum(head, 0)[rank].to(torch.int32)
    x = torch.randn(n, case["F"], generator=gen, device=DEV, dtype=dtype)
    grad = torch.randn(n_c, case["F"], generator=gen, device=DEV, dtype=dtype)
    return lift, n_c, x, grad


def _weights_grad(case, seed, m_c):
    return torch.randn(m_c, generator=_gen(seed + 1), device=DEV, dtype=DTYPES[case["dtype"]])


# ---- the cases --------------------------------------------------------------------------------

_CONTEXT = []


def _context():
    """The program's context, kept for all of its calls."""
    if not _CONTEXT:
        _CONTEXT.append(api.Context())
    return _CONTEXT[0]


def _as_csr(g):
    return api.CSR(g["rowptr"], g["col"], g["w"])


def prepare(case, seed):
    op = case["op"]
    s = dict(case=case, ctx=api.Context() if case.get("repeat") else _context(), keep={})
    if op == "pool":
        s["lift"], s["n_c"], s["x"], s["grad"] = _pool_inputs(case, _gen(seed))
        s["x"].requires_grad_(True)
    elif op == "batch":
        g, s["ptr"] = _batch(case, _gen(seed))
        s["csr"], s["w"] = _as_csr(g), g["w_und"].requires_grad_(True)
        s["keep"]["a"] = torch.zeros(g["m"], dtype=g["w"].dtype, device=DEV)
    elif op in ("contract", "weights"):
        g, s["lift"], s["n_c"] = _mesh_and_lift(case, seed)
        s["csr"] = _as_csr(g)
        if op == "weights":
            level = s["ctx"].contract(s["csr"], s["lift"], s["n_c"])
            s["plan"] = api.ContractionPlan.from_levels(s["ctx"], [level])
            s["w"] = g["w_und"].requires_grad_(True)
            s["grad"] = _weights_grad(case, seed, level.m_c)
    else:
        s["csr"] = _as_csr(_graph(case, _gen(seed)))
        if op == "coarsen":
            s["keep"]["col"] = torch.zeros_like(s["csr"].col)
            s["keep"]["w"] = torch.zeros_like(s["csr"].w)
    return s


def _keep(s, name, t):
    """The caller's own array, large enough for any coarse graph, with the result in front."""
    s["keep"][name][:t.shape[0]].copy_(t)
    return s["keep"][name]


def run(s):
    case, ctx = s["case"], s["ctx"]
    op = case["op"]
    if op == "coarsen":
        csr = s["csr"]
        lift, n_c, _ = ctx.coarsen(csr, max(1, csr.n // case["ratio"]), levels=case["levels"],
                                   reorder=case["reorder"])
        last = ctx.level(case["levels"] - 1)
        return dict(lift=lift, n_c=n_c, rowptr=last.rowptr_c, mass=last.mass,
                    col=_keep(s, "col", last.col_c), w=_keep(s, "w", last.w_c))
    if op == "batch":
        lift, ptr_c, _ = ctx.coarsen_batched(s["csr"], s["ptr"], 8, 3)
        plan = api.ContractionPlan.from_levels(ctx, ctx.levels())
        a = api.contract_weights(s["w"], plan)
        grad, = torch.autograd.grad(a.sum(), s["w"])
        return dict(lift=lift, ptr_c=ptr_c, a=_keep(s, "a", a.detach()), grad=grad)
    if op == "score":
        return dict(score=ctx.score(s["csr"]))
    if op == "contract":
        lv = ctx.contract(s["csr"], s["lift"], s["n_c"])
        return dict(emap=lv.emap, a=lv.a_und, self_mass=lv.self_mass, rowptr=lv.rowptr_c,
                    col=lv.col_c, w=lv.w_c, perm=lv.perm, seg=lv.seg)
    if op == "weights":
        a = api.contract_weights(s["w"], s["plan"])
        grad, = torch.autograd.grad(a, s["w"], s["grad"])
        return dict(a=a.detach(), grad=grad)
    xc = api.pool_features(s["x"], s["lift"], s["n_c"], ctx)
    grad, = torch.autograd.grad(xc, s["x"], s["grad"])
    return dict(xc=xc.detach(), grad=grad)


def _sizes(case):
    """(n, m) of the case's graph; of a batch, the means of its sizes and of both degrees."""
    if case["op"] == "batch":
        n = case["B"] * (20000 - 200) / math.log(100.0)
        return n, 4.6 * n
    if case.get("graph") == "rgg":
        return case["n"], EDGES_PER_NODE * case["n"]
    if case.get("graph") == "tri":
        x, y = case["nx"], case["ny"]
        return x * y, (x - 1) * y + x * (y - 1) + (x - 1) * (y - 1)
    k = case["k"]
    return k ** 3, 3 * (k - 1) * k * k + 3 * (k - 1) ** 2 * k + (k - 1) ** 3


def work(case):
    """Every input read once, every output written once; one addition per union coordinate of
    every edge's score and one per weight or feature summed."""
    s = 8 if case["dtype"] == "float64" else 4
    if case["op"] == "pool":
        n, F = case["n"], case["F"]
        return {"bytes": 2.0 * n * F * s + 2.0 * n / case["ratio"] * F * s + 8.0 * n,
                "flops": 2.0 * n * F}
    n, m = _sizes(case)
    csr = 8.0 * (n + 1) + 2.0 * m * (4 + s)
    union = 3.2 * m / n  # two rows of 2m/n entries less the coordinates they share
    if case["op"] == "coarsen":
        levels, r = case["levels"], case["ratio"]
        return {"bytes": csr + 4.0 * n + csr / r,
                "flops": sum(m / 2 ** l for l in range(levels)) * union}
    if case["op"] == "batch":
        return {"bytes": csr + 4.0 * n + 2.0 * m * s + m / 8 * s, "flops": 1.75 * m * union}
    if case["op"] == "score":
        return {"bytes": csr + m * s, "flops": m * union}
    if case["op"] == "contract":
        n_c, m_c = n / 8, m / 5
        return {"bytes": csr + 4.0 * n + 8.0 * m + n_c * (8 + s) + m_c * (s + 4 + 2 * (4 + s)),
                "flops": float(m)}
    return {"bytes": m * (4.0 + s) + m * (4.0 + s) + 0.6 * m * (4 + 2 * s), "flops": float(m)}


# ---- the same in 64 bits ------------------------------------------------------------------------

def _exact_score(g):
    """sum over the union of both rows of |p_ax - p_bx|, p = w / degree."""
    n, m = g["n"], g["m"]
    rowptr, col = g["rowptr"], g["col"].long()
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), rowptr[1:] - rowptr[:-1])
    w = g["w"].double()
    p = w / torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, rows, w)[rows]
    key = rows * n + col  # ascending
    out = torch.empty(m, dtype=torch.float64, device=DEV)
    step = 1 << 22
    for e0 in range(0, m, step):
        a, b = g["eu"][e0:e0 + step], g["ev"][e0:e0 + step]
        cnt = rowptr[a + 1] - rowptr[a]
        e = torch.repeat_interleave(torch.arange(a.shape[0], device=DEV), cnt)
        j = torch.arange(e.shape[0], device=DEV) - (torch.cumsum(cnt, 0) - cnt - rowptr[a])[e]
        want = b[e] * n + col[j]
        at = torch.searchsorted(key, want).clamp_(max=key.shape[0] - 1)
        pb = torch.where(key[at] == want, p[at], torch.zeros_like(p[at]))
        f = torch.zeros(a.shape[0], dtype=torch.float64, device=DEV)
        f.index_add_(0, e, (p[j] - pb).abs() - pb)
        out[e0:e0 + step] = f + 1.0  # row b's entries sum to 1, the shared ones counted above
    return out


def _exact_coarse(g, lift, n_c):
    """Coarse edges in (U, V) order: their keys, the coarse edge of every fine edge (-1 inside a
    super-node) and the fine weights in 64 bits."""
    U, V = lift.long()[g["eu"]], lift.long()[g["ev"]]
    inter = U != V
    key = torch.minimum(U, V) * n_c + torch.maximum(U, V)
    keys, inv = torch.unique(key[inter], return_inverse=True)
    emap = torch.full_like(U, -1)
    emap[inter] = inv
    return keys, emap, U, inter, g["w_und"].double()


def exact(case, seed):
    op = case["op"]
    if op in ("coarsen", "batch"):  # merge decisions: no 64-bit value to compare with
        return None
    if op == "pool":
        lift, n_c, x, grad = _pool_inputs(case, _gen(seed))
        lift = lift.long()
        cnt = torch.bincount(lift, minlength=n_c).double()[:, None]
        xc = torch.zeros(n_c, case["F"], dtype=torch.float64, device=DEV)
        for i in range(0, case["n"], 1 << 20):
            xc.index_add_(0, lift[i:i + (1 << 20)], x[i:i + (1 << 20)].double())
        return dict(xc=xc / cnt, grad=(grad.double() / cnt)[lift])
    if op == "score":
        return dict(score=_exact_score(_graph(case, _gen(seed))))
    g, lift, n_c = _mesh_and_lift(case, seed)
    keys, emap, U, inter, w = _exact_coarse(g, lift, n_c)
    a = torch.zeros(keys.shape[0], dtype=torch.float64, device=DEV)
    a.index_add_(0, emap[inter], w[inter])
    if op == "weights":
        grad_a = _weights_grad(case, seed, keys.shape[0]).double()
        return dict(a=a, grad=torch.where(inter, grad_a[emap.clamp(min=0)],
                                          torch.zeros((), dtype=torch.float64, device=DEV)))
    mass = torch.zeros(n_c, dtype=torch.float64, device=DEV)
    mass.index_add_(0, U[~inter], w[~inter])
    lo, hi = torch.div(keys, n_c, rounding_mode="floor"), keys % n_c
    both = torch.sort(torch.cat([lo * n_c + hi, hi * n_c + lo]))[1]
    return dict(emap=None, a=a, self_mass=mass, rowptr=None, col=None,
                w=torch.cat([a, a])[both], perm=None, seg=None)
