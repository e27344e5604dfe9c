"""GPU kernels at the sizes where their tiles, groups and dispatch rules end, against the oracle
(bit-exact: the library's sums run in the oracle's order)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2204_11757_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2204_11757_gb300 import api
    with api.Context() as c:
        yield c


def _bits(a):
    return a.view(np.uint32 if a.dtype.itemsize == 4 else np.uint64) if a.dtype.kind == "f" else a


# rows of 1 to 59 entries (a group of lanes copies 1 to 30 chunks of a row), edge counts around a
# warp's tile of 32, a path (rows of 2), and rows whose tile exceeds the stage
@pytest.mark.parametrize("n,p", [(2, 1.0), (9, 0.9), (12, 0.5), (33, 1.0), (60, 1.0), (300, 0.1),
                                 (1000, 0.006), (3000, 0.004)])
def test_binary32_scores_packed_and_in_place(ctx, n, p):
    from paper_2204_11757_gb300 import api
    g = I.random_graph(n, p, seed=n, weight="float", dtype=np.float32, connected=True)
    ref = O.score(g)
    csr = api.CSR.from_graph(g)
    assert np.array_equal(_bits(ctx.score(csr).cpu().numpy()), _bits(ref))
    for schedule in (1, 3):
        ctx.coarsen(csr, g.n, levels=1, schedule=schedule)
        assert np.array_equal(_bits(ctx.level(0).score.cpu().numpy()), _bits(ref))


# super-nodes of up to 256 members are gathered in one pass, larger ones (or too much ranking)
# go through the sort and the tree; features around the 16-byte accesses and the lanes of a row
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("F", [1, 2, 4, 31, 64, 132])
@pytest.mark.parametrize("sizes", [[1], [256], [257, 1, 0, 3], [0, 5, 256, 255, 2, 1, 33, 0] * 3,
                                   [7, 9] * 200, [65, 64, 63] * 30, [256] * 40])
def test_pooling_routes(ctx, dtype, F, sizes):
    rng = np.random.default_rng(F)
    lift = rng.permutation(np.repeat(np.arange(len(sizes)), sizes)).astype(np.int32)
    n, n_c = lift.shape[0], len(sizes)
    x = (rng.standard_normal((n, F)) * 10.0 ** rng.integers(-3, 4, size=(n, 1))).astype(dtype)
    g = rng.standard_normal((n_c, F)).astype(dtype)
    lt = torch.from_numpy(lift).cuda()

    def put(a, shift):  # a tensor whose data starts `shift` elements into its storage
        t = torch.zeros(a.size + shift, dtype=torch.from_numpy(a).dtype, device="cuda")
        t[shift:] = torch.from_numpy(a.ravel()).cuda()
        return t[shift:].view(a.shape)

    ref, ref_g = O.pool_features(lift, n_c, x), O.pool_backward(lift, n_c, g)
    for shift in (0, 1):
        xc = ctx.pool_features(lt, n_c, put(x, shift)).cpu().numpy()
        assert np.array_equal(_bits(xc), _bits(ref))
        gx = ctx.pool_features_backward(lt, n_c, put(g, shift)).cpu().numpy()
        assert np.array_equal(_bits(gx), _bits(ref_g))


# the one-kernel merge selection: one CTA and many, the tail's item count, the score prefix's edge
# count (65,536), one target per relabelling rule (n / 8), nothing to merge, everything to merge, a
# disconnected graph (the target is not reached), equal scores (the edge id decides)
@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.int32])
@pytest.mark.parametrize("n,p", [(2, 1.0), (40, 0.2), (513, 0.01), (1025, 0.004), (3000, 0.002),
                                 (6000, 0.0036), (6000, 0.0038), (20000, 0.0006)])
def test_selection_at_the_edges_of_its_phases(ctx, n, p, dtype):
    from paper_2204_11757_gb300 import api
    weight = "unit" if dtype == np.int32 else "float"
    g = I.random_graph(n, p, seed=n, weight=weight, dtype=dtype, connected=n != 6000)
    csr = api.CSR.from_graph(g)
    for target in sorted({1, max(1, n // 256), max(1, n // 8 - 1), max(1, n // 8), max(1, n // 2),
                          max(1, n - 1), n}):
        ref = O.coarsen_level(g, target)
        lift, n_c, st = ctx.coarsen(csr, target, levels=1)
        assert n_c == ref.n_c and st == (1 if ref.n_c > target else 0)
        assert np.array_equal(lift.cpu().numpy(), ref.lift)
    f = ctx.score(csr)
    target = max(1, n // 3)
    ref = O.coarsen_level(g, target)
    lift, merged, n_c, st = ctx.select_merges(csr, f, target)
    assert n_c == ref.n_c and int(merged.sum()) == n - n_c
    assert np.array_equal(lift.cpu().numpy(), ref.lift)


# segments and super-nodes around the 256 terms from which the tables of the long sums take over:
# the contraction and the carried mass decide from the bucket sizes whether to look for them
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("leaves", [255, 256, 257, 258])
def test_long_segments_found_from_bucket_sizes(ctx, dtype, leaves):
    from paper_2204_11757_gb300 import api
    # two hubs with a fan of light leaves each, a chain between the leaves of both: merging leaves
    # one coarse edge of `leaves` fine edges and, a level later, super-nodes of about that many
    rng = np.random.default_rng(leaves)
    a, b = 0, leaves + 1
    eu = np.concatenate([np.full(leaves, a), np.full(leaves, b), 1 + np.arange(leaves), [a]])
    ev = np.concatenate([1 + np.arange(leaves), b + 1 + np.arange(leaves),
                         b + 1 + np.arange(leaves), [b]])
    g = I.csr_from_edges(2 * leaves + 2, eu, ev, rng.uniform(0.5, 2, eu.shape[0]).astype(dtype))
    for ratio in (4, 32):
        ref, total = O.coarsen(g, ratio, "halving")
        lift, n_c, _ = ctx.coarsen(api.CSR.from_graph(g), ref[-1].target, levels=len(ref))
        assert np.array_equal(lift.cpu().numpy(), total)
        for lv, r in zip(ctx.levels(), ref):
            assert np.array_equal(_bits(lv.w_c.cpu().numpy()), _bits(r.coarse.graph.w))
            assert np.array_equal(_bits(lv.self_mass.cpu().numpy()), _bits(r.coarse.self_mass))
            assert np.array_equal(_bits(lv.score.cpu().numpy()), _bits(r.f))
    lift = np.repeat(np.int32([0, 1]), leaves + 1)
    lv = ctx.contract(api.CSR.from_graph(g), torch.from_numpy(lift).cuda(), 2)
    c = O.contract(g, lift, 2)
    assert np.array_equal(_bits(lv.a_und.cpu().numpy()), _bits(c.a_und))
    assert np.array_equal(_bits(lv.self_mass.cpu().numpy()), _bits(c.self_mass))


# long sums (rows' degrees, coarse weights, self-masses) streamed by one CTA: lengths around the first
# 32 terms and the blocks of 1,024 after them, the limit of 65,536 terms, terms over 60 binades, exact
# half-grid ties, and leading zeros (the masses carried into a giant super-node)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("L", [257, 1055, 1056, 1057, 2080, 4100, 65535, 65536, 65537])
def test_streamed_long_sums(ctx, dtype, L):
    from paper_2204_11757_gb300 import api
    rng = np.random.default_rng(L)
    ties = I.star_ties(12, dtype).w_und  # 1 + eps, 1 - eps in turn
    for w in (rng.uniform(0.5, 2.0, L), np.exp2(rng.uniform(-40, 20, L)),
              np.resize(np.asarray(ties), L), np.full(L, 0.1)):
        w = w.astype(dtype)
        g = I.csr_from_edges(L + 1, np.zeros(L, np.int64), 1 + np.arange(L), w)
        if L < 5000:  # the hub's degree is in every score (the oracle's time grows with L^2)
            f = ctx.score(api.CSR.from_graph(g)).cpu().numpy()
            assert np.array_equal(_bits(f), _bits(O.score(g)))
        lift = np.r_[np.int32(0), np.ones(L, np.int32)]
        for lt, n_c in ((lift, 2), (np.zeros(L + 1, np.int32), 1)):
            lv = ctx.contract(api.CSR.from_graph(g), torch.from_numpy(lt).cuda(), n_c)
            c = O.contract(g, lt, n_c)
            assert np.array_equal(_bits(lv.a_und.cpu().numpy()), _bits(c.a_und))
            assert np.array_equal(_bits(lv.self_mass.cpu().numpy()), _bits(c.self_mass))
            if n_c == 2:
                a = ctx.contract_forward(lv.perm, lv.seg, lv.m_c, torch.from_numpy(w).cuda())
                assert np.array_equal(_bits(a.cpu().numpy()), _bits(c.a_und))


# one giant super-node per level whose members mostly carry no mass yet
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_streamed_masses_of_a_giant(ctx, dtype):
    from paper_2204_11757_gb300 import api
    rng = np.random.default_rng(3)
    n = 3000
    eu = np.r_[np.zeros(n - 1, np.int64), 1 + np.arange(n - 2)]
    ev = np.r_[1 + np.arange(n - 1), 2 + np.arange(n - 2)]
    g = I.csr_from_edges(n, eu, ev, rng.uniform(0.5, 2.0, eu.shape[0]).astype(dtype))
    ref, total = O.coarsen(g, 64, "halving")
    lift, n_c, _ = ctx.coarsen(api.CSR.from_graph(g), ref[-1].target, levels=len(ref))
    assert np.array_equal(lift.cpu().numpy(), total)
    for lv, r in zip(ctx.levels(), ref):
        assert np.array_equal(_bits(lv.score.cpu().numpy()), _bits(r.f))
        assert np.array_equal(_bits(lv.w_c.cpu().numpy()), _bits(r.coarse.graph.w))


# the flat normalise and diagonal kernels march over tiles of 2,048 and 1,024 stored entries: entry
# counts around a tile, rows longer than a tile's share, more rows in a tile than shared memory
# holds (a path: 1,024), runs of empty rows longer than a block, long rows between short ones
def _flat_graphs(dtype):
    rng = np.random.default_rng(5)
    out = []
    for m in (511, 512, 513, 1023, 1024, 1025, 5000):  # paths: 2 m entries
        out.append((m + 1, np.arange(m), 1 + np.arange(m)))
    gaps = np.cumsum(rng.integers(1, 900, 60))         # a path over a few nodes of many
    out.append((int(gaps[-1]) + 700, gaps[:-1], gaps[1:]))
    u = np.r_[np.zeros(2500, np.int64), np.full(300, 2000), 1 + np.arange(2400)]
    v = np.r_[1 + np.arange(2500), 2101 + np.arange(300), 2 + np.arange(2400)]
    key = np.unique(np.minimum(u, v) * 4000 + np.maximum(u, v))
    out.append((3000, key // 4000, key % 4000))
    for n, eu, ev in out:
        w = np.ones(eu.shape[0]) if dtype == np.int32 else rng.uniform(0.1, 2.0, eu.shape[0])
        yield I.csr_from_edges(n, eu, ev, w.astype(dtype))


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.int32])
def test_flat_kernels_at_tile_edges(ctx, dtype):
    from paper_2204_11757_gb300 import api, native as N
    for g in _flat_graphs(dtype):
        csr = api.CSR.from_graph(g)
        assert np.array_equal(_bits(ctx.score(csr).cpu().numpy()), _bits(O.score(g)))
        ref, total = O.coarsen(g, 4, "halving")
        lift, n_c, _ = ctx.coarsen(csr, ref[-1].target, levels=len(ref))
        assert np.array_equal(lift.cpu().numpy(), total)
        for lv, r in zip(ctx.levels(), ref):
            assert np.array_equal(_bits(lv.score.cpu().numpy()), _bits(r.f))
            assert np.array_equal(_bits(lv.w_c.cpu().numpy()), _bits(r.coarse.graph.w))
        # without scores the mirrors are looked up edge by edge: one weight changed on one side
        lt = torch.from_numpy(ref[0].lift).cuda()
        assert ctx.contract(csr, lt, ref[0].n_c).m_c == ref[0].coarse.m_c
        for j in (0, g.col.shape[0] - 1):
            w = g.w.copy()
            w[j] = w[j] + 1
            bad = api.CSR.from_numpy(g.rowptr, g.col, w)
            with pytest.raises(N.SpcError) as e:
                ctx.contract(bad, lt, ref[0].n_c)
            assert e.value.status == -2  # SPC_ERR_NOT_SYMMETRIC


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [2, 31, 33, 4095, 4096, 4097, 4096 * 5 + 1, 4096 * 40 - 1])
@pytest.mark.parametrize("values", [1, 3, 40, 0])
def test_sort_ranks_and_look_back(ctx, dtype, n, values):
    """Equal keys keep their order whether a warp's 32 share one digit, a few or none, in partial
    tiles and over more tiles than a look-back window."""
    rng = np.random.default_rng(n + values)
    f = rng.random(n) if values == 0 else rng.integers(0, values, n) * 0.37
    f = f.astype(dtype)
    order = ctx.sort_fitness(torch.from_numpy(f).cuda()).cpu().numpy()
    assert np.array_equal(order, np.argsort(f, kind="stable").astype(np.int32))


@pytest.mark.parametrize("dtype", [np.int32, np.float32, np.float64])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 97, 1000])
@pytest.mark.parametrize("shape", ["stars", "cliques"])
def test_lower_rows_over_groups_of_32(ctx, dtype, n, shape):
    """Coarse rows' lower entries, rows pooled 32 to a warp: empty rows, rows on both sides of 32
    entries next to one another, a last group that is not full."""
    from paper_2204_11757_gb300 import api
    rng = np.random.default_rng(n)
    if shape == "stars":  # every 13th row holds many lower entries, the others none
        e = [(u, v) for v in range(12, n, 13) for u in range(max(0, v - 70), v)]
        e = e or [(0, 1)]
    else:
        e = [(u, v) for v in range(n) for u in range(max(0, v - int(rng.integers(0, 40))), v)]
        e = e or [(0, 1)]
    eu, ev = (np.array(x, dtype=np.int32) for x in zip(*e))
    w = rng.integers(1, 9, eu.shape[0]) if dtype == np.int32 else rng.random(eu.shape[0]) + 0.1
    g = I.csr_from_edges(n, eu, ev, w.astype(dtype))
    lift = np.arange(n, dtype=np.int32)  # nothing merged: the coarse graph is the graph itself
    lv = ctx.contract(api.CSR.from_graph(g), torch.from_numpy(lift).cuda(), n)
    assert np.array_equal(lv.rowptr_c.cpu().numpy(), g.rowptr)
    assert np.array_equal(lv.col_c.cpu().numpy(), g.col)
    assert np.array_equal(_bits(lv.w_c.cpu().numpy()), _bits(g.w))


@pytest.mark.parametrize("dtype", [np.int32, np.float64])
@pytest.mark.parametrize("size", [1, 9, 63, 64, 65, 200, 300])
def test_buckets_across_the_ranking_tiles(ctx, dtype, size):
    """Coarse edges from buckets around the 64 items that are ranked in a tile, and longer ones, with
    several fine edges to most of them, over a few tiles of 1,024 positions."""
    from paper_2204_11757_gb300 import api
    rng = np.random.default_rng(size)
    n_c, per = max(8, 5000 // size), 24
    n = n_c * per  # super-node U holds the nodes U, U + n_c, ...
    a = np.repeat(np.arange(n_c), size)
    b = (a + 1 + rng.integers(0, min(n_c - 1, max(1, size // 2)), a.shape[0])) % n_c
    x = a + n_c * rng.integers(0, per, a.shape[0])
    y = b + n_c * rng.integers(0, per, a.shape[0])
    lo, hi = np.minimum(x, y).astype(np.int64), np.maximum(x, y)
    key = np.unique(lo * n + hi)
    eu, ev = key // n, key % n
    w = rng.integers(1, 9, eu.shape[0]) if dtype == np.int32 else rng.random(eu.shape[0]) + 0.1
    g = I.csr_from_edges(n, eu, ev, w.astype(dtype))
    lift = (np.arange(n) % n_c).astype(np.int32)
    c = O.contract(g, lift, n_c)
    lv = ctx.contract(api.CSR.from_graph(g), torch.from_numpy(lift).cuda(), n_c)
    assert np.array_equal(lv.emap.cpu().numpy(), c.emap)
    inter = np.flatnonzero(c.emap >= 0)
    perm = inter[np.argsort(c.emap[inter], kind="stable")]
    assert np.array_equal(lv.perm.cpu().numpy()[:perm.size], perm)
    assert np.array_equal(lv.seg.cpu().numpy(), np.searchsorted(c.emap[perm], np.arange(lv.m_c + 1)))
    assert np.array_equal(_bits(lv.a_und.cpu().numpy()), _bits(c.a_und))
    assert np.array_equal(lv.rowptr_c.cpu().numpy(), c.graph.rowptr)
    assert np.array_equal(lv.col_c.cpu().numpy(), c.graph.col)
    assert np.array_equal(_bits(lv.w_c.cpu().numpy()), _bits(c.graph.w))


@pytest.mark.parametrize("dtype", [np.int32, np.float32, np.float64])
@pytest.mark.parametrize("blocks,extra,clique", [(1, 0, 10), (1, 1, 64), (1, 0, 65), (3, 1, 10),
                                                 (5, 1, 140), (90, 1, 10)])
def test_huge_buckets_among_short_ones(ctx, dtype, blocks, extra, clique):
    """Buckets of 2,048 and 2,049 inter edges and intra buckets on both sides of 2,048 (cliques of 64
    and 65 have 2,016 and 2,080 edges), fewer than half of the edges: sorted apart from the ranked
    ones."""
    from paper_2204_11757_gb300 import api
    rng = np.random.default_rng(blocks + extra)
    eu, ev, lift, n, U = [], [], [], 0, 0
    for q in range(blocks):  # a complete bipartite block: one bucket, one or two coarse edges
        A, B = n + np.arange(32), n + 32 + np.arange(64)
        eu.append(np.repeat(A, 64))
        ev.append(np.tile(B, 32))
        if extra:
            eu.append(A[:1])
            ev.append(B[-1:] + 1)  # into whatever comes next
        lift += [U] * 32 + [U + 1] * 64
        n, U = n + 96, U + 2
    for _ in range(2):
        iu, iv = np.triu_indices(clique, 1)
        eu.append(n + iu)
        ev.append(n + iv)
        lift += [U] * clique
        n, U = n + clique, U + 1
    k = 30000 + 3000 * blocks
    C = n + np.arange(k)
    eu.append(C)
    ev.append(np.roll(C, -1))
    lift += list(U + np.arange(k) // 2)
    n, U = n + k, U + k // 2
    perm = rng.permutation(n)  # node numbers in any order
    eu, ev = perm[np.concatenate(eu)], perm[np.concatenate(ev)]
    lift, old = np.empty(n, dtype=np.int32), lift
    lift[perm] = old
    w = rng.integers(1, 99, eu.shape[0]) if dtype == np.int32 else rng.random(eu.shape[0]) + 0.1
    g = I.csr_from_edges(n, eu, ev, w.astype(dtype))
    c = O.contract(g, lift, U)
    ctx.time_kernel("*")
    try:
        lv = ctx.contract(api.CSR.from_graph(g), torch.from_numpy(lift).cuda(), U)
        prof = ctx.kernel_profile()
    finally:
        ctx.time_kernel(None)
    assert any("k_huge_put" in k for k in prof) == bool(extra or clique > 64)
    assert not any("k_classify" in k for k in prof)
    assert np.array_equal(lv.emap.cpu().numpy(), c.emap)
    assert np.array_equal(_bits(lv.a_und.cpu().numpy()), _bits(c.a_und))
    assert np.array_equal(_bits(lv.self_mass.cpu().numpy()), _bits(c.self_mass))
    assert np.array_equal(lv.rowptr_c.cpu().numpy(), c.graph.rowptr)
    assert np.array_equal(lv.col_c.cpu().numpy(), c.graph.col)
    assert np.array_equal(_bits(lv.w_c.cpu().numpy()), _bits(c.graph.w))


def _sparse(n, dtype, connected=True):
    """About 3 n random edges, and a path through all nodes in random order when connected."""
    rng = np.random.default_rng(n)
    e = rng.integers(0, n, (2, 3 * n))
    if connected:
        q = rng.permutation(n)
        e = np.concatenate([e, [q[:-1], q[1:]]], axis=1)
    lo, hi = e.min(axis=0), e.max(axis=0)
    key = np.unique((lo * n + hi)[lo != hi])
    w = np.ones(key.size) if dtype == np.int32 else rng.uniform(0.1, 2.0, key.size)
    return I.csr_from_edges(n, key // n, key % n, w.astype(dtype))


def _batch_checked(ctx, graphs, ratio, schedule, levels):
    from paper_2204_11757_gb300 import api
    b = I.batch_of(graphs)
    res = O.coarsen_batch(b, ratio, schedule)
    gp = torch.from_numpy(b.graph_ptr).cuda()
    lift, gpc, _ = ctx.coarsen_batched(api.CSR.from_graph(b.graph), gp, ratio, levels=levels)
    lift, gpc = lift.cpu().numpy(), gpc.cpu().numpy()
    for i, (levels_ref, total) in enumerate(res):
        n0, n1 = b.graph_ptr[i], b.graph_ptr[i + 1]
        assert gpc[i + 1] - gpc[i] == levels_ref[-1].n_c
        assert np.array_equal(lift[n0:n1] - gpc[i], total)


# one CTA per graph: the node counts at which the classes of shared memory end (4,708, 10,444 and
# 19,968 nodes with 32-bit scores, 3,364, 7,460 and 14,260 with 64-bit ones; past the last the batch
# goes through the launches over all graphs), more graphs than SMs and fewer, tiny ones among them
@pytest.mark.parametrize("dtype,sizes", [
    (np.float32, [4708, 4709, 10444, 10445, 19968]), (np.float32, [4708]), (np.float32, [19969]),
    (np.float64, [3364, 3365, 7460, 7461, 14260]), (np.float64, [14261]), (np.int32, [3364, 3365])])
@pytest.mark.parametrize("many", [False, True])
def test_small_graphs_at_the_classes_of_shared_memory(ctx, dtype, sizes, many):
    rng = np.random.default_rng(len(sizes))
    graphs = [_sparse(n, dtype, connected=bool(n & 1)) for n in sizes]
    tiny = [_sparse(int(n), dtype) for n in rng.integers(2, 60, 400 if many else 5)]
    for ratio, levels in ((2, 1), (16, 1), (8, 3)):
        _batch_checked(ctx, tiny[:3] + graphs + tiny[3:], ratio, "halving" if levels > 1 else "one",
                       levels)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,p", [(8192, 0), (8193, 0), (700, 0.5), (700, 0.57)])
def test_one_small_graph_at_its_limits(ctx, dtype, n, p):
    """8,192 nodes, 131,072 edges (p = 0.5: 122,325, p = 0.57: 139,450), few distinct scores."""
    from paper_2204_11757_gb300 import api
    g = (I.random_graph(n, p, seed=n, weight="float", dtype=dtype, connected=True) if p
         else _sparse(n, dtype))
    csr = api.CSR.from_graph(g)
    rng = np.random.default_rng(n)
    for f in (O.score(g), (rng.integers(1, 4, g.m) * 0.25).astype(O.score(g).dtype)):
        for target in (1, n // 3, n - 5):
            lift, merged, n_c, _ = ctx.select_merges(csr, torch.from_numpy(f).cuda(), target)
            ref, ref_n = O.relabel(O.greedy_merge(g, O.sort_fitness(f), target)[0])
            assert n_c == ref_n and int(merged.sum()) == n - n_c
            assert np.array_equal(lift.cpu().numpy(), ref)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("leaves", [3, 40, 126, 127, 128, 129, 200])
def test_masses_carried_by_buckets_and_by_sort(ctx, dtype, leaves):
    """Members of super-nodes listed by buckets up to 64 squared members a node, else sorted: fans of
    leaves that merge into their hubs, beside a path as long."""
    from paper_2204_11757_gb300 import api
    rng = np.random.default_rng(leaves)
    hubs, s = 6, leaves + 1
    eu = [np.repeat(np.arange(hubs) * s, leaves), hubs * s + np.arange(hubs * s - 1),
          np.arange(hubs) * s]
    ev = [np.repeat(np.arange(hubs) * s, leaves) + np.tile(1 + np.arange(leaves), hubs),
          hubs * s + 1 + np.arange(hubs * s - 1), hubs * s + np.arange(hubs)]
    eu, ev = np.concatenate(eu), np.concatenate(ev)
    g = I.csr_from_edges(2 * hubs * s, eu, ev, rng.uniform(0.5, 2, eu.shape[0]).astype(dtype))
    ref, total = O.coarsen(g, 16, "halving")
    lift, _, _ = ctx.coarsen(api.CSR.from_graph(g), ref[-1].target, levels=len(ref))
    assert np.array_equal(lift.cpu().numpy(), total)
    for lv, r in zip(ctx.levels(), ref):
        assert np.array_equal(_bits(lv.self_mass.cpu().numpy()), _bits(r.coarse.self_mass))
        assert np.array_equal(_bits(lv.score.cpu().numpy()), _bits(r.f))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_batches_that_are_not_block_diagonal(ctx, dtype):
    """Edges between two graphs of a batch merge across them: such a batch takes the launches over
    all graphs, as one with a graph too large for shared memory does (an added path of 20,001
    nodes), with the same partition."""
    from paper_2204_11757_gb300 import api
    a, c = _sparse(3000, dtype), _sparse(5000, dtype)
    eu = np.concatenate([a.eu, 3000 + c.eu, [17, 2999]])
    ev = np.concatenate([a.ev, 3000 + c.ev, [3001, 7000]])
    w = np.concatenate([a.w_und, c.w_und, np.full(2, 1.5, dtype)]).astype(dtype)
    path = np.arange(20000)
    wide_u, wide_v = np.concatenate([eu, 8000 + path]), np.concatenate([ev, 8001 + path])
    ww = np.concatenate([w, np.ones(20000, dtype)])
    g, wide = I.csr_from_edges(8000, eu, ev, w), I.csr_from_edges(28001, wide_u, wide_v, ww)
    lift, _, _ = ctx.coarsen_batched(api.CSR.from_graph(g),
                                     torch.tensor([0, 3000, 8000]).cuda(), 4, levels=2)
    ref, _, _ = ctx.coarsen_batched(api.CSR.from_graph(wide),
                                    torch.tensor([0, 3000, 8000, 28001]).cuda(), 4, levels=2)
    assert np.array_equal(lift.cpu().numpy(), ref.cpu().numpy()[:8000])


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [20011, 262144, 262145])
def test_deep_trees_of_random_graphs(ctx, dtype, n):
    """Graphs without locality, whose trees are flattened between rounds (up to 2^18 nodes) and before
    every further slab (a target of n / 16 takes several)."""
    from paper_2204_11757_gb300 import api
    g = _sparse(n, dtype)
    csr = api.CSR.from_graph(g)
    for target in (n // 2, n // 16):
        ref = O.coarsen_level(g, target)
        lift, n_c, _ = ctx.coarsen(csr, target, levels=1)
        assert n_c == ref.n_c
        assert np.array_equal(lift.cpu().numpy(), ref.lift)


@pytest.mark.parametrize("dtype,work", [(np.float32, 20000), (np.float64, 14000), (np.int32, 14000)])
def test_one_graph_on_both_sides_of_its_rule(ctx, dtype, work):
    """One graph is selected in one CTA while its nodes and edges are few (an edge counts up to four
    times per merge wanted), or when it is halved at best and has at most 30,000 edges."""
    from paper_2204_11757_gb300 import api

    def check(g, target, one_cta):
        csr = api.CSR.from_graph(g)
        ref = O.coarsen_level(g, target)
        ctx.time_kernel("*")
        try:
            lift, n_c, _ = ctx.coarsen(csr, target, levels=1)
            prof = ctx.kernel_profile()
        finally:
            ctx.time_kernel(None)
        assert any("k_select_small" in k for k in prof) == one_cta
        assert any("k_select_coop" in k for k in prof) == (not one_cta)
        assert n_c == ref.n_c
        assert np.array_equal(lift.cpu().numpy(), ref.lift)

    def graph(n, m):  # a path and the first edges of a denser one
        rng = np.random.default_rng(m)
        e = rng.integers(0, n, (2, 2 * m))
        key = np.unique(np.minimum(e[0], e[1]) * n + np.maximum(e[0], e[1]))
        key = key[(key // n + 1 < key % n)]  # no self-loop, no edge of the path
        key = np.r_[np.arange(n - 1) * n + np.arange(n - 1) + 1,
                    rng.permutation(key)[:m - (n - 1)]]
        w = np.ones(m) if dtype == np.int32 else rng.uniform(0.1, 2.0, m)
        return I.csr_from_edges(n, key // n, key % n, w.astype(dtype))

    n = 5000
    check(graph(n, work - n), 1, True)
    check(graph(n, work - n + 1), 1, False)
    k = (work - n) // 4  # four edges per merge
    check(graph(n, 40000), n - k, True)
    check(graph(n, 40000), n - k - 1, False)
    check(graph(8192, 30000), 4096, True)
    check(graph(8192, 30000), 4095, False)
    check(graph(8192, 30001), 4096, False)
    check(graph(8193, 9000), 8000, False)


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.int32])
@pytest.mark.parametrize("larger", [[], [300, 4000], [300, 4000, 9000, 12000]])
def test_batches_of_tiny_graphs(ctx, dtype, larger):
    """Graphs of up to 64 nodes in CTAs of their own (1,000 and more of them), on both sides of 512 edges
    and of the 64 nodes, with few distinct scores, without edges, of one node."""
    rng = np.random.default_rng(len(larger))
    shapes = [_sparse(int(n), dtype, connected=bool(n & 1)) for n in (2, 3, 5, 17, 31, 63, 64, 65, 70)]
    shapes += [I.complete_graph(n, dtype) for n in (32, 33, 64, 65)]  # 496, 528, 2,016, 2,080 edges
    shapes += [I.random_graph(60, 0.3, 1, weight="int", dtype=dtype), I.path_graph(40, dtype)]
    none = np.zeros(0, np.int64)
    shapes += [I.csr_from_edges(n, none, none, none.astype(dtype)) for n in (1, 6)]
    graphs = [shapes[i] for i in rng.integers(0, len(shapes), 1500)]
    graphs += [_sparse(n, dtype) for n in larger]
    for ratio, levels in ((2, 1), (8, 1), (4, 2)):
        _batch_checked(ctx, graphs, ratio, "halving" if levels > 1 else "one", levels)


def test_batches_of_ten_thousand_graphs(ctx):
    """Of very many graphs a block looks at eight together, a warp at each but the larger ones: every
    graph is merged as the same graph in a small batch, which the oracle checks; an edge that leaves
    its graph is seen wherever it is."""
    from paper_2204_11757_gb300 import api
    shapes = [_sparse(2 + i % 4, np.float32) for i in range(96)]
    shapes[17], shapes[40], shapes[41] = (_sparse(n, np.float32) for n in (1500, 300, 1100))
    shapes[70] = _sparse(1023, np.float32)
    _batch_checked(ctx, shapes, 2, "one", 1)
    small = I.batch_of(shapes)
    lift, gpc, _ = ctx.coarsen_batched(api.CSR.from_graph(small.graph),
                                       torch.from_numpy(small.graph_ptr).cuda(), 2, levels=1)
    g, n, nnz, n_c = small.graph, small.graph.n, small.graph.col.shape[0], int(gpc[-1])
    for reps in (100, 127):  # 9,600 and 12,192 graphs
        big = api.CSR.from_numpy(
            np.r_[0, (g.rowptr[1:][None, :] + nnz * np.arange(reps)[:, None]).ravel()],
            (g.col[None, :] + n * np.arange(reps)[:, None]).ravel().astype(np.int32),
            np.tile(g.w, reps))
        gp = np.r_[0, (small.graph_ptr[1:][None, :] + n * np.arange(reps)[:, None]).ravel()]
        want = (lift.cpu().numpy()[None, :] + n_c * np.arange(reps)[:, None]).ravel()
        for split in (None, 17, 40 + 96 * (reps - 1)):  # the graph divided in two: its edges leave it
            ptr = gp if split is None else np.r_[gp[:split + 1], gp[split] + 200, gp[split + 1:]]
            ctx.time_kernel("*")
            try:
                blift, bgpc, _ = ctx.coarsen_batched(big, torch.from_numpy(ptr).cuda(), 2, levels=1)
                prof = ctx.kernel_profile()
            finally:
                ctx.time_kernel(None)
            assert any("k_select_small" in k for k in prof) == (split is None)
            if split is None:
                assert np.array_equal(blift.cpu().numpy(), want)
                assert int(bgpc[-1]) == n_c * reps


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("L", [257, 1056, 1057, 5000, 65536, 65537])
def test_long_sums_of_any_terms(ctx, dtype, L):
    """A caller's own weights: of any sign, infinite, NaN, subnormal, and of few mantissa bits, whose
    additions are ties; left to right, as numpy accumulates."""
    rng = np.random.default_rng(L)
    top, low = (1e306, 1e-310) if dtype == np.float64 else (1e36, 1e-41)
    one_inf, opposite, nan = (np.ones(L) for _ in range(3))
    one_inf[L // 2] = np.inf
    opposite[[L // 3, L // 2]] = np.inf, -np.inf
    nan[L // 2] = np.nan
    late = rng.uniform(0.5, 2.0, L)
    late[-3] = -3.0 * L
    with np.errstate(all="ignore"):
        data = [rng.standard_normal(L), -rng.uniform(0.5, 2.0, L), -np.zeros(L), late,
                np.where(rng.random(L) < 0.01, -1, 1) * rng.uniform(0.5, 2.0, L),
                rng.uniform(0, 1, L).astype(np.float16), rng.uniform(0, 1, L) * low,
                rng.uniform(0.5, 1, L) * top, one_inf, opposite, nan,
                np.resize([1.0, 2.0 ** -24, 3 * 2.0 ** -24, 2.0 ** -53, 3 * 2.0 ** -53], L),
                rng.integers(0, 2, L) * 0.5 + rng.integers(0, 3, L) * 2.0 ** 30]
        perm = torch.from_numpy(rng.permutation(L + 40).astype(np.int32)).cuda()
        seg = torch.tensor([0, 40, L + 40], dtype=torch.int32).cuda()
        for d in data:
            w = np.empty(L + 40, dtype)
            w[perm.cpu().numpy()] = np.r_[np.ones(40), d].astype(dtype)
            ref = dtype(0) + np.add.accumulate(d.astype(dtype))[-1]
            a = ctx.contract_forward(perm, seg, 2, torch.from_numpy(w).cuda()).cpu().numpy()
            assert a[0] == 40
            assert _bits(a[1:]) == _bits(np.array([ref])) or (np.isnan(a[1]) and np.isnan(ref))


@pytest.mark.parametrize("F", [1, 2, 3, 40, 130])
def test_pooled_gradients_of_any_size(ctx, F):
    """Binary64 gradients are divided by one reciprocal per row where a lane has several: the same
    quotients as IEEE division, zeros, subnormals, huge and infinite values among them."""
    rng = np.random.default_rng(F)
    lift = rng.permutation(np.repeat(np.arange(40), np.arange(1, 41))).astype(np.int32)
    g = rng.standard_normal((40, F)) * np.exp2(rng.integers(-1070, 1020, (40, F)))
    g.ravel()[::7] = rng.choice([0.0, -0.0, np.inf, -np.inf, 5e-324, 1.7e308], g.ravel()[::7].shape)
    gx = ctx.pool_features_backward(torch.from_numpy(lift).cuda(), 40, torch.from_numpy(g).cuda())
    ref = g[lift] / np.arange(1, 41)[lift][:, None].astype(np.float64)
    assert np.array_equal(_bits(gx.cpu().numpy()), _bits(ref))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_batches_that_are_not_block_diagonal_against_the_merge_loop(ctx, dtype):
    """The launches over all graphs on a batch with edges between graphs: of the minimum spanning forest
    of the whole batch, each graph's lightest edges (an edge belongs to its smaller end's graph) up
    to its own merges, found here by the merge loop itself."""
    from paper_2204_11757_gb300 import api
    a, c = _sparse(3000, dtype), _sparse(5000, dtype)
    eu = np.concatenate([a.eu, 3000 + c.eu, [17, 2999]])
    ev = np.concatenate([a.ev, 3000 + c.ev, [3001, 7000]])
    w = np.concatenate([a.w_und, c.w_und, np.full(2, 1.5, dtype)]).astype(dtype)
    g, gp, ratio = I.csr_from_edges(8000, eu, ev, w), np.array([0, 3000, 8000]), 4
    assert g.m <= 65536  # one slab: the whole batch's forest

    def find(p, x):
        while p[x] != x:
            p[x] = p[p[x]]
            x = p[x]
        return x

    forest, merged = list(range(g.n)), list(range(g.n))
    left = [n - max(1, n // ratio) for n in np.diff(gp)]
    for e in np.lexsort((np.arange(g.m), O.score(g))):
        u, v = int(g.eu[e]), int(g.ev[e])
        ru, rv = find(forest, u), find(forest, v)
        if ru == rv:
            continue
        forest[max(ru, rv)] = min(ru, rv)
        b = 0 if u < 3000 else 1
        if left[b] > 0:
            left[b] -= 1
            ru, rv = find(merged, u), find(merged, v)
            merged[max(ru, rv)] = min(ru, rv)
    root = np.array([find(merged, x) for x in range(g.n)])
    is_root = root == np.arange(g.n)
    ids = np.r_[0, np.cumsum(is_root)]
    lift, gpc, _ = ctx.coarsen_batched(api.CSR.from_graph(g), torch.from_numpy(gp).cuda(), ratio,
                                       levels=1)
    assert np.array_equal(lift.cpu().numpy(), ids[root])
    assert np.array_equal(gpc.cpu().numpy(), ids[gp])
