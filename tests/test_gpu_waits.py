"""Waits that give up, over every entry point (needs a GPU).  The context's wait limit is lowered, so
that the look-backs of the scans, the sorts and the contraction's ranking, the union-find walks and
the grid barriers of the selection reach it.  A call then returns SPC_ERR_TIMEOUT or, when every wait
of it was short enough, its result; the next call with the default limit is exact.  Nothing here
faults or hangs the GPU: while a limit is set the calls stop after a kernel whose wait gave up, so
nothing indexes with what it left unwritten."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2204_11757_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

LIMITS = (1, 2, 3, 5, 9, 17, 40, 200, 5000)


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as ge
    ge.build()
    from paper_2204_11757_gb300 import api as A
    return A


def _sparse(n, degree, dtype, seed):
    rng = np.random.default_rng(seed)
    e = rng.integers(0, n, (2, n * degree // 2))
    q = rng.permutation(n)
    e = np.concatenate([e, [q[:-1], q[1:]]], axis=1)
    lo, hi = e.min(axis=0), e.max(axis=0)
    key = np.unique((lo * n + hi)[lo != hi])
    w = np.ones(key.size) if dtype == np.int32 else rng.uniform(0.1, 2.0, key.size)
    return I.csr_from_edges(n, key // n, key % n, w.astype(dtype))


def _hubs(dtype):
    return I.hub_graph(20000, [9000, 4000, 700, 300], 3, dtype=dtype, base_p=0.0003)


def _flat(r):
    """The arrays of a result, in order."""
    if isinstance(r, torch.Tensor):
        return [r.cpu().numpy()]
    if isinstance(r, (list, tuple)):
        return [a for x in r for a in _flat(x)]
    return [np.asarray(r)]


def _coarsen(graph, levels, **options):
    def make(api, c):
        csr, n_c = api.CSR.from_graph(graph()), max(1, graph().n >> levels)
        return lambda: c.coarsen(csr, n_c, levels=levels, **options)
    return make


def _batch(sizes, dtype):
    def make(api, c):
        b = I.batch_of([_sparse(n, 6, dtype, n) for n in sizes])
        csr, gp = api.CSR.from_graph(b.graph), torch.from_numpy(b.graph_ptr).cuda()
        return lambda: c.coarsen_batched(csr, gp, 4, levels=2)
    return make


def _contract(n_c, dtype):
    def make(api, c):
        g = _sparse(60000, 8, dtype, 1)
        lift = np.random.default_rng(n_c).integers(0, n_c, g.n)
        lift[:n_c] = np.arange(n_c)
        csr, lt = api.CSR.from_graph(g), torch.from_numpy(lift.astype(np.int32)).cuda()

        def run():
            lv = c.contract(csr, lt, n_c)
            return lv.emap, lv.a_und, lv.self_mass, lv.rowptr_c, lv.col_c, lv.w_c
        return run
    return make


def _select(dtype):
    def make(api, c):
        g = _sparse(60000, 8, dtype, 2)
        csr, f = api.CSR.from_graph(g), torch.from_numpy(O.score(g)).cuda()
        return lambda: c.select_merges(csr, f, 20000)
    return make


def _weights(L):
    def make(api, c):
        seg = torch.tensor([0, 300, 300 + L], dtype=torch.int32).cuda()
        perm = torch.from_numpy(np.random.default_rng(L).permutation(300 + L).astype(np.int32)).cuda()
        w = torch.from_numpy(np.random.default_rng(1).uniform(0.1, 2.0, 300 + L)).cuda()
        return lambda: c.contract_forward(perm, seg, 2, w)
    return make


def _pool(n_c):
    def make(api, c):
        rng = np.random.default_rng(n_c)
        lift = torch.from_numpy(rng.integers(0, n_c, 200000).astype(np.int32)).cuda()
        x = torch.from_numpy(rng.standard_normal((200000, 3))).cuda()
        return lambda: c.pool_features(lift, n_c, x)
    return make


CALLS = {
    "coarsen_f32": _coarsen(lambda: _sparse(60000, 12, np.float32, 5), 4),
    "coarsen_f64": _coarsen(lambda: _sparse(60000, 6, np.float64, 6), 5),
    "coarsen_i32": _coarsen(lambda: I.tri_mesh_2d(300, 201, 1), 4),
    "coarsen_reordered": _coarsen(lambda: _sparse(60000, 12, np.float32, 5), 3, reorder=True),
    "coarsen_hubs_f32": _coarsen(lambda: _hubs(np.float32), 4),
    "coarsen_hubs_f64": _coarsen(lambda: _hubs(np.float64), 4),
    "coarsen_hubs_reordered": _coarsen(lambda: _hubs(np.float64), 2, reorder=True),
    "coarsen_star": _coarsen(lambda: I.star_ties(17, np.float64, chords=30000), 2),
    "batch_small": _batch([9000, 300, 5000] * 4, np.float32),
    "batch_general": _batch([30000, 300, 5000], np.float64),
    "contract_short_buckets": _contract(20000, np.float32),
    "contract_huge_buckets": _contract(9, np.float64),
    "select_f32": _select(np.float32),
    "select_f64": _select(np.float64),
    "weights_streamed": _weights(60000),
    "weights_tables": _weights(300000),
    "pool_short": _pool(50000),
    "pool_hubs": _pool(3),
}


@pytest.mark.parametrize("name", list(CALLS))
def test_calls_whose_waits_give_up(api, name):
    from paper_2204_11757_gb300 import native as N
    with api.Context() as c:
        run = CALLS[name](api, c)
        want = _flat(run())
        run()
        codes = []
        for limit in LIMITS:
            c.set_wait_limit(limit)
            try:
                got = _flat(run())
                codes.append(0)
            except N.SpcError as e:
                codes.append(e.status)
            finally:
                c.set_wait_limit(0)
            assert codes[-1] in (0, -7), codes  # SPC_ERR_TIMEOUT
            if codes[-1] == 0:
                assert all(np.array_equal(a, b) for a, b in zip(got, want))
        for _ in range(3):
            got = _flat(run())
            assert len(got) == len(want)
            assert all(np.array_equal(a, b) for a, b in zip(got, want))


def test_the_rankings_look_back_gives_up(api):
    """4,096 nodes, nothing merged, 190 tiles of 1,024 edges: the scans of the call run in one CTA, so
    the ranking's look-back is the only wait that can give up."""
    from paper_2204_11757_gb300 import native as N
    g = _sparse(4096, 96, np.float64, 7)
    lift = torch.arange(g.n, dtype=torch.int32).cuda()
    with api.Context() as c:
        csr = api.CSR.from_graph(g)
        codes = []
        for _ in range(20):
            c.set_wait_limit(1)
            c.time_kernel("k_bucket_rank_inter")
            try:
                c.contract(csr, lift, g.n)
                codes.append(0)
            except N.SpcError as e:
                codes.append(e.status)
            finally:
                c.set_wait_limit(0)
            assert c.kernel_time()[0] == 1
            c.time_kernel(None)
            lv = c.contract(csr, lift, g.n)
            assert np.array_equal(lv.rowptr_c.cpu().numpy(), g.rowptr)
            assert np.array_equal(lv.col_c.cpu().numpy(), g.col)
            assert np.array_equal(lv.w_c.cpu().numpy().view(np.uint64), g.w.view(np.uint64))
        assert set(codes) <= {0, -7} and -7 in codes, codes
