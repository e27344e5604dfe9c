"""The captured schedule of a repeated coarsening when other calls on the context come between:
it is replayed only while everything it takes for granted still holds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2204_11757_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as ge
    ge.build()
    from paper_2204_11757_gb300 import api as A
    return A


class Repeated:
    """One coarsening call made again and again on one context."""

    def __init__(self, api, ctx, graph, levels):
        self.ctx, self.csr, self.levels = ctx, api.CSR.from_graph(graph), levels
        self.ref, self.total = O.coarsen(graph, 1 << levels, "halving")

    def run(self, replayed):
        lift, n_c, _ = self.ctx.coarsen(self.csr, self.ref[-1].target, levels=self.levels)
        assert self.ctx.last_call_replayed == replayed
        assert n_c == self.ref[-1].n_c
        assert np.array_equal(lift.cpu().numpy(), self.total)
        for lv, r in zip(self.ctx.levels(), self.ref):
            assert np.array_equal(lv.w_c.cpu().numpy().view(np.uint64),
                                  r.coarse.graph.w.view(np.uint64))
            assert np.array_equal(lv.emap.cpu().numpy(), r.coarse.emap)


def _mesh(nx, ny, seed):
    return I.tri_mesh_2d(nx, ny, seed, jitter=0.3, weight="inv_len", dtype=np.float64)


def _other_call(api, ctx, op, g):
    csr = api.CSR.from_graph(g)
    if op == "contract":
        lift = (np.arange(g.n) // 2).astype(np.int32)
        lv = ctx.contract(csr, torch.from_numpy(lift).cuda(), int(lift[-1]) + 1)
        assert np.array_equal(lv.emap.cpu().numpy(), O.contract(g, lift, int(lift[-1]) + 1).emap)
    elif op == "score":
        assert np.array_equal(ctx.score(csr).cpu().numpy().view(np.uint64),
                              O.score(g).view(np.uint64))
    elif op == "select":
        f = O.score(g)
        lift, _, _, _ = ctx.select_merges(csr, torch.from_numpy(f).cuda(), g.n // 2)
        assert np.array_equal(lift.cpu().numpy(), O.coarsen_level(g, g.n // 2).lift)
    else:
        f = np.random.default_rng(1).random(g.m)
        order = ctx.sort_fitness(torch.from_numpy(f).cuda()).cpu().numpy()
        assert np.array_equal(order, np.argsort(f, kind="stable"))


@pytest.mark.parametrize("op", ["contract", "score", "select", "sort"])
def test_a_larger_call_between_drops_the_captured_schedule(api, op):
    """The larger call grows workspace blocks, so the addresses inside the captured schedule are
    no longer the context's: the next call runs host-driven and is captured anew."""
    with api.Context() as c:
        r = Repeated(api, c, _mesh(60, 51, 2), 3)
        for replayed in (False, True, True):
            r.run(replayed)
        _other_call(api, c, op, _mesh(180, 170, 3))
        for replayed in (False, True, True):
            r.run(replayed)
        _other_call(api, c, op, _mesh(181, 170, 4))
        _other_call(api, c, op, _mesh(50, 40, 5))
        for replayed in (False, True):
            r.run(replayed)


@pytest.mark.parametrize("op", ["contract", "score", "select", "sort"])
def test_a_smaller_call_between_keeps_the_captured_schedule(api, op):
    with api.Context() as c:
        r = Repeated(api, c, _mesh(181, 170, 4), 4)
        r.run(False)
        r.run(True)
        _other_call(api, c, op, _mesh(60, 51, 2))
        r.run(True)
        _other_call(api, c, op, _mesh(50, 40, 5))
        r.run(True)


def _selection_gives_up(ctx, csr, f, n_c):
    """A stand-alone selection of one large graph whose grid barrier gives up: the wait limit is
    raised from one poll until the selection's kernel is reached (at small limits the scans before
    it give up first); a phase of it takes longer than a few polls."""
    from paper_2204_11757_gb300 import native as N
    stopped = 0
    for limit in (1, 2, 4, 8, 12, 16, 24, 32) * 4:
        ctx.set_wait_limit(limit)
        ctx.time_kernel("k_select_coop")
        try:
            ctx.select_merges(csr, f, n_c)
            code = 0
        except N.SpcError as e:
            code = e.status
        finally:
            ctx.set_wait_limit(0)
        reached = ctx.kernel_time()[0] > 0
        ctx.time_kernel(None)
        assert code in (0, -7)  # SPC_ERR_TIMEOUT
        stopped += 1 if reached and code == -7 else 0
        if stopped == 3:
            return
    raise AssertionError("no selection reached its grid barrier and gave up")


@pytest.mark.parametrize("recorded_only", [True, False])
def test_a_selection_that_gave_up_leaves_a_repeated_call_right(api, recorded_only):
    """A grid barrier that gives up leaves the selection's counters and its barrier word nonzero;
    the next call clears them, whether it runs host-driven, is captured or is replayed."""
    g = _mesh(181, 170, 4)
    assert g.n > 8192  # past the one-CTA selection
    with api.Context() as c:
        r = Repeated(api, c, g, 4)
        r.run(False)
        if not recorded_only:
            r.run(True)
        f = torch.from_numpy(O.score(g)).cuda()
        _selection_gives_up(c, r.csr, f, g.n // 3)
        r.run(True)
        r.run(True)
        _selection_gives_up(c, r.csr, f, g.n // 3)
        lift, _, n_c, _ = c.select_merges(r.csr, f, g.n // 2)
        assert n_c == g.n // 2
        assert np.array_equal(lift.cpu().numpy(), r.ref[0].lift)
        r.run(True)


@pytest.mark.parametrize("device", ["cuda", "cpu"])
@pytest.mark.parametrize("levels", [1, 3])
def test_a_selection_keeps_the_last_coarsening(api, levels, device):
    """The retained levels, and a result taken from them, hold until the next coarsening call,
    whatever graph a stand-alone selection runs on in between."""
    g, big = _mesh(60, 51, 2), _mesh(181, 170, 4)
    with api.Context() as c:
        r = Repeated(api, c, g, levels)
        r.run(False)
        with_mass = c.take_result().tensors()
        f = torch.from_numpy(O.score(big)).to(device)
        lift, _, _, _ = c.select_merges(api.CSR.from_graph(big, device=device), f, big.n // 2)
        assert np.array_equal(lift.cpu().numpy(), O.coarsen_level(big, big.n // 2).lift)
        for lv, x in zip(c.levels(), r.ref):
            assert np.array_equal(lv.lift.cpu().numpy(), x.lift)
            assert np.array_equal(lv.score.cpu().numpy().view(np.uint64), x.f.view(np.uint64))
            assert np.array_equal(lv.emap.cpu().numpy(), x.coarse.emap)
        again = c.take_result().tensors()
        assert with_mass.keys() == again.keys()
        for name, t in with_mass.items():
            assert (t is None and again[name] is None) or torch.equal(t, again[name]), name


def test_pooling_between_keeps_the_captured_schedule(api):
    """A training step coarsens and pools: pooling on growing sizes, by both of its routes, touches no
    block that a coarsening uses."""
    with api.Context() as c:
        r = Repeated(api, c, _mesh(181, 170, 4), 4)
        r.run(False)
        r.run(True)
        for n, n_c in ((3000, 900), (90000, 20000), (300000, 3)):
            lift = (np.arange(n) % n_c).astype(np.int32)
            x = np.random.default_rng(n).standard_normal((n, 5))
            xc = c.pool_features(torch.from_numpy(lift).cuda(), n_c, torch.from_numpy(x).cuda())
            assert np.array_equal(xc.cpu().numpy(), O.pool_features(lift, n_c, x))
            r.run(True)
