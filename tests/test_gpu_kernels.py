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
