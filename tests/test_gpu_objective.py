"""The objective reads every edge once, from the upper part of its lower end's
row, and graphs above 2^24 vertices compare 4-bit signatures of the cluster
ids before the ids: both against the oracle at the sizes where the row lists,
the warps' shared adds and the signature words can go wrong.  Exact integers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1507_05086_gb300 as cc
    cc.load()
    return cc


def _graph(gg, n, m, seed):
    """m random edges, the first and the last vertex isolated when there is
    room, one hub row that lies wholly above its vertex and one wholly below."""
    rng = np.random.default_rng(seed)
    lo, hi = (1, n - 1) if n > 4 else (0, n)
    u, v = rng.integers(lo, hi, m), rng.integers(lo, hi, m)
    if n > 4:
        spokes = np.arange(lo, hi, max(1, n // 3000))
        u = np.concatenate([u, np.full(spokes.size, lo), np.full(spokes.size, hi - 1)])
        v = np.concatenate([v, spokes, spokes])
    keep = u != v
    return gg.from_edges(n, u[keep].astype(np.int32), v[keep].astype(np.int32))


@pytest.mark.parametrize("n, m", [(1, 0), (2, 3), (7, 9), (31, 40), (33, 64), (129, 500), (4097, 60_000),
                                  (100_003, 700_000), (2**24, 300_000), (2**24 + 13, 300_000)])
def test_objective_equals_oracle(cc, gg, ora, n, m):
    g = _graph(gg, n, m, n)
    rng = np.random.default_rng(n + 1)
    labellings = [np.arange(n), np.full(n, n - 1), rng.integers(0, max(1, n // 50), n),
                  np.where(rng.random(n) < 0.4, n // 2, rng.integers(0, n, n))]   # one giant cluster, the rest spread
    with cc.Graph(g.off, g.col) as graph:
        for lab in labellings:
            lab = lab.astype(np.int32)
            assert graph.disagreements(lab) == ora.disagreements(g.off, g.col, lab)
        order = ora.permutation(n, 5)
        lab, _, d = graph.cluster("c4", 0.5, 5)
        assert np.array_equal(lab, ora.kwik(g.off, g.col, order))
        assert d == ora.disagreements(g.off, g.col, lab)
