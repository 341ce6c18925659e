"""Delta of every round is the exact largest residual degree, although degrees
are recounted only where a vertex can hold the maximum.  Graphs at the sizes
where that can go wrong: as many equal degrees as the coordinator looks at by
itself (8192) and as every block lists (512), one more and one less, rows at
the length from which the whole grid counts them (1024), windows around the
selection's inline limit, degrees that fall far below their bounds.  Labels,
rounds and every round's statistics equal the oracle's; exact integers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STAT_FIELDS = ("n_alive", "delta", "k", "centers", "removed", "blocked")


@pytest.fixture(scope="module")
def cc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1507_05086_gb300 as cc
    cc.load()
    return cc


def _ring(n, half):
    """Every vertex joined to the `half` next ones: all degrees equal."""
    v = np.arange(n)
    return n, np.repeat(v, half), (np.repeat(v, half) + np.tile(np.arange(1, half + 1), n)) % n


def _stars(count, leaves):
    """Disjoint stars of near-equal size: nothing but hub rows can hold Delta."""
    size = leaves + (np.arange(count) % 3) - 1
    n = int(count + size.sum())
    return n, np.repeat(np.arange(count), size), np.arange(count, n)


def _cliques(count, size):
    """Disjoint cliques: a center's round takes whole blocks of equal degrees away."""
    i, j = np.triu_indices(size, 1)
    base = (np.arange(count) * size)[:, None]
    return count * size, (base + i).ravel(), (base + j).ravel()


def _shared(hubs, length, n):
    """Hubs over the same leaves: attaching one hub's leaves empties all others."""
    leaves = hubs + np.arange(length)
    return n, np.repeat(np.arange(hubs), length), np.tile(leaves, hubs)


CASES = [("ring", _ring, a) for a in ((3, 1), (31, 2), (33, 2), (511, 3), (513, 3), (1025, 2), (8191, 2), (8193, 2),
                                      (30_011, 4))]
CASES += [("stars", _stars, a) for a in ((1, 1024), (7, 1025), (40, 1024), (600, 1025), (1100, 30))]
CASES += [("cliques", _cliques, a) for a in ((700, 12), (1, 300), (9000, 3))]
CASES += [("shared", _shared, a) for a in ((30, 1023, 4000), (30, 5000, 9000), (700, 900, 2000))]


@pytest.mark.parametrize("name, make, args", CASES, ids=["%s%s" % (n, a) for n, _, a in CASES])
def test_delta_equals_oracle(cc, gg, ora, name, make, args):
    n, u, v = make(*args)
    relabel = np.random.default_rng(n).permutation(n).astype(np.int32)
    g = gg.from_edges(n, relabel[u], relabel[v])
    with cc.Graph(g.off, g.col) as graph:
        for algo, a in (("c4", 1), ("cw", 2)):
            for eps in (0.05, 0.5, 1.0):
                order = ora.permutation(n, 3)
                olab, orr, _, ost = ora.rounds(g.off, g.col, order, a, eps, 1, stats_cap=1_000_000)
                lab, r, d, st = graph.cluster(algo, eps, 3, stats_cap=1_000_000)
                assert np.array_equal(lab, olab) and r == orr and d == ora.disagreements(g.off, g.col, olab), (algo, eps)
                for f in STAT_FIELDS:
                    assert np.array_equal(st[f], ost[f]), (algo, eps, f)
        D, R = cc.batch_jobs([graph], "cw", 0.5, np.array([3], np.uint64), 2)
        for j in range(2):
            lab, r, d = graph.cluster("cw", 0.5, 3 + j)
            assert D[0, j] == d and R[0, j] == r
