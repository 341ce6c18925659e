"""Windows whose tiles hold rows of more than 8192 entries beside shorter ones.
The block lists the short rows itself and leaves the long ones to the grid, and
both are booked in the same tallies of the round.  2500 hubs share 8200 leaves;
once one of them is a center the leaves are gone, and the other hubs stay with
long rows of few alive entries, some in every tile of windows of thousands of
vertices.  Labels, rounds and statistics equal the oracle's; exact integers (a
round whose tallies do not add up ends in an error)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STAT_FIELDS = ("n_alive", "delta", "k", "centers", "removed", "blocked")
RING, HUBS, LEAVES = 200_000, 2500, 8200


@pytest.fixture(scope="module")
def cc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1507_05086_gb300 as cc
    cc.load()
    return cc


def test_long_rows_in_every_tile_equal_oracle(cc, gg, ora):
    rng = np.random.default_rng(1)
    v = np.arange(RING)
    hub = RING + np.arange(HUBS)
    leaf = RING + HUBS + np.arange(LEAVES)
    src = [np.repeat(v, 2), np.repeat(hub, LEAVES), np.repeat(hub, 3)]
    dst = [(np.repeat(v, 2) + np.tile([1, 2], RING)) % RING, np.tile(leaf, HUBS), rng.integers(0, RING, 3 * HUBS)]
    n = RING + HUBS + LEAVES
    relabel = rng.permutation(n).astype(np.int32)
    g = gg.from_edges(n, relabel[np.concatenate(src)], relabel[np.concatenate(dst)])
    kind = np.zeros(n, np.int8)
    kind[relabel[hub]], kind[relabel[leaf]] = 1, 2
    # orders in which a hub comes well before the first leaf (rounds of 24 at first)
    orders = []
    for seed in range(1000):
        order = ora.permutation(n, seed)
        first = [int(np.argmax(kind[order] == k)) for k in (1, 2)]
        if first[0] + 60 < first[1]:
            orders.append((seed, order))
            if len(orders) == 3:
                break
    assert len(orders) == 3
    with cc.Graph(g.off, g.col) as graph:
        for seed, order in orders:
            for algo, a in (("c4", 1), ("cw", 2)):
                olab, orr, _, ost = ora.rounds(g.off, g.col, order, a, 0.9, 1, stats_cap=100_000)
                # the case is there: hubs are left for long windows
                assert int((ost["k"] > 10_000).sum()) >= 1 and ost["delta"][ost["k"] > 10_000].max() < 100
                lab, r, d, st = graph.cluster(algo, 0.9, seed, stats_cap=100_000)
                assert np.array_equal(lab, olab) and r == orr, (algo, seed)
                assert d == ora.disagreements(g.off, g.col, olab), (algo, seed)
                for f in STAT_FIELDS:
                    assert np.array_equal(st[f], ost[f]), (algo, seed, f)
