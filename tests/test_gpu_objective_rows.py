"""Which walk counts the edges inside clusters depends on how many upper entries
the rows have per unit of 32 (below 6: all entries in batches of 128; else units,
or rows with signatures above 2^24 vertices).  Rings of 1 to 9 neighbours on
either side, so that the upper parts lie around that line, below and above 2^24
vertices, with a hub row and isolated vertices between.  Exact integers."""
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


CASES = [(ring, n, half) for ring, n in ((19, 19), (127, 130), (4099, 9001), (70_001, 70_002))
         for half in (1, 2, 5, 6, 7, 9)] + [(200_003, 2**24 + 13, half) for half in (2, 9)]


@pytest.mark.parametrize("ring, n, half", CASES)
def test_objective_around_the_line(cc, gg, ora, ring, n, half):
    rng = np.random.default_rng(ring + half)
    place = np.sort(rng.choice(n, ring, replace=False))        # the others are isolated
    v = np.arange(ring)
    u, w = np.repeat(v, half), (np.repeat(v, half) + np.tile(np.arange(1, half + 1), ring)) % ring
    spokes = v[2::max(3, ring // 400)]
    u, w = np.concatenate([u, np.ones_like(spokes)]), np.concatenate([w, spokes])
    g = gg.from_edges(n, place[u].astype(np.int32), place[w].astype(np.int32))
    lab = np.arange(n, dtype=np.int32)
    blocks = lab.copy()
    blocks[place] = place[v - v % 11]                            # eleven neighbours each
    half_one = np.where(rng.random(n) < 0.5, n - 1, lab).astype(np.int32)
    with cc.Graph(g.off, g.col) as graph:
        for x in (lab, blocks, half_one, np.zeros(n, np.int32)):
            assert graph.disagreements(x) == ora.disagreements(g.off, g.col, x)
        for algo, a in (("cw", 2), ("c4", 1)):
            olab, rounds, _, _ = ora.rounds(g.off, g.col, ora.permutation(n, 7), a, 0.5, 1)
            labels, r, d = graph.cluster(algo, 0.5, 7)
            assert np.array_equal(labels, olab) and r == rounds and d == ora.disagreements(g.off, g.col, olab)
        labels, _, d = graph.cluster("c4-async", 0.5, 7)
        assert np.array_equal(labels, olab) and d == ora.disagreements(g.off, g.col, olab)
