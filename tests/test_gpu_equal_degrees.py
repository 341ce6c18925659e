"""Of picked rows with many entries a few are recounted first, and vertices whose
bound is not above the largest degree found are left out.  Cliques of one size and
of nearly one size, some joined to each other, and rings, with small and large eps:
lists of more and of less than 24576 entries per block, by the whole GPU and by one
block.  Labels, rounds and every round's statistics equal the oracle's; exact."""
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


def _cliques(gg, count, size, spread, chords):
    rng = np.random.default_rng(count)
    sizes = size + rng.integers(0, spread + 1, count)
    start = np.concatenate([[0], np.cumsum(sizes)])
    n = int(start[-1])
    u, v = [rng.integers(0, n, chords)], [rng.integers(0, n, chords)]
    for c in range(count):
        i, j = np.triu_indices(sizes[c], 1)
        u.append(start[c] + i)
        v.append(start[c] + j)
    u, v = np.concatenate(u), np.concatenate(v)
    relabel = rng.permutation(n).astype(np.int32)
    return gg.from_edges(n, relabel[u[u != v]], relabel[v[u != v]])


@pytest.mark.parametrize("count, size, spread, chords", [(300, 100, 0, 0), (200, 250, 0, 0), (200, 240, 20, 0),
                                                         (400, 100, 3, 5000), (4000, 12, 0, 0), (50, 1100, 2, 100)])
def test_equal_degrees_equal_oracle(cc, gg, ora, count, size, spread, chords):
    g = _cliques(gg, count, size, spread, chords)
    with cc.Graph(g.off, g.col) as graph:
        want = {}
        for algo, a in (("c4", 1), ("cw", 2)):
            for eps in (0.02, 0.5):
                olab, orr, _, ost = ora.rounds(g.off, g.col, ora.permutation(g.n, 4), a, eps, 1, stats_cap=100_000)
                want[algo, eps] = (orr, ora.disagreements(g.off, g.col, olab))
                lab, r, d, st = graph.cluster(algo, eps, 4, stats_cap=100_000)
                assert np.array_equal(lab, olab) and (r, d) == want[algo, eps], (algo, eps)
                for f in STAT_FIELDS:
                    assert np.array_equal(st[f], ost[f]), (algo, eps, f)
        if g.n <= 65_536:
            with cc.Server() as server:          # one block per request
                tickets = {k: server.submit(graph, k[0], k[1], 4) for k in want}
                for k, t in tickets.items():
                    assert server.wait(t)[:2] == want[k], k
