"""Batched jobs get teams of one block to batch_team_blocks by their sizes and
their number, and a team whose queue is dry takes jobs of the smaller classes.
Numbers of jobs around the blocks of the GPU, equal and mixed sizes: every job
equals the same clustering run by itself; exact integers."""
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


SMALL, MEDIUM, LARGE = 300, 20_000, 150_000
# graphs (vertices, how many), orders each
BATCHES = [([(1, 1)], 1), ([(SMALL, 1)], 1), ([(LARGE, 1)], 3), ([(MEDIUM, 3), (SMALL, 5)], 2),
           ([(SMALL, 19)], 8), ([(SMALL, 151)], 2), ([(SMALL, 101)], 3), ([(SMALL, 61)], 5),
           ([(LARGE, 1), (MEDIUM, 4), (2, 3), (SMALL, 60)], 6), ([(LARGE, 2), (MEDIUM, 40), (SMALL, 100)], 5)]


@pytest.mark.parametrize("team_blocks", [2, 8, 12])
@pytest.mark.parametrize("sizes, orders", BATCHES, ids=[str(b) for b in BATCHES])
def test_every_job_equals_its_own_clustering(cc, gg, sizes, orders, team_blocks):
    default = cc.get_batch_tuning()
    n = [m for m, count in sizes for _ in range(count)]
    made = {m: [gg.chung_lu(m, min(12.0, m / 8), seed=3 + s) for s in range(2)] if m > 2 else
            [gg.from_edges(m, np.zeros(m - 1), np.ones(m - 1))] * 2 for m, _ in sizes}
    graphs = [cc.Graph(made[m][i % 2].off, made[m][i % 2].col) for i, m in enumerate(n)]
    rng = np.random.default_rng(len(n))
    graphs = [graphs[i] for i in rng.permutation(len(graphs))]
    seeds = np.arange(len(graphs), dtype=np.uint64) % 7 * 16
    try:
        cc.set_batch_tuning(dict(default, batch_team_blocks=team_blocks))
        known = {}
        for algo in ("cw", "c4"):
            D, R = cc.batch_jobs(graphs, algo, 0.5, seeds, orders)
            for i, g in enumerate(graphs):
                for j in range(orders):
                    key = (g.n, g.nnz, algo, int(seeds[i]) + j)
                    if key not in known:
                        _, r, d = g.cluster(algo, 0.5, int(seeds[i]) + j)
                        known[key] = (d, r)
                    assert (D[i, j], R[i, j]) == known[key], key
    finally:
        cc.set_batch_tuning(default)
        for g in graphs:
            g.close()
