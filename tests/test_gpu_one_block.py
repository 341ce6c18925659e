"""Jobs that one block runs by itself.  Its heavy list has no limit: lists above
2048 vertices are looked at 2048 at a time, and after every step the whole block
decides whether to recount.  Lists of equal degrees around one and two steps
(2047 .. 2049, 4095 .. 4097), around the length from which they are not made
inside the barrier (8192), and of many steps; few and many vertices of the
largest degree among them.  Labels, rounds and disagreements equal the oracle's;
exact integers."""
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


def _ring(gg, n, half, chords):
    """Every vertex joined to the `half` next ones, `chords` random edges more."""
    rng = np.random.default_rng(n)
    v = np.arange(n)
    u = np.concatenate([np.repeat(v, half), rng.integers(0, n, chords)])
    w = np.concatenate([(np.repeat(v, half) + np.tile(np.arange(1, half + 1), n)) % n, rng.integers(0, n, chords)])
    keep = u != w
    relabel = rng.permutation(n).astype(np.int32)
    return gg.from_edges(n, relabel[u[keep]], relabel[w[keep]])


@pytest.mark.parametrize("n, half, chords", [(2047, 2, 0), (2048, 2, 0), (2049, 2, 0), (4095, 1, 0), (4097, 3, 0),
                                             (8191, 2, 0), (8193, 2, 0), (30_000, 4, 0), (65_536, 2, 0),
                                             (30_000, 4, 30), (30_000, 2, 15_000), (65_535, 8, 300_000)])
def test_long_heavy_lists_equal_oracle(cc, gg, ora, n, half, chords):
    import torch
    g = _ring(gg, n, half, chords)
    reqs = [(algo, a, eps, seed) for algo, a in (("c4", 1), ("cw", 2)) for eps in (0.05, 0.5, 1.0) for seed in (1, 8)]
    labels = torch.full((len(reqs), n), -1, dtype=torch.int32, device="cuda")
    with cc.Graph(g.off, g.col) as graph:
        with cc.Server() as server:              # one block for every request of up to 65536 vertices
            tickets = [server.submit(graph, algo, eps, seed, labels_out=labels[i])
                       for i, (algo, _, eps, seed) in enumerate(reqs)]
            done = [server.wait(t)[:2] for t in tickets]
        torch.cuda.synchronize()
    got = labels.cpu().numpy()
    for i, (algo, a, eps, seed) in enumerate(reqs):
        lab, rounds, _, _ = ora.rounds(g.off, g.col, ora.permutation(n, seed), a, eps, 1)
        assert np.array_equal(got[i], lab), reqs[i]
        assert done[i] == (rounds, ora.disagreements(g.off, g.col, lab)), reqs[i]


def test_batch_of_one_block_teams_equals_oracle(cc, gg, ora):
    """As many equal jobs as the GPU has blocks: every one gets a single block."""
    n = 12_000
    g = _ring(gg, n, 3, 4000)
    with cc.Graph(g.off, g.col) as graph:
        for algo, a in (("c4", 1), ("cw", 2)):
            D, R = cc.batch_jobs([graph], algo, 0.5, np.array([5], np.uint64), 320)
            for j in range(0, 320, 4):
                lab, rounds, _, _ = ora.rounds(g.off, g.col, ora.permutation(n, 5 + j), a, 0.5, 1)
                assert R[0, j] == rounds and D[0, j] == ora.disagreements(g.off, g.col, lab), (algo, j)
