"""Selection and attachment of a window run in one pass: blocks attach while
others still count, so a vertex may be reached before its own block makes it
active, C4 tells blocked actives by the ranks of pi, and rows of more than 8192
entries are left to a second pass.  Windows around the inline limit and of
several tiles per block, rows around 8192 that are still alive when windows are
long, removal tags that come round again (more than 15 rounds).  Labels, rounds
and statistics equal the oracle's; exact."""
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


def _ring_and_hubs(gg, n, half, hubs, leaves, seed):
    """A ring of n vertices (each joined to the `half` next ones) and hubs whose
    shared leaves fall to the first hub that becomes a center; every hub also
    knows three vertices of the ring, so the others stay with long rows."""
    rng = np.random.default_rng(seed)
    v = np.arange(n)
    src = [np.repeat(v, half)]
    dst = [(np.repeat(v, half) + np.tile(np.arange(1, half + 1), n)) % n]
    for h in range(hubs):
        length = leaves - hubs // 2 + h
        src += [np.full(length, n + h), np.full(3, n + h)]
        dst += [n + hubs + np.arange(length), rng.choice(n, 3, replace=False)]
    total = n + hubs + leaves + hubs
    relabel = rng.permutation(total).astype(np.int32)
    return gg.from_edges(total, relabel[np.concatenate(src)], relabel[np.concatenate(dst)])


@pytest.mark.parametrize("n, half, hubs, leaves", [(1500, 1, 0, 0), (9000, 3, 4, 60), (60_000, 2, 10, 8189),
                                                   (400_000, 1, 3, 20_000), (700_001, 2, 0, 0)])
def test_fused_selection_equals_oracle(cc, gg, ora, n, half, hubs, leaves):
    g = _ring_and_hubs(gg, n, half, hubs, leaves, n)
    with cc.Graph(g.off, g.col) as graph:
        for algo, a, eps in (("cw", 2, 0.1), ("cw", 2, 0.9), ("cw-est", 4, 0.9), ("c4", 1, 0.1), ("c4", 1, 0.9),
                             ("c4-est", 3, 0.9)):
            order = ora.permutation(g.n, 11)
            olab, orr, _, ost = (ora.rounds_bsp(g.off, g.col, order, a - 2, eps, 11, stats_cap=1_000_000) if a > 2 else
                                 ora.rounds(g.off, g.col, order, a, eps, 1, stats_cap=1_000_000))
            lab, r, d, st = graph.cluster(algo, eps, 11, stats_cap=1_000_000)
            assert np.array_equal(lab, olab) and r == orr and d == ora.disagreements(g.off, g.col, olab), (algo, eps)
            for f in STAT_FIELDS:
                assert np.array_equal(st[f], ost[f]), (algo, eps, f)


def test_second_window_of_a_round_in_small_teams(cc, gg, ora):
    """Teams of two blocks fuse windows of up to 4096 entries.  In the last rounds
    of 7000 cliques a window of that length holds a handful of alive vertices;
    when it holds too few, the round goes on with a longer one whose vertices the
    first window's centers may have reached."""
    i, j = np.triu_indices(10, 1)
    base = (np.arange(7000) * 10)[:, None]
    g = gg.from_edges(70_000, (base + i).ravel(), (base + j).ravel())
    default = cc.get_batch_tuning()
    with cc.Graph(g.off, g.col) as graph:
        try:
            cc.set_batch_tuning(dict(default, batch_team_blocks=2))
            for first in range(0, 600, 150):
                D, R = cc.batch_jobs([graph], "cw", 0.5, np.array([first], np.uint64), 150)
                for q in range(150):
                    lab, r, _, _ = ora.rounds(g.off, g.col, ora.permutation(g.n, first + q), 2, 0.5, 1)
                    assert R[0, q] == r and D[0, q] == ora.disagreements(g.off, g.col, lab), first + q
        finally:
            cc.set_batch_tuning(default)
