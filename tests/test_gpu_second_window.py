"""A C4 round whose first window holds too few alive vertices goes on with a second
one: its actives are blocked by the first window's actives too, and the first one's
centers may have attached them already.  Teams of two blocks over 7000 cliques of
ten, whose last rounds have such windows, and the whole GPU over a graph whose
low ranks leave early; rounds, costs and statistics equal the oracle's; exact."""
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


def _cliques(gg, count, size):
    i, j = np.triu_indices(size, 1)
    base = (np.arange(count) * size)[:, None]
    return gg.from_edges(count * size, (base + i).ravel(), (base + j).ravel())


def test_c4_second_window_in_small_teams(cc, gg, ora):
    g = _cliques(gg, 7000, 10)
    default = cc.get_batch_tuning()
    with cc.Graph(g.off, g.col) as graph:
        try:
            cc.set_batch_tuning(dict(default, batch_team_blocks=2))
            for first in range(0, 600, 150):
                D, R = cc.batch_jobs([graph], "c4", 0.5, np.array([first], np.uint64), 150)
                for q in range(150):
                    lab, r, _, _ = ora.rounds(g.off, g.col, ora.permutation(g.n, first + q), 1, 0.5, 1)
                    assert R[0, q] == r and D[0, q] == ora.disagreements(g.off, g.col, lab), first + q
        finally:
            cc.set_batch_tuning(default)


@pytest.mark.parametrize("count, size", [(700, 40), (3000, 100), (20_000, 10)])
def test_windows_of_whole_gpu_rounds(cc, gg, ora, count, size):
    g = _cliques(gg, count, size)
    with cc.Graph(g.off, g.col) as graph:
        for seed in range(8):
            for algo, a in (("c4", 1), ("cw", 2)):
                olab, orr, _, ost = ora.rounds(g.off, g.col, ora.permutation(g.n, seed), a, 0.9, 1, stats_cap=100_000)
                lab, r, d, st = graph.cluster(algo, 0.9, seed, stats_cap=100_000)
                assert np.array_equal(lab, olab) and r == orr and d == ora.disagreements(g.off, g.col, olab)
                for f in STAT_FIELDS:
                    assert np.array_equal(st[f], ost[f]), (algo, seed, f)
