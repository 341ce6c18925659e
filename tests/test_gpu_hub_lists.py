"""32 rows with more than 2^31 entries together: 32 hubs over 70M shared leaves.
The objective walks them as one window of rows, whose starts lie further apart
than 32 bits tell.  Labellings whose cost is known in closed form; exact."""
import pytest

pytestmark = pytest.mark.gpu

HUBS, LEAVES = 32, 70_000_000


@pytest.fixture(scope="module")
def cc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1507_05086_gb300 as cc
    cc.load()
    return cc


def test_objective_and_rounds_over_hubs(cc):
    import torch
    n, m = HUBS + LEAVES, HUBS * LEAVES
    col = torch.empty(2 * m, dtype=torch.int32, device="cuda")
    col[:m].view(HUBS, LEAVES).copy_(torch.arange(HUBS, n, dtype=torch.int32, device="cuda"))
    col[m:].view(LEAVES, HUBS).copy_(torch.arange(HUBS, dtype=torch.int32, device="cuda"))
    v = torch.arange(n + 1, dtype=torch.int64, device="cuda")
    off = torch.where(v <= HUBS, v * LEAVES, m + (v - HUBS) * HUBS)
    with cc.Graph(off, col) as graph:
        # one cluster
        lab = torch.zeros(n, dtype=torch.int32, device="cuda")
        assert graph.disagreements(lab) == n * (n - 1) // 2 - m
        # every leaf with hub (leaf mod 32), the first hub's share left out
        leaf = torch.arange(LEAVES, dtype=torch.int32, device="cuda")
        lab[:HUBS] = torch.arange(HUBS, dtype=torch.int32, device="cuda")
        lab[HUBS:] = leaf % HUBS
        lab[HUBS:][leaf % HUBS == 0] = HUBS
        size = torch.bincount(lab.long(), minlength=HUBS + 1).tolist()[:HUBS + 1]
        inside = int((leaf % HUBS != 0).sum())
        assert graph.disagreements(lab) == m - 2 * inside + sum(s * (s - 1) // 2 for s in size)
        # the first vertex of pi is a leaf: it takes every hub, and nothing else is left
        for algo in ("cw", "c4"):
            labels, rounds, cost = graph.cluster(algo, 0.5, 1, labels_out=torch.empty(n, dtype=torch.int32, device="cuda"))
            first = int(labels[0])
            assert first >= HUBS and rounds == 2
            assert torch.equal(labels[:HUBS], torch.full((HUBS,), first, dtype=torch.int32, device="cuda"))
            assert cost == m - 2 * HUBS + (HUBS + 1) * HUBS // 2
    del col, off
    torch.cuda.empty_cache()
