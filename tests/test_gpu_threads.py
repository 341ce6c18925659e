"""Different graphs may be used from different host threads at once: graphs whose
permutations take kernels of different scratch sizes (10K to 17M vertices: one
scatter with few or many buckets, two levels), each clustered over and over by a
thread of its own, give the results that they give alone; exact integers."""
import threading

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


@pytest.mark.parametrize("sizes", [(10_000, 4_000_000), (10_000, 700_000, 17_000_000), (17_000_000, 70_000_000)])
def test_threads_with_graphs_of_different_sizes(cc, sizes):
    """Rings: every vertex joined to the next one."""
    import torch
    graphs = []
    for n in sizes:
        v = torch.arange(n, dtype=torch.int64, device="cuda")
        pair = torch.stack([(v - 1) % n, (v + 1) % n], 1).sort(1).values
        graphs.append(cc.Graph(torch.arange(n + 1, dtype=torch.int64, device="cuda") * 2,
                               pair.to(torch.int32).flatten()))
        del v, pair
    torch.cuda.synchronize()
    seeds = (3, 4)
    alone = [[g.cluster("cw", 1.0, s, want_labels=False)[1:] for s in seeds] for g in graphs]
    problems, slow_done = [], threading.Event()

    def work(i, times):
        try:
            t = 0
            while t < times or (i == 0 and not slow_done.is_set()):
                k = t % len(seeds)
                got = graphs[i].cluster("cw", 1.0, seeds[k], want_labels=False)[1:]
                if got != alone[i][k]:
                    problems.append((sizes[i], seeds[k], got, alone[i][k]))
                    return
                t += 1
        except Exception as e:                  # a refused launch
            problems.append((sizes[i], repr(e)))

    threads = [threading.Thread(target=work, args=(i, 40)) for i in range(len(graphs))]
    for t in threads:
        t.start()
    for t in threads[1:]:
        t.join()
    slow_done.set()
    threads[0].join()
    for g in graphs:
        g.close()
    assert not problems, problems
