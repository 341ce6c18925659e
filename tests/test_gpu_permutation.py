"""The permutation at the sizes where its plan changes: one bucket, the first
split, a full chunk and one more, fewer vertices per bucket while there are few
buckets, the last size sorted in one level of buckets and the first in two."""
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


@pytest.mark.parametrize("n", [2, 511, 1023, 1024, 2047, 2049, 4097, 155_647, 622_593, 2**22 - 1, 2**22 + 4097, 2**24 + 4095,
                               2**24 + 4097])
def test_permutation_equals_oracle(cc, gg, ora, n):
    off = np.zeros(n + 1, np.int64)
    off[1], off[2:] = 1, 2
    with cc.Graph(off, np.array([1, 0], np.int32)) as graph:
        for seed in (0, 2**63 + 5):
            assert np.array_equal(graph.permutation(seed), ora.permutation(n, seed))
