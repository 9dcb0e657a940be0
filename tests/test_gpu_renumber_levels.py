"""The device vertex order on frontiers around the size up to which the
search's levels run on the device in a row (8192), and around the shares of a
group, against the plain queue search."""
import numpy as np
import pytest

from paper_2401_11029_gb300 import gen
from test_gpu_renumber import check_order

pytestmark = pytest.mark.gpu


def layered(sizes, extra, seed):
    """Trees whose levels have the given sizes (level 0: the roots), extra
    edges inside levels and to the next one, ids and edges shuffled; the roots
    keep the smallest ids, so that they start the search."""
    rng = np.random.default_rng(seed)
    first = np.concatenate([[0], np.cumsum(sizes)])
    n = int(first[-1])
    src, dst = [], []
    for k in range(1, len(sizes)):
        src.append(first[k - 1] + rng.integers(0, sizes[k - 1], sizes[k]))
        dst.append(np.arange(first[k], first[k + 1]))
        a = rng.integers(0, sizes[k], extra)
        src.append(first[k] + a)
        dst.append(first[k] + rng.integers(0, sizes[k], extra))
    src, dst = np.concatenate(src), np.concatenate(dst)
    ids = np.concatenate([np.arange(sizes[0]), sizes[0] + rng.permutation(n - sizes[0])])
    at = rng.permutation(src.size)
    flip = rng.random(src.size) < 0.5
    s, d = ids[src][at], ids[dst][at]
    s, d = np.where(flip, d, s), np.where(flip, s, d)
    return gen.Graph(n=n, labels=["a"], src=s.astype(np.uint32),
                     lab=np.zeros(s.size, np.uint32), dst=d.astype(np.uint32))


@pytest.mark.parametrize("sizes", [
    [1, 2, 3], [1, 1023, 1024, 1025, 2], [3, 8191, 1], [2, 300, 8192, 8193, 40, 8192, 1],
    [9000, 100, 1], [9000, 9000, 9000], [1, 100, 8193], [5, 7, 20_000, 6, 1, 1, 1, 30]])
@pytest.mark.parametrize("extra", [0, 700])
def test_frontiers_around_the_cluster_limit(sizes, extra):
    check_order("S -> a\n", layered(sizes, extra, seed=len(sizes) + extra))
