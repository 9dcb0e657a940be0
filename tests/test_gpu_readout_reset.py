"""The read-out over the map of non-empty rows, and the reset that clears the
rows in use and every pair set in one launch, at the sizes where their units,
words and chunks end.  Under `S -> a` the pairs of S are the `a` edges, so the
expected result is the sorted edge list itself."""
import numpy as np
import pytest

from common import keys_of
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver

pytestmark = pytest.mark.gpu


def rows_graph(n, lens, labels, seed):
    """Per label, rows of the given lengths (cut to n) in turn, columns drawn
    without repetition."""
    rng = np.random.default_rng(seed)
    src, lab, dst = [], [], []
    for li in range(len(labels)):
        for i in range(n):
            k = min(n, lens[(i * 7 + li) % len(lens)])
            src.append(np.full(k, i))
            lab.append(np.full(k, li))
            dst.append(rng.choice(n, size=k, replace=False))
    src, lab, dst = (np.concatenate(x).astype(np.uint32) for x in (src, lab, dst))
    at = rng.permutation(src.size)
    return gen.Graph(n=n, labels=labels, src=src[at], lab=lab[at], dst=dst[at])


def edges_of(g, label):
    e = g.lab == g.labels.index(label)
    return np.unique(keys_of(g.src[e], g.dst[e]))


SHORT = [0, 1, 0, 2, 3, 0, 17, 1, 31, 32, 33, 0, 5]
LONG = [0, 1, 64, 500, 0, 1023, 1024, 1025, 2, 40]


@pytest.mark.parametrize("n,lens", [(1, SHORT), (31, SHORT), (32, SHORT), (33, SHORT),
                                    (1023, SHORT), (1025, SHORT), (1100, LONG),
                                    (3001, [0] * 40 + [1, 2]), (40_003, [0] * 900 + [3, 1])])
@pytest.mark.parametrize("keep", [0, 1])
def test_rows_of_every_length(n, lens, keep):
    text = "S -> a\nT -> b\nU -> c\n"
    g = rows_graph(n, lens, ["a", "b"], seed=n)
    with Solver(text, keep_vertex_order=keep) as s:
        s.load(g)
        s.solve()
        got = s.pairs_many(["T", "U", "S", "T"])
        assert np.array_equal(got["S"], edges_of(g, "a"))
        assert np.array_equal(got["T"], edges_of(g, "b"))
        assert got["U"].size == 0


def test_read_out_without_room_for_the_map():
    import torch
    text = "S -> a\nT -> b\n"
    g = rows_graph(2500, SHORT, ["a", "b"], seed=5)
    with Solver(text) as s:
        s.load(g)
        total = s.solve()["total_pairs"]
        peak = s.solve()["peak_device_bytes"]
    # room for the lists of the call, but less than the map's rule asks for
    budget = peak + 4 * total + (1 << 18)
    assert total > 30_000 and 17 * total + (1 << 16) > budget - peak
    with Solver(text, mem_budget_bytes=budget) as s:
        s.load(g)
        s.solve()
        src = torch.empty(total, dtype=torch.int32, device="cuda")
        dst = torch.empty(total, dtype=torch.int32, device="cuda")
        off = cflr.cflr_get_pairs_device_many(s.ctx, [0, 1], src.data_ptr(), dst.data_ptr(), total)
        keys = keys_of(src.cpu().numpy().view(np.uint32), dst.cpu().numpy().view(np.uint32))
        assert np.array_equal(keys[:int(off[1])], edges_of(g, "a"))
        assert np.array_equal(keys[int(off[1]):], edges_of(g, "b"))


@pytest.mark.parametrize("slots", [1, 2047, 2048, 2049, 4500])
def test_reset_clears_every_set_and_row(slots):
    # set 0 spans several clearing chunks, the others are of the smallest size
    text = "".join(f"S{i} -> a{i}\n" for i in range(slots))
    rng = np.random.default_rng(slots)
    n, big = 300, 6000
    pick = rng.choice(n * n, size=big, replace=False)
    lab = np.concatenate([np.zeros(big, np.int64), rng.integers(0, slots, size=2 * slots)])
    src = np.concatenate([pick // n, rng.integers(0, n, size=2 * slots)]).astype(np.uint32)
    dst = np.concatenate([pick % n, rng.integers(0, n, size=2 * slots)]).astype(np.uint32)
    g = gen.Graph(n=n, labels=[f"a{i}" for i in range(slots)], src=src,
                  lab=lab.astype(np.uint32), dst=dst)
    names = [f"S{i}" for i in sorted({0, 1 % slots, slots // 2, slots - 1,
                                      min(2047, slots - 1), min(2048, slots - 1)})]
    with Solver(text, form=cflr.CFLR_FORM_GRAPH) as s:
        s.load(g)
        first = s.solve()["total_pairs"]
        for _ in range(2):
            cflr.cflr_reset(s.ctx)
            assert s.solve()["total_pairs"] == first
            got = s.pairs_many(names)
            for x in names:
                assert np.array_equal(got[x], edges_of(g, "a" + x[1:])), x
