"""The union passes (room, append, pack) against the oracle at the sizes where
their paths change: rows that get 1 to 5, 32 or 33, 256 or 257 new entries at a
time, in one word or in a word each, and more long rows moving at once than
their list holds.  Under `S -> a | S b`, with `b` edges that shift a column by
one block, every row gets the same number of new pairs in each iteration."""
import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import gen
from paper_2401_11029_gb300.cflr import Solver

pytestmark = pytest.mark.gpu

TEXT = "S -> a | S b\n"


def shift_graph(rows, width, stride, steps):
    cols = rows + stride * np.arange(width * (steps + 1))
    n = int(cols[-1]) + 1
    src = [np.repeat(np.arange(rows), width), cols[:-width]]
    dst = [np.tile(cols[:width], rows), cols[width:]]
    lab = [np.zeros(rows * width, np.uint32), np.ones(cols.size - width, np.uint32)]
    return gen.Graph(n=n, labels=["a", "b"], src=np.concatenate(src).astype(np.uint32),
                     lab=np.concatenate(lab), dst=np.concatenate(dst).astype(np.uint32))


def check(g, **cfg):
    want = oracle.solve(TEXT, g)
    with Solver(TEXT, **cfg) as s:
        s.load(g)
        s.solve()
        got = s.pairs("S")
    assert np.array_equal(got, want.pairs["S"])


@pytest.mark.parametrize("width", [1, 2, 3, 4, 5, 8, 31, 32, 33, 128, 256, 257, 600])
@pytest.mark.parametrize("stride", [1, 7, 32])
def test_new_entries_per_row(width, stride):
    g = shift_graph(37, width, stride, 6)
    check(g, keep_vertex_order=1)
    check(g, keep_vertex_order=1, initial_capacity=32)    # pool growth inside the union


def test_more_long_rows_move_than_the_list_holds():
    # 3000 rows grow past 256 tiles in step; the smallest first buffers keep
    # the list at touched / 64 + 1024 rows
    check(shift_graph(3000, 8, 32, 66), keep_vertex_order=1, initial_capacity=32)
