"""Growth of several pair sets at once: all in one pass, one at a time under a
memory budget, with recorded steps, and across the contexts of a batch (each
with a stream of its own)."""
import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver
from test_gpu_union import shift_graph

pytestmark = pytest.mark.gpu


def text_of(sets):
    # `sets` closures that advance in step and so outgrow their sets together
    return "".join(f"S{k} -> a | S{k} b\n" for k in range(sets))


@pytest.mark.parametrize("sets", [1, 2, 7, 65])
@pytest.mark.parametrize("config", [{}, {"witness": 1}, {"mem_budget_bytes": 4 << 30},
                                    {"form": cflr.CFLR_FORM_GRAPH}])
def test_sets_grow_together(sets, config):
    g = shift_graph(40, 100, 5, 9)
    want = oracle.solve(text_of(1), g).pairs["S0"]
    with Solver(text_of(sets), **config) as s:
        s.load(g)
        assert s.solve()["regrow_sets"] >= sets
        for k in range(sets):
            assert np.array_equal(s.pairs(f"S{k}"), want)
        if config.get("witness"):
            ids = s.label_ids(g.labels)
            names = {int(i): lab for i, lab in zip(ids, g.labels)}
            for key in want[:: want.size // 7]:
                u, v = int(key >> 32), int(key & 0xFFFFFFFF)
                path = s.path("S0", u, v, names)
                assert path[0][0] == u and path[-1][2] == v
                assert [lab for _, lab, _ in path] == ["a"] + ["b"] * (len(path) - 1)


def test_sets_of_a_batch_grow_together():
    graphs = [shift_graph(20 + 5 * k, 60 + 20 * k, 5, 9) for k in range(5)]
    text = text_of(3)
    solvers = [Solver(text, witness=k & 1) for k in range(5)]
    try:
        for s, g in zip(solvers, graphs):
            s.load(g)
        cflr.cflr_solve_batch([s.ctx for s in solvers])
        for s, g in zip(solvers, graphs):
            want = oracle.solve(text_of(1), g).pairs["S0"]
            for k in range(3):
                assert np.array_equal(s.pairs(f"S{k}"), want)
    finally:
        for s in solvers:
            s.close()


def test_large_sets_beside_small_ones():
    # S grows past 16 MB, the other closures stay below it
    big, small = shift_graph(200, 200, 5, 9), shift_graph(40, 100, 5, 9)
    text = "S -> a | S b\nT -> c | T d\nU -> c | U d\n"
    g = gen.Graph(n=big.n, labels=["a", "b", "c", "d"],
                  src=np.concatenate([big.src, small.src]),
                  lab=np.concatenate([big.lab, small.lab + 2]),
                  dst=np.concatenate([big.dst, small.dst]))
    want = oracle.solve(text, g)
    with Solver(text) as s:
        s.load(g)
        assert s.solve()["regrow_sets"] >= 3
        for x in "STU":
            assert np.array_equal(s.pairs(x), want.pairs[x])
