"""Batches led from another stream than their contexts': loads and resets that
leave millions of delta rows queued on private streams, and a batch at once
(results against the oracle).  The order itself is shown by
test_host_runtime.py."""
import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver

pytestmark = pytest.mark.gpu

TEXT = "S -> A B\nA -> a\nB -> b\n"


def many_rows(n, m, seed):
    """m random 'a' edges and m / 16 'b' edges: the first delta lists nearly
    every vertex in both orientations."""
    rng = np.random.default_rng(seed)
    mb = m // 16
    src, dst = (rng.integers(0, n, m + mb, dtype=np.uint32) for _ in range(2))
    lab = np.r_[np.zeros(m, np.uint32), np.ones(mb, np.uint32)]
    return gen.Graph(n=n, labels=["a", "b"], src=src, lab=lab, dst=dst)


@pytest.mark.parametrize("form", [cflr.CFLR_FORM_BATCHED, cflr.CFLR_FORM_GRAPH])
def test_batches_right_after_loads_and_resets(form):
    graphs = [many_rows(n, 3 * n, 40 + k) for k, n in enumerate((700_001, 300_007, 1_000, 50))]
    want = [oracle.solve(TEXT, g) for g in graphs]
    leader = Solver(TEXT, form=form)
    solvers = [Solver(TEXT, form=form) for _ in graphs]
    try:
        leader.load(graphs[3])
        leader.solve()
        for turn in range(12):
            for s, g in zip(solvers, graphs):
                if turn == 0:
                    s.load(g)
                else:
                    cflr.cflr_reset(s.ctx)
            # led by a context that only lends its buffers, or by each in turn
            lead = turn % (len(solvers) + 1)
            order = [leader] + solvers if lead == 0 else solvers[lead - 1:] + solvers[:lead - 1]
            stats = cflr.cflr_solve_batch([s.ctx for s in order])
            assert all(st["converged"] for st in stats)
            for s, w in zip(solvers, want):
                for name in ("S", "A", "B"):
                    assert np.array_equal(s.pairs(name), w.pairs[name]), (turn, name)
    finally:
        for s in [leader] + solvers:
            s.close()
