"""One context through graphs of different sizes, resets, schedules, batches and
grammars: the tables, the captured loop and the grammar's part that it keeps
must follow every change (results against the oracle)."""
import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver

pytestmark = pytest.mark.gpu

FICA = gen.grammar_text("fica")


def alias(n, seed):
    return gen.fica_like(n=n, n_a=2 * n, n_d=3 * n // 4, seed=seed)


def same(s, want):
    names = want.grammar.nts[:want.grammar.n_user]
    got = s.pairs_many(names)
    for x in names:
        assert np.array_equal(got[x], want.pairs[x]), x


@pytest.mark.parametrize("form", [cflr.CFLR_FORM_BATCHED, cflr.CFLR_FORM_GRAPH])
@pytest.mark.parametrize("capacity", [0, 64])
def test_graphs_resets_and_schedules(form, capacity):
    graphs = [alias(n, 60 + k) for k, n in enumerate((300, 2500, 40, 1200))]
    want = [oracle.solve(FICA, g) for g in graphs]
    with Solver(FICA, form=form, initial_capacity=capacity) as s:
        for k in (0, 1, 2, 1, 3):
            s.load(graphs[k])
            s.solve()
            same(s, want[k])
            for limits in ((128, 1024, 4096), (64, 256, 2048)):
                t = cflr.cflr_get_tuning(s.ctx)
                cflr.cflr_set_tuning(s.ctx, t["probe_ratio"], limits, t["ctas_per_sm"])
                cflr.cflr_reset(s.ctx)
                s.solve()
                same(s, want[k])


def test_leading_batches_between_own_solves():
    graphs = [alias(n, 70 + k) for k, n in enumerate((500, 900, 1300))]
    want = [oracle.solve(FICA, g) for g in graphs]
    solvers = [Solver(FICA, form=cflr.CFLR_FORM_GRAPH) for _ in graphs]
    try:
        for s, g in zip(solvers, graphs):
            s.load(g)
        for lead in (0, 1, 0, 2):
            order = solvers[lead:] + solvers[:lead]
            for s in solvers:
                cflr.cflr_reset(s.ctx)
            cflr.cflr_solve_batch([s.ctx for s in order])
            for s, w in zip(solvers, want):
                same(s, w)
            cflr.cflr_reset(solvers[lead].ctx)
            solvers[lead].solve()
            same(solvers[lead], want[lead])
    finally:
        for s in solvers:
            s.close()


def test_another_grammar_in_the_same_context():
    g1, g2 = alias(700, 80), gen.fsjpt_like(n=900, n_edges=3600, fields=64, seed=81)
    text2 = gen.grammar_text("fsjpt")
    w1, w2 = oracle.solve(FICA, g1), oracle.solve(text2, g2)
    with Solver(FICA, form=cflr.CFLR_FORM_GRAPH) as s:
        for text, g, w in ((FICA, g1, w1), (text2, g2, w2), (FICA, g1, w1)):
            cflr.cflr_load_grammar(s.ctx, text)
            s.load(g)
            s.solve()
            same(s, w)
            cflr.cflr_reset(s.ctx)
            s.solve()
            same(s, w)


def test_iteration_limit_then_more():
    g = alias(900, 90)
    want = oracle.solve(FICA, g)
    with Solver(FICA, form=cflr.CFLR_FORM_GRAPH, max_iterations=2) as s:
        for _ in range(2):
            s.load(g)
            for _ in range(40):
                if cflr.cflr_solve_batch([s.ctx], allow_limit=True)[0]["converged"]:
                    break
            same(s, want)
