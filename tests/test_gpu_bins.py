"""Which accumulator a work-list group takes, against the oracle: groups of the
hash-table bins move to the bitmap bin where their table would be no smaller
than the row's bitmap, so vertex counts on both sides of that line are run
with groups of each bin's sizes, in the default and in narrower schedules."""
import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver
from test_gpu_union import TEXT, shift_graph

pytestmark = pytest.mark.gpu


def padded(g, n):
    assert g.n <= n
    return gen.Graph(n=n, labels=g.labels, src=g.src, lab=g.lab, dst=g.dst)


@pytest.mark.parametrize("limits", [None, (128, 512, 513), (64, 256, 2048), (128, 1024, 3000)])
@pytest.mark.parametrize("width", [40, 100, 130, 300, 700, 1500])
# the rows' words beside 2 << lg for tables of 2^lg slots, lg 9, 11, 13
@pytest.mark.parametrize("n", [32 * 1024, 32 * 1024 + 1, 32 * 4096, 32 * 4096 + 1, 32 * 16384 + 1])
def test_groups_on_both_sides_of_the_bitmap_line(n, width, limits):
    g = padded(shift_graph(5, width, 3, 4), n)
    want = oracle.solve(TEXT, g)
    with Solver(TEXT, keep_vertex_order=1, form=cflr.CFLR_FORM_GRAPH) as s:
        if limits:
            t = cflr.cflr_get_tuning(s.ctx)
            cflr.cflr_set_tuning(s.ctx, t["probe_ratio"], limits, t["ctas_per_sm"])
        s.load(g)
        s.solve()
        assert np.array_equal(s.pairs("S"), want.pairs["S"])


@pytest.mark.parametrize("limits", [(128, 512, 513), (64, 256, 2048), (32, 64, 4096)])
def test_families_in_narrow_bins(limits):
    # tagged families stay in the hash bins whatever the row's bitmap takes
    text = gen.grammar_text("fsjpt")
    g = gen.fsjpt_like(n=6000, n_edges=24_000, fields=64, seed=13)
    want = oracle.solve(text, g)
    with Solver(text) as s:
        t = cflr.cflr_get_tuning(s.ctx)
        cflr.cflr_set_tuning(s.ctx, t["probe_ratio"], limits, t["ctas_per_sm"])
        s.load(g)
        s.solve()
        got = s.pairs_many(["PT", "FT"])
        for x in ("PT", "FT"):
            assert np.array_equal(got[x], want.pairs[x]), x


@pytest.mark.parametrize("n_wide", [32 * 16384 + 1, 32 * 51200 + 1])
def test_a_small_instance_beside_a_wide_one(n_wide):
    """The bitmap bin's launch is laid out for the batch's widest rows (beyond
    51200 words its bitmaps are in global memory): beside them the groups of a
    small instance keep their hash tables."""
    text = gen.grammar_text("fica")
    small = gen.fica_like(n=3000, n_a=6000, n_d=2250, seed=7)
    wide = gen.fica_like(n=300, n_a=600, n_d=225, seed=8)
    wide = padded(wide, n_wide)
    want = [oracle.solve(text, g) for g in (small, wide)]
    solvers = [Solver(text, form=cflr.CFLR_FORM_GRAPH) for _ in want]
    try:
        for s, g in zip(solvers, (small, wide)):
            s.load(g)
        alone = solvers[0].solve()["groups"]
        assert alone[1] == alone[2] == 0 and alone[3] > 0
        for s in solvers:
            cflr.cflr_reset(s.ctx)
        beside = cflr.cflr_solve_batch([s.ctx for s in solvers])[0]["groups"]
        assert beside[1] > 0
        for s, w in zip(solvers, want):
            for name in w.grammar.nts[:w.grammar.n_user]:
                assert np.array_equal(s.pairs(name), w.pairs[name]), name
    finally:
        for s in solvers:
            s.close()
