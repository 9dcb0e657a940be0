"""The frame of an iteration: pair sets checked inside the reset pass (up to
2048 non-terminals) or by a launch of their own, and the product bins on side
streams that contexts take from a shared store."""
import threading

import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver
from test_gpu_union import TEXT, shift_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slots", [2, 2047, 2048, 2049, 3000])
@pytest.mark.parametrize("form", [cflr.CFLR_FORM_BATCHED, cflr.CFLR_FORM_GRAPH])
def test_sets_grow_with_many_non_terminals(slots, form):
    # S and the wrapper <b> beside idle non-terminals; S outgrows its first set
    text = TEXT + "".join(f"X{i} -> x{i}\n" for i in range(slots - 2))
    g = shift_graph(40, 200, 5, 9)
    want = oracle.solve(TEXT, g)
    with Solver(text, form=form) as s:
        assert s.n_nt == slots
        s.load(g)
        first = s.solve()
        assert first["regrow_sets"] > 0
        assert np.array_equal(s.pairs("S"), want.pairs["S"])
        cflr.cflr_reset(s.ctx)
        assert s.solve()["iterations"] == first["iterations"]
        assert np.array_equal(s.pairs("S"), want.pairs["S"])


def test_contexts_of_several_threads():
    # more contexts at a time than side streams are kept for, twice over
    text = gen.grammar_text("fica")
    graphs = [gen.fica_like(n=500 + 37 * k, n_a=1000 + 74 * k, n_d=375 + 20 * k, seed=50 + k)
              for k in range(24)]
    want = [oracle.solve(text, g).pairs["M"] for g in graphs]
    bad = []

    def work(ks):
        try:
            for _ in range(2):
                open_ = []
                for k in ks:
                    s = Solver(text, form=cflr.CFLR_FORM_GRAPH if k % 2 else cflr.CFLR_FORM_BATCHED)
                    open_.append((k, s))
                    s.load(graphs[k])
                for k, s in open_:
                    s.solve()
                for k, s in open_:
                    if not np.array_equal(s.pairs("M"), want[k]):
                        bad.append(k)
                    s.close()
        except Exception as exc:
            bad.append(exc)

    threads = [threading.Thread(target=work, args=(range(t, 24, 4),)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
