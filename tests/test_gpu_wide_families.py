"""Indexed families of more than 64 members (optimisation 4) against the
oracle, at member counts around the ends of occupancy words: families whose
members write different non-terminals (Figs. wcnf:fsca, wcnf:cscvf) and one
non-terminal (Fig. wcnf:fsjpt)."""
import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver

pytestmark = pytest.mark.gpu


def check(text, g, **cfg):
    want = oracle.solve(text, g)
    names = want.grammar.nts
    with Solver(text, **cfg) as s:
        s.load(g)
        s.solve()
        got = s.pairs_many(names)
    for x in names:
        assert np.array_equal(got[x], want.pairs[x]), x


@pytest.mark.parametrize("form", [cflr.CFLR_FORM_BATCHED, cflr.CFLR_FORM_GRAPH])
@pytest.mark.parametrize("members", [64, 65, 95, 96, 97, 142, 300])
def test_members_with_non_terminals_of_their_own(members, form):
    check(gen.grammar_text("fsca", index_hi=members - 1),
          gen.fsca_like(n=700, n_edges=1000, fields=members, seed=members), form=form)


@pytest.mark.parametrize("members", [65, 128, 511])
def test_call_sites(members):
    check(gen.grammar_text("cscvf", index_hi=members - 1),
          gen.cscvf_like(n=2500, n_edges=4200, calls=members, seed=members))


@pytest.mark.parametrize("members", [65, 100])
def test_members_writing_one_non_terminal(members):
    check(gen.grammar_text("fsjpt", index_hi=members - 1),
          gen.fsjpt_like(n=1500, n_edges=6000, fields=members, seed=members),
          form=cflr.CFLR_FORM_GRAPH)


def test_dense_rows_split_and_span_blocks():
    # delta rows of many entries and members with long rows: the families grow
    # past the hash bins (split into members) and past 32 items per step
    labels = ["d", "d_r", "a", "a_r"] + [f"{p}_{i}" for p in ("f", "f_r") for i in range(70)]
    check(gen.grammar_text("fsca", index_hi=69),
          gen.random_graph(n=220, n_edges=14_000, labels=labels, seed=3))
