"""The work-list pass against the oracle: rows of 1 to 1100 delta entries read by
1 to 70 productions, so that uses of several rows share a turn, a row's uses
take several turns, and long rows go to the warp or the CTA pass."""
import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver
from test_gpu_union import TEXT, shift_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("uses", [1, 3, 31, 33, 70])
@pytest.mark.parametrize("width", [1, 2, 5, 11, 16, 17, 32, 33, 70, 1100])
def test_uses_and_entries(uses, width):
    # T_i -> S x_i, with x_i edges at every (i + 2)-th column
    g = shift_graph(9, width, 3, 3)
    src, lab, dst = [g.src], [g.lab], [g.dst]
    cols = np.arange(9, g.n)
    for i in range(uses):
        at = cols[::i + 2]
        src.append(at)
        dst.append((at * 7 + i) % g.n)
        lab.append(np.full(at.size, 2 + i))
    g = gen.Graph(n=g.n, labels=["a", "b"] + [f"x{i}" for i in range(uses)],
                  **{k: np.concatenate(v).astype(np.uint32)
                     for k, v in (("src", src), ("lab", lab), ("dst", dst))})
    text = TEXT + "".join(f"T{i} -> S x{i}\n" for i in range(uses)) + "U -> S\n"
    want = oracle.solve(text, g)
    names = want.grammar.nts[:want.grammar.n_user]
    for form in (cflr.CFLR_FORM_GRAPH, cflr.CFLR_FORM_PLAIN):
        if form == cflr.CFLR_FORM_PLAIN and uses > 3:
            continue
        with Solver(text, form=form) as s:
            s.load(g)
            s.solve()
            got = s.pairs_many(names)
        for x in names:
            assert np.array_equal(got[x], want.pairs[x]), x
