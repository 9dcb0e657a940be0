"""The walks over gathered tile lists against the oracle: lists of 0 to 9, 31 to
33 and 63 to 65 tiles side by side, so that quads and pairs end inside and at
the ends of lists and windows, in the bitmap bin (small rows), the hash bins
(wide rows) and the first bin."""
import numpy as np
import pytest

import oracle
from paper_2401_11029_gb300 import cflr, gen
from paper_2401_11029_gb300.cflr import Solver

pytestmark = pytest.mark.gpu

TEXT = "S -> A B\nA -> a\nB -> b\n"


@pytest.mark.parametrize("lens", [list(range(10)), [1], [2, 3], [4, 5, 0], [31, 32, 33, 1],
                                  [63, 64, 65, 2, 0, 7]])
@pytest.mark.parametrize("degree", [1, 3, 31, 33, 130])
@pytest.mark.parametrize("n,limits", [(8192, None), (300_000, None), (300_000, (16, 32, 4096)),
                                      (300_000, (2, 4096 // 8, 4096))])
def test_list_lengths(lens, degree, n, limits):
    rng = np.random.default_rng(degree + len(lens))
    rows, mids = 12, 200
    src, lab, dst = [], [], []
    for i in range(rows):                       # A: row i -> `degree` middle vertices
        k = rows + rng.choice(mids, size=degree, replace=False)
        src.append(np.full(degree, i))
        dst.append(k)
        lab.append(np.zeros(degree, np.int64))
    for m in range(mids):                       # B: middle m -> so many words, 1 to 4 bits each
        words = rng.choice(8192 // 32 - 8, size=lens[m % len(lens)], replace=False) + 8
        for w in words:
            bits = rng.choice(32, size=rng.integers(1, 5), replace=False)
            src.append(np.full(bits.size, rows + m))
            dst.append(32 * w + bits)
            lab.append(np.ones(bits.size, np.int64))
    g = gen.Graph(n=n, labels=["a", "b"], src=np.concatenate(src).astype(np.uint32),
                  lab=np.concatenate(lab).astype(np.uint32),
                  dst=np.concatenate(dst).astype(np.uint32))
    want = oracle.solve(TEXT, g)
    for witness in (0, 1):
        with Solver(TEXT, keep_vertex_order=1, witness=witness) as s:
            if limits:
                t = cflr.cflr_get_tuning(s.ctx)
                cflr.cflr_set_tuning(s.ctx, t["probe_ratio"], limits, t["ctas_per_sm"])
            s.load(g)
            s.solve()
            assert np.array_equal(s.pairs("S"), want.pairs["S"])
