"""The commit takes a candidate per thread when its grid holds all of them and
two rounds of the CTA otherwise: candidate counts around both lines."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_11029_gb300.cflr import Solver
from test_gpu_union import TEXT, shift_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 8, 9, 16, 17, 33])
def test_few_candidates(rows):
    g = shift_graph(rows, 32, 5, 4)
    with Solver(TEXT, keep_vertex_order=1) as s:
        s.load(g)
        s.solve()
        assert np.array_equal(s.pairs("S"), oracle.solve(TEXT, g).pairs["S"])


@pytest.mark.parametrize("share", [0.5, 0.97, 1.0, 1.03, 2.1])
def test_candidates_around_the_grid(share):
    grid = 8 * 256 * torch.cuda.get_device_properties(0).multi_processor_count
    g = shift_graph(int(share * grid) // 64, 64, 5, 3)
    with Solver(TEXT, keep_vertex_order=1) as s:
        s.load(g)
        s.solve()
        assert np.array_equal(s.pairs("S"), oracle.solve(TEXT, g).pairs["S"])
