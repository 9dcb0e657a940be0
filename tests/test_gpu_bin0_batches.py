"""Bin 0 takes its groups one at a time below eight a warp, and in batches of
two, four and eight from 8, 16 and 32 a warp on: group counts on both sides of
each line, with one CTA of eight warps per SM so that small graphs reach them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_11029_gb300 import cflr
from paper_2401_11029_gb300.cflr import Solver
from test_gpu_union import TEXT, shift_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_warp", [1, 8, 16, 32, 33])
@pytest.mark.parametrize("off", [-1, 0, 1])
@pytest.mark.parametrize("witness", [0, 1])
def test_groups_around_the_batch_lines(per_warp, off, witness):
    warps = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    g = shift_graph(per_warp * warps + off, 2, 3, 3)      # a group per row and iteration
    want = oracle.solve(TEXT, g).pairs["S"]
    with Solver(TEXT, keep_vertex_order=1, witness=witness) as s:
        t = cflr.cflr_get_tuning(s.ctx)
        cflr.cflr_set_tuning(s.ctx, t["probe_ratio"], t["bin_limit"],
                             [1] + list(t["ctas_per_sm"])[1:])
        s.load(g)
        s.solve()
        assert np.array_equal(s.pairs("S"), want)
