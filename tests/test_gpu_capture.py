"""Calls captured into a CUDA graph: once any evaluation has planned the pair, every
other one finds its plans, tables and buffers in place (allocations are refused
while a stream captures).  A whole evaluation and a single call may take different
y passes of one source; a replay repeats the call bit for bit."""

import pytest
import torch

import workloads
from tests.pair_setup import gpu_pair

pytestmark = pytest.mark.gpu

CALLS = {
    "demag": lambda mm, out: mm.lib.mm_compute_demag(mm.ctx, 0, out.data_ptr()),
    "stray": lambda mm, out: mm.lib.mm_compute_stray_field(mm.ctx, 1, out.data_ptr()),
    "whole": lambda mm, out: mm.lib.mm_compute_torque(mm.ctx, 0, None, out.data_ptr()),
}


@pytest.mark.parametrize("n", [(140, 33, 1), (296, 33, 1), (40, 33, 3), (12, 9, 6), (9, 7, 12)])
@pytest.mark.parametrize("first,captured", [("demag", "whole"), ("whole", "stray"), ("stray", "demag")])
def test_a_planned_pair_can_be_captured(n, first, captured):
    fp, m0, m1 = workloads.film_pair_plain(n, 2, 3)
    fp.u0 = (0.3, -0.2, 0.0)
    stream = torch.cuda.Stream()
    mm = gpu_pair(fp, m0, m1, mech=False, stream=stream)
    out = torch.zeros(mm.shapes[0], dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    assert CALLS[first](mm, out) == 0
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        status = CALLS[captured](mm, out)
    assert status == 0, mm.lib.mm_last_error(mm.ctx)
    graph.replay()
    torch.cuda.synchronize()
    got = out.clone()
    assert CALLS[captured](mm, out) == 0
    torch.cuda.synchronize()
    assert torch.equal(got, out)
    mm.close()
