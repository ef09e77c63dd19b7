"""FP64 batches that FM_KERNEL_AUTO sends level-wise where no scratch can be had:
under a stream capture on a context that has solved nothing, the schedule without
scratch runs (one sample a warp or CTA), its results bit for bit."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

LEVELWISE, RESIDENT = 1, 2


@pytest.mark.parametrize("n,per_sm", [(16, 8), (32, 4)])
def test_a_batch_beyond_the_schedule_line_can_be_captured(n, per_sm):
    import paper_1910_04727_gb300 as fm
    S = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + 1
    K = torch.tensor(W.smooth_lognormal_field(n, S=8, tag=5100 + n), device="cuda").repeat(S // 8 + 1, 1, 1)[:S].contiguous()
    c = fm.Context(1, n, 8)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = c.fmg_solve_batch(K, want_p=True)
    graph.replay()
    torch.cuda.synchronize()
    other = fm.Context(1, n, 8)
    for x, y in zip(out, other.fmg_solve_batch(K, want_p=True, kernel=RESIDENT)):
        assert torch.equal(x, y)
    for x, y in zip(c.fmg_solve_batch(K, want_p=True), other.fmg_solve_batch(K, want_p=True, kernel=LEVELWISE)):
        assert torch.equal(x, y)   # outside a capture: the schedule of the rule
