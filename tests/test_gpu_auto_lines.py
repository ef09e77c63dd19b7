"""FM_KERNEL_AUTO in FP64 on both sides of its line, for every grid and form that
has one: the resident kernel at the line, the level-wise schedule one sample past
it, and the bits of that schedule asked for by name."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

LEVELWISE, RESIDENT = 1, 2


@pytest.mark.parametrize("n,per_sm,converged", [(16, 8, 0), (32, 4, 0), (64, 1, 0), (16, 32, 1), (32, 12, 1),
                                                (64, 2, 1)])
def test_the_schedule_on_both_sides_of_the_line(n, per_sm, converged):
    import paper_1910_04727_gb300 as fm
    line = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    c = fm.Context(1, n, 8, converged=converged, tol=1e-10, max_cycles=100)
    base = torch.tensor(W.smooth_lognormal_field(n, S=16, tag=5400 + n), device="cuda")
    for S, kernel in ((line, RESIDENT), (line + 1, LEVELWISE)):
        K = base.repeat(S // 16 + 1, 1, 1)[:S].contiguous()
        c.profile_begin()
        got = c.fmg_solve_batch(K, want_p=True)
        torch.cuda.synchronize()
        ran = {k for k, v in c.profile_end().items() if v["launches"]}
        assert ("fmg_resident" in ran) == (kernel == RESIDENT)
        for x, y in zip(got, c.fmg_solve_batch(K, want_p=True, kernel=kernel)):
            assert torch.equal(x, y)
