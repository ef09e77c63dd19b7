"""Autotuned FP64 contexts keep the rule for batches of few cells: strips chosen on
the tuner's large batch do not march the rows of one sample; a shape set by hand
does stay."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _families(c, K):
    c.profile_begin()
    out = c.fmg_solve_batch(K, want_p=True, kernel=1)
    torch.cuda.synchronize()
    return {k for k, v in c.profile_end().items() if v["launches"]}, out


@pytest.mark.parametrize("n", [64, 256])
def test_one_sample_after_tuning(n):
    import paper_1910_04727_gb300 as fm
    c = fm.Context(1, n, 8)
    K = torch.tensor(W.smooth_lognormal_field(n, S=1, tag=5300 + n), device="cuda")
    plain, want = _families(c, K)
    assert "rbgs_strip" not in plain
    c.autotune(precision=0, nsweeps=2, n_min=64, n_max=n)
    tuned, got = _families(c, K)
    assert "rbgs_strip" not in tuned
    by_hand = fm.Context(1, n, 8)
    by_hand.set_smoother_shape(n, -1, 0, 0)
    shapes, got2 = _families(by_hand, K)
    assert "rbgs_strip" in shapes
    for x, y, z in zip(want, got, got2):
        assert torch.equal(x, y) and torch.equal(x, z)
