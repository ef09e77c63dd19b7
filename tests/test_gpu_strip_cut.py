"""Batches that the strips cut into whole waves of uncut samples and a last wave
of row segments (segments of a third, a half and other fractions of a grid)
against one launch per colour: the same bits."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,converged", [(0, 0), (1, 1)])
@pytest.mark.parametrize("n,S", [(64, 2500), (64, 1300), (128, 1300), (256, 333), (256, 97)])
def test_a_cut_batch_equals_colour_launches(precision, converged, n, S):
    import paper_1910_04727_gb300 as fm
    c = fm.Context(2, 8, 16, precision=precision, converged=converged, tol=1e-9, qtol=0.0,
                   max_cycles=200)
    K = torch.tensor(W.smooth_lognormal_field(n, S=min(S, 40), tag=4900 + n), device="cuda")
    K = K.repeat((S + len(K) - 1) // len(K), 1, 1)[:S].contiguous()
    out = []
    for tile in (-1, 0):
        for m in [4 << k for k in range(8) if (4 << k) <= n]:
            if m >= 32 or tile == 0:
                c.set_smoother_shape(m, tile, 0)
        out.append([x.cpu().numpy() for x in c.fmg_solve_batch(K, want_p=True, kernel=1)])
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)
