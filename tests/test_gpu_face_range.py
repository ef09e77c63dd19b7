"""FP64 faces next to the end of the exponent range: a coefficient above 2^1022,
whose sum with its neighbour has a reciprocal below the normal numbers, between
neighbours of ordinary size.  The oracle divides; tolerance 1e-10, the FP64 bar."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import lib as OL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [1, 2])
@pytest.mark.parametrize("n", [16, 32])
def test_a_cell_above_the_reciprocals_range(kernel, n):
    import paper_1910_04727_gb300 as fm
    K = 0.02 * W.smooth_lognormal_field(n, S=4, tag=5500 + n)
    assert K.max() < 1.0                # 2 a b stays finite
    K[:, 7, 5] = 6e307                  # odd row and column: in no injected grid
    c = fm.Context(1, n, 8)
    qf, qc, p = c.fmg_solve_batch(torch.tensor(K, device="cuda"), want_p=True, kernel=kernel)
    of, oc, _, _ = OL.fmg_solve_batch(K, OL.params())
    assert np.all(np.isfinite(of)) and np.all(np.isfinite(p.cpu().numpy()))
    assert np.max(np.abs(qf.cpu().numpy() - of) / np.abs(of)) < 1e-10
    assert np.max(np.abs(qc.cpu().numpy() - oc) / np.abs(oc)) < 1e-10
