"""FP64 set-up of the level-wise schedule against the oracle at its edges:
coarsest grids of 2, 3 and 4 cells (the banded inverse), one sample to just
past a block of 32, both boundary cases, coefficients whose products leave
the range of the square-root form of the geometric mean, and batches on both
sides of FM_KERNEL_AUTO's schedule line.  Tolerance 1e-10, the FP64 bar (the
two sides round in a different order)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import lib as OL

pytestmark = pytest.mark.gpu


def _check(c, K, prm, n0, **kw):
    qf, qc, _ = c.fmg_solve_batch(torch.tensor(K, device="cuda"), **kw)
    of, oc, _, _ = OL.fmg_solve_batch(K, prm, n0=n0)
    assert np.max(np.abs(qf.cpu().numpy() - of) / np.abs(of)) < 1e-10
    assert np.max(np.abs(qc.cpu().numpy() - oc) / np.abs(oc)) < 1e-10


@pytest.mark.parametrize("n0,case", [(2, 2), (3, 1), (4, 2), (4, 1)])
@pytest.mark.parametrize("S", [1, 33])
def test_coarse_inverse_and_child_means(n0, case, S):
    import paper_1910_04727_gb300 as fm
    c = fm.Context(1, 4 * n0, 8, n_coarsest=n0, bc_case=case, pS=0.3, pN=0.7)
    for scale in (1.0, 1e90, 1e-90):   # products of four leave 1e280 and 1e-280
        K = W.smooth_lognormal_field(8 * n0, S=S, tag=4300 + n0) * scale
        _check(c, K, OL.params(bc_case=case, pS=0.3, pN=0.7), n0, kernel=1)


@pytest.mark.parametrize("exponent", [480, -481])
def test_coefficients_on_both_sides_of_the_short_reciprocal(exponent):
    import paper_1910_04727_gb300 as fm
    c = fm.Context(1, 16, 8)
    K = W.smooth_lognormal_field(64, S=5, tag=4500) * 2.0 ** exponent
    _check(c, K, OL.params(), 4, kernel=1)


@pytest.mark.parametrize("n,per_sm,converged", [(16, 8, 0), (32, 4, 0), (64, 1, 0), (64, 4, 1)])
def test_auto_schedule_on_both_sides_of_its_line(n, per_sm, converged):
    import paper_1910_04727_gb300 as fm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    c = fm.Context(1, n, 8, converged=bool(converged), tol=1e-13, max_cycles=300)
    for S in (per_sm * sms, per_sm * sms + 1):
        K = W.smooth_lognormal_field(n, S=8, tag=4400 + n)
        K = np.concatenate([K] * (S // 8 + 1))[:S]
        qf, qc, _ = c.fmg_solve_batch(torch.tensor(K, device="cuda"))
        of, oc, _, _ = OL.fmg_solve_batch(K[:8], OL.params(converged=bool(converged), tol=1e-13, max_cycles=300))
        idx = np.arange(S) % 8
        assert np.max(np.abs(qf.cpu().numpy() - of[idx]) / np.abs(of[idx])) < 1e-10
        assert np.max(np.abs(qc.cpu().numpy() - oc[idx]) / np.abs(oc[idx])) < 1e-10
