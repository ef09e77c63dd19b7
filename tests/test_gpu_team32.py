"""The register-resident 32 x 32 mixed kernel (a sample on five warps): the pressure
of every sample it reports converged solves that sample's system (the bound of
test_gpu_refine_kernels: tol ||b|| and the rounding of two residuals), for one
sample to past the CTAs in flight, both boundary cases, one to three sweeps,
with and without Q^c; all converge with two sweeps.  A sample that is not finite
leaves the others' bits alone.
"""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_refine_kernels import _system

pytestmark = pytest.mark.gpu

RESIDENT, TOL = 2, 1e-12


def _ctx(case):
    import paper_1910_04727_gb300 as fm
    return fm.Context(2, 16, 16, precision=1, converged=1, tol=TOL, qtol=0.0, max_cycles=200, bc_case=case,
                      pW=1.0, pE=0.0, pS=0.3, pN=0.7)


@pytest.mark.parametrize("case", [1, 2])
@pytest.mark.parametrize("nu1,nu2", [(2, 2), (1, 1), (3, 2)])
@pytest.mark.parametrize("want_qc", [True, False])
@pytest.mark.parametrize("S", [1, 5, 701])
def test_the_returned_pressure_solves_its_system(case, nu1, nu2, want_qc, S):
    c = _ctx(case)
    K = W.smooth_lognormal_field(32, S=S, tag=3400 + S)
    qf, _, p, st = c.fmg_solve_batch(torch.tensor(K, device="cuda"), want_qc=want_qc, want_p=True, want_status=True,
                                     kernel=RESIDENT, nu1=nu1, nu2=nu2)
    qf, p, st = qf.cpu().numpy(), p.cpu().numpy(), st.cpu().numpy()
    assert (nu1, nu2) == (1, 1) or not st.any()
    for i in np.flatnonzero(st == 0):
        D, w, e, s, t, b = _system(K[i], case)
        q = np.pad(p[i], 1)
        r = b - (D * p[i] - w * q[1:-1, :-2] - e * q[1:-1, 2:] - s * q[:-2, 1:-1] - t * q[2:, 1:-1])
        bound = TOL * np.linalg.norm(b) + 12 * np.finfo(float).eps * np.linalg.norm(D * p[i])
        assert np.linalg.norm(r) <= bound
        flux = 2 * K[i][:, -1] * p[i][:, -1]
        Q = p[i][15:17, 15:17].mean() if case == 1 else flux.sum()
        assert abs(Q - qf[i]) <= 1e-12 * (np.abs(flux).sum() + abs(Q))


def test_a_sample_that_is_not_finite_leaves_the_others_alone():
    c = _ctx(2)
    K = torch.tensor(W.smooth_lognormal_field(32, S=70, tag=3500), device="cuda")
    want = c.fmg_solve_batch(K, want_p=True, want_status=True, kernel=RESIDENT)
    bad = [0, 33, 34, 69]
    K2 = K.clone()
    K2[0, 3, 5] = float("nan")
    K2[33, 0, 0] = float("inf")
    K2[34] *= 1e200
    K2[69, 31, 31] = float("nan")
    got = c.fmg_solve_batch(K2, want_p=True, want_status=True, kernel=RESIDENT)
    keep = np.setdiff1d(np.arange(70), bad)
    for x, y in zip(got, want):
        assert np.array_equal(x.cpu().numpy()[keep], y.cpu().numpy()[keep])
    assert (got[3].cpu().numpy()[bad] != 0).all()
