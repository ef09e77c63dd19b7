"""Residual tests, prolongation and the energy-optimal step of the level-wise
schedule at the edges of their work splits: grids that are not powers of two,
odd coarse rows, one window of columns and several with a ragged last one,
chunks with one band and with many, both boundary cases, one sample and a few.

A solve that reports convergence has ||b - A p|| <= tol ||b||; the test forms
A p from the coefficients itself.  Bound: tol ||b|| and the rounding of two
residuals of six operations each, 12 eps || |D p| ||.  The QoI is that of the
returned pressure to 1e-12.
"""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

LEVELWISE, TOL = 1, 1e-12
PW, PE, PS, PN = 1.0, 0.0, 0.3, 0.7


def _system(K, case):
    """D, faces (west, east, south, north) and rhs of one field."""
    n = K.shape[0]
    te, tn = 2 * K[:, :-1] * K[:, 1:] / (K[:, :-1] + K[:, 1:]), 2 * K[:-1] * K[1:] / (K[:-1] + K[1:])
    w, e = np.zeros((n, n)), np.zeros((n, n))
    s, t = np.zeros((n, n)), np.zeros((n, n))
    w[:, 1:], e[:, :-1], s[1:], t[:-1] = te, te, tn, tn
    b, edge = np.zeros((n, n)), np.zeros((n, n))
    sides = [(np.s_[:, 0], PW), (np.s_[:, -1], PE)] + ([(np.s_[0], PS), (np.s_[-1], PN)] if case == 1 else [])
    for side, g in sides:
        edge[side] += 2 * K[side]
        b[side] += 2 * K[side] * g
    return w + e + s + t + edge, w, e, s, t, b


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", [1, 2])
@pytest.mark.parametrize("energy", [False, True])
@pytest.mark.parametrize("n0,n,S", [(2, 8, 3), (3, 24, 1), (3, 96, 3), (4, 64, 5), (4, 256, 1)])
def test_the_returned_pressure_solves_its_system(precision, case, energy, n0, n, S):
    import paper_1910_04727_gb300 as fm
    c = fm.Context(2, n0 * 2, 16, n_coarsest=n0, precision=precision, converged=1, tol=TOL, qtol=0.0, max_cycles=300,
                   bc_case=case, pW=PW, pE=PE, pS=PS, pN=PN, energy_step=energy)
    K = W.smooth_lognormal_field(n, S=S, tag=4700 + n)
    qf, _, p, st = c.fmg_solve_batch(torch.tensor(K, device="cuda"), want_p=True, want_status=True, kernel=LEVELWISE)
    assert not st.cpu().numpy().any()
    p, qf = p.cpu().numpy(), qf.cpu().numpy()
    for i in range(S):
        D, w, e, s, t, b = _system(K[i], case)
        q = np.pad(p[i], 1)
        r = b - (D * p[i] - w * q[1:-1, :-2] - e * q[1:-1, 2:] - s * q[:-2, 1:-1] - t * q[2:, 1:-1])
        bound = TOL * np.linalg.norm(b) + 12 * np.finfo(float).eps * np.linalg.norm(D * p[i])
        assert np.linalg.norm(r) <= bound
        h = n // 2
        Q = p[i][h - 1:h + 1, h - 1:h + 1].mean() if case == 1 else np.sum(2 * K[i][:, -1] * (p[i][:, -1] - PE))
        assert abs(Q - qf[i]) <= 1e-12 * np.abs(2 * K[i][:, -1] * (p[i][:, -1] - PE)).sum() + 1e-12 * abs(Q)
