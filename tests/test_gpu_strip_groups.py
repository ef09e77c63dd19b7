"""Warp groups, windows and merged cycles of the column-strip smoother.

Strips sweep in the colour launches' order, so every solve is the same bit
for bit whichever shape runs: one warp a row (64 columns), two and four warps
exchanging their border columns, several windows on wider grids, samples
packed into a warp below 64 columns, and the post-smoothing of one V-cycle
merged with the pre-smoothing of the next (nu1 = nu2; any number of cycles
between residual tests, so that the merged passes end in either buffer).
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import lib as OL

pytestmark = pytest.mark.gpu

LEVELWISE = 1


def _grids(n):
    return [4 << k for k in range(20) if (4 << k) <= n]


@pytest.mark.parametrize("nu1,nu2,cycles,case,energy", [(2, 2, 1, 2, False), (2, 2, 4, 1, False), (2, 2, 5, 2, False),
                                                        (1, 1, 3, 2, False), (1, 2, 2, 1, False), (2, 2, 4, 2, True),
                                                        (1, 1, 3, 1, True)])
def test_strip_groups_equal_colour_launches(nu1, nu2, cycles, case, energy):
    import paper_1910_04727_gb300 as fm
    c = fm.Context(2, 16, 16, precision=1, converged=True, tol=1e-10, max_cycles=60, nu1=nu1, nu2=nu2, nu0=cycles,
                   ir_cycles=cycles, bc_case=case, pS=0.3, pN=0.7, energy_step=energy)
    for n, S in [(16, 5), (32, 3), (64, 5), (128, 3), (256, 2), (512, 2), (1024, 1)]:
        K = torch.tensor(W.smooth_lognormal_field(n, S=S, tag=4100 + n), device="cuda")
        out = []
        for tile in (-1, 0):
            for m in _grids(n):
                c.set_smoother_shape(m, tile)
            out.append(c.fmg_solve_batch(K, want_p=True, kernel=LEVELWISE))
        for a, b in zip(*out):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True), n


def test_strip_rows_that_are_no_power_of_two_against_the_oracle():
    """Coarsest grids of 3 cells: rows of 48 and 96 columns leave lanes of a
    group idle, 192 is three warps.  Fixed FP64 schedule (1e-10: the rounding
    order alone) and the mixed form (1e-8, the mixed bar)."""
    import paper_1910_04727_gb300 as fm
    for precision, bar in ((0, 1e-10), (1, 1e-8)):
        c = fm.Context(1, 48, 8, n_coarsest=3, precision=precision, converged=bool(precision), tol=1e-12,
                       max_cycles=200)
        for n, S in [(48, 5), (96, 3), (192, 2)]:
            K = W.smooth_lognormal_field(n, S=S, tag=4200 + n)
            qf, qc, _ = c.fmg_solve_batch(torch.tensor(K, device="cuda"), kernel=LEVELWISE)
            prm = OL.params(converged=True, tol=1e-13, max_cycles=300) if precision else OL.params()
            of, oc, _, _ = OL.fmg_solve_batch(K, prm, n0=3)
            assert np.max(np.abs(qf.cpu().numpy() - of) / np.abs(of)) < bar, n
            assert np.max(np.abs(qc.cpu().numpy() - oc) / np.abs(oc)) < bar, n


@pytest.mark.parametrize("n,S", [(16, 1), (16, 37), (32, 3), (32, 301), (64, 5)])
@pytest.mark.parametrize("nu1,nu2", [(2, 2), (1, 2), (3, 2)])
@pytest.mark.parametrize("precision,energy", [(0, False), (1, False), (1, True)])
def test_default_shapes_of_small_grids_give_the_register_regions_bits(n, S, nu1, nu2, precision, energy):
    import paper_1910_04727_gb300 as fm
    K = torch.tensor(W.smooth_lognormal_field(n, S=S, tag=3700 + n), device="cuda")
    got = []
    for shape in (None, 32):
        c = fm.Context(1, n, 8, precision=precision, converged=precision, tol=1e-12, qtol=0.0, max_cycles=100,
                       energy_step=energy)
        for g in (16, 32):
            if shape is not None:
                c.set_smoother_shape(g, shape, 0, precision)
        got.append(c.fmg_solve_batch(K, want_p=True, want_status=True, kernel=1, nu1=nu1, nu2=nu2))
    for x, y in zip(*got):
        assert torch.equal(x, y)


@pytest.mark.parametrize("n,S", [(64, 255), (64, 256), (128, 127), (128, 128), (256, 1)])
@pytest.mark.parametrize("converged", [0, 1])
def test_fp64_batches_on_both_sides_of_the_strip_line(n, S, converged):
    import paper_1910_04727_gb300 as fm
    K = torch.tensor(W.smooth_lognormal_field(n, S=min(S, 8), tag=3800 + n), device="cuda")
    K = K.repeat((S + 7) // 8, 1, 1)[:S].contiguous()
    got = []
    for shape in (None, -1):
        c = fm.Context(1, n, 8, converged=converged, tol=1e-10, max_cycles=100)
        for g in (64, 128, 256):
            if shape is not None:
                c.set_smoother_shape(g, shape, 0, 0)
        got.append(c.fmg_solve_batch(K, want_p=True, want_status=True, kernel=1))
    for x, y in zip(*got):
        assert torch.equal(x, y)
