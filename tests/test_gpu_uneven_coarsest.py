"""Uneven batches whose coarsest grid has 2 or 3 cells a side: the register and
shared-memory kernels of one sample a CTA take powers of two only, so groups of
12, 24 and 48 cells go level-wise, with their scratch sized before the capture.
Every group's results are those of its own call, bit for bit, on a context that
has solved nothing before."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0,grids", [(3, (12, 24, 48, 96)), (2, (8, 16, 32, 64)), (4, (16, 64, 128))])
@pytest.mark.parametrize("precision,converged", [(0, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("energy", [False, True])
def test_groups_equal_their_own_calls(n0, grids, precision, converged, energy):
    import paper_1910_04727_gb300 as fm
    if energy and not converged:
        pytest.skip("the energy step needs the converged mode")
    kw = dict(n_coarsest=n0, precision=precision, converged=converged, tol=1e-10, max_cycles=100,
              energy_step=energy)
    Ks = [torch.tensor(W.smooth_lognormal_field(n, S=S, tag=5000 + n), device="cuda")
          for n, S in zip(grids, (7, 5, 3, 2))]
    outs = fm.Context(1, 4 * n0, 8, **kw).solve_uneven(Ks, want_status=True)
    c = fm.Context(1, 4 * n0, 8, **kw)
    for K, got in zip(Ks, outs):
        want = c.fmg_solve_batch(K, want_status=True)
        for x, y in zip(got, (want[0], want[1], want[3])):
            assert torch.equal(x, y)
