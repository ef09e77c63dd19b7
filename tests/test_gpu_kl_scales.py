"""FP64 fields with a mode that carries a large constant of the logarithm (units of
permeability far from 1), which puts the product of the rows' scales past the line
of the split: the sum g is large too, so the digits left out stay below its own
rounding.  Tolerance: one ulp of g in the exponent, the rounding of the sum, and
2^-51 for the exponential.  (The plain sum of 128 products is some ten ulps off.)"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("constant", [-690.0, -120.0, -41.0, 41.0, 300.0])
@pytest.mark.parametrize("M", [40, 128, 512])
def test_a_large_constant_mode(constant, M):
    import paper_1910_04727_gb300 as fm
    r = np.random.default_rng([75, M])
    B, xi = 0.1 * r.standard_normal((256, M)) / np.sqrt(1 + np.arange(M)), r.standard_normal((70, M))
    B[:, 0], xi[:, 0] = constant, 1.0
    c = fm.Context(1, 16, M, kl_mode=1)
    c.kl_basis_set(B)
    K = c.kl_field_batch(0, torch.tensor(xi, device="cuda")).cpu().numpy().reshape(70, 256)
    g = xi.astype(np.longdouble) @ B.T.astype(np.longdouble)
    err = np.abs(K.astype(np.longdouble) / np.exp(g) - 1).astype(float)
    assert np.all(err <= np.spacing(np.abs(g).astype(float)) + 2.0 ** -51)
