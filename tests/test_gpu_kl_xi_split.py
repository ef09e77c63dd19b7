"""BF16x3 fields of one mode with a unit basis entry: K = exp(hi + lo), hi and lo the
coefficient's first two BF16 parts (round to nearest even, numpy).  The FP32 sum of the two
rounds by 2^-24 |xi| and the FP32 exponential by two ulps: 1e-6 for |xi| <= 4 (a wrong
last bit of lo is 4e-6 at 1).  Ties, carries, signed zeros, subnormals and values far out."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _bf16(v):
    m, e = np.frexp(v)
    return np.ldexp(np.rint(m * 256), e - 8)


@pytest.mark.parametrize("S", [5, 4096, 5001])
def test_coefficient_parts(S):
    import paper_1910_04727_gb300 as fm
    r = np.random.default_rng(81)
    xi = r.uniform(-4, 4, S) * 2.0 ** -r.integers(0, 12, S)
    ties = [1 + 2.0 ** -8, 1 + 3 * 2.0 ** -8, 2 - 2.0 ** -9, 1 + 2.0 ** -8 + 2.0 ** -52, 1.0 + 2.0 ** -17 + 2.0 ** -9,
            -(2 - 2.0 ** -52), 0.0, -0.0, 5e-324, 1e-300, -1e-40, 2.0 ** -63, 2.0 ** -64, 3.999999999999999]
    xi[:min(S, len(ties))] = ties[:S]
    c = fm.Context(1, 4, 1, kl_mode=3)
    c.kl_basis_set(np.ones((16, 1)))
    K = c.kl_field_batch(0, torch.tensor(xi[:, None], device="cuda")).cpu().numpy().reshape(S, 16)
    hi = _bf16(xi)
    want = np.exp(hi + _bf16(xi - hi))
    assert np.max(np.abs(K / want[:, None] - 1)) <= 1e-6
    bad = np.array([np.inf, -np.inf, np.nan, 1e39, 0.5])
    K = c.kl_field_batch(0, torch.tensor(bad[:, None], device="cuda")).cpu().numpy().reshape(5, 16)
    assert np.isnan(K[:4]).all()
    assert np.max(np.abs(K[4] / np.exp(0.5) - 1)) <= 1e-6
