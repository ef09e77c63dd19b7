"""FP64 fields by exact digit products on the tensor cores.

Against numpy at the edges of its tiles (32 modes, 32 samples, 128 cells) and
of its range (512 modes; 513 take the FP64 contraction).  Tolerance: the sum
of M products rounds below M 2^-53 sum |B xi| in either form and the
exponential below two ulps, so |K - ref| / ref <= 2 M 2^-53 sum |B xi| + 2^-51
covers both sides.  Rows that are not split (values not finite, far scales),
calls on several streams and calls under stream capture give what the plain
sum gives.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _ctx(n, B):
    import paper_1910_04727_gb300 as fm
    c = fm.Context(1, n, B.shape[1], kl_mode=1)
    c.kl_basis_set(B)
    return c


def _check(K, B, xi):
    M = B.shape[1]
    g = xi.astype(np.longdouble) @ B.T.astype(np.longdouble)
    ref = np.exp(g)
    bound = 2 * M * 2.0 ** -53 * (np.abs(xi) @ np.abs(B.T)) + 2.0 ** -51
    err = np.abs((K.reshape(len(xi), -1).astype(np.longdouble) - ref) / ref).astype(float)
    assert np.all(err <= bound), float(np.max(err / bound))


@pytest.mark.parametrize("n,M,S", [(4, 1, 1), (4, 31, 33), (8, 32, 32), (16, 33, 31), (16, 64, 65), (32, 128, 1),
                                   (8, 512, 40), (8, 513, 40), (64, 129, 3)])
def test_fields_at_the_edges(n, M, S):
    r = np.random.default_rng([71, n, M, S])
    B = 0.4 * r.standard_normal((n * n, M)) / np.sqrt(1 + np.arange(M))
    B[1] = 0.0
    B[2] *= 1e-9
    B[3, 0] *= 2.0 ** 12 / np.sqrt(M)
    xi = r.standard_normal((S, M)) * np.where(np.arange(S) % 7 == 3, 1e-3, 1.0)[:, None]
    _check(_ctx(n, B).kl_field_batch(0, torch.tensor(xi, device="cuda")).cpu().numpy(), B, xi)


def test_rows_that_are_not_split():
    r = np.random.default_rng(72)
    B, xi = 0.3 * r.standard_normal((64, 40)), r.standard_normal((9, 40))
    xi[2, 3], xi[4, 1], xi[6] = np.inf, np.nan, 0.0
    xi[5] *= 1e80
    B[11] *= 1e-90
    K = _ctx(8, B).kl_field_batch(0, torch.tensor(xi, device="cuda")).cpu().numpy().reshape(9, 64)
    with np.errstate(all="ignore"):
        ref = np.exp(xi @ B.T)
    for s in range(9):
        assert np.array_equal(np.isnan(K[s]), np.isnan(ref[s]))
        fin = np.isfinite(ref[s]) & (ref[s] != 0)
        assert np.array_equal(K[s][~fin & ~np.isnan(ref[s])], ref[s][~fin & ~np.isnan(ref[s])])
        if s != 5:
            np.testing.assert_allclose(K[s][fin], ref[s][fin], rtol=1e-13)


@pytest.mark.parametrize("scale", [2.0 ** 12, 2.0 ** 40, 2.0 ** 150])
def test_a_large_entry_against_a_zero_coefficient_costs_no_digits(scale):
    r = np.random.default_rng(74)
    B, xi = 0.3 * r.standard_normal((64, 40)), r.standard_normal((33, 40))
    B[5, 7] = scale
    xi[:, 7] = 0.0
    xi[9, 2], B[:, 2] = scale, 0.0
    _check(_ctx(8, B).kl_field_batch(0, torch.tensor(xi, device="cuda")).cpu().numpy(), B, xi)


def test_streams_and_capture():
    r = np.random.default_rng(73)
    B = 0.3 * r.standard_normal((256, 48))
    c = _ctx(16, B)
    xis = [torch.tensor(r.standard_normal((700 + 40 * q, 48)), device="cuda") for q in range(6)]
    want = [c.kl_field_batch(0, x) for x in xis]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in xis]
    got = []
    for s, x in zip(streams, xis):   # more streams than kept buffers, all in flight together
        with torch.cuda.stream(s):
            got.append([c.kl_field_batch(0, x) for _ in range(3)])
    torch.cuda.synchronize()
    for w, g in zip(want, got):
        for k in g:
            torch.testing.assert_close(k, w, rtol=1e-13, atol=0.0)
    out = torch.empty_like(want[0])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.kl_field_batch(0, xis[0], out=out)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    torch.testing.assert_close(out, want[0], rtol=1e-13, atol=0.0)
