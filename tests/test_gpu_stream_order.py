"""Calls of one context on several streams that share its scratch: the library
orders them, so every result is that of the same call alone, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _overlapped(call, inputs, rounds=4):
    """call(x) for every input on a stream of its own, `rounds` times, all in flight together."""
    streams = [torch.cuda.Stream() for _ in inputs]
    torch.cuda.synchronize()
    got = [[] for _ in inputs]
    for _ in range(rounds):
        for i, (s, x) in enumerate(zip(streams, inputs)):
            with torch.cuda.stream(s):
                got[i].append(call(x))
    torch.cuda.synchronize()
    return got


@pytest.mark.parametrize("kl_mode", [2, 3])
def test_tensor_core_fields(kl_mode):
    import paper_1910_04727_gb300 as fm
    r = np.random.default_rng([92, kl_mode])
    c = fm.Context(1, 64, 96, kl_mode=kl_mode)
    c.kl_basis_set(0.2 * r.standard_normal((64 * 64, 96)))
    xis = [torch.tensor(r.standard_normal((3000 - 500 * q, 96)), device="cuda") for q in range(4)]
    want = [c.kl_field_batch(0, x) for x in xis]
    for w, ks in zip(want, _overlapped(lambda x: c.kl_field_batch(0, x), xis)):
        for k in ks:
            assert torch.equal(k, w)
    # a captured call beside them keeps its place: it is replayed after they are done
    out, graph = torch.empty_like(want[1]), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.kl_field_batch(0, xis[1], out=out)
    assert torch.equal(c.kl_field_batch(0, xis[0]), want[0])
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want[1])


@pytest.mark.parametrize("n,S,kw", [(16, 4000, {}), (64, 600, {}), (64, 400, dict(kernel=1)),
                                    (128, 40, dict(precision=1, converged=1, tol=1e-10, max_cycles=100))])
def test_level_wise_solves(n, S, kw):
    import paper_1910_04727_gb300 as fm
    import workloads as W
    c = fm.Context(1, n, 8)
    Ks = [torch.tensor(W.smooth_lognormal_field(n, S=8, tag=5600 + n + q), device="cuda").repeat(S // 8 - q, 1, 1)
          for q in range(4)]
    want = [c.fmg_solve_batch(K, want_p=True, **kw) for K in Ks]
    for w, outs in zip(want, _overlapped(lambda K: c.fmg_solve_batch(K, want_p=True, **kw), Ks, rounds=3)):
        for out in outs:
            for x, y in zip(w, out):
                assert torch.equal(x, y)
