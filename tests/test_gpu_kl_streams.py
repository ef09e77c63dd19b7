"""FP64 fields are the same bits on every stream, however many a program makes and
destroys, and under capture; a call takes no device memory, so it neither waits for
the device nor disturbs a capture that runs on another stream."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _ctx(n, M, tag):
    import paper_1910_04727_gb300 as fm
    r = np.random.default_rng([91, tag])
    c = fm.Context(1, n, M, kl_mode=1)
    c.kl_basis_set(0.3 * r.standard_normal((n * n, M)))
    return c, lambda S: torch.tensor(r.standard_normal((S, M)), device="cuda")


def test_streams_that_come_and_go_give_the_same_bits():
    c, draw = _ctx(16, 48, 1)
    xi = draw(700)
    want = c.kl_field_batch(0, xi)
    torch.cuda.synchronize()
    for _ in range(12):
        s = torch.cuda.ExternalStream(_new_stream())
        with torch.cuda.stream(s):
            got = c.kl_field_batch(0, xi)
        s.synchronize()
        assert torch.equal(got, want)
        _destroy_stream(s.cuda_stream)


def test_overlapping_streams_give_the_same_bits():
    c, draw = _ctx(32, 64, 2)
    xis = [draw(900 + 70 * q) for q in range(7)]
    want = [c.kl_field_batch(0, x) for x in xis]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in xis]
    got = []
    for s, x in zip(streams, xis):
        with torch.cuda.stream(s):
            got.append([c.kl_field_batch(0, x) for _ in range(3)])
    torch.cuda.synchronize()
    for w, g in zip(want, got):
        for k in g:
            assert torch.equal(k, w)


def test_captured_fields_are_the_same_bits():
    c, draw = _ctx(16, 48, 3)
    xi = draw(333)
    want = c.kl_field_batch(0, xi)
    out = torch.empty_like(want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.kl_field_batch(0, xi, out=out)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


def test_a_call_takes_no_device_memory():
    c, draw = _ctx(4, 300, 4)
    small, large = draw(40), draw(60000)
    out = torch.empty((60000, 4, 4), dtype=torch.float64, device="cuda")
    c.kl_field_batch(0, small, out=out[:40])
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    c.kl_field_batch(0, large, out=out)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == before


def test_a_call_beside_another_streams_capture():
    c, draw = _ctx(16, 48, 5)
    xi, x = draw(500), torch.ones(1000, device="cuda")
    out = torch.empty((500, 16, 16), dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):   # captures in the global mode
        y = x * 2
        with torch.cuda.stream(side):
            c.kl_field_batch(0, xi, out=out)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, 2 * x)
    assert torch.equal(out, c.kl_field_batch(0, xi))


def _runtime():
    import ctypes
    lib = ctypes.CDLL("libcudart.so.13")
    return lib


def _new_stream():
    import ctypes
    h = ctypes.c_void_p()
    assert _runtime().cudaStreamCreateWithFlags(ctypes.byref(h), 1) == 0
    return h.value


def _destroy_stream(handle):
    import ctypes
    assert _runtime().cudaStreamDestroy(ctypes.c_void_p(handle)) == 0
