"""FP64 r2c of many components: as many as have their line exponents in 4 MiB share
the three passes (more, and the remainder of a larger number, in groups of that
many), with each component's result that of a call of its own, bit for bit."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def _kernels(stream, call):
    """Nodes of the graph that `call` queues on the stream."""
    rt = None
    for name in ("libcudart.so.13", "libcudart.so.12", "libcudart.so"):
        try:
            rt = ctypes.CDLL(name)
            break
        except OSError:
            continue
    s, g, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert rt.cudaStreamBeginCapture(s, 2) == 0   # relaxed
    call()
    assert rt.cudaStreamEndCapture(s, ctypes.byref(g)) == 0
    assert rt.cudaGraphGetNodes(g, None, ctypes.byref(n)) == 0
    assert rt.cudaGraphDestroy(g) == 0
    return n.value


@pytest.mark.parametrize("dims,ncomp,groups", [((16, 16, 16), 64, 1), ((12, 8, 18), 300, 1), ((64, 64, 64), 168, 1),
                                               ((64, 64, 64), 170, 2), ((256, 256, 256), 4, 1),
                                               ((512, 384, 256), 4, 2)])
def test_components_share_the_passes(ns, dims, ncomp, groups):
    import torch
    nx, ny, nz = dims
    stream = torch.cuda.Stream()
    ctx = ns.ns_init([dict(n=8, dt=1e-3)], ns.NS_FP64, stream)
    try:
        with torch.cuda.stream(stream):
            u = torch.randn((ncomp,) + dims, dtype=torch.float64, device="cuda")
            out, one = (torch.empty((m, nx, ny, nz // 2 + 1), dtype=torch.complex128, device="cuda")
                        for m in (ncomp, 1))
        ns.ns_fft_r2c_grid(ctx, nx, ny, nz, ncomp, u, out)
        for c in (0, 2, ncomp // 2, ncomp - 1):
            ns.ns_fft_r2c_grid(ctx, nx, ny, nz, 1, u[c:c + 1], one)
            ns.ns_sync(ctx)
            assert torch.equal(out[c], one[0]), c
        n = _kernels(stream, lambda: ns.ns_fft_r2c_grid(ctx, nx, ny, nz, ncomp, u, out))
        assert n == 3 * groups
    finally:
        ns.ns_destroy(ctx)
