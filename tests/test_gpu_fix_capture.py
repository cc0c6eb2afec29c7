"""Captured FP64 transforms have line exponents of their own: graphs replayed at the
same time on different streams, and beside the context's own calls, give each its
own result, bit for bit; buffers come back when their graphs are gone; and where
there are none (guard bands on), the passes exchange doubles."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _fields(dims, nc, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    u = torch.randn((nc,) + dims, generator=g, dtype=torch.float64, device="cuda")
    return u, torch.zeros((nc,) + dims[:2] + (dims[2] // 2 + 1,), dtype=torch.complex128, device="cuda")


def _capture(ns, ctx, stream, dims, u, out, calls=1):
    import torch
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for _ in range(calls):
            ns.ns_fft_r2c_grid(ctx, *dims, u.shape[0], u, out)
    return graph


@pytest.mark.parametrize("dims,nc", [((128, 128, 128), 3), ((64, 96, 48), 7)])
def test_replayed_side_by_side(ns, dims, nc):
    import torch
    stream = torch.cuda.Stream()
    ctx = ns.ns_init([dict(n=8, dt=1e-3)], ns.NS_FP64, stream)
    graphs = []
    try:
        sets = [_fields(dims, nc, i) for i in range(3)]
        want = []
        for u, out in sets:
            torch.cuda.synchronize()
            ns.ns_fft_r2c_grid(ctx, *dims, nc, u, out)
            ns.ns_sync(ctx)
            want.append(out.clone())
            out.zero_()
        torch.cuda.synchronize()
        graphs = [_capture(ns, ctx, stream, dims, u, out, calls=2) for u, out in sets[:2]]
        others = [torch.cuda.Stream(), torch.cuda.Stream()]
        for _ in range(40):
            for graph, s in zip(graphs, others):
                with torch.cuda.stream(s):
                    graph.replay()
            ns.ns_fft_r2c_grid(ctx, *dims, nc, *sets[2])
        torch.cuda.synchronize()
        for (_, out), w in zip(sets, want):
            assert torch.equal(out, w)
    finally:
        del graphs
        ns.ns_destroy(ctx)


def test_buffers_come_back(ns):
    """More captures than the buffers of all of them would fit, one after the other."""
    import torch
    dims = (512, 512, 16)   # 3.1 MiB of exponents each, 256 MiB in all
    stream = torch.cuda.Stream()
    ctx = ns.ns_init([dict(n=8, dt=1e-3)], ns.NS_FP64, stream)
    try:
        u, out = _fields(dims, 3, 5)
        torch.cuda.synchronize()
        ns.ns_fft_r2c_grid(ctx, *dims, 3, u, out)
        ns.ns_sync(ctx)
        want = out.clone()
        for _ in range(100):
            out.zero_()
            torch.cuda.synchronize()
            graph = _capture(ns, ctx, stream, dims, u, out)
            graph.replay()
            torch.cuda.synchronize()
            del graph
        assert torch.equal(out, want)   # doubles between the passes round otherwise
    finally:
        ns.ns_destroy(ctx)


def test_without_buffers():
    env = dict(os.environ, NS_GUARD="1")
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-p", "no:cacheprovider",
                        "tests/test_gpu_fix.py::test_capture_without_exponent_buffers"], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]
