"""The FP64 transforms' block fixed-point passes at the edges of their range,
through ns_fft_r2c_grid / ns_fft_c2r_grid against the FP64 oracle: every
radix plan (axis lengths with one to four stages, with and without powers of
three, the shortest and the longest), tiles with fewer columns than a CTA,
lines far outside the range of the FP32 scale sum, zero lines, non-finite
entries, results at the ends of the double range.

Tolerance: a line pass has a relative L2 error of at most 3.4e-16 (flat lines
of 1024 points), three passes 6e-16 in quadrature, and the oracle's own FP64
recursion about as much; 2e-15 leaves a factor of two."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TOL = 2e-15
DIMS = [(8, 8, 8), (12, 18, 24), (16, 36, 54), (54, 32, 162), (108, 8, 486), (1024, 8, 16), (8, 972, 12),
        (12, 16, 1024), (48, 64, 96), (288, 16, 72), (8, 768, 8), (36, 512, 10 + 2)]


def _both(ns, u, uh):
    """(r2c of u, c2r of uh) for arrays [ncomp][nx][ny][nz], [..][nz/2+1]."""
    import torch
    nc, nx, ny, nz = u.shape
    ud, xd = torch.from_numpy(u).cuda(), torch.from_numpy(uh).cuda()
    out, back = torch.empty_like(xd), torch.empty_like(ud)
    ctx = ns.ns_init([dict(n=8, dt=1e-3)], ns.NS_FP64)
    try:
        ns.ns_fft_r2c_grid(ctx, nx, ny, nz, nc, ud, out)
        ns.ns_fft_c2r_grid(ctx, nx, ny, nz, nc, xd, back)
        ns.ns_sync(ctx)
    finally:
        ns.ns_destroy(ctx)
    return out.cpu().numpy(), back.cpu().numpy()


def _inputs(dims, seed, nc=1):
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((nc,) + dims)
    return u, np.fft.rfftn(rng.standard_normal((nc,) + dims), axes=(1, 2, 3))


def _rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("log2", [0, -90, 95, -500, 500, -990])
def test_scales(ns, dims, log2):
    """The result follows a power-of-two scale of the input."""
    u, x = _inputs(dims, 1 + sum(dims))
    f = 2.0 ** log2
    X, v = _both(ns, u * f, x * f)
    assert _rel(X / f, oracle.fft3_r2c(u)) < TOL
    assert _rel(v / f, oracle.fft3_c2r(x)) < TOL


@pytest.mark.parametrize("dims", [(16, 12, 24), (96, 8, 48)])
def test_mixed_lines(ns, dims):
    """Planes and lines of very different magnitude in one CTA, zero lines among them."""
    u, x = _inputs(dims, 7)
    u[:, :, ::3] *= 2.0 ** -150
    u[:, 1::4] = 0
    x[:, :, :, 1::2] *= 2.0 ** -160
    x[:, :, ::5, ::3] = 0
    x[0, :, :, 0] = x[0, :, :, -1] = 0
    X, v = _both(ns, u, x)
    assert _rel(X, oracle.fft3_r2c(u)) < TOL
    assert _rel(v, oracle.fft3_c2r(x)) < TOL
    z, w = _both(ns, np.zeros_like(u), np.zeros_like(x))
    assert not z.any() and not w.any()


def test_ends_of_the_double_range(ns):
    dims = (8, 12, 16)
    u, x = np.zeros((1,) + dims), np.zeros((1, 8, 12, 9), dtype=complex)
    for a in (2.0 ** 1022, -2.0 ** -1022, 2.0 ** -1060, 2.0 ** -1074):
        u[0, 0, 0, 0] = a
        x[0, 0, 0, 0] = a
        X, v = _both(ns, u, x)
        assert (X == a).all() and (v == a).all(), a
    u[...] = 2.0 ** 1020
    X, _ = _both(ns, u, x)
    # 16 * 2^1020 overflows in the z pass; an infinity makes its later lines NaN
    assert not np.isfinite(X[0, 0, 0, 0].real)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_entries_spread(ns, bad):
    u, x = _inputs((16, 24, 12), 5, nc=2)
    u[1, 3, 5, 7] = bad
    x[1, 3, 5, 2] = bad
    X, v = _both(ns, u, x)
    assert np.isfinite(X[0]).all() and np.isfinite(v[0]).all()
    assert not np.isfinite(X[1]).any() and not np.isfinite(v[1]).any()


def test_capture_without_exponent_buffers(ns):
    """Under capture nothing is allocated: a grid larger than any before keeps
    doubles between its passes (and, replayed, gives the same transform)."""
    import torch
    stream = torch.cuda.Stream()
    ctx = ns.ns_init([dict(n=8, dt=1e-3)], ns.NS_FP64, stream)
    try:
        for dims in ((24, 8, 16), (8, 24, 16)):   # the tables of 8, 16, 24
            small = torch.zeros((1,) + dims, dtype=torch.float64, device="cuda")
            o = torch.empty((1,) + dims[:2] + (9,), dtype=torch.complex128, device="cuda")
            torch.cuda.synchronize()
            ns.ns_fft_r2c_grid(ctx, *dims, 1, small, o)
            ns.ns_sync(ctx)
        u, _ = _inputs((24, 24, 24), 3, nc=4)
        ud = torch.zeros(u.shape, dtype=torch.float64, device="cuda")
        out = torch.empty((4, 24, 24, 13), dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            ns.ns_fft_r2c(ctx, 24, 4, ud, out)
        ud.copy_(torch.from_numpy(u))
        graph.replay()
        torch.cuda.synchronize()
        ref = oracle.fft3_r2c(u)
        assert _rel(out.cpu().numpy(), ref) < TOL
        ns.ns_fft_r2c(ctx, 24, 4, ud, out)   # the ordinary way, components in groups of three
        ns.ns_sync(ctx)
        assert _rel(out.cpu().numpy(), ref) < TOL
    finally:
        ns.ns_destroy(ctx)
