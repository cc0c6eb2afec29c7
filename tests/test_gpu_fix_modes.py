"""Single modes and points of the FP64 transforms: a rounding with a preferred
sign adds up in phase over the lines of a transform and shows in the lowest modes
(r2c) and next to the grid's origin (c2r), where the L2 norm does not see it.  The
modes on the three axes against sums in extended precision.

Tolerance, in units of the rms mode or point: three passes have an L2 error of at
most 6e-16, so an unbiased mode's error is a Gaussian of that size at most, and
the largest of some thousand is within four times that."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 4 * 6e-16
LD, CLD = np.longdouble, np.clongdouble
DIMS = [(256, 256, 256), (96, 144, 192), (8, 512, 486), (1024, 16, 256)]


def _dft(p, sign):
    """The transform of one vector in extended precision."""
    n = len(p)
    t = np.outer(np.arange(n), np.arange(n)) % n
    a = LD("6.283185307179586476925286766559005768") * np.arange(n, dtype=LD) / LD(n)
    c, s = np.cos(a)[t], LD(sign) * np.sin(a)[t]
    return c @ p.real - s @ p.imag, s @ p.real + c @ p.imag


def _axis(a, ax):
    return a[tuple(slice(None) if i == ax else 0 for i in range(3))]


def _others(ax):
    return tuple(i for i in range(3) if i != ax)


@pytest.mark.parametrize("dims", DIMS)
def test_axis_modes_and_points(ns, dims):
    import torch
    rng = np.random.default_rng(sum(dims))
    nz = dims[2]
    u = rng.standard_normal(dims)
    half = dims[:2] + (nz // 2 + 1,)
    x = rng.standard_normal(half) + 1j * rng.standard_normal(half)
    ud, xd = torch.from_numpy(u).cuda()[None], torch.from_numpy(x).cuda()[None]
    X, v = torch.empty_like(xd), torch.empty_like(ud)
    ctx = ns.ns_init([dict(n=8, dt=1e-3)], ns.NS_FP64)
    try:
        ns.ns_fft_r2c_grid(ctx, *dims, 1, ud, X)
        ns.ns_fft_c2r_grid(ctx, *dims, 1, xd, v)
        ns.ns_sync(ctx)
    finally:
        ns.ns_destroy(ctx)
    X, v = X[0].cpu().numpy(), v[0].cpu().numpy()
    w = np.full(nz // 2 + 1, 2.0)
    w[0] = w[-1] = 1.0
    rms_mode, rms_point = np.sqrt(np.prod(dims)), np.sqrt(np.sum(w * np.abs(x) ** 2))
    for ax in range(3):
        got = _axis(X, ax)
        re, im = _dft(np.add.reduce(u, axis=_others(ax), dtype=LD).astype(CLD), -1)
        k = np.arange(len(got))
        err = np.hypot((got.real - re[k]).astype(float), (got.imag - im[k]).astype(float))
        assert err.max() < TOL * rms_mode, (ax, int(err.argmax()))
        p = np.zeros(dims[ax], dtype=CLD)
        s = np.add.reduce(x * w, axis=_others(ax), dtype=CLD)
        p[:len(s)] = s
        err = np.abs((_axis(v, ax) - _dft(p, +1)[0]).astype(float))
        assert err.max() < TOL * rms_point, (ax, int(err.argmax()))
