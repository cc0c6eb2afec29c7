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


@pytest.mark.parametrize("dims", [(256, 16, 16), (144, 12, 8), (486, 8, 12), (1024, 8, 8), (16, 162, 8)])
def test_coherent_lines_at_the_limit_of_the_range(ns, dims):
    """A plane wave puts every entry of a line in phase at one output, which comes as
    near to the largest representable value as the line's scale allows (amplitudes
    between two powers of two): nothing overflows.  Error of the modes over that
    output: the input's rounding, three passes and the result's, 2^-53 each at most;
    eight of them."""
    import torch
    nx, ny, nz = dims
    x, y = np.arange(nx)[:, None, None], np.arange(ny)[None, :, None]
    nc = 32
    amp = 2.0 ** (np.arange(nc) / nc)
    u, want = np.empty((nc,) + dims), np.zeros((nc, nx, ny, nz // 2 + 1), dtype=complex)
    for c in range(nc):
        kx, ky = (7 * c + 1) % (nx // 2 - 1) + 1, (3 * c + 1) % (ny // 2 - 1) + 1
        ph = 0.2 * c
        turn = LD("6.283185307179586476925286766559005768") / LD(nx * ny)
        wave = np.cos(((kx * x * ny + ky * y * nx) % (nx * ny)).astype(LD) * turn + LD(ph))
        u[c] = (LD(amp[c]) * wave).astype(float)
        a = 0.5 * amp[c] * np.prod(dims) * np.exp(1j * ph)
        want[c, kx, ky, 0], want[c, -kx, -ky, 0] = a, np.conj(a)
    ud = torch.from_numpy(u).cuda()
    X, v = torch.empty((nc, nx, ny, nz // 2 + 1), dtype=torch.complex128, device="cuda"), torch.empty_like(ud)
    ctx = ns.ns_init([dict(n=8, dt=1e-3)], ns.NS_FP64)
    try:
        ns.ns_fft_r2c_grid(ctx, *dims, nc, ud, X)
        ns.ns_fft_c2r_grid(ctx, *dims, nc, torch.from_numpy(want).cuda(), v)
        ns.ns_sync(ctx)
    finally:
        ns.ns_destroy(ctx)
    peak = 0.5 * amp * np.prod(dims)
    assert (np.abs(X.cpu().numpy() - want).max(axis=(1, 2, 3)) <= 8 * 2.0 ** -53 * peak).all()
    back = v.cpu().numpy() / np.prod(dims)
    assert (np.abs(back - u).max(axis=(1, 2, 3)) <= 8 * 2.0 ** -53 * amp).all()
