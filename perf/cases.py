"""The work this library is run for, as cases that can be timed and checked.

Two families, both through the public Python layer over the C ABI:

* time integration (`Solver.set_state` / `set_states` -> `step` ->
  `get_state`): a user loads a spectral state, advances it and reads it back.
  The FP64 form also reads the energy spectrum, as the monitoring of a run
  does.  The FP32 form's states come back through the same complex128 buffers
  and are kept in single precision, the precision they were computed in;
* the standalone 3D transforms (`fft_r2c`, `fft_c2r`, their grid forms, and
  the allocation-free c2r).

Buffers stay on the device throughout.  Inputs are seeded: turbulence-like
solenoidal fields (a k^-5/3 shell spectrum with an exponential tail, rms 1)
for the solver, Gaussian fields for the transforms.
"""
from __future__ import annotations

import math

import torch

from paper_1003_4322_gb300 import _native as nat
from paper_1003_4322_gb300.solver import Solver

# even 2^a 3^b lengths of the range that is drawn from
SIZES = (32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324, 384, 432, 512)


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------ cases

def _solver_case(prec, n, steps, ny=0, nz=0, lx=1.0, ly=1.0, lz=1.0, start="turbulent", nu=2e-3, dt=1e-3,
                 force_amp=0.0, force_k=0, dealias=0, rot=0.0, mhd=0, eta=0.0, count=1):
    return dict(kind="solver", prec=prec, n=n, ny=ny or n, nz=nz or n, lx=lx, ly=ly, lz=lz, steps=steps, start=start,
                nu=nu, dt=dt, force_amp=force_amp, force_k=force_k, dealias=dealias, rot=rot, mhd=mhd, eta=eta,
                count=count)


def listed():
    return [
        # the smallest run that is used in earnest (a check or a teaching
        # case): a forced 32^3 box in FP64, ten steps; launches and latency
        dict(_solver_case("fp64", 32, 10, nu=0.01, force_amp=0.5, force_k=3), name="step64_32"),
        # Taylor-Green at 256^3 in FP64: the common validation run
        dict(_solver_case("fp64", 256, 2, start="taylor-green", nu=1 / 1600, dt=2e-3), name="step64_256_tg"),
        # 512^3 forced turbulence in FP64: the production run of the plain form
        dict(_solver_case("fp64", 512, 1, force_amp=0.5, force_k=3), name="step64_512_forced"),
        # a rotating box of another aspect ratio in FP64: ragged axes with
        # factors of three, the spherical dealiasing rule
        dict(_solver_case("fp64", 96, 2, ny=144, nz=192, lx=1.0, ly=1.5, lz=2.0, nu=5e-3, force_amp=0.5, force_k=2,
                          dealias=1, rot=1.0), name="step64_box96x144x192"),
        # a single small run in FP32: latency of the step graph
        dict(_solver_case("fp32", 64, 20, nu=5e-3), name="step32_64"),
        # 512^3 forced turbulence in FP32: the production run of the fused form
        dict(_solver_case("fp32", 512, 4, force_amp=0.5, force_k=3), name="step32_512_forced"),
        # a parameter study: 48 runs at 64^3, 96^3 and 128^3, advanced together
        dict(_solver_case("fp32", 0, 5, nu=5e-3, count=48), name="step32_ensemble48"),
        # forced MHD turbulence at 256^3 in FP32
        dict(_solver_case("fp32", 256, 4, force_amp=0.5, force_k=3, mhd=1, eta=2e-3), name="step32_mhd256"),
        # a flat box in FP32
        dict(_solver_case("fp32", 512, 4, nz=256, lz=0.5, force_amp=0.5, force_k=4), name="step32_box512x512x256"),
        # post-processing transforms of a vector field: FP32 at 512^3, FP64 at
        # 256^3, and the smallest one, the allocation-free c2r at 64^3
        dict(kind="fft", prec="fp32", nx=512, ny=512, nz=512, ncomp=3, name="fft32_512"),
        dict(kind="fft", prec="fp64", nx=256, ny=256, nz=256, ncomp=3, name="fft64_256"),
        dict(kind="noalloc", n=64, ncomp=3, name="fft32_noalloc64"),
    ]


def _pick(rng, lo, hi):
    """A supported length in [lo, hi], spread evenly over its logarithm."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ok = [s for s in SIZES if lo <= s <= hi]
    return min(ok, key=lambda s: abs(math.log(s / x)))


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "fp64", "fp32", "fp32", "fp32", "ensemble", "fft32", "fft64", "noalloc"])
    if kind == "noalloc":
        return dict(kind="noalloc", n=_pick(rng, 32, 128), ncomp=rng.randint(4, 40))
    if kind in ("fft32", "fft64"):
        hi = 512 if kind == "fft32" else 384
        nx = _pick(rng, 32, hi)
        ny, nz = (nx, nx) if rng.random() < 0.5 else (_pick(rng, 32, hi), _pick(rng, 32, hi))
        return dict(kind="fft", prec="fp32" if kind == "fft32" else "fp64", nx=nx, ny=ny, nz=nz,
                    ncomp=rng.randint(1, 3))
    if kind == "ensemble":
        return _solver_case("fp32", 0, rng.randint(2, 6), nu=rng.uniform(5e-3, 2e-2), count=rng.randint(2, 48))
    # a run of either form: what a user sets is drawn with it
    hi = 384 if kind == "fp64" else 512
    n = _pick(rng, 32, hi)
    opt = dict(nu=rng.uniform(1e-3, 1e-2), dt=1e-3)
    what = rng.choice(["plain", "forced", "rotating", "mhd", "box", "spherical", "shifted"])
    if what in ("mhd", "shifted"):
        n = min(n, 256)
    if what == "forced":
        opt.update(force_amp=0.5, force_k=rng.randint(1, 4))
    elif what == "rotating":
        opt.update(rot=rng.uniform(0.5, 4.0))
    elif what == "mhd":
        opt.update(mhd=1, eta=rng.uniform(1e-3, 1e-2))
    elif what == "box":
        opt.update(ny=_pick(rng, 32, hi), nz=_pick(rng, 32, hi), lx=rng.choice([0.5, 1.0, 2.0]),
                   ly=rng.choice([1.0, 1.5]), lz=rng.choice([0.5, 1.0, 2.0]), dealias=rng.randint(0, 1))
    elif what == "spherical":
        opt.update(dealias=1)
    elif what == "shifted":
        opt.update(dealias=2)
    points = n * opt.get("ny", n) * opt.get("nz", n) * (2 if what in ("mhd", "shifted") else 1)
    return _solver_case(kind, n, max(1, min(rng.randint(2, 6), 24_000_000 // points)), **opt)


# ------------------------------------------------------------------ states

def _runs(case):
    """The run parameters of a case, one dict per run."""
    keys = ("nu", "dt", "force_amp", "force_k", "dealias", "rot", "mhd", "eta")
    base = {k: case[k] for k in keys}
    if case["count"] == 1:
        return [dict(base, n=case["n"], ny=case["ny"], nz=case["nz"], lx=case["lx"], ly=case["ly"], lz=case["lz"])]
    sizes = (64, 96, 128)   # three resolutions, each with its share of the viscosities
    cnt = case["count"]
    return [dict(base, n=sizes[3 * i // cnt], nu=base["nu"] * (1 + i / cnt)) for i in range(cnt)]


def _grid(run):
    n = run["n"]
    return ((n, run.get("ny", n), run.get("nz", n)), (run.get("lx", 1.0), run.get("ly", 1.0), run.get("lz", 1.0)))


def _indices(dims):
    """Signed grid indices along the three axes, broadcastable."""
    nx, ny, nz = dims
    f = lambda n: torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=_dev()).round()  # noqa: E731
    mz = torch.arange(nz // 2 + 1, dtype=torch.float64, device=_dev())
    return f(nx)[:, None, None], f(ny)[None, :, None], mz[None, None, :]


def _waves(run):
    dims, l = _grid(run)
    return [m / li for m, li in zip(_indices(dims), l)]


def _mask(run):
    dims, _ = _grid(run)
    m, D = _indices(dims), math.lcm(*dims)
    keep = torch.ones((), dtype=torch.bool, device=_dev())
    for mi, n in zip(m, dims):
        keep = keep & (mi.abs() * 2 < n if run["dealias"] == 2 else mi.abs() * 3 < n)
    if run["dealias"]:
        r2 = sum((3 * mi * (D // n)) ** 2 for mi, n in zip(m, dims))   # exact in 53 bits
        keep = keep & (r2 < run["dealias"] * D * D)
    return keep


def _random_field(run, seed, rms):
    """A solenoidal field with a turbulent spectrum: normalised coefficients
    in the half layout, complex128."""
    dims, l = _grid(run)
    g = torch.Generator(device=_dev())
    g.manual_seed(seed)
    a = torch.stack([torch.fft.rfftn(torch.randn(dims, generator=g, dtype=torch.float64, device=_dev()),
                                     norm="forward") for _ in range(3)])
    k = _waves(run)
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    safe = torch.where(k2 > 0, k2, torch.ones_like(k2))
    tail = min(n / li for n, li in zip(dims, l)) / 9.0
    a *= safe ** (-11.0 / 12.0) * torch.exp(-safe.sqrt() / tail) * _mask(run) * (k2 > 0)
    a -= torch.stack([ki.expand(k2.shape) for ki in k]) * ((k[0] * a[0] + k[1] * a[1] + k[2] * a[2]) / safe)
    w = torch.full((dims[2] // 2 + 1,), 2.0, dtype=torch.float64, device=_dev())
    w[0] = w[-1] = 1.0
    a *= rms / math.sqrt(float((w * (a.real ** 2 + a.imag ** 2)).sum()) / 3.0)
    return a


def _taylor_green(run, seed):
    """(sin x cos y cos z, -cos x sin y cos z, 0) with a small perturbation."""
    n = run["n"]
    x = torch.arange(n, dtype=torch.float64, device=_dev()) * (2 * math.pi / n)
    s, c = torch.sin(x), torch.cos(x)
    u = torch.zeros((3, n, n, n), dtype=torch.float64, device=_dev())
    u[0] = s[:, None, None] * c[None, :, None] * c[None, None, :]
    u[1] = -c[:, None, None] * s[None, :, None] * c[None, None, :]
    return torch.fft.rfftn(u, dim=(1, 2, 3), norm="forward") * _mask(run) + _random_field(run, seed, 1e-2)


def _states(case, seed):
    """Initial states: per run a list of fields (velocity, and the magnetic
    field of an MHD run with its mean along z)."""
    out = []
    for i, run in enumerate(_runs(case)):
        s = 1000 * seed + 2 * i
        fields = [_taylor_green(run, s) if case["start"] == "taylor-green" else _random_field(run, s, 1.0)]
        if run["mhd"]:
            b = _random_field(run, s + 1, 0.7)
            b[2, 0, 0, 0] = 0.5
            fields.append(b)
        out.append(fields)
    return out


def _gauss(shape, dtype, seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, dtype=dtype, device=_dev())


def _fft_inputs(case, seed):
    """A real field for r2c and a half-layout spectrum for c2r."""
    if case["kind"] == "noalloc":
        dims, dt = (case["n"],) * 3, torch.float32
    else:
        dims, dt = (case["nx"], case["ny"], case["nz"]), torch.float32 if case["prec"] == "fp32" else torch.float64
    u = _gauss((case["ncomp"],) + dims, dt, 2 * seed)
    x = torch.fft.rfftn(_gauss((case["ncomp"],) + dims, dt, 2 * seed + 1), dim=(1, 2, 3), norm="ortho")
    return u, x.contiguous()


# ------------------------------------------------------------------ interface

def prepare(case, seed):
    if case["kind"] == "noalloc":
        _, x = _fft_inputs(case, seed)
        n = case["n"]
        st = dict(kind="noalloc", n=n, ncomp=case["ncomp"], x=x, v=torch.empty((case["ncomp"], n, n, n), device=_dev()))
        # a program makes its first call on a device at start-up
        nat.ns_fft_c2r_noalloc(n, case["ncomp"], x, st["v"])
        return st
    if case["kind"] == "fft":
        u, x = _fft_inputs(case, seed)
        dims = (case["nx"], case["ny"], case["nz"])
        s = Solver([dict(n=8, nu=0.0, dt=1.0)], prec=case["prec"])
        st = dict(kind="fft", cube=len(set(dims)) == 1, s=s, u=u, x=x, uh=torch.empty_like(x), v=torch.empty_like(u))
        run(st)   # a program's plan: the tables and launch shapes of these lengths
        s.sync()
        return st
    states = _states(case, seed)
    s = Solver(_runs(case), prec=case["prec"])
    out = [[torch.empty_like(f) for f in fields] for fields in states]
    st = dict(kind="solver", s=s, a=states, out=out, steps=case["steps"], prec=case["prec"])
    if case["count"] > 1:
        st["first"] = [fields[0] for fields in states]
    return st


def run(state):
    s = state.get("s")
    if state["kind"] == "noalloc":
        nat.ns_fft_c2r_noalloc(state["n"], state["ncomp"], state["x"], state["v"])
        return [state["v"]]
    if state["kind"] == "fft":
        if state["cube"]:
            s.fft_r2c(state["u"], state["uh"])
            s.fft_c2r(state["x"], state["v"])
        else:
            s.fft_r2c_grid(state["u"], state["uh"])
            s.fft_c2r_grid(state["x"], state["v"])
        return [state["uh"], state["v"]]
    if "first" in state:
        s.set_states(state["first"])
    else:
        for f, a in enumerate(state["a"][0]):
            s.set_field(f, a)
    s.step(state["steps"])
    if state["prec"] == "fp64":
        energy, enstrophy, spec = s.energy_spectrum()
        return [s.get_field(f, 0, o) for f, o in enumerate(state["out"][0])] + [energy, enstrophy, spec]
    return [s.get_field(f, r, o).to(torch.complex64) for r, fields in enumerate(state["out"])
            for f, o in enumerate(fields)]


def work(case):
    """Inputs read once and outputs written once; the flops of the line
    transforms (5 n log2 n each, half for real lines) that the retained modes
    need, which are all but a few per cent of the arithmetic."""
    if case["kind"] == "noalloc":
        n, v = case["n"], case["n"] ** 3 * case["ncomp"]
        return dict(bytes=4.0 * v * (1 + 2 / n) + 4.0 * v, flops=2.5 * v * 3 * math.log2(n))
    if case["kind"] == "fft":
        V = case["nx"] * case["ny"] * case["nz"] * case["ncomp"]
        b = 4 if case["prec"] == "fp32" else 8
        return dict(bytes=2.0 * b * V * (2 + 2 / case["nz"]),
                    flops=2 * 2.5 * V * math.log2(case["nx"] * case["ny"] * case["nz"]))
    byt = flo = 0.0
    for r in _runs(case):
        (nx, ny, nz), _ = _grid(r)
        V, fields = nx * ny * nz, 2 if r["mhd"] else 1
        kept = min(1.0, math.sqrt(2) * 2 / 3) if r["dealias"] == 2 else 2 / 3   # per axis
        byt += 2 * fields * 3 * 16.0 * nx * ny * (nz // 2 + 1) * kept ** 3 + \
            (24.0 if case["prec"] == "fp32" else 0.0) * fields * nx * ny * (nz // 2 + 1)
        lines = 18 if r["mhd"] else 9 * (2 if r["dealias"] == 2 else 1)
        flo += case["steps"] * 2 * lines * 2.5 * V * (kept ** 2 * math.log2(nx) + kept * math.log2(ny) + math.log2(nz))
    return dict(bytes=byt, flops=flo)


# ------------------------------------------------------------------ in 64 bits

def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _curl(k, a):
    return 1j * torch.stack([k[1] * a[2] - k[2] * a[1], k[2] * a[0] - k[0] * a[2], k[0] * a[1] - k[1] * a[0]])


def _advance(run, fields, steps):
    """Integrating-factor Heun steps of the rotational-form equations (with
    the Lorentz force and the induction equation for two fields)."""
    dims, _ = _grid(run)
    k, m, keep = _waves(run), _indices(dims), _mask(run)
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    safe = torch.where(k2 > 0, k2, torch.ones_like(k2))
    inv = lambda a: torch.fft.irfftn(a, s=dims, dim=(1, 2, 3), norm="forward")  # noqa: E731
    fwd = lambda u: torch.fft.rfftn(u, dim=(1, 2, 3), norm="forward")  # noqa: E731
    E = [torch.exp(-c * k2 * run["dt"]) for c in (run["nu"], run["eta"])]
    f = None
    if run["force_k"] > 0 and run["force_amp"] != 0.0:
        x, y, z = (2 * math.pi * li * torch.arange(n, dtype=torch.float64, device=_dev()) / n
                   for n, li in zip(*_grid(run)))
        x, y, z, kf = x[:, None, None], y[None, :, None], z[None, None, :], run["force_k"]
        one = torch.ones(dims, dtype=torch.float64, device=_dev())
        f = run["force_amp"] * fwd(torch.stack([(torch.sin(kf * p) + torch.cos(kf * q)) * one
                                                for p, q in ((z, y), (x, z), (y, x))])) * keep * (k2 > 0)

    def product(a):
        """The transformed products of the nonlinear terms, dealiased."""
        u = inv(a[0])
        n = _cross(u, inv(_curl(k, a[0])))
        if len(a) == 1:
            return [fwd(n)]
        b = inv(a[1])
        n += _cross(inv(_curl(k, a[1])), b)
        return [fwd(n), fwd(_cross(u, b))]

    def rate(a):
        p = product(a)
        if run["dealias"] == 2:   # also on the grid shifted by half a spacing
            sh = torch.exp(1j * math.pi * (m[0] / dims[0] + m[1] / dims[1] + m[2] / dims[2]))
            p = [0.5 * (p[0] + product([a[0] * sh])[0] * sh.conj())]
        n = p[0] * keep
        if run["rot"] != 0.0:
            n[0] += 2 * run["rot"] * a[0][1]
            n[1] -= 2 * run["rot"] * a[0][0]
        n -= torch.stack([ki.expand(k2.shape) for ki in k]) * ((k[0] * n[0] + k[1] * n[1] + k[2] * n[2]) / safe)
        n *= (k2 > 0)
        if f is not None:
            n += f
        return [n] + [_curl(k, q) * keep for q in p[1:]]

    dt = run["dt"]
    a = [x * keep for x in fields]
    for _ in range(steps):
        a1 = [e * (x + dt * n) for e, x, n in zip(E, a, rate(a))]
        a = [0.5 * (e * x + x1 + dt * n) for e, x, x1, n in zip(E, a, a1, rate(a1))]
    return a


def _diagnostics(run, a):
    """Energy, enstrophy and shell spectrum (shells round-half-up(|k| / k_min))."""
    dims, l = _grid(run)
    k = _waves(run)
    k2 = (k[0] ** 2 + k[1] ** 2 + k[2] ** 2).flatten()
    w = torch.ones(dims[2] // 2 + 1, dtype=torch.float64, device=_dev())
    w[0] = w[-1] = 0.5
    e = (w * (a.real ** 2 + a.imag ** 2)).sum(0).flatten()
    lm = max(l)
    bins = math.ceil(math.sqrt(sum((n // 2 / li) ** 2 for n, li in zip(dims, l))) * lm) + 1
    shell = torch.floor(k2.sqrt() * lm + 0.5).long()
    spec = torch.zeros(bins, dtype=torch.float64, device=_dev()).index_add_(0, shell, e)
    return [float(e.sum()), float((k2 * e).sum()), spec.cpu().numpy()]


def exact(case, seed):
    if case["kind"] in ("fft", "noalloc"):
        u, x = _fft_inputs(case, seed)
        dims = u.shape[1:]
        v = torch.fft.irfftn(x.to(torch.complex128), s=dims, dim=(1, 2, 3), norm="forward")
        if case["kind"] == "noalloc":
            return [v]
        return [torch.fft.rfftn(u.double(), dim=(1, 2, 3)), v]
    out = []
    for run_, fields in zip(_runs(case), _states(case, seed)):
        a = _advance(run_, fields, case["steps"])
        out += a
        if case["prec"] == "fp64":
            # an MHD run's spectrum is that of its velocity
            out += _diagnostics(run_, a[0])
    return out
