"""FP64 runs transform u and its curl through the same launches where their buffers
hold six components, and one after the other where they hold three (larger grids,
or little free memory).  The lines are the same either way, so the states and
spectra agree bit for bit, on cubes, boxes, with rotation, MHD, the phase shift and
with every line transformed."""
import numpy as np
import pytest

from paper_1003_4322_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = [
    (dict(n=32, force_amp=0.5, force_k=3), "1"),
    (dict(n=54, dealias=1, rot=1.5), "1"),
    (dict(n=24, ny=16, nz=36, lx=1.5, ly=1.0, lz=0.75, dealias=1), "1"),
    (dict(n=24, ny=16, nz=36, lx=1.5, ly=1.0, lz=0.75), "0"),
    (dict(n=36, ny=16, nz=24, lx=2.0, ly=1.0, lz=1.0, force_amp=0.3, force_k=2, dealias=2), "1"),
    (dict(n=24, mhd=1, eta=0.03), "1"),
    (dict(n=16, ny=12, nz=24, lx=1.0, ly=0.75, lz=1.5, mhd=1, eta=0.03), "0"),
]


def _run(ns, run, both, monkeypatch):
    from paper_1003_4322_gb300.solver import Solver
    monkeypatch.setenv("NS_PLAIN_BOTH", both)
    dims = (run["n"], run.get("ny", run["n"]), run.get("nz", run["n"]))
    fields = range(1 + run.get("mhd", 0))
    with Solver([run], prec="fp64") as s:
        for f in fields:
            s.set_field(f, 1e-3 * inputs.random_hermitian_half_grid(dims, 3, seed=80 + f))
        s.step(3)
        out = [s.get_field(f) for f in fields] + list(s.energy_spectrum())
        names = {name for name, _, _ in ns.ns_kernel_census(s.ctx, 1)}
    return out, names


@pytest.mark.parametrize("i", range(len(CASES)))
def test_three_components_at_a_time(ns, i, monkeypatch):
    run, prune = CASES[i]
    monkeypatch.setenv("NS_PLAIN_PRUNE", prune)
    run = dict(run, nu=0.02, dt=2e-3)
    six, names6 = _run(ns, run, "1", monkeypatch)
    three, names3 = _run(ns, run, "0", monkeypatch)
    assert {"curl_x_inverse6", "fft_y_inverse6", "fft_z_c2r6"} <= names6
    assert {"fft_x_inverse", "curl_x_inverse"} <= names3 and not any(n.endswith("6") for n in names3)
    assert np.abs(six[0]).max() > 0
    for a, b in zip(six, three):
        assert np.array_equal(a, b)
