"""The shell-spectrum kernels against the FP64 oracle at the edges of their
dispatch: cubes and boxes by rows (from the smallest grid to one with a long
kz row, shells one or many modes wide), and boxes so elongated that their
shells no longer fit the row kernel's shared histogram (above 4096 shells),
which take the gather kernel.  Sums of at most 1e6 FP64 terms: 1e-12."""
import numpy as np
import pytest

import oracle
from paper_1003_4322_gb300 import inputs

pytestmark = pytest.mark.gpu

RUNS = [
    dict(n=8), dict(n=54, dealias=1), dict(n=48, dealias=2), dict(n=8, ny=12, nz=384),
    dict(n=16, ny=16, nz=16, lz=200.0), dict(n=16, ny=12, nz=16, lx=700.0), dict(n=96, ny=8, nz=8, lx=0.25),
]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("i", range(len(RUNS)))
def test_spectra_against_oracle(ns, prec, i):
    from paper_1003_4322_gb300.solver import Solver
    run = dict(RUNS[i], nu=0.01, dt=1e-3)
    dims = (run["n"], run.get("ny", run["n"]), run.get("nz", run["n"]))
    a = inputs.random_hermitian_half_grid(dims, 3, seed=40 + i)
    p = oracle.Params(**run)
    with Solver([run], prec=prec) as s:
        s.set_state(a)
        a = s.get_state()   # as the context holds it
        e, om, spec = s.energy_spectrum()
        h, hspec = s.helicity()
        eb, omb, specb = s.energy_spectra()
    er, omr, sr = oracle.diagnostics(a, p)
    hr, hsr = oracle.helicity(a, p)
    assert spec.shape == sr.shape
    tol = 1e-12
    assert abs(e - er) < tol * er and abs(om - omr) < tol * omr
    assert np.abs(spec - sr).max() < tol * er
    scale = np.sqrt(er * omr)
    assert abs(h - hr) < tol * scale and np.abs(hspec - hsr).max() < tol * scale
    assert eb[0] == e and omb[0] == om and np.array_equal(specb[0], spec)
