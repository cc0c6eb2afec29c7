"""The plain FP64 update's branches against the FP64 oracle: forcing on the
axes' rows of cubes and boxes (another index on every axis, the largest kept
one), from rest, so that nothing but the forced modes carries the result; and
halving where the exponent cannot be lowered (subnormal states)."""
import numpy as np
import pytest

import oracle
from paper_1003_4322_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("run", [dict(n=16, force_k=1), dict(n=16, force_k=5), dict(n=32, force_k=3, dealias=1),
                                 dict(n=16, ny=24, nz=36, lx=1.0, ly=2.0, lz=3.0, force_k=2),
                                 dict(n=36, ny=16, nz=24, lx=2.0, ly=1.0, lz=1.0, force_k=5, dealias=2)])
def test_forcing_from_rest(ns, run):
    from paper_1003_4322_gb300.solver import Solver
    run = dict(run, nu=0.02, dt=1e-2, force_amp=0.7)
    dims = (run["n"], run.get("ny", run["n"]), run.get("nz", run["n"]))
    a = np.zeros((3, dims[0], dims[1], dims[2] // 2 + 1), dtype=np.complex128)
    want = oracle.step(a, oracle.Params(**run), 2)
    with Solver([run], prec="fp64") as s:
        s.set_state(a)
        s.step(2)
        got = s.get_state()
    assert np.abs(want).max() > 1e-3
    # two steps: a few roundings of each forced mode
    assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max()


@pytest.mark.parametrize("scale", [3e-323, 1e-318, 4e-308])
def test_halving_of_subnormal_states(ns, scale):
    from paper_1003_4322_gb300.solver import Solver
    run = dict(n=16, nu=0.02, dt=1e-2)
    a = inputs.random_hermitian_half_grid((16, 16, 16), 3, seed=8)
    a *= scale / np.abs(a).max()
    with Solver([run], prec="fp64") as s:
        s.set_state(a)
        a = s.get_state()
        want = oracle.step(a, oracle.Params(**run), 1)
        s.step(1)
        got = s.get_state()
    assert np.abs(a).max() > 0
    want[:, 0, 0, 0] = 0   # the update sets the mean of u to zero; the oracle carries it
    # E a, its sum with a_1 and the half: at most half a unit each, in either program
    assert np.abs((got - want).view(np.float64)).max() <= max(4 * 5e-324, 4e-16 * scale)
