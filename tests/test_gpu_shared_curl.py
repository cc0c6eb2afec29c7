"""Pass A of the fused form with shared transforms (the curl's transforms
formed from the velocity's, fused_kA3.cu) in every compiled shape, forced
through NS_FORCE_STRIDED, against the plain FP64 form: the smallest compiled
cubes, radix-3 lengths, a grid on a box (scaled wavenumbers, ragged last
column tile) and MHD (the pass on the magnetic block).  The FP32 solver
tolerance of the other tests, 2e-5, on modes of every direction."""
import numpy as np
import pytest

from paper_1003_4322_gb300 import inputs
from tests.spectral_ref import rel_l2

pytestmark = pytest.mark.gpu

RUNS = [dict(n=64), dict(n=96, rot=1.5), dict(n=128, dealias=1), dict(n=96, ny=96, nz=48, lx=1.0, ly=2.0, lz=0.5),
        dict(n=64, mhd=1, eta=3e-3)]
SHAPES = [(E, ct) for E in (8, 12, 16, 32) for ct in (8, 16)]


@pytest.mark.parametrize("i", range(len(RUNS)))
def test_against_fp64(ns, i, monkeypatch):
    from paper_1003_4322_gb300.solver import Solver
    run = dict(RUNS[i], nu=2e-3, dt=1e-3)
    dims = (run["n"], run.get("ny", run["n"]), run.get("nz", run["n"]))
    fields = [1e-3 * inputs.random_hermitian_half_grid(dims, 3, seed=60 + i + f) for f in range(1 + run.get("mhd", 0))]

    def go(prec):
        with Solver([run], prec=prec) as s:
            d = ns.ns_describe_run(s.ctx, 0).get("passes", {}).get("A_x_inverse_curl")
            for f, a in enumerate(fields):
                s.set_field(f, a)
            s.step(2)
            return d, np.concatenate([s.get_field(f) for f in range(len(fields))])

    _, ref = go("fp64")
    tried = 0
    for E, ct in SHAPES:
        monkeypatch.setenv("NS_FORCE_STRIDED", f"3,{E},{ct}")
        d, got = go("fp32")
        if (d["kernel"], d["E"], d["cols_per_cta"]) != ("constant geometry, shared transforms", E, ct):
            continue
        tried += 1
        assert rel_l2(got, ref) < 2e-5, (E, ct)
    assert tried
