"""Plan files (NS_PLAIN_CACHE, NS_PLAN_CACHE) with entries that the kernels do
not take: more columns per CTA than a pass has threads for, FP64 z passes of
one line per transform, shared transforms on another pass than A.  Such an
entry is passed over: the run tunes as without a file, gives the same state,
and writes an entry that it takes."""
import json
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CODE = """
import sys
import numpy as np
from paper_1003_4322_gb300 import inputs
from paper_1003_4322_gb300.solver import Solver
with Solver([dict(n=64, nu=2e-3, dt=1e-3)], prec=sys.argv[1]) as s:
    s.set_field(0, 1e-3 * inputs.random_hermitian_half_grid((64, 64, 64), 3, seed=5))
    s.step(2)
    np.save(sys.argv[2], s.get_field(0))
"""


def advance(prec, out, monkeypatch, var=None, path=None):
    for v in ("NS_PLAIN_CACHE", "NS_PLAN_CACHE"):
        monkeypatch.delenv(v, raising=False)
    if var:
        monkeypatch.setenv(var, str(path))
    subprocess.run([sys.executable, "-c", CODE, prec, str(out)], check=True, timeout=120)
    return np.load(out)


@pytest.mark.parametrize("entry", ["64 8 4 32 8 8 108 108", "64 8 8 8 8 24 108 108", "64 8 8 8 8 8 4 108",
                                   "64 8 8 8 8 8 108 4"])
def test_fp64_entry_passed_over(ns, entry, tmp_path, monkeypatch):
    f = tmp_path / "plain.txt"
    f.write_text(entry + "\n")
    got = advance("fp64", tmp_path / "a.npy", monkeypatch, "NS_PLAIN_CACHE", f)
    ref = advance("fp64", tmp_path / "b.npy", monkeypatch)
    # two steps of transforms of 2^-60 of a line's largest value each
    assert np.abs(got - ref).max() <= 1e-14 * np.abs(ref).max()
    _, b, ei, ci, ef, cf, ec, er = map(int, f.read_text().split())
    assert b == 8 and ec >= 100 and er >= 100
    for E, ct in ((ei, ci), (ef, cf)):
        assert ct & (ct - 1) == 0 and 64 // E * ct <= 256


@pytest.mark.parametrize("i,triple", [(1, [3, 8, 8]), (0, [3, 5, 8])])
def test_fused_entry_passed_over(ns, i, triple, tmp_path, monkeypatch):
    t = [[0, 8, 8] for _ in range(4)] + [[0, 8, 1], [0, 0, 0]]
    t[i] = triple
    f = tmp_path / "plans.json"
    f.write_text('{\n  "64": ' + json.dumps(t) + "\n}\n")
    got = advance("fp32", tmp_path / "a.npy", monkeypatch, "NS_PLAN_CACHE", f)
    ref = advance("fp32", tmp_path / "b.npy", monkeypatch)
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()   # other plans, other roundings
    assert json.loads(f.read_text())["64"][i] != triple
