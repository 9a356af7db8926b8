"""The first thing a process does: every scheme variant's tile sweeps (blocks of
256 threads along x, y and z, pencils of more than 64 cells, with and without
the floor, need their shared-memory limit raised by the call itself), and an
ensemble on each x path with no single box made before it."""
import subprocess
import sys

import pytest

from paper_1004_1680_gb300.build import ROOT

pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
from paper_1004_1680_gb300 import mhd
from paper_1004_1680_gb300 import initial_conditions as ic
b = mhd.Box(100, 96, 68)
b.set_scheme({limiter!r}, {freezing!r})
b.set_pressure_floor({floor})
b.set_state(ic.turbulence((100, 96, 68), seed=1, dtype=torch.float32, kmin=1.0, kmax=2.0, mach=0.6).contiguous().cuda())
b.run(2, 0.7)
s = b.get_state()
assert b.time() > 0.0 and bool(torch.isfinite(s).all())
"""


@pytest.mark.parametrize("limiter, freezing, floor", [("vanleer", "bound", 0.0), ("minmod", "bound", 1e-3),
                                                      ("superbee", "bound", 0.0), ("vanleer", "fast", 1e-3),
                                                      ("vanleer", "pencil", 0.0)])
def test_variant_in_a_fresh_process(limiter, freezing, floor):
    subprocess.run([sys.executable, "-c", PROGRAM.format(limiter=limiter, freezing=freezing, floor=floor)], check=True, cwd=ROOT)


ENSEMBLE = """
import torch
from paper_1004_1680_gb300 import mhd
from paper_1004_1680_gb300 import initial_conditions as ic
dims = [(48, 40, 36), (8, 12, 100), (36, 96, 1)]
e = mhd.Ensemble(dims)
e.set_tuning({xpath}, {segdiv})
for b, d in enumerate(dims):
    e.set_state(b, ic.turbulence(d, seed=b, dtype=torch.float32, kmin=1.0, kmax=2.0, mach=0.5).contiguous().cuda())
e.run(2, 0.7)
assert (e.times() > 0.0).all() and all(bool(torch.isfinite(e.get_state(b)).all()) for b in range(3))
"""


@pytest.mark.parametrize("xpath, segdiv", [(1, 1), (1, 2), (2, 1), (2, 4)])
def test_ensemble_in_a_fresh_process(xpath, segdiv):
    subprocess.run([sys.executable, "-c", ENSEMBLE.format(xpath=xpath, segdiv=segdiv)], check=True, cwd=ROOT)
