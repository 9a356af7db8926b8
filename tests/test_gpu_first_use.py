"""Every scheme variant's tile sweeps as the first thing a process does: blocks of
256 threads along x, y and z (pencils of more than 64 cells), with and without
the floor, need their shared-memory limit raised by the call itself."""
import subprocess
import sys

import pytest

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
    subprocess.run([sys.executable, "-c", PROGRAM.format(limiter=limiter, freezing=freezing, floor=floor)], check=True)
