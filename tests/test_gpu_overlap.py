"""Sweeps that are launched while the one before them drains, against the same
sweeps one at a time (an event recorded between two launches, as the trace does,
keeps the second from starting early).  Bitwise: the overlap changes no
arithmetic, so a difference is a value that was read too early or out of an L1
that still held an older one.  Rows of 236 and 100 cells share 32-byte pieces
between neighbouring rows, the floor acts (marching sweeps then read cells
back), and the boxes take marching, row and tile sweeps, ghost layers and x
rows beyond the row sweeps' 1024 cells."""
import pytest
import torch

from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims, walls, floor", [
    ((236, 150, 98), (0, 0, 0), 0.5), ((236, 150, 98), (0, 1, 2), 0.5), ((236, 150, 98), (0, 0, 0), 0.0),
    ((100, 160, 100), (0, 0, 0), 0.5), ((128, 128, 128), (0, 0, 0), 0.5), ((1028, 64, 32), (0, 0, 0), 0.5),
    ((64, 64, 64), (2, 0, 1), 0.5), ((64, 64, 64), (0, 0, 0), 0.0), ((32, 32, 32), (0, 0, 0), 0.5)])
def test_overlapped_steps_equal_serial_ones(dims, walls, floor):
    from paper_1004_1680_gb300 import mhd
    nx, ny, nz = dims
    st = to_gpu(ic.turbulence(dims, seed=83, dtype=torch.float64, kmin=1.0, kmax=3.0, mach=0.6))
    out = []
    modes = ("periodic", "outflow", "reflecting")
    for traced in (True, False):
        b = mhd.Box(nx, ny, nz, gamma=G)
        for axis, mode in enumerate(walls):
            b.set_boundary(axis, modes[mode])
        b.set_pressure_floor(floor)
        b.set_state(st)
        if traced:
            b.profile(1000)
        b.run(4, 0.7)
        out.append((b.get_state(), b.time(), b.cfl_dt()))
        b.close()
    assert torch.equal(out[0][0], out[1][0]) and out[0][1:] == out[1][1:]
