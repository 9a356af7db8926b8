"""Marching sweeps whose last pencil segment is shorter than the others.

The library picks segment lengths that need not divide the pencil; a box whose
pencils are whole (`set_segments` with the extents) runs the same arithmetic,
so a few steps must match it bitwise.  The extents cover one long and one
short segment, nearly equal ones, staged and register-load sweeps, the
exchanged copy for x, partial tiles of pencils and the floor variant.
"""
import pytest
import torch

from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, to_gpu

pytestmark = pytest.mark.gpu

CASES = [
    ((160, 160, 160), {}),
    ((200, 200, 200), {}),
    ((132, 158, 162), {"floor": 1e-3}),
    ((64, 36, 100), {"tma": False, "xpath": 1}),
    ((100, 62, 45), {"tma": False, "xpath": 2}),
    ((116, 40, 88), {"tma": False, "xpath": 2, "floor": 1e-3}),
    ((120, 60, 92), {"freezing": "pencil"}),
]


@pytest.fixture(scope="module")
def mhd():
    from paper_1004_1680_gb300 import mhd as m
    m.load()
    return m


@pytest.mark.parametrize("dims,cfg", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_ragged_segments_match_whole_pencils(mhd, dims, cfg):
    x = to_gpu(ic.turbulence(dims, seed=5, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.6))
    out = []
    for whole in (False, True):
        b = mhd.Box(*dims, gamma=G)
        if "tma" in cfg:
            b.set_tma(cfg["tma"])
            b.set_xpath(cfg["xpath"])
        if "floor" in cfg:
            b.set_pressure_floor(cfg["floor"])
        if "freezing" in cfg:
            b.set_scheme(freezing=cfg["freezing"])
        # x alike in both (forced whole, it marches); y and z in the library's segments or whole
        b.set_segments(*(n if n % 4 == 0 and (whole or d == 0) else 0 for d, n in enumerate(dims)))
        b.set_state(x)
        b.run(2, 0.7)
        out.append(b.get_state().clone())
        b.close()
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0], out[1])
