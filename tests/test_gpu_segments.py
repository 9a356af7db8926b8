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


@pytest.mark.parametrize("xpath", [1, 2])
def test_ragged_ensemble_segments_match_single_boxes(mhd, xpath):
    """Members of very different extents: one segment length for all leaves
    whole pencils, equal segments and short last ones."""
    dims = [(36, 20, 44), (84, 40, 36), (8, 4, 12), (48, 52, 100), (120, 12, 20), (32, 32, 31)]
    states = [to_gpu(ic.turbulence(d, seed=90 + i, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.6))
              for i, d in enumerate(dims)]
    ens = mhd.Ensemble(dims, gamma=G)
    ens.set_tuning(xpath, 1)
    ens.set_pressure_floor(1e-3)
    for i, x in enumerate(states):
        ens.set_state(i, x)
    ens.run(2, 0.7)
    for i, (d, x) in enumerate(zip(dims, states)):
        b = mhd.Box(*d, gamma=G)
        b.set_tma(False)
        b.set_xpath(xpath)
        b.set_segments(*(n if n % 4 == 0 else 0 for n in d))
        b.set_pressure_floor(1e-3)
        b.set_state(x)
        b.run(2, 0.7)
        assert torch.equal(ens.get_state(i), b.get_state()), d
        b.close()
    ens.close()


@pytest.mark.parametrize("nx,exchanged", [(132, True), (128, False)], ids=["ragged_rows", "whole_rows"])
def test_given_x_segments_choose_the_x_path(mhd, nx, exchanged):
    """A given segment length of x keeps tile sweeps off: beyond 2,097,152 cells
    rows that are not whole go through the exchanged copy, whole ones along x,
    and the automatic choice is bitwise the requested one."""
    dims = (nx, 132, 128)
    x = to_gpu(ic.turbulence(dims, seed=7, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.6))
    out = []
    for path in (0, 2 if exchanged else 1):
        b = mhd.Box(*dims, gamma=G)
        b.set_segments(nx, 0, 0)
        b.set_xpath(path)
        b.set_state(x)
        b.profile(200)
        b.run(1, 0.7)
        assert (b.profile_read()["transpose"][0] > 0) == exchanged
        out.append(b.get_state().clone())
        b.set_segments(0, 0, 0)  # tiles are open again: along x unless requested otherwise
        b.profile(200)
        b.run(1, 0.7)
        assert (b.profile_read()["transpose"][0] > 0) == (path == 2)
        b.close()
    assert torch.equal(out[0], out[1])
