"""Tile sweeps (a block holds its pencils' stencil on chip, 4 cells per thread)
against the marching sweeps.

A tile sweep does the arithmetic of the marching sweep it replaces, cell by
cell, square root included, so a single sweep must match it bitwise.
`set_segments` forces the marching sweep along an axis whose extent is a
multiple of 4; other extents are compared with the register-load sweeps of
`set_tma(False)`, which share the magnetic arithmetic bitwise and the fluid
arithmetic but for the square root (1e-6 of the field scales, as for the staged
sweeps).  The extents cover whole pencils and segments, partial tiles, the
shortest pencils and extents of one.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, field_scales, from_gpu, rel_err, to_gpu

pytestmark = pytest.mark.gpu

DIMS = [(32, 32, 32), (4, 1, 1), (4, 5, 3), (8, 4, 36), (12, 7, 33), (20, 44, 64), (36, 62, 9), (48, 97, 18),
        (260, 5, 40), (100, 34, 129), (128, 16, 8), (512, 8, 4)]


@pytest.fixture(scope="module")
def mhd():
    from paper_1004_1680_gb300 import mhd as m
    m.load()
    return m


def state(dims, seed):
    return ic.turbulence(dims, seed=seed, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.6)


def boxes(mhd, st64, forced):
    """A box as it is by default, and one whose `forced` axes march."""
    nz, ny, nx = st64.shape[1:]
    a, b = mhd.Box(nx, ny, nz, gamma=G), mhd.Box(nx, ny, nz, gamma=G)
    n = (nx, ny, nz)
    if all(n[d] % 4 == 0 for d in forced):
        b.set_segments(*(n[d] if d in forced else 0 for d in range(3)))
        exact = True
    else:
        b.set_tma(False)
        b.set_xpath(1)
        exact = False
    a.set_state(to_gpu(st64))
    b.set_state(to_gpu(st64))
    return a, b, exact


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("kind", [0, 1])
def test_tile_sweep_matches_the_marching_sweep(mhd, dims, axis, kind):
    st = state(dims, 71)
    a, b, exact = boxes(mhd, st, [axis])
    tau = 0.35 / oracle.cfl_rate(ic.as_oracle_input(st), G)
    a.sweep(axis, kind, tau)
    b.sweep(axis, kind, tau)
    if exact or kind == 1:
        assert torch.equal(a.get_state(), b.get_state())
        assert a.cfl_dt() == b.cfl_dt()
    else:
        s = b.get_state().double().cpu().numpy()
        assert np.all(rel_err(a.get_state().double().cpu().numpy(), s, field_scales(s)) < 1e-6)


@pytest.mark.parametrize("dims", [(32, 32, 32), (20, 44, 64), (48, 96, 20), (4, 4, 4)])
@pytest.mark.parametrize("floor", [0.0, 0.5])
def test_tile_steps_match_the_marching_steps(mhd, dims, floor):
    """Runs with the fused CFL rate, the fused z pair (whole pencils: one tile
    launch) and the pressure floor (0.5 acts on this state)."""
    st = state(dims, 73)
    a, b, exact = boxes(mhd, st, [0, 1, 2])
    assert exact
    for box in (a, b):
        box.set_pressure_floor(floor)
        box.run(3, 0.7)
    assert torch.equal(a.get_state(), b.get_state())
    assert a.time() == b.time()


def test_tile_step_parity_with_oracle(mhd):
    """One full step of an odd box, within the one-step bound of the oracle."""
    st = state((44, 37, 50), 79)
    s = ic.as_oracle_input(st)
    box = mhd.Box(44, 37, 50, gamma=G)
    box.set_state(to_gpu(st))
    dt = oracle.cfl_dt(s, G, 0.7)
    box.step(dt)
    oracle.step(s, dt, G)
    assert np.all(rel_err(from_gpu(box.get_state()), s, field_scales(s)) < 1e-4)
