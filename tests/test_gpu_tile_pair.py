"""The two z magnetic sweeps of a step in one tile launch (whole pencils of up to
40 cells) against the marching sweeps: the shortest pencils, whose cells have
several periodic images in the block, and boxes above 120,000 cells, which take
tiles of 16 x 4 pencils (whole ones, and ones cut by the box along x or y).

With pencils along y and z shorter than the staged sweeps' 16 cells and rows
that are not whole warps every fluid sweep takes the same square root as the
register-load sweeps, so the comparison is bitwise; segments of whole pencils
give the marching sweeps of multiples of 4."""
import numpy as np
import pytest
import torch

from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, field_scales, rel_err, to_gpu

pytestmark = pytest.mark.gpu


def state(dims, seed):
    return ic.turbulence(dims, seed=seed, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.6)


def two_boxes(st64, marching, limiter="vanleer", cubic=False):
    from paper_1004_1680_gb300 import mhd
    nz, ny, nx = st64.shape[1:]
    out = []
    for m in (False, True):
        b = mhd.Box(nx, ny, nz, gamma=G)
        b.set_scheme(limiter)
        if cubic:  # cubic cells, whatever the extents
            b.set_resolution(1.0, 1.0, 1.0)
        if m:
            marching(b)
        b.set_pressure_floor(0.05)
        b.set_state(to_gpu(st64))
        b.run(3, 0.7)
        out.append((b.get_state(), b.time()))
        b.close()
    return out


@pytest.mark.parametrize("dims", [(36, 12, 1), (36, 12, 2), (100, 15, 2), (36, 12, 3), (36, 12, 4), (68, 9, 2), (100, 14, 7)])
def test_shortest_pencils(dims):
    """Fast flow along z (most of the signal speed) over a weak field that differs
    from cell to cell."""
    nx, ny, nz = dims
    gen = torch.Generator().manual_seed(5)
    st = torch.ones((8, nz, ny, nx), dtype=torch.float64)
    st[1:3] = 0.0
    st[3] = 3.0 * torch.randn((nz, ny, nx), generator=gen, dtype=torch.float64)
    st[5:8] = 0.1 * torch.randn((3, nz, ny, nx), generator=gen, dtype=torch.float64)
    st[4] = 0.5 * st[3] ** 2 + 1.0

    def marching(b):
        b.set_tma(False)
        b.set_xpath(1)
    a, b = two_boxes(st, marching, cubic=True)
    assert torch.isfinite(a[0]).all() and a[1] > 0.0
    assert bool((a[0] == b[0]).all()) and a[1] == b[1]


@pytest.mark.parametrize("dims, limiter", [((128, 128, 32), "vanleer"), ((96, 96, 36), "vanleer"), ((100, 64, 20), "minmod"),
                                           ((100, 64, 20), "vanleer")])
def test_pairs_of_wide_tiles(dims, limiter):
    a, b = two_boxes(state(dims, 93), lambda m: m.set_segments(*dims), limiter)
    assert torch.isfinite(a[0]).all() and a[1] > 0.0
    assert bool((a[0] == b[0]).all()) and a[1] == b[1]


def test_pair_of_cut_wide_tiles():
    """62 rows cut the last tile; the fluid sweeps may differ by the square root."""
    def marching(b):
        b.set_tma(False)
        b.set_xpath(1)
    a, b = two_boxes(state((68, 62, 36), 95), marching)
    s = b[0].double().cpu().numpy()
    assert np.all(rel_err(a[0].double().cpu().numpy(), s, field_scales(s)) < 1e-5)
