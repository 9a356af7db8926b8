"""The magnetic row sweep on rows of any multiple of 4 cells: idle lanes past a
row's end, a last tile of fewer rows and a last segment of fewer planes, tiles of
four and of two rows.  Its arithmetic is the register-load sweep's cell by cell, so
it must match `set_tma(False)` bitwise."""
import pytest
import torch

import oracle
from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, to_gpu

pytestmark = pytest.mark.gpu

DIMS = [(236, 151, 40), (200, 98, 90), (300, 103, 80), (100, 141, 128), (128, 130, 100), (384, 97, 50),
        (1000, 67, 80), (1024, 61, 64)]


@pytest.fixture(scope="module")
def mhd():
    from paper_1004_1680_gb300 import mhd as m
    m.load()
    return m


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("limiter", ["vanleer", "minmod"])
def test_ragged_rows_match_the_register_sweep(mhd, dims, limiter):
    st = ic.turbulence(dims, seed=7, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.6)
    x = to_gpu(st)
    tau = 0.3 / oracle.cfl_rate(ic.as_oracle_input(st), G)
    out = []
    for tma in (True, False):
        b = mhd.Box(*dims, gamma=G)
        b.set_xpath(1)
        b.set_tma(tma)
        b.set_scheme(limiter=limiter)
        b.set_state(x)
        b.sweep(0, 1, tau)
        out.append(b.get_state().clone())
        b.close()
    assert not torch.equal(out[0], x)
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("dims", [(516, 67, 60), (572, 99, 61), (636, 64, 64)])
def test_tiles_of_three_rows_match_the_register_sweep(mhd, dims):
    """Rows of 513 to 639 cells: a last tile of one row, of three and again of one."""
    test_ragged_rows_match_the_register_sweep(mhd, dims, "vanleer")
