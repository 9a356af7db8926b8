"""The kernels that sum FP32 values in FP32 words (fp32_sums.cuh): diagnostics
of boxes that take one cell per lane (odd rows, unaligned fields) or two, and
sums that leave FP32's range within a block."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mhd():
    from paper_1004_1680_gb300 import mhd as m
    m.load()
    return m


@pytest.mark.parametrize("dims", [(1, 3, 2), (4, 1, 1), (7, 5, 3), (33, 9, 4), (4, 300, 3), (130, 66, 5),
                                  (256, 100, 40)])
def test_diagnostics_of_odd_boxes(mhd, dims):
    """Sums within 1e-13 of the absolute sum, extrema the FP64 values of their
    formulas (the bounds of the parity test)."""
    st = ic.turbulence(dims, seed=5, dtype=torch.float32, kmin=1.0, kmax=3.0).contiguous()
    got = mhd.diagnostics_static(st.cuda(), gamma=G)
    s = st.double().numpy()
    ref = oracle.diagnostics(s, G)
    for q in range(8):
        assert abs(got[q] - math.fsum(s[q].ravel().tolist())) <= 1e-13 * np.abs(s[q]).sum() + 1e-300
    assert got[8] == pytest.approx(ref[8], rel=1e-9, abs=1e-300)
    assert got[9] == pytest.approx(ref[9], rel=1e-12)


def test_diagnostics_past_a_blocks_range(mhd):
    """A momentum whose block total leaves FP32's range (a lane's does not)."""
    st = ic.turbulence((64, 32, 40), seed=7, dtype=torch.float32, kmin=1.0, kmax=3.0).contiguous()
    st[1] = 1e35
    got = mhd.diagnostics_static(st.cuda(), gamma=G)
    for q in range(8):
        s = st[q].double().numpy()
        assert abs(got[q] - math.fsum(s.ravel().tolist())) <= 1e-13 * np.abs(s).sum()
