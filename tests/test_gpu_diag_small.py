"""Diagnostics of states far below one: the extrema are the FP64 values of their
formulas where FP32 squares of the momenta underflow (1e-12 and 1e-9, as for
states near one), the sums within 1e-13 of the absolute sum."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(7, 5, 3), (64, 32, 20), (33, 40, 64)])
@pytest.mark.parametrize("rho, v", [(1e-18, 1.0), (1e-25, 1.0), (1e-30, 1.0), (1e-34, 1.0), (1e-24, 1e6), (1e-12, 1e-8)])
def test_small_states(dims, rho, v):
    """Densities around rho, speeds around v."""
    from paper_1004_1680_gb300 import mhd
    st = ic.turbulence(dims, seed=2, dtype=torch.float64, kmin=1.0, kmax=3.0)
    st[0] *= rho
    st[1:4] *= rho * v
    st[4] *= rho * v * v
    st[5:8] *= math.sqrt(rho) * v
    st = st.float().contiguous()
    got = mhd.diagnostics_static(st.cuda(), gamma=G)
    s = st.double().numpy()
    ref = oracle.diagnostics(s, G)
    for q in range(8):
        assert abs(got[q] - math.fsum(s[q].ravel().tolist())) <= 1e-13 * np.abs(s[q]).sum() + 1e-300
    assert got[8] == pytest.approx(ref[8], rel=1e-9, abs=1e-300)
    assert got[9] == pytest.approx(ref[9], rel=1e-12, abs=0.0)
