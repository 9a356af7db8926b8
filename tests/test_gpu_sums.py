"""The kernels that sum FP32 values in FP32 words (fp32_sums.cuh): diagnostics
of boxes that take one cell per lane (odd rows, unaligned fields) or two, the
restriction for ratios with and without vector loads and with several windows
per cell, and the values FP32 words cannot hold (infinities, sums and squares
past FP32's range), which fall back to FP64."""
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


@pytest.mark.parametrize("r, coarse", [(2, (6, 5, 4)), (3, (5, 4, 3)), (4, (33, 3, 2)), (8, (3, 2, 4)), (16, (2, 1, 2)),
                                       (1, (8, 3, 2))])
def test_restrict_ratios(mhd, r, coarse):
    """Every mean is the FP64 mean rounded to FP32 (half a unit in the last
    place, and 1e-6 of one for the last addition)."""
    n = tuple(r * x for x in coarse)
    g = torch.Generator().manual_seed(9)
    st = torch.randn((8, n[2], n[1], n[0]), generator=g) * torch.logspace(-3, 3, 8).view(8, 1, 1, 1)
    got = mhd.restrict(st.cuda(), r).cpu().double().numpy()
    ref = oracle.restrict(st.double().numpy(), r)
    assert np.all(np.abs(got - ref) <= 0.500001 * np.spacing(np.abs(ref).astype(np.float32)))


@pytest.mark.parametrize("r", [2, 3, 4])
def test_restrict_outside_the_words_range(mhd, r):
    n = 6 * r
    st = torch.full((8, n, n, n), 3e38)
    st[0, :r] = math.inf
    got = mhd.restrict(st.cuda(), r).cpu()
    assert torch.all(got[0, 0] == math.inf)
    assert torch.all(got[1:] == st[1, 0, 0, 0])


@pytest.mark.parametrize("scale", [1.0, 1e25, 1e-25, 1e18])
def test_loss_range(mhd, scale):
    """Differences far from what the weights expect: the loss is the FP64 sum
    of the squares of the FP32 differences (1e-12)."""
    n = (16, 16, 5)
    g = torch.Generator().manual_seed(11)
    d, t = (torch.randn((8, n[2], n[1], n[0]), generator=g) * scale for _ in range(2))
    w = [0.1 * (q + 1) for q in range(8)]
    got = float(mhd.cnn_loss(d.cuda(), t.cuda(), w).item())
    diff = (d - t).double().numpy()
    ref = sum(float(np.float32(w[q])) * math.fsum((diff[q] ** 2).ravel().tolist()) for q in range(8))
    assert got == pytest.approx(ref, rel=1e-12)


def test_projection_means_past_fp32_sums(mhd):
    """Box totals past FP32's range still give the FP64 mean."""
    n = (16, 16, 4)
    y = torch.zeros((n[0] * n[1] * n[2], 8))
    y[:, 0] = 2e38
    d = mhd.cnn_project(y.cuda(), n, [1.0] * 6).cpu()
    assert torch.all(d[0] == 0.0) and torch.all(torch.isfinite(d))
