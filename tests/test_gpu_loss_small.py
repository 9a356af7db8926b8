"""The loss of differences whose squares FP32 cannot hold: down to the smallest
FP32 values the loss is the FP64 sum of the squares of the FP32 differences
(1e-12), also where one field's differences are tiny and another's are not, and
zero where they are zero."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-22, 1e-24, 1e-30, 1e-38, 2.0 ** -149, 0.0])
@pytest.mark.parametrize("one_field", [False, True])
def test_small_differences(scale, one_field):
    from paper_1004_1680_gb300 import mhd
    n = (16, 16, 5)
    gen = torch.Generator().manual_seed(11)
    d = torch.randn((8, n[2], n[1], n[0]), generator=gen, dtype=torch.float64) * scale
    if scale == 2.0 ** -149:
        d = d.sign() * scale
    if one_field:
        d[:3] = 0.0
        d[4:] = 0.0
    d = d.float()
    w = [0.1 * (q + 1) for q in range(8)]
    got = float(mhd.cnn_loss(d.cuda(), torch.zeros_like(d).cuda(), w).item())
    x = d.double().numpy()
    ref = sum(float(np.float32(w[q])) * math.fsum((x[q] ** 2).ravel().tolist()) for q in range(8))
    assert got == pytest.approx(ref, rel=1e-12, abs=0.0)
