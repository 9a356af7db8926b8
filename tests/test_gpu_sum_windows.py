"""Sums of more cells than one window per thread holds (39.8 M): the projection's
means, their adjoint's and the loss, against FP64 sums (the bounds of
test_gpu_sums.py; half a unit of the mean's FP32 rounding and one more)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

N3 = (512, 400, 200)  # 41 M cells


def test_sums_of_a_large_grid():
    from paper_1004_1680_gb300 import mhd
    nx, ny, nz = N3
    gen = torch.Generator(device="cuda").manual_seed(3)
    y = torch.randn((nx * ny * nz, 8), generator=gen, device="cuda")
    y[:, 0] += 1.0
    scale = [1.0, 2.0, 0.5, 1.0, 1.0, 0.25]
    d = mhd.cnn_project(y, N3, scale)
    for q in range(5):
        mean = (y[:, q] * scale[q]).double().mean().float()
        assert torch.equal(d[q].flatten(), y[:, q] * scale[q] - mean) or \
            (d[q].flatten() - (y[:, q] * scale[q] - mean)).abs().max() <= 2.0 ** -23 * (1 + abs(float(mean)))
    t = torch.randn(d.shape, generator=gen, device="cuda")
    g = torch.empty_like(d)
    w = [1e-7 * (q + 1) for q in range(8)]
    loss = float(mhd.cnn_loss(d, t, w, g=g).item())
    ref = sum(float(torch.tensor(w[q])) * float(((d[q] - t[q]).double() ** 2).sum()) for q in range(8))
    assert loss == pytest.approx(ref, rel=1e-11)
    gy = mhd.cnn_project_backward(g, scale)
    for q in range(5):
        want = (scale[q] * (g[q] - g[q].double().mean().float())).flatten()
        assert (gy[:, q].float() - want).abs().max() <= 2.0 ** -8 * want.abs().max()
