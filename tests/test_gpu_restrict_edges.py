"""Restriction of nothing, and of fields that start off the vector loads'
alignment (the general kernel)."""
import ctypes

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 2, 3, 4])
def test_no_cells(r):
    from paper_1004_1680_gb300 import mhd
    lib = mhd.load()
    t = torch.full((8, 16), 7.0, device="cuda")
    p = (ctypes.c_void_p * 8)(*[t[q].data_ptr() for q in range(8)])
    for dims in ((0, 12, 12), (12, 0, 12), (12, 12, 0)):
        assert lib.mhd_restrict(*dims, r, p, p, None) == mhd.MHD_OK
    torch.cuda.synchronize()
    assert bool((t == 7.0).all())


@pytest.mark.parametrize("r", [2, 4])
def test_unaligned_fields(r):
    """Half a unit in the last place (and 1e-6 of one), as for aligned fields."""
    from paper_1004_1680_gb300 import mhd
    n = (6 * r, 3 * r, 5 * r)
    cells = n[0] * n[1] * n[2]
    gen = torch.Generator().manual_seed(4)
    st = torch.randn((8, n[2], n[1], n[0]), generator=gen)
    buf = torch.zeros(8 * (cells + 1) + 1, device="cuda")
    fine = buf[1:1 + 8 * (cells + 1)].view(8, cells + 1)[:, :cells]
    fine.copy_(st.view(8, cells))
    got = mhd.restrict(fine.as_strided((8, n[2], n[1], n[0]), (cells + 1, n[0] * n[1], n[0], 1)), r).cpu().double().numpy()
    ref = oracle.restrict(st.double().numpy(), r)
    assert np.all(np.abs(got - ref) <= 0.500001 * np.spacing(np.abs(ref).astype(np.float32)))
