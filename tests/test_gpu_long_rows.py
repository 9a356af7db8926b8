"""Boxes with rows of more than 1024 cells: steps by default, along x and through the
exchanged layout agree to FP32 rounding (1e-5 of the field scales after two
steps), and large ones whose exchanged layout is staged throughout take it by
themselves (bitwise the requested path, with its transposes in the trace)."""
import numpy as np
import pytest
import torch

from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, field_scales, rel_err, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims, exchanged", [((1028, 12, 20), False), ((2048, 64, 32), False), ((2048, 128, 32), True),
                                             ((1280, 256, 28), False), ((1100, 100, 80), False), ((8192, 32, 32), True)])
def test_x_path_of_long_rows(dims, exchanged):
    from paper_1004_1680_gb300 import mhd
    st = to_gpu(ic.turbulence(dims, seed=97, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.6))
    out = {}
    for path in (0, 1, 2):
        b = mhd.Box(*dims, gamma=G)
        b.set_xpath(path)
        b.set_state(st)
        b.profile(200)
        b.run(2, 0.7)
        out[path] = (b.get_state(), b.profile_read()["transpose"][0])
        b.close()
    assert (out[0][1] > 0) == exchanged and out[1][1] == 0 and out[2][1] > 0
    assert torch.equal(out[0][0], out[2 if exchanged else 1][0])
    s = out[1][0].double().cpu().numpy()
    assert np.all(rel_err(out[2][0].double().cpu().numpy(), s, field_scales(s)) < 1e-5)
