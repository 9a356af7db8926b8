"""The FP64 sweeps' split of long pencils: the longest whole ones (512 cells, one
pencil per block), the shortest that take segments, ragged last segments, and
blocks with idle threads.  Against the FP64 oracle, the single-sweep bound of
test_gpu_fp64.py (1e-13 of the field scales)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, field_scales, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("long", [129, 171, 256, 257, 511, 512, 513, 1013, 1100])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_sweeps(long, axis):
    from paper_1004_1680_gb300 import mhd
    dims = [5, 3, 4]
    dims[axis] = long
    st = ic.turbulence(dims, seed=23, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.5)
    tau = 0.3 / oracle.cfl_rate(np.ascontiguousarray(st.numpy()), G)
    box = mhd.Box64(*dims)
    for kind in (0, 1):
        s = np.ascontiguousarray(st.numpy())
        box.set_state(st.cuda())
        box.sweep(axis, kind, tau)
        (oracle.fluid_sweep(s, axis, tau, G) if kind == 0 else oracle.mag_sweep(s, axis, tau))
        assert np.all(rel_err(box.get_state().cpu().numpy(), s, field_scales(st.numpy())) < 1e-13)
    box.close()
