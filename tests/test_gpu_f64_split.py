"""The FP64 sweeps' split of a pencil over threads: whole pencils, segments with
halo cells, ragged last segments, the shortest pencils, odd extents along every
axis, and quotients whose operands take the division (zero momenta, densities
far from one).  Against the FP64 oracle, the single-sweep bound of
test_gpu_fp64.py (1e-13 of the field scales)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, field_scales, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("long", [1, 2, 3, 7, 64, 65, 117, 200])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("kind", [0, 1])
def test_sweeps(long, axis, kind):
    from paper_1004_1680_gb300 import mhd
    dims = [5, 6, 7]
    dims[axis] = long
    st = ic.turbulence(dims, seed=19, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.5)
    st[2] = 0.0                                  # zero momenta
    st[0, 0], st[4, 0] = 1e-200, 1e-200 * st[4, 0]
    st[1:4, 0] *= 1e-200
    st[5:8] *= 0.0 if long == 7 else 1e-3
    s = np.ascontiguousarray(st.numpy())
    tau = 1e-3
    box = mhd.Box64(*dims)
    box.set_state(st.cuda())
    box.sweep(axis, kind, tau)
    (oracle.fluid_sweep(s, axis, tau, G) if kind == 0 else oracle.mag_sweep(s, axis, tau))
    got = box.get_state().cpu().numpy()
    box.close()
    fine = np.isfinite(s)
    assert np.array_equal(fine, np.isfinite(got))
    assert np.all(rel_err(np.where(fine, got, 0.0), np.where(fine, s, 0.0), field_scales(st.numpy())) < 1e-13)
