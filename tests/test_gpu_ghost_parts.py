"""Ghost layers in a step: filled 4 cells at a time where rows allow it, and only
the fields that the sweep before has written.  The same sweeps called one by one
refill every field (also after the sweep, for the CFL rate); a step must match them
bitwise once its own ghost layers are refilled."""
import pytest
import torch

from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mhd():
    from paper_1004_1680_gb300 import mhd as m
    m.load()
    return m


def mapped(u, modes):
    """The ghost layers of every non-periodic axis, cell by cell from their definition."""
    g = 4
    for axis, mode in enumerate(modes):
        if mode == "periodic":
            continue
        v = torch.movedim(u, 3 - axis, 1)  # [field][axis][..][..]
        n = v.shape[1]
        lo, hi = g, n - g
        w = v.clone()
        for c in list(range(lo)) + list(range(hi, n)):
            out = mode == "outflow"
            s = (lo if out else 2 * lo - 1 - c) if c < lo else (hi - 1 if out else 2 * hi - 1 - c)
            f = (lo if out else 2 * lo - c) if c < lo else (hi if out or c == hi else 2 * hi - c)
            sign = 1.0 if out else -1.0
            for q in range(8):
                if q == 5 + axis:
                    w[q][c] = v[q][f] * (sign if f != c else 1.0)
                else:
                    w[q][c] = v[q][s] * (sign if q == 1 + axis else 1.0)
        u = torch.movedim(w, 1, 3 - axis)
    return u


@pytest.mark.parametrize("modes", [("periodic", "outflow", "reflecting"), ("reflecting", "outflow", "periodic"),
                                   ("outflow", "reflecting", "outflow"), ("reflecting", "periodic", "periodic")])
@pytest.mark.parametrize("dims", [(20, 17, 24), (36, 16, 13), (12, 12, 16), (72, 70, 66)])
def test_fill_and_step(mhd, modes, dims):
    x = to_gpu(ic.turbulence(dims, seed=3, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.6))
    boxes = [mhd.Box(*dims, gamma=G) for _ in range(2)]
    for b in boxes:
        for a, m in enumerate(modes):
            if m != "periodic":
                b.set_boundary(a, m)
        b.set_state(x)
    boxes[0].fill_ghosts()
    assert torch.equal(boxes[0].get_state(), mapped(x, modes).contiguous())
    tau = 0.2 / max(dims)
    boxes[0].step(2 * tau)  # (a step is two sweeps of tau along every axis)
    for axis, kind in [(0, 0), (0, 1), (1, 0), (1, 1), (2, 0), (2, 1), (2, 1), (2, 0), (1, 1), (1, 0), (0, 1), (0, 0)]:
        boxes[1].sweep(axis, kind, tau)
    for b in boxes:
        b.fill_ghosts()
    assert torch.equal(boxes[0].get_state(), boxes[1].get_state())
    for b in boxes:
        b.close()
