"""Overlapped launches under a user's stream capture, and two boxes at work on two
streams: bitwise the results of plain calls."""
import pytest
import torch

from paper_1004_1680_gb300 import initial_conditions as ic
from tests.parity_util import G, to_gpu

pytestmark = pytest.mark.gpu

BOXES = [((32, 32, 32), ()), ((64, 64, 64), ()), ((40, 36, 44), (0, 2)), ((236, 50, 44), (0,)), ((128, 64, 64), ()),
         ((100, 96, 2), ())]


def box(mhd, dims, open_axes, seed):
    st = to_gpu(ic.turbulence(dims, seed=seed, dtype=torch.float64, kmin=1.0, kmax=2.0, mach=0.5))
    b = mhd.Box(*dims, gamma=G)
    for a in open_axes:
        b.set_boundary(a, "outflow")
    b.set_pressure_floor(0.05)
    b.set_state(st)
    return b


@pytest.mark.parametrize("dims, open_axes", BOXES)
def test_captured_run_replays_as_plain_runs(dims, open_axes):
    from paper_1004_1680_gb300 import mhd
    plain, captured = box(mhd, dims, open_axes, 3), box(mhd, dims, open_axes, 3)
    for b in (plain, captured):
        b.run(2, 0.6)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        captured.set_stream(torch.cuda.current_stream())
        captured.run(2, 0.6)          # an even number of steps leaves the two copies where they were
    for _ in range(3):
        g.replay()
        plain.run(2, 0.6)
    torch.cuda.synchronize()
    captured.set_stream(torch.cuda.current_stream())
    assert torch.equal(captured.get_state(), plain.get_state()) and captured.time() == plain.time()


@pytest.mark.parametrize("pair", [(0, 1), (1, 2), (3, 0), (4, 5)])
def test_two_boxes_on_two_streams(pair):
    from paper_1004_1680_gb300 import mhd
    alone = []
    for k in pair:
        b = box(mhd, *BOXES[k], 11 + k)
        b.run(12, 0.6)
        alone.append((b.get_state(), b.time()))
    both = [box(mhd, *BOXES[k], 11 + k) for k in pair]
    streams = [torch.cuda.Stream() for _ in pair]
    torch.cuda.synchronize()
    for b, s in zip(both, streams):
        b.set_stream(s)
    for _ in range(6):
        for b in both:
            b.run(2, 0.6)
    torch.cuda.synchronize()
    for b, (state, t) in zip(both, alone):
        assert torch.equal(b.get_state(), state) and b.time() == t
