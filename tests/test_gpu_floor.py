"""The pressure floor of the fluid sweeps at its edge.

A sweep with a vanishing step leaves the state but for the floor, so the energy
must come out as max(e, |m|^2 / 2 rho + |b|^2 / 2 + p_floor / (gamma - 1)).  The
pressures lie below, at (to a few roundings) and above the floor, the densities
span six decades and the kinetic energy up to a thousand times the thermal one.
The bound holds the roundings of the face means, the squares, the quotient and
the two sums (8 x 2^-24 of a sum of terms >= 0).
"""
import pytest
import torch

from tests.parity_util import G

pytestmark = pytest.mark.gpu

FLOOR = 0.25
BOUND = 8 * 2.0 ** -24


@pytest.fixture(scope="module")
def mhd():
    from paper_1004_1680_gb300 import mhd as m
    m.load()
    return m


def state(dims):
    nx, ny, nz = dims
    gen = torch.Generator().manual_seed(11)
    u = torch.empty((8, nz, ny, nx), dtype=torch.float64)
    u[0] = 10.0 ** (6 * torch.rand((nz, ny, nx), generator=gen, dtype=torch.float64) - 3)
    u[1:4] = torch.randn((3, nz, ny, nx), generator=gen, dtype=torch.float64) * u[0].sqrt() * 10
    u[5:8] = torch.randn((3, nz, ny, nx), generator=gen, dtype=torch.float64)
    u = u.float()
    kinds = torch.randint(0, 6, (nz, ny, nx), generator=gen)
    eps = (torch.rand((nz, ny, nx), generator=gen, dtype=torch.float64) - 0.5) * 2e-6
    p = torch.tensor([0.0, 0.5, 1.0, 1.0, 1.5, 40.0], dtype=torch.float64)[kinds] * FLOOR
    rest = floor_energy(u) - FLOOR / (G - 1)
    u[4] = ((rest + p / (G - 1)) * (1 + eps)).float()
    return u


def floor_energy(u):
    v = u.double()
    b = [0.5 * (v[5 + d] + torch.roll(v[5 + d], -1, dims=2 - d)) for d in range(3)]
    return (v[1:4] ** 2).sum(0) / (2 * v[0]) + sum(x * x for x in b) / 2 + FLOOR / (G - 1)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("dims,cfg", [((128, 8, 8), {}), ((36, 20, 44), {}), ((64, 32, 16), {"whole": True}),
                                      ((64, 32, 16), {"tma": False})], ids=lambda v: str(v).replace(" ", ""))
def test_floor_edge(mhd, dims, cfg, axis):
    u = state(dims)
    b = mhd.Box(*dims, gamma=G)
    if cfg.get("whole"):
        b.set_segments(*dims)
    if "tma" in cfg:
        b.set_tma(False)
        b.set_xpath(1)
    b.set_pressure_floor(FLOOR)
    b.set_state(u.cuda())
    b.sweep(axis, 0, 1e-20)
    got = b.get_state().cpu()
    assert torch.equal(got[0], u[0]) and torch.equal(got[5:], u[5:])
    bound = floor_energy(u)
    want = torch.maximum(u[4].double(), bound)
    assert ((got[4].double() - want).abs() <= BOUND * want).all()
    # cells clearly above the floor keep their energy as it was
    above = u[4].double() > bound * (1 + 1e-5)
    assert above.any() and torch.equal(got[4][above], u[4][above])
