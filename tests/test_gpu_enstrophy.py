"""lb_enstrophy against 0.5 sum |curl u|^2 of the same FP32 velocity field in FP64.

The kernel forms each component of the curl as a sum of two floats with a
relative error below 2^-44 and keeps FP64 where the square would lose that, so
the sum is held to 2^-40 of its value (64 bits for the few hundred thousand
additions are far below). Velocities from large to those whose squares leave
the FP32 range; rows of whole float4 and not, below, at and above what a block
takes; walls.
"""
import numpy as np
import pytest

from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _curl_sum(u, walls):
    """0.5 sum w |curl u|^2, u [D, nz, ny, nx] float64."""
    d, *shape = u.shape

    def diff(b, a):
        ax = 2 - a
        f = u[b]
        out = 0.5 * (np.roll(f, -1, ax) - np.roll(f, 1, ax))
        if (walls >> a) & 1:
            f, o = np.moveaxis(f, ax, 0), np.moveaxis(out, ax, 0)
            o[0] = 0.5 * (-3.0 * f[0] + 4.0 * f[1] - f[2])
            o[-1] = 0.5 * (3.0 * f[-1] - 4.0 * f[-2] + f[-3])
        return out

    c = (diff(1, 0) - diff(0, 1)) ** 2
    if d == 3:
        c = c + (diff(2, 1) - diff(1, 2)) ** 2 + (diff(0, 2) - diff(2, 0)) ** 2
    for a in range(d):
        if (walls >> a) & 1:
            w = np.moveaxis(c, 2 - a, 0)
            w[0] *= 0.5
            w[-1] *= 0.5
    return 0.5 * float(c.sum())


@pytest.mark.parametrize("lattice,shape,walls", [
    (B.D3Q27, (40, 30, 20), 0), (B.D3Q27, (256, 9, 5), 0), (B.D3Q19, (300, 17, 8), 0),
    (B.D2Q9, (257, 33, 1), 0), (B.D2Q9, (1, 7, 1), 0), (B.D2Q9, (65, 65, 1), 3),
    (B.D3Q27, (24, 20, 18), 5), (B.D3Q19, (1100, 5, 4), 0), (B.D3Q27, (515, 6, 4), 2),
])
@pytest.mark.parametrize("size", [0.05, 1e-9, 1e-20])
def test_enstrophy_of_the_velocity_field(lattice, shape, walls, size):
    with B.Solver(lattice, shape, 0.7, walls=walls) as s:
        gen = torch.Generator(device="cuda").manual_seed(11)
        dims = (s.nz, s.ny, s.nx)
        rho = torch.ones(dims, device="cuda")
        u = size * torch.randn((s.d,) + dims, device="cuda", generator=gen)
        s.init_fields(rho, u, B.INIT_EQ)
        got = s.enstrophy()
        ref = _curl_sum(s.moments()[1].cpu().numpy().astype(np.float64), walls)
        assert abs(got - ref) <= 2.0 ** -40 * ref, (got, ref)
        assert s.enstrophy() == got
