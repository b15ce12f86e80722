"""Runs of updates on the moments against the same number of single updates, bit
for bit, where FP32 runs out of range.

Populations that underflow or are about to, in the whole grid and where a flow
decays into rest; zeros of both signs; momenta next to zero in a density other
than one; densities far from one, of zero, and the largest below one with
momenta that are powers of two. NaN (a density of zero) counts as equal to NaN.
"""
import pytest

from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _scaled(shape, gen, lo, hi):
    e = torch.empty(shape, device="cuda", dtype=torch.float64).uniform_(lo, hi, generator=gen)
    return (torch.randn(shape, device="cuda", generator=gen) * torch.exp2(e)).float()


def _populations(kind, q, dims, gen):
    shape = (q,) + dims
    if isinstance(kind, tuple):
        return _scaled(shape, gen, *kind)
    if kind == "zeros of both signs":
        m = torch.randint(0, 3, shape, device="cuda", generator=gen)
        df = _scaled(shape, gen, -149, -120)
        df[m == 0], df[m == 1] = 0.0, -0.0
        return df
    if kind == "decays into rest":
        x = torch.arange(dims[2], device="cuda", dtype=torch.float64)
        return (_scaled(shape, gen, -8, -6) * torch.exp2(-2 * (x - dims[2] / 2).abs())).float()
    rand = torch.rand(dims, device="cuda", generator=gen)
    if kind == "momenta next to zero":
        df = _scaled(shape, gen, -149, -95)
        df[q // 2] = 0.01 + 0.01 * rand
    elif kind == "densities far from one":
        df = 0.01 * _scaled(shape, gen, -1, 1)
        df[q // 2] = torch.where(rand < 0.3, 1e7 * rand, torch.where(rand < 0.6, 1e-3, 0.5) * rand)
    elif kind == "densities of zero":
        df = 0.01 * _scaled(shape, gen, -1, 1)
        hole = rand < 1e-5
        df[:, hole] = 0.0
        df[q // 2, hole] = -1.0
        df[q // 2 + 1, hole], df[q // 2 - 1, hole] = 0.01, -0.01
    else:  # rho = 1 - 2^-24, momentum +-2^-k along x
        df = torch.zeros(shape, device="cuda")
        df[q // 2] = -2.0 ** -24
        j = torch.exp2(-torch.randint(3, 12, dims, device="cuda", generator=gen).float())
        df[q // 2 + 1], df[q // 2 - 1] = 0.5 * j, -0.5 * j
        df[0], df[-1] = 0.3 * j * rand, 0.3 * j * rand
        df[q // 2] -= 0.6 * j * rand
    return df


@pytest.mark.parametrize("kind", [
    (-149, -140), (-130, -120), (-128, -124), (-149, -110), (-110, -100), "zeros of both signs",
    "decays into rest", "momenta next to zero", "densities far from one", "densities of zero",
    "just below one",
])
@pytest.mark.parametrize("lattice,shape,steps,collision", [
    (B.D2Q9, (128, 128, 1), 8, B.COLLIDE_RR), (B.D2Q9, (701, 500, 1), 13, B.COLLIDE_RR),
    (B.D2Q9, (1900, 1300, 1), 21, B.COLLIDE_RR),
    (B.D3Q27, (128, 128, 128), 5, B.COLLIDE_RR), (B.D3Q27, (128, 128, 128), 5, B.COLLIDE_REG2),
    (B.D3Q19, (150, 200, 180), 9, B.COLLIDE_RR), (B.D3Q19, (150, 200, 180), 9, B.COLLIDE_REG2),
])
def test_runs_equal_single_updates_out_of_range(lattice, shape, steps, collision, kind):
    gen = torch.Generator(device="cuda").manual_seed(3)
    df = _populations(kind, lattice, shape[::-1], gen).contiguous()
    for tau, first in ((0.61, 0), (1.7, 1)):
        with B.Solver(lattice, shape, tau, collision=collision) as a, \
                B.Solver(lattice, shape, tau, collision=collision) as b:
            for s in (a, b):
                s.set_populations(df)
                if first:
                    s.step(1)
            a.step(steps)
            for _ in range(steps):
                b.step(1)
            x, y = a.populations(), b.populations()
            same = x.view(torch.int32) == y.view(torch.int32)
            assert (same | (x.isnan() & y.isnan())).all(), (tau, first)
