"""lb_enstrophy where the two differences of a curl component cancel.

A velocity component of one of the four neighbours that make a difference is
large and the other some 2^-25 of it, so that the rounding errors of the
differences are themselves numbers of full length, and the two differences of a
component agree to all but a part of 2^-8 to 2^-22. What is left is then a
matter of those rounding errors; the enstrophy is held to 2^-40 of the value
that the same FP32 field has in FP64, as for fields without cancellation.
"""
import numpy as np
import pytest

import test_gpu_enstrophy as E
from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FACES = {B.D2Q9: ((5, 3), (7, 1)), B.D3Q19: ((10, 8), (12, 6), (16, 2)),
         B.D3Q27: ((14, 12), (16, 10), (22, 4))}  # populations of velocity +-1 along each axis


@pytest.mark.parametrize("lattice,shape", [
    (B.D2Q9, (24, 24, 1)), (B.D2Q9, (36, 100, 1)), (B.D3Q27, (12, 16, 20)), (B.D3Q19, (20, 24, 16)),
])
@pytest.mark.parametrize("left", [8, 14, 18, 20, 22])
def test_enstrophy_of_differences_that_cancel(lattice, shape, left):
    rng = np.random.default_rng(5)
    nx, ny, nz = shape
    d = 2 if nz == 1 else 3
    k = np.indices(shape[::-1]).sum(0) % 4
    big = rng.uniform(0.02, 0.04)
    u = np.stack([
        np.where(k == 1, big * (1 + 2.0 ** -left * rng.standard_normal(k.shape)),
                 np.where(k == 3, rng.uniform(-1, 1, k.shape) * 2.0 ** rng.uniform(-32, -28, k.shape),
                          0.0)) for _ in range(d)]).astype(np.float32)
    with B.Solver(lattice, shape, 0.7) as s:
        df = np.zeros((s.q, nz, ny, nx), np.float32)
        for a, (plus, minus) in enumerate(FACES[lattice]):  # rho = 1, momentum u, exactly
            df[plus], df[minus] = 0.5 * u[a], -0.5 * u[a]
        s.set_populations(torch.from_numpy(df).cuda())
        got = s.enstrophy()
        assert np.array_equal(s.moments()[1].cpu().numpy().reshape(u.shape), u)
        ref = E._curl_sum(u.astype(np.float64), 0)
        assert abs(got - ref) <= 2.0 ** -40 * ref, (got, ref)
