"""Rows of features and targets on grids that do not fill the writing blocks.

Every feature row is compared with the rows of the neighbouring cells bit for
bit (a neighbour's moments are that neighbour's own), the features of the cell
itself and the targets with the reference at the tolerances of the tests on an
even grid; the buffers start 16 bytes and 4 bytes from a boundary and are
followed by words that must stay as they are.
"""
import numpy as np
import pytest

import test_gpu_closure as T
from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("offset", [4, 1])
@pytest.mark.parametrize("shape", [(33, 9, 5), (32, 4, 3), (5, 3, 7), (65, 6, 4), (3, 5, 1)])
def test_rows_of_odd_grids(shape, offset):
    nx, ny, nz = shape
    n = nx * ny * nz
    rng = np.random.default_rng(70)
    mean, inv = rng.standard_normal(10) * 1e-3, rng.uniform(10, 100, 10)
    out_scale = rng.uniform(1e-3, 1e-2, 17)
    net = B.MLP()
    net.set_scaling(mean, inv, out_scale)
    df = T._random_d3q27(shape, 71)
    Xb = torch.full((offset + n * 144 + 64,), 7, device="cuda", dtype=torch.int32)
    Tb = torch.full((offset + n * 32 + 64,), 7.0, device="cuda")
    X, Y = Xb[offset:offset + n * 144], Tb[offset:offset + n * 32]
    with B.Solver(B.D3Q27, shape, 0.7) as s:
        s.set_populations(torch.from_numpy(df).cuda())
        lib = s._lib
        assert lib.lb_closure_features(s.handle, net.handle, B._ptr(X)) == B.LB_OK
        assert lib.lb_closure_targets(s.handle, net.handle, B._ptr(Y)) == B.LB_OK
        torch.cuda.synchronize()
    net.close()
    assert (Xb[:offset] == 7).all() and (Xb[offset + n * 144:] == 7).all()
    assert (Tb[:offset] == 7).all() and (Tb[offset + n * 32:] == 7).all()
    bits = X.cpu().numpy().view(np.uint16).reshape(nz, ny, nx, 288)
    centre = bits[..., 130:140]
    for nb in range(27):
        shift = (-(nb // 9 - 1), -((nb // 3) % 3 - 1), -(nb % 3 - 1))
        assert np.array_equal(bits[..., 10 * nb:10 * nb + 10], np.roll(centre, shift, (0, 1, 2)))
    assert not bits[..., 270:].any()
    f = T.f64_state(T.O.D3Q27, df)
    Xo = T.C.features(T.C.moment_field(f), mean.astype(np.float32).astype(np.float64),
                      inv.astype(np.float32).astype(np.float64))
    got = (bits.astype(np.uint32) << 16).view(np.float32).astype(np.float64).reshape(n, 288)
    ulp = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(Xo), 1e-30))) - 7)
    assert np.all(np.abs(got - Xo) <= ulp + 1e-3)
    To = T.C.targets(f) / out_scale.astype(np.float32)
    Y = Y.cpu().numpy().astype(np.float64).reshape(n, 32)
    assert np.abs(Y[:, :17] - To).max() <= 1e-6 / out_scale.min()
    assert not Y[:, 17:].any()
