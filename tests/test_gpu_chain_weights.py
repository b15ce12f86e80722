"""Closure updates right after the weights have changed.

The network kernel of an update reads the weights before it waits for the
kernel in front of it, the feature source, which has waited for whatever wrote
them. Training steps and updates follow one another on one stream without a
synchronisation, on a grid whose feature source is itself launched early (2^19
cells or fewer) and on larger ones, with rows of whole tiles and without;
against the same calls with a synchronisation after each, bit for bit.
"""
import numpy as np
import pytest

from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run(shape, wait):
    gen = torch.Generator().manual_seed(1)
    net = B.MLP((0.05 * torch.randn(B.MLP_PARAMS, generator=gen)).numpy())
    net.set_scaling(np.zeros(10), np.full(10, 20.0), np.full(17, 1e-5))
    gen = torch.Generator(device="cuda").manual_seed(2)
    X = torch.randn((300, B.MLP_IN), device="cuda", generator=gen).to(torch.bfloat16)
    T = torch.randn((300, B.MLP_OUT), device="cuda", generator=gen)
    with B.Solver(B.D3Q27, shape, 0.62) as s:
        dims = shape[::-1]
        s.init_fields(1 + 0.01 * torch.rand(dims, device="cuda", generator=gen),
                      0.02 * torch.randn((3,) + dims, device="cuda", generator=gen), B.INIT_EQ)
        s.set_closure(net, bound=1e6)
        torch.cuda.synchronize()
        for _ in range(25):
            net.train_step(X, T, 0.05, want_loss=False)
            if wait:
                torch.cuda.synchronize()
            s.step(1)
            if wait:
                torch.cuda.synchronize()
        out = s.populations()
        params = net.get_params()
    net.close()
    return out, params


@pytest.mark.parametrize("shape", [(16, 16, 16), (128, 16, 16), (128, 64, 64), (128, 96, 96),
                                   (100, 90, 80)])
def test_updates_take_the_weights_of_the_step_before(shape):
    ref, params = _run(shape, wait=True)
    for _ in range(3):
        got, p = _run(shape, wait=False)
        assert np.array_equal(p, params)
        assert torch.equal(got, ref)
