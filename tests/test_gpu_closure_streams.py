"""A closure set on a context whose stream does not wait for the default stream.

What lb_set_closure allocates is zeroed before the call returns, whatever the
default stream still has to do: with that stream busy for about as long as the
updates take, the updates that follow at once on a stream of their own, and the
count of the cells that fell back, are those of a context left to itself.
"""
import numpy as np
import pytest

from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _net():
    gen = torch.Generator().manual_seed(1)
    net = B.MLP((0.05 * torch.randn(B.MLP_PARAMS, generator=gen)).numpy())
    net.set_scaling(np.zeros(10), np.full(10, 20.0), np.full(17, 1e-5))
    return net


@pytest.mark.parametrize("shape", [(128, 64, 64), (130, 62, 61)])
def test_updates_right_after_the_closure_is_set(shape):
    gen = torch.Generator(device="cuda").manual_seed(3)
    dims = shape[::-1]
    rho = 1 + 0.01 * torch.rand(dims, device="cuda", generator=gen)
    u = 0.02 * torch.randn((3,) + dims, device="cuda", generator=gen)
    net, steps = _net(), 40

    def updates(s):
        s.set_closure(net, bound=0.05)  # exceeded by some of the cells
        s.step(steps)

    with B.Solver(B.D3Q27, shape, 0.62) as s:
        s.init_fields(rho, u, B.INIT_EQ)
        torch.cuda.synchronize()
        updates(s)
        ref, count = s.populations(), s.closure_fallbacks()
    assert 0 < count
    side = torch.cuda.Stream()
    for cycles in (2e5, 1e6, 4e6):
        with B.Solver(B.D3Q27, shape, 0.62, stream=side) as s:
            s.init_fields(rho, u, B.INIT_EQ)
            torch.cuda.synchronize()
            torch.cuda._sleep(int(cycles))  # on the default stream
            updates(s)
            assert s.closure_fallbacks() == count
            got = torch.empty_like(ref)
            assert s._lib.lb_get_populations(s.handle, B._ptr(got)) == B.LB_OK
            torch.cuda.synchronize()
            assert torch.equal(got, ref), cycles
    net.close()
