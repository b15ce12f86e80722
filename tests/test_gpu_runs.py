"""Runs of updates on the moments (lb_step(n) of FP32 grids) against the same
number of single updates.

Both carry out the same FP32 operations in the same order, so the stores agree
bit for bit; no tolerance is needed. 3-D shapes: partial tiles in x (also rows
of fewer cells than a tile), in y and in z segments, both lattices, both
regularized models, runs from and to either parity, and the fewest updates a
run takes over. 2-D shapes: halos wider than the grid, each block shape of the
tile kernel and the row-streaming kernel.
"""
import numpy as np
import pytest

from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _init(s, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (s.nz, s.ny, s.nx)
    rho = 1.0 + 0.01 * torch.randn(shape, device="cuda", generator=gen)
    u = 0.03 * torch.randn((s.d,) + shape, device="cuda", generator=gen)
    s.init_fields(rho, u)


def _state(s):
    buf = torch.empty(s.state_bytes(), dtype=torch.uint8, device="cuda")
    return buf, s.get_state(buf)


@pytest.mark.parametrize("lattice,shape,steps", [
    (B.D3Q27, (250, 151, 101), 5), (B.D3Q27, (31, 200, 200), 4), (B.D3Q27, (640, 130, 16), 6),
    (B.D3Q27, (97, 118, 120), 20), (B.D3Q19, (150, 200, 180), 16), (B.D3Q19, (62, 287, 201), 12),
])
@pytest.mark.parametrize("collision", [B.COLLIDE_RR, B.COLLIDE_REG2])
@pytest.mark.parametrize("first", [0, 1])
def test_runs_equal_single_updates(lattice, shape, steps, collision, first):
    with B.Solver(lattice, shape, 0.61, collision=collision) as a, \
            B.Solver(lattice, shape, 0.61, collision=collision) as b:
        for s in (a, b):
            _init(s, 5)
            for _ in range(first):  # the run starts at the odd parity
                s.step(1)
        free = torch.cuda.mem_get_info()[0]
        a.step(steps)
        scratch = free - torch.cuda.mem_get_info()[0]
        assert scratch >= 80 * a.n, "the run was expected to work on the moments"
        for _ in range(steps):
            b.step(1)
        (fa, pa), (fb, pb) = _state(a), _state(b)
        assert pa == pb == (first + steps) % 2
        assert torch.equal(fa, fb)
        assert a.info()["steps"] == b.info()["steps"]
        a.step(1)  # and the store goes on from there
        b.step(1)
        assert torch.equal(_state(a)[0], _state(b)[0])


@pytest.mark.parametrize("shape,steps", [
    ((1, 1), 6), ((5, 3), 20), ((4, 9), 21), ((128, 128), 50), ((100, 37), 23), ((37, 100), 24),
    ((64, 4000), 9), ((251, 251), 40), ((300, 200), 4), ((701, 500), 13), ((1001, 1001), 21),
    ((1900, 1300), 31), ((2300, 1700), 6), ((1400, 3000), 17),
])
@pytest.mark.parametrize("first", [0, 1])
def test_flat_runs_equal_single_updates(shape, steps, first):
    with B.Solver(B.D2Q9, (*shape, 1), 0.61) as a, B.Solver(B.D2Q9, (*shape, 1), 0.61) as b:
        for s in (a, b):
            _init(s, 7)
            for _ in range(first):
                s.step(1)
        free = torch.cuda.mem_get_info()[0]
        a.step(steps)
        scratch = free - torch.cuda.mem_get_info()[0]
        if a.n > 1 << 20:
            assert scratch >= 48 * a.n, "the run was expected to work on the moments"
        for _ in range(steps):
            b.step(1)
        (fa, pa), (fb, pb) = _state(a), _state(b)
        assert pa == pb == (first + steps) % 2
        assert torch.equal(fa, fb)
        a.step(7)
        for _ in range(7):
            b.step(1)
        assert torch.equal(_state(a)[0], _state(b)[0])
        assert a.info()["steps"] == b.info()["steps"]


def test_run_at_rest_and_uniform_flow():
    """df = 0 stays 0 and a uniform flow stays uniform, bit for bit."""
    with B.Solver(B.D3Q27, (128, 128, 128), 0.6) as s:
        s.step(7)
        assert not torch.any(s.populations())
        rho = torch.full((128,) * 3, 1.01, device="cuda")
        u = torch.zeros((3, 128, 128, 128), device="cuda")
        u[0], u[1] = 0.05, -0.02
        s.init_fields(rho, u, B.INIT_EQ)
        s.step(8)
        df = s.populations().reshape(27, -1)
        assert torch.equal(df, df[:, :1].expand_as(df))


def test_a_run_that_diverges_is_reported():
    with B.Solver(B.D3Q27, (128, 128, 128), 0.6) as s:
        df = torch.zeros((27, 128, 128, 128), device="cuda")
        df[13, 60, 61, 62] = float("nan")
        s.set_populations(df)
        s.step(6)
        with pytest.raises(B.LBError) as e:
            s.diagnostics()
        assert e.value.code == B.LB_EDIVERGED
        assert np.isnan(s.moments()[0].cpu().numpy()).any()
