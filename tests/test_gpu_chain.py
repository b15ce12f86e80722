"""Kernels launched while the one before them ends: the same results every time.

Closure updates, training steps and runs of D2Q9 updates, each many times over
without a synchronisation, alone, with other work on the stream in between that
writes what the next kernel reads, and replayed from a captured graph, against
the same calls with a synchronisation after each, bit for bit.
"""
import ctypes

import numpy as np
import pytest

from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _net(seed):
    gen = torch.Generator().manual_seed(seed)
    net = B.MLP((0.05 * torch.randn(B.MLP_PARAMS, generator=gen)).numpy())
    net.set_scaling(np.zeros(10), np.full(10, 20.0), np.full(17, 1e-5))
    return net


def _solver(lattice, shape, **kw):
    s = B.Solver(lattice, shape, 0.62, **kw)
    gen = torch.Generator(device="cuda").manual_seed(3)
    dims = (s.nz, s.ny, s.nx)
    s.init_fields(1 + 0.01 * torch.rand(dims, device="cuda", generator=gen),
                  0.02 * torch.randn((s.d,) + dims, device="cuda", generator=gen), B.INIT_EQ)
    return s


@pytest.mark.parametrize("shape", [(16, 16, 16), (64, 40, 30), (128, 32, 16)])
def test_closure_updates(shape):
    net = _net(1)
    with _solver(B.D3Q27, shape) as a, _solver(B.D3Q27, shape) as b:
        for s in (a, b):
            s.set_closure(net, bound=1e6)
        for k in range(30):
            a.step(1)
            torch.cuda.synchronize()
        b.step(30)
        assert torch.equal(a.populations(), b.populations())
        # captured: two updates a replay
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        b.set_stream(stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            b.step(2)
        for _ in range(5):
            graph.replay()
        torch.cuda.synchronize()
        for k in range(10):
            a.step(1)
            torch.cuda.synchronize()
        assert torch.equal(a.populations(), b.populations())
    net.close()


@pytest.mark.parametrize("rows", [100, 8192, 40000])
def test_training_steps(rows):
    gen = torch.Generator(device="cuda").manual_seed(rows)
    Xs = torch.randn((12, rows, B.MLP_IN), device="cuda", generator=gen).to(torch.bfloat16)
    Ts = torch.randn((12, rows, B.MLP_OUT), device="cuda", generator=gen)
    a, b = _net(2), _net(2)
    X, T = torch.empty_like(Xs[0]), torch.empty_like(Ts[0])
    for k in range(12):
        a.train_step(Xs[k], Ts[k], 1e-3, want_loss=False)
        torch.cuda.synchronize()
    for k in range(12):  # one buffer, written between the steps
        X.copy_(Xs[k])
        T.copy_(Ts[k])
        b.train_step(X, T, 1e-3, want_loss=False)
    assert np.array_equal(a.get_params(), b.get_params())
    for k in range(12):
        a.train_step(Xs[k], Ts[k], 1e-3, want_loss=False)
        torch.cuda.synchronize()
        b.train_step(Xs[k], Ts[k], 1e-3, want_loss=False)
    assert np.array_equal(a.get_params(), b.get_params())
    assert np.array_equal(a.forward(Xs[0]).cpu().numpy(), b.forward(Xs[0]).cpu().numpy())
    a.close()
    b.close()


@pytest.mark.parametrize("shape", [(128, 128, 1), (700, 500, 1), (2048, 1024, 1)])
def test_runs_of_updates(shape):
    with _solver(B.D2Q9, shape) as a, _solver(B.D2Q9, shape) as b:
        for k in range(6):
            a.step(16)
            torch.cuda.synchronize()
        b.step(16)
        rho, u, _ = b.moments()
        b.step(48)
        b.step(32)
        assert torch.equal(a.populations(), b.populations())


@pytest.mark.parametrize("lattice,shape,walls", [(B.D2Q9, (65, 65, 1), 3), (B.D3Q27, (20, 18, 16), 2)])
def test_captured_between_copies_and_a_second_stream(lattice, shape, walls):
    """Chained kernels in a captured graph whose neighbours are copies and a
    kernel of another stream that joins."""
    with _solver(lattice, shape, walls=walls) as a, _solver(lattice, shape, walls=walls) as b:
        state = torch.empty(a.state_bytes(), dtype=torch.uint8, device="cuda")
        a.get_state(state)
        first = state.clone()
        a.step(6)
        ref = a.populations()
        net = _net(4)
        gen = torch.Generator(device="cuda").manual_seed(9)
        Xs = torch.randn((300, B.MLP_IN), device="cuda", generator=gen).to(torch.bfloat16)
        T = torch.randn((300, B.MLP_OUT), device="cuda", generator=gen)
        X = torch.zeros_like(Xs)
        stream, side = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()
        b.set_stream(stream)
        net._lib.lb_mlp_set_stream(net.handle, ctypes.c_void_p(stream.cuda_stream))
        keep, out = torch.empty_like(first), torch.empty_like(ref)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            side.wait_stream(stream)
            with torch.cuda.stream(side):
                X.copy_(Xs)
            keep.copy_(first)
            b.step(4)
            stream.wait_stream(side)
            net.train_step(X, T, 1e-3, want_loss=False)
            b.step(2)
        b.set_state(first, 0)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(b.populations(), ref) and torch.equal(X, Xs)
        other = _net(4)
        other.train_step(Xs, T, 1e-3, want_loss=False)
        assert np.array_equal(net.get_params(), other.get_params())
        net.close()
        other.close()
