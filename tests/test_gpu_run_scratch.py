"""The scratch of runs of updates: given back, refused, looked for again, and the
route that lb_step takes with and without it.
"""
import threading

import pytest

from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GB = 1 << 30
BOX = (300, 300, 256)  # D3Q27: 2.3 GB of populations, 1.8 GB of scratch


def _init(s, seed=5):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dims = (s.nz, s.ny, s.nx)
    rho = 1.0 + 0.01 * torch.rand(dims, device="cuda", generator=gen)
    u = 0.03 * torch.randn((s.d,) + dims, device="cuda", generator=gen)
    s.init_fields(rho, u)
    torch.cuda.synchronize()
    s._keep = None


def _free():
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _leave(nbytes):
    """A tensor that takes all free memory but nbytes."""
    return torch.empty(_free() - nbytes, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("lattice,shape,steps,route", [
    (B.D2Q9, (1, 1, 1), 6, B.RUN_TILES), (B.D2Q9, (5, 3, 1), 20, B.RUN_TILES),
    (B.D2Q9, (128, 128, 1), 50, B.RUN_TILES), (B.D2Q9, (251, 251, 1), 40, B.RUN_TILES),
    (B.D2Q9, (701, 500, 1), 13, B.RUN_TILES), (B.D2Q9, (2300, 1700, 1), 6, B.RUN_ROWS),
    (B.D2Q9, (128, 128, 1), 3, B.RUN_SINGLE), (B.D3Q27, (128, 128, 128), 5, B.RUN_MOMENTS),
    (B.D3Q27, (64, 64, 64), 20, B.RUN_SINGLE), (B.D3Q19, (150, 200, 180), 16, B.RUN_MOMENTS),
])
def test_route(lattice, shape, steps, route):
    with B.Solver(lattice, shape, 0.7) as s:
        assert s.run_info() == {"route": B.RUN_SINGLE, "bytes": 0, "limit": -1}
        s.step(steps)
        info = s.run_info()
        assert info["route"] == route and (info["bytes"] > 0) == (route != B.RUN_SINGLE)
        s.step(0)
        assert s.run_info() == info
        s.step(1)
        assert s.run_info()["route"] == B.RUN_SINGLE


def test_limit():
    with B.Solver(B.D3Q27, BOX, 0.61) as a, B.Solver(B.D3Q27, BOX, 0.61) as b:
        for s in (a, b):
            _init(s)
        a.step(8)
        held = a.run_info()["bytes"]
        assert held >= 80 * a.n
        before = _free()
        a.set_run_limit(held - 1)
        assert a.run_info() == {"route": B.RUN_MOMENTS, "bytes": 0, "limit": held - 1}
        assert _free() - before >= held - GB // 64
        a.step(8)
        assert a.run_info()["route"] == B.RUN_SINGLE and a.run_info()["bytes"] == 0
        a.set_run_limit(held)
        a.step(8)
        assert a.run_info() == {"route": B.RUN_MOMENTS, "bytes": held, "limit": held}
        b.set_run_limit(0)
        b.step(24)
        assert b.run_info()["route"] == B.RUN_SINGLE
        assert torch.equal(a.populations(), b.populations())


def test_refused_while_memory_is_short_and_looked_for_again():
    with B.Solver(B.D3Q27, BOX, 0.61) as s:
        _init(s)
        hog = _leave(4 * GB)  # the scratch would take more than a quarter
        s.step(8)
        assert s.run_info()["route"] == B.RUN_SINGLE
        del hog
        _free()
        s.step(8)
        assert s.run_info()["route"] == B.RUN_MOMENTS


def test_a_context_that_needs_the_memory_gets_it():
    with B.Solver(B.D3Q27, BOX, 0.61) as a, B.Solver(B.D3Q27, BOX, 0.61) as b:
        for s in (a, b):
            _init(s)
        b.set_run_limit(0)
        hog = _leave(9 * GB)
        a.step(8)
        assert a.run_info()["bytes"] > 0
        left = _free()
        big = (300, 300, (left + GB // 2) // (108 * 90000))
        with B.Solver(B.D3Q27, big, 0.7) as c:  # without the scratch it does not fit
            assert c.state_bytes() > left and a.run_info()["bytes"] == 0
            a.step(8)  # no room now: update by update
            assert a.run_info()["route"] == B.RUN_SINGLE
        a.step(8)
        assert a.run_info()["route"] == B.RUN_MOMENTS
        del hog
        b.step(24)
        assert torch.equal(a.populations(), b.populations())


def test_scratch_taken_away_while_another_thread_steps():
    shape, rounds = (128, 128, 128), 30
    with B.Solver(B.D3Q27, shape, 0.61) as a, B.Solver(B.D3Q27, shape, 0.61) as b:
        for s in (a, b):
            _init(s)
        hog = _leave(9 * GB)
        done = threading.Event()
        taken = []

        def steps():
            for _ in range(rounds):
                a.step(8)
                taken.append(a.run_info()["route"])
                torch.cuda.current_stream().synchronize()
            done.set()

        worker = threading.Thread(target=steps)
        worker.start()
        while not done.is_set():  # each wants more than there is and takes the scratch first
            with pytest.raises(B.LBError) as e:
                B.Solver(B.D3Q27, (300, 300, 1200), 0.7)
            assert e.value.code == B.LB_ENOMEM
        worker.join()
        del hog
        assert taken.count(B.RUN_MOMENTS) > 0
        b.set_run_limit(0)
        b.step(8 * rounds)
        assert torch.equal(a.populations(), b.populations())
