"""16-bit stores on rows that are not whole 16-byte chunks (two cells to a thread).

One update from either parity, correctly rounded, in the comparison and at the
tolerance of the other 16-bit kernels: rows of two cells and of an odd number
(whose odd update goes one cell to a thread), of less and more than a block
takes, several rows to a block with some left over, a grid of an odd number of
cells and one too small for this kernel.
"""
import pytest

import oracle as O
import test_gpu_lowprec as T
from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage", [B.STORE_F16, B.STORE_BF16])
@pytest.mark.parametrize("parity", [0, 1])
@pytest.mark.parametrize("collision", [B.COLLIDE_RR, B.COLLIDE_REG2, B.COLLIDE_BGK])
@pytest.mark.parametrize("lattice,shape", [
    (O.D2Q9, (250, 600, 1)), (O.D2Q9, (602, 240, 1)), (O.D2Q9, (1046, 140, 1)),
    (O.D2Q9, (15, 9400, 1)), (O.D2Q9, (15, 9401, 1)), (O.D2Q9, (2, 3, 1)),
    (O.D3Q19, (26, 60, 50)), (O.D3Q19, (530, 13, 11)), (O.D3Q19, (4, 150, 120)),
    (O.D3Q27, (66, 30, 25)), (O.D3Q27, (250, 19, 10)), (O.D3Q27, (2, 301, 80)),
])
def test_one_update(storage, parity, collision, lattice, shape):
    T.test_one_update_is_correctly_rounded(storage, parity, collision, lattice, shape)


@pytest.mark.parametrize("storage", [B.STORE_F16, B.STORE_BF16])
@pytest.mark.parametrize("lattice,shape,copies", [
    (O.D2Q9, (250, 50, 1), 12), (O.D3Q19, (30, 20, 11), 10), (O.D3Q27, (26, 18, 10), 10),
])
def test_updates_equal_those_of_one_cell_to_a_thread(storage, lattice, shape, copies):
    """A periodic pattern repeated along the last axis fills a store that takes
    two cells to a thread, the pattern alone one that does not: populations bit
    for bit over updates from both parities."""
    _, q = O.dims_of(lattice)
    axis = -2 if shape[2] == 1 else -3
    long = (shape[0], shape[1] * copies, 1) if axis == -2 else shape[:2] + (shape[2] * copies,)
    assert q * shape[0] * shape[1] * shape[2] < 1250000 <= q * long[0] * long[1] * long[2]
    df = torch.from_numpy(T.W.random_populations(q, shape, seed=5, amp=0.05).astype("float32")).cuda()

    def repeated(t):
        return torch.cat([t] * copies, dim=axis)

    with B.Solver(lattice, shape, 0.63, storage=storage) as a, \
            B.Solver(lattice, long, 0.63, storage=storage) as b:
        a.set_populations(df)
        b.set_populations(repeated(df).contiguous())
        for _ in range(3):
            a.step(1)
            b.step(1)
            assert torch.equal(repeated(a.populations()), b.populations())
