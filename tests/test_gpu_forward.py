"""The forward pass over many tiles: a row's output does not depend on the batch.

Batches of less than a tile and with a ragged last tile, with one tile to a
group of threads, to a block and several to each are compared bit for bit with
the same rows taken a few at a time, the sizes that the tests against the
reference cover; the words after the outputs must stay as they are.
"""
import pytest

from paper_1505_06900_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m", [1, 127, 129, 128 * 152 + 1, 128 * 304, 128 * 304 + 77, 131073])
def test_rows_do_not_depend_on_the_batch(m):
    gen = torch.Generator().manual_seed(m)
    params = (0.1 * torch.randn(B.MLP_PARAMS, generator=gen)).numpy()
    X = torch.randn((m, B.MLP_IN), generator=gen).cuda().to(torch.bfloat16)
    net = B.MLP(params)
    out = torch.full((m + 8, B.MLP_OUT), 7.0, device="cuda")
    assert net._lib.lb_mlp_forward(net.handle, B._ptr(X), m, B._ptr(out)) == B.LB_OK
    torch.cuda.synchronize()
    assert (out[m:] == 7.0).all()
    rows = {0, 1, 126, 127, 128, m // 2, m - 129, m - 128, m - 2, m - 1}
    for r in sorted(q for q in rows if 0 <= q < m):
        n = min(m - r, 3)
        assert torch.equal(net.forward(X[r:r + n].contiguous()), out[r:r + n]), r
    net.close()
