"""The training step at the limits of its inputs: row counts near 2^31, targets without a finite loss."""
import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    from paper_1907_06821_gb300 import build as b
    b.build()
    import paper_1907_06821_gb300 as m
    return m


@pytest.fixture
def ctx(fs):
    with fs.Context((10.0, 10.0, 10.0), (16, 16, 16), 3.0, (0, 0, 0), np.zeros((16, 16, 16))) as c:
        theta = mlp.init_params(3)
        theta[-129:] = np.random.default_rng(3).uniform(-0.1, 0.1, 129)
        c.precond_weights(theta.astype(np.float32))
        yield c


def _rows(seed, n):
    rng = np.random.default_rng(seed)
    return [torch.as_tensor(v.astype(np.float32), device="cuda")
            for v in (rng.normal(0, 0.5, (n, 4)), rng.normal(0, 0.5, n), rng.uniform(0.1, 1, n))]


def test_row_counts_near_2_31(ctx):
    """Rows of weight zero add nothing: the gradient of 2^31 - 4,096 rows of which the first and the
    last 100 carry weight is that of the 200 rows.  The step of a persistent block and of the weight
    sum (9,728 and 8,192 rows) beyond the last row passes 2^31.  Tolerance: the sums are taken in
    another order, FP32 products, 64 * 2^-24 of the largest entry (52 GB of device memory)."""
    n, w = (1 << 31) - 4096, 100
    if torch.cuda.mem_get_info()[0] < 70 << 30:
        pytest.skip("needs 70 GB of free device memory")
    small = _rows(1, 2 * w)
    big = []
    for v in small:
        b = torch.zeros((n,) + tuple(v.shape[1:]), dtype=torch.float32, device="cuda")
        b[:w], b[-w:] = v[:w], v[w:]
        big.append(b)
    loss, g = ctx.precond_loss_grad(*big)
    loss0, g0 = ctx.precond_loss_grad(*small)
    del big, b
    torch.cuda.empty_cache()
    assert abs(loss - loss0) < 64 * 2.0 ** -24 * loss0
    assert (g - g0).abs().max().item() < 64 * 2.0 ** -24 * g0.abs().max().item()


@pytest.mark.parametrize("rows", [50, 20000])  # one block; more than one tile per block
def test_infinite_loss(ctx, rows):
    """A loss beyond the FP32 range is infinite, not a NaN, and so are the gradients of the output
    layer for an infinite target (FP32 has them as sums of infinities of one sign)."""
    F, zt, wt = _rows(4, rows)
    zt[7] = 3e25
    torch.cuda.synchronize()
    assert ctx.precond_loss_grad(F, zt, wt)[0] == float("inf")
    zt[7] = float("inf")
    torch.cuda.synchronize()
    loss, g = ctx.precond_loss_grad(F, zt, wt)
    assert loss == float("inf")
    assert g[-1].item() == -float("inf") and torch.isinf(g[-129:]).all()
    zt[7] = float("nan")
    torch.cuda.synchronize()
    loss, g = ctx.precond_loss_grad(F, zt, wt)
    assert np.isnan(loss) and torch.isnan(g[-129:]).all()
