"""Loss and gradients of the warm-start network at the row counts where its
tiles and blocks end: one row, a warp's 16 and a block's 128 rows less and more
one, more rows than one pass of the grid. A batch's loss and gradient are the
row-weighted means of its parts', here computed row by row (128 rows at a time
for the largest). Every row's forward pass is the same in both; dy carries the
scale 1/m into its BF16 rounding, so the gradients agree to 2^-8 a product."""
import numpy as np
import pytest

from paper_2011_00459_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


@pytest.mark.parametrize("m", [1, 7, 15, 16, 17, 127, 128, 129, 300, 40000])
def test_gradients_at_the_edges_of_tiles(tds, m):
    g = S.rng(50 + m)
    X = g.normal(0, 1, (m, 10)).astype(np.float32)
    T = g.normal(0, 1, (m, 3)).astype(np.float32)
    net = tds.Net(seed=3)

    def run(a, b):
        loss, grad = net.loss_grad(X[a:b], T[a:b])
        return float(loss.item()), grad.cpu().numpy().astype(np.float64)

    loss, grad = run(0, m)
    part = 1 if m <= 300 else 128
    parts = [(min(a + part, m) - a, *run(a, min(a + part, m))) for a in range(0, m, part)]
    mean_loss = sum(k * v for k, v, _ in parts) / m
    mean = sum(k * v for k, _, v in parts) / m
    assert loss == pytest.approx(mean_loss, rel=1e-5)  # FP32 sums in another order
    assert np.linalg.norm(grad - mean) <= 1e-2 * np.linalg.norm(mean)
