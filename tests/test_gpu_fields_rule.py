"""The choice between gather and scatter looks at the grid's own scene: the
same launches and the same fields for a scene alone, as one of a batch, and
with a reserve of dormant slots."""
import numpy as np
import pytest

from tests.parity_cases import packed_scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


def fields(g, grid, R):
    before = g.stats()["kernel_launches"]
    out = [t.cpu().numpy() for t in g.coarse_grain(grid, 1, R)]
    return g.stats()["kernel_launches"] - before, out


@pytest.mark.parametrize("l0,q", [(0.016, 1.0), (0.016, 0.5), (0.05, 1.0)])
def test_a_scene_alone_in_a_batch_and_with_a_reserve(tds, l0, q):
    scenes = [packed_scene(1000, 100 + k, tool=False) for k in range(30)]
    sc = scenes[7]
    lo, hi = sc["x"].min(0) - 2 * l0, sc["x"].max(0) + 2 * l0
    dims = [int(d) for d in np.ceil((hi - lo) / l0)]
    alone = tds.Scene(sc)
    count, want = fields(alone, tds.make_grid(lo, l0, dims), q * l0)
    alone.close()
    reserve = dict(sc)
    for k in ("x", "v", "w"):
        reserve[k] = np.concatenate([sc[k], np.zeros((29000, 3), np.float32)])
    reserve["r"] = np.concatenate([sc["r"], np.zeros(29000, np.float32)])
    batch, single = tds.Batch(scenes), tds.Scene(reserve)
    for g, scene in ((batch, 7), (single, 0)):
        c, got = fields(g, tds.make_grid(lo, l0, dims, scene), q * l0)
        assert c == count
        for a, b in zip(got, want):  # (sums in another order)
            assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max()
        g.close()
