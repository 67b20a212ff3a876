"""The ways tds_coarse_grain computes a field, against the FP64 oracle: the
sorted gather (well filled grids), the scatter (sparse ones) and the voxel
kernel with and without scratch for its grid; grids of odd extents, smaller
than the bed (particles outside count in the border voxels' sums), a single
voxel, smoothing lengths from half a voxel to many, one scene of a batch."""
import numpy as np
import pytest

from oracle import fields as F
from tests.parity_cases import packed_scene

pytestmark = pytest.mark.gpu

TOL = 1e-5  # of the field's maximum, as the fields' own tests


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


# (voxel, smoothing length over it (0: voxel kernel), extents; None: the bed and a margin)
CASES = [(0.05, 0.5, None), (0.05, 1.0, None), (0.1, 3.0, None), (0.012, 1.0, None), (0.05, 16.0, (3, 2, 5)),
         (0.07, 1.3, (5, 3, 2)), (1.0, 0.4, (1, 1, 1)), (0.05, 0.0, None), (0.07, 0.0, (5, 3, 2)), (0.009, 0.0, None)]


@pytest.mark.parametrize("l0,ratio,dims", CASES)
def test_every_way_matches_the_oracle(tds, l0, ratio, dims):
    scenes = [packed_scene(300, 71), packed_scene(1500, 72)]
    sc = scenes[1]
    x = sc["x"]
    lo = (x.min(0) + (0.1 if dims else -2 * l0)).astype(np.float32)
    dims = dims or tuple(int(d) for d in np.ceil((x.max(0) + 2 * l0 - lo) / l0))
    b = tds.Batch(scenes)
    rho, p, u = (t.cpu().numpy() for t in b.coarse_grain(tds.make_grid(lo, l0, dims, 1), int(ratio > 0), ratio * l0))
    b.close()
    m = sc["density"] * 4.0 / 3.0 * np.pi * np.asarray(sc["r"], np.float64) ** 3
    ro, po, uo = F.coarse_grain(x, sc["v"], m, lo, l0, dims, int(ratio > 0), ratio * l0)
    assert np.abs(rho - ro).max() <= TOL * ro.max()
    assert np.abs(p - po).max() <= TOL * np.abs(po).max()
    big = ro > 1e-3 * ro.max()
    assert np.abs(u[big] - uo[big]).max() <= 1e-4 * max(np.abs(uo[big]).max(), 1e-3)
    assert np.array_equal(u[rho == 0], np.zeros_like(u[rho == 0]))
