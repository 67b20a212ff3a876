"""Gaussian fields on a grid over a part of the bed: at every voxel the values
of a grid over the whole bed (they depend on the particles around it, not on
the grid's border), whichever particles lie far outside it or just within
reach of its border voxels."""
import numpy as np
import pytest

from tests.parity_cases import packed_scene

pytestmark = pytest.mark.gpu

TOL = 1e-5  # of the field's maximum: sums in another order


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


@pytest.mark.parametrize("q", [0.4, 0.5, 1.0, 2.3])
@pytest.mark.parametrize("at,dims", [((0, 0, 0), (12, 12, 12)), ((7, 5, 6), (6, 8, 7)), ((9, 9, 9), (9, 9, 9)), ((3, 15, 2), (20, 3, 20))])
def test_a_region_is_a_part_of_the_whole(tds, q, at, dims):
    l0 = 0.0625  # (exact: the voxels' centres are the same numbers)
    sc = packed_scene(12000, 81, tool=False)
    lo = np.floor(sc["x"].min(0) / l0) * l0 - l0
    whole = [int(d) for d in np.ceil((sc["x"].max(0) + l0 - lo) / l0)]
    dims = [min(d, w - a) for d, w, a in zip(dims, whole, at)]
    assert min(dims) >= 3
    g = tds.Scene(sc)
    full = [t.cpu().numpy() for t in g.coarse_grain(tds.make_grid(lo, l0, whole), 1, q * l0)]
    part = [t.cpu().numpy() for t in g.coarse_grain(tds.make_grid(lo + l0 * np.array(at), l0, dims), 1, q * l0)]
    g.close()
    cut = tuple(slice(a, a + d) for a, d in zip(at[::-1], dims[::-1]))
    for name, a, b in zip(("rho", "p", "u"), part, full):
        if name != "u":
            assert np.abs(a - b[cut]).max() <= TOL * np.abs(b).max(), name
    heavy = full[0][cut] > 1e-3 * full[0].max()
    assert np.abs(part[2] - full[2][cut])[heavy].max() <= 1e-4 * np.abs(full[2][cut][heavy]).max()
    assert np.array_equal(part[0] > 0, full[0][cut] > 0)
