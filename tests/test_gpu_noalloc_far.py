"""tds_find_pair_contacts_noalloc with particles so far away that the cells
between would overflow an integer, or at infinity: the pairs of the rest are
those found without them."""
import numpy as np
import pytest

from tests.parity_cases import packed_scene
from tests.test_zz_no_alloc import Inputs, env, step_pair_keys  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu

INF = float("inf")


@pytest.mark.parametrize("far", [(1e30, 1e30, 0.0), (1e12, -1e12, 0.1), (2.7e8, 2.7e8, 0.0), (3e38, -3e38, 3e38),
                                 (INF, 0.0, 0.0), (INF, -INF, 0.1), (INF, INF, INF)])
def test_far_particles_change_nothing(env, far):  # noqa: F811
    torch, tds, L = env
    scene = packed_scene(900, 31, cohesion=1000.0, iters=5)
    ref = step_pair_keys(tds, scene)
    assert len(ref) > 900
    x = np.concatenate([scene["x"], [far]]).astype(np.float32)
    r = np.concatenate([scene["r"], [0.025]]).astype(np.float32)
    keys, m = Inputs(torch, x, r, 20000).call(torch, L, True)
    assert m == len(ref)
    assert np.array_equal(np.sort(keys), ref)
