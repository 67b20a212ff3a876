"""A particle with more contacts than the search keeps per particle (it is then
searched again for the list) and more colours than one mask word holds: a large
sphere in a shell of small ones, against the oracle, first and last in id order
(it owns all of the contacts, or none)."""
import numpy as np
import pytest

from paper_2011_00459_gb300 import scenes as S
from tests.parity_cases import rel_impulse_error

pytestmark = pytest.mark.gpu

IMPULSE_TOL = 1e-4  # the parity tests' bound


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


@pytest.mark.parametrize("k", [3, 63, 64, 65, 100])
@pytest.mark.parametrize("first", [True, False])
def test_a_large_sphere_among_small_ones(tds, orc, k, first):
    g = np.random.Generator(np.random.PCG64(k))
    i = np.arange(k) + 0.5  # a Fibonacci lattice on the sphere: no two small ones touch
    z, phi = 1.0 - 2.0 * i / k, np.pi * (1.0 + 5.0 ** 0.5) * i
    d = np.stack([np.sqrt(1 - z * z) * np.cos(phi), np.sqrt(1 - z * z) * np.sin(phi), z], 1)
    x = np.concatenate([[[0.0, 0.0, 0.0]], d * (0.22 - g.uniform(1e-5, 1e-4, (k, 1)))])
    r = np.concatenate([[0.2], np.full(k, 0.02)])
    v = np.concatenate([[[0.0, 0.0, 0.0]], -0.05 * d + g.normal(0, 0.01, (k, 3))])
    if not first:
        x, r, v = x[::-1], r[::-1], v[::-1]
    scene = S.with_particles(S.base_params(gravity=(0.0, 0.0, 0.0), iters=10), x, r, v)
    ref = orc.step(scene, orc.State(scene))
    assert ref["n_contacts"] == k and ref["n_colours"] == k
    s = tds.Scene(scene)
    s.step(1)
    c = s.read_contacts()
    s.close()
    assert np.array_equal(c["keys"], ref["keys"])
    assert np.array_equal(c["colour"].astype(np.int64), ref["colour"].astype(np.int64))
    assert rel_impulse_error(c["lam"], ref["lam"]) <= IMPULSE_TOL
