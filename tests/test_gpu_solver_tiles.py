"""The solver's row tiles at their edges: buckets of fewer than 32 contacts,
warps without a tile, with one, with as many as their ring holds or one more,
and with more than 32 (their list is then read in groups). Every case against
the oracle, and bit for bit the same whatever the number of solver CTAs, the
synchronisation between colours and the CTA shape."""
import numpy as np
import pytest

from tests.parity_cases import packed_scene, rel_impulse_error

pytestmark = pytest.mark.gpu

IMPULSE_TOL = 1e-3  # the second step's bound: its inputs carry the first step's FP32 rounding


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


@pytest.mark.parametrize("n,tool", [(1, False), (2, False), (9, False), (60, True), (700, True), (6000, True)])
def test_tiles_of_every_count(tds, orc, n, tool):
    scene = packed_scene(n, 90 + n, iters=12, tool=tool)
    st = orc.State(scene)
    ref = [orc.step(scene, st) for _ in range(2)][-1]  # a cold start, then a warm one
    want = None
    for cfg in (dict(), dict(pgs_blocks=1), dict(pgs_blocks=2), dict(pgs_blocks=3, pgs_sync=0),
                dict(pgs_blocks=1, pgs_threads=256, pgs_per_thread=1), dict(pgs_threads=512, pgs_per_thread=3),
                dict(pgs_blocks=1, pgs_threads=768, pgs_per_thread=1)):
        g = tds.Scene(scene)
        g.set_launch_config(**cfg)
        g.step(2)
        c, p, s = g.read_contacts(), g.read_particles(), g.stats()
        g.close()
        got = [c["keys"], c["colour"], c["lam"], p["x"], p["v"], p["w"], np.float32(s["residual"])]
        if want is None:
            want = got
            assert np.array_equal(c["keys"], ref["keys"])
            if ref["n_contacts"]:
                assert rel_impulse_error(c["lam"], ref["lam"]) <= IMPULSE_TOL
        for a, b in zip(want, got):
            assert np.array_equal(a, b), cfg
