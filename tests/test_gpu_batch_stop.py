"""A batch whose beds stop at their own residual: the row tiles of stopped beds
leave the solver's lists. Bit for bit the beds' solo runs, with lists that
start above a warp's ring and end in it or empty, tiles shared by beds that
stop at different sweeps, beds without contacts, and every kind of wait."""
import numpy as np
import pytest

from tests.parity_cases import packed_scene

pytestmark = pytest.mark.gpu

SIZES = (60, 1, 9, 700, 30, 1500)
TOL, EVERY, CAP, STEPS = 1e-3, 3, 400, 2


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


@pytest.fixture(scope="module")
def alone(tds):
    out = []
    for k, n in enumerate(SIZES):
        g = tds.Scene(packed_scene(n, 61 + k, iters=CAP, tol=TOL, mu_t=0.4 + 0.1 * k))
        g.set_solver(CAP, TOL, EVERY)
        g.step(STEPS)
        s, p = g.stats(), g.read_particles()
        g.close()
        out.append((s["iterations"], np.float32(s["residual"]), p))
    return out


@pytest.mark.parametrize("cfg", [dict(), dict(pgs_blocks=1), dict(pgs_blocks=2, pgs_sync=0), dict(pgs_blocks=5),
                                 dict(pgs_blocks=1, pgs_threads=256, pgs_per_thread=1),
                                 dict(pgs_blocks=3, pgs_threads=512, pgs_per_thread=3)], ids=str)
def test_stopped_beds_leave_the_lists(tds, alone, cfg):
    b = tds.Batch([packed_scene(n, 61 + k, iters=CAP, tol=TOL, mu_t=0.4 + 0.1 * k) for k, n in enumerate(SIZES)])
    b.set_solver(CAP, TOL, EVERY)
    b.set_launch_config(**cfg)
    b.step(STEPS)
    solve = b.read_solve()
    for q, (sweeps, residual, p) in enumerate(alone):
        mine = b.read_scene(q)
        assert (solve["sweeps"][q], solve["residual"][q]) == (sweeps, residual), q
        for key in ("x", "v", "w"):
            assert np.array_equal(mine[key], p[key]), (q, key)
    b.close()
    assert len({s for s, _, _ in alone}) > 2
