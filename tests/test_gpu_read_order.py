"""Read-back of a bed larger than the scattered read-back takes: as given before
its first step (slots in id order), by id after steps (slots in cell order), and
in a scene that another's state was loaded into."""
import numpy as np
import pytest

from paper_2011_00459_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def test_before_and_after_steps():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    n = 70001
    x, r, v, w = S.packed_block(n, 0.02, 0.03, 5)
    o = np.random.Generator(np.random.PCG64(1)).permutation(n)
    scene = S.with_particles(S.base_params(iters=1, gravity=(0.0, 0.0, 0.0), dt=1e-7), x[o], r[o], v[o], w[o])
    g = tds.Scene(scene)
    p = g.read_particles()
    assert all(np.array_equal(p[k], scene[k]) for k in "xvw") and np.array_equal(g.read_radii(), scene["r"])
    g.step(2)  # 1e-7 s: the particles stay where they are, to 1e-5
    p = g.read_particles()
    assert np.abs(p["x"] - scene["x"]).max() < 1e-5 and np.array_equal(g.read_radii(), scene["r"])
    h = tds.Scene(scene)
    h.load_state(g.save_state())
    q = h.read_particles()
    assert all(np.array_equal(p[k], q[k]) for k in "xvw") and np.array_equal(h.read_radii(), scene["r"])
    g.close()
    h.close()
