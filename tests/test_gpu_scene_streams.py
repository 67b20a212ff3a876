"""Several scenes, each on its own stream, stepped in turn without waiting for
one another: their solver CTAs share the SMs. Every scene gets the bits it has
alone, with few and with many warps a CTA."""
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


SIZES = [3, 40, 500, 501, 2000, 2000, 5000, 9000]
BLOCKS = [0, 0, 36, 5, 0, 61, 0, 152]


def scene(q):
    return packed_scene(SIZES[q], 200 + q, iters=15, tol=1e-30 if q % 2 else 0.0)  # (odd ones: with residual checks)


def result(g):
    p = g.read_particles()
    return [p["x"], p["v"], p["w"], np.float32(g.stats()["residual"])]


@pytest.mark.parametrize("graph", [False, True])
def test_alone_and_together(tds, graph):
    import torch

    alone = []
    for q in range(len(SIZES)):
        g = tds.Scene(scene(q))
        g.step(6)
        alone.append(result(g))
        g.close()
    gs = [tds.Scene(scene(q), stream=torch.cuda.Stream()) for q in range(len(SIZES))]
    for g, b in zip(gs, BLOCKS):
        g.set_graph(graph)
        g.set_launch_config(pgs_blocks=b)
    for _ in range(6):
        for g in gs:
            g.step(1)
    for q, g in enumerate(gs):
        assert all(np.array_equal(a, b) for a, b in zip(alone[q], result(g))), q
        g.close()
