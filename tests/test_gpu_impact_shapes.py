"""The impact stage under every compiled solver shape with all of the shape's
co-resident CTAs (the stage's own kernel holds fewer per SM than some of
them): the same bits as with the default shape, with launches and from a
graph."""
import numpy as np
import pytest

from tests.test_gpu_impact import impact_block

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


def stepped(tds, graph, **cfg):
    import torch

    g = tds.Scene(impact_block(53), stream=torch.cuda.Stream())
    try:
        if cfg:
            g.set_launch_config(**cfg)
            g.set_launch_config(**dict(cfg, pgs_blocks=g.launch_config()["max_pgs_blocks"]))
        g.set_graph(graph)
        g.step(2)
        p = g.read_particles()
        assert g.stats()["impacts"] > 0
        return [p["x"], p["v"], p["w"]]
    finally:
        g.close()


@pytest.mark.parametrize("graph", [False, True])
def test_every_shape_at_its_most_ctas(tds, graph):
    want = stepped(tds, False)
    for threads, per in tds.SHAPES:
        got = stepped(tds, graph, pgs_threads=threads, pgs_per_thread=per)
        assert all(np.array_equal(a, b) for a, b in zip(want, got)), (threads, per)
