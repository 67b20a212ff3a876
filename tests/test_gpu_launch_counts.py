"""Solver CTA counts that tds_set_launch_config takes: without a chosen shape up
to two per SM, lowered to what fits; with one, its co-resident CTAs at most."""
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


def test_counts(tds):
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    scene = packed_scene(300, 61, iters=8)
    g, h = tds.Scene(scene), tds.Scene(scene)
    fits = g.launch_config()["max_pgs_blocks"]
    assert fits == sms  # the default shape: one CTA per SM
    for asked in (1, fits, fits + 1, 2 * sms):
        g.set_launch_config(pgs_blocks=asked)
        assert g.launch_config()["pgs_blocks"] == min(asked, fits)
    with pytest.raises(tds.TdsError):
        g.set_launch_config(pgs_blocks=2 * sms + 1)
    assert g.launch_config()["pgs_blocks"] == fits
    g.step(2)
    h.step(2)
    a, b = g.read_particles(), h.read_particles()
    assert all(np.array_equal(a[k], b[k]) for k in "xvw")
    with pytest.raises(tds.TdsError):  # a chosen shape: what fits and no more
        h.set_launch_config(pgs_threads=512, pgs_per_thread=2, pgs_blocks=fits + 1)
    h.set_launch_config(pgs_threads=416, pgs_per_thread=1, pgs_blocks=2 * sms)
    assert h.launch_config()["pgs_blocks"] == 2 * sms
    h.set_launch_config(pgs_threads=512, pgs_per_thread=2)
    assert h.launch_config()["pgs_blocks"] == fits
    with pytest.raises(tds.TdsError):
        h.set_launch_config(pgs_blocks=2 * sms)
    g.close()
    h.close()
