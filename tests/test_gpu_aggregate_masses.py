"""Aggregate bodies of particles whose FP32 record 1/m is denormal, near the
largest number, infinite or zero (radii far from any soil's): the body's mass
is the record's reciprocal in FP64."""
import numpy as np
import pytest

from paper_2011_00459_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


@pytest.mark.parametrize("r", [1e-16, 1e-15, 7.1e-15, 1e-14, 1.2e-14, 1e-9, 0.03, 1e6, 1e11, 3.2e11, 3.5e11, 1e12, 1e13, 1e14, 1e20])
def test_mass_is_the_records_reciprocal(tds, r):
    p = S.base_params()
    with np.errstate(all="ignore"):
        r32 = np.float32(r)
        record = np.float32(1.0 / (np.float64(np.float32(p["density"])) * 4.0 / 3.0 * np.pi * np.float64(r32) ** 3))
        want = 1.0 / np.float64(record)
    g = tds.Scene(S.with_particles(p, [[0.0, 0.0, 0.0]], [r32], [[1.0, 2.0, 3.0]]))
    a = g.aggregate_bodies([{"planes": S.box_planes((0, 0, 0), (1, 1, 1))}])[0]
    g.close()
    assert a["count"] == (want > 0.0)  # (without mass there is no body, as ever)
    if np.isinf(want) or want == 0.0:
        assert a["mass"] == want
    else:
        assert a["mass"] == pytest.approx(want, rel=1e-15)
        assert np.abs(a["vel"] - [1.0, 2.0, 3.0]).max() <= 1e-14
