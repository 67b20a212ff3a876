"""Aggregate bodies where the lanes' running sums and the solve for omega can
go wrong: zones that alternate from particle to particle, warps with part of a
zone, zones of no, one, two and three particles and of a straight line (a
singular inertia, so the pseudo-inverse), sizes around a warp's stretch."""
import numpy as np
import pytest

from oracle import aggregate as AG
from paper_2011_00459_gb300 import scenes as S

pytestmark = pytest.mark.gpu

REL = 1e-6  # FP32 reciprocals of the masses, as the aggregates' own tests


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


def bodies(tds, x, v, r, zones):
    p = S.base_params()
    g = tds.Scene(S.with_particles(p, x, r, v))
    got = g.aggregate_bodies(zones)
    g.close()
    return got, AG.aggregate(np.asarray(x, np.float32), np.asarray(v, np.float32), np.asarray(r, np.float32), p["density"], zones)


def close(a, b, scale):
    return np.abs(np.asarray(a) - np.asarray(b)).max() <= REL * max(np.abs(b).max(), scale)


@pytest.mark.parametrize("n", [1, 31, 33, 128, 129, 1000, 40001])
def test_zones_that_alternate(tds, n):
    g = np.random.Generator(np.random.PCG64(n))
    x = g.uniform(-1.0, 1.0, (n, 3))
    x[:, 2] = np.arange(n) % 5 + g.uniform(-0.3, 0.3, n)  # the zone of particle i is i mod 5 (the fifth: none)
    v, r = g.normal(0, 1, (n, 3)), g.uniform(0.02, 0.05, n)
    zones = [{"planes": S.box_planes((0, 0, k), (2, 2, 0.4))} for k in range(4)]
    got, ref = bodies(tds, x, v, r, zones)
    for a, b in zip(got, ref):
        assert a["count"] == b["count"]
        if b["count"]:
            assert a["mass"] == pytest.approx(b["mass"], rel=REL)
            assert close(a["com"], b["com"], 1.0) and close(a["vel"], b["vel"], 1.0)
            assert close(a["inertia"], b["inertia"], 0.0)
        if b["count"] > 20:  # (a few particles: omega hangs on the smallest eigenvalue)
            assert np.abs(a["omega"] - b["omega"]).max() <= 10 * REL * max(np.abs(b["omega"]).max(), 1e-3)


@pytest.mark.parametrize("k", [1, 2, 3, 7])
@pytest.mark.parametrize("line", [False, True])
def test_singular_and_small_bodies(tds, k, line):
    """k particles spinning about their centre: omega without the component
    that a body of no extent about an axis cannot have."""
    g = np.random.Generator(np.random.PCG64(10 * k + line))
    d = np.linspace(-1, 1, k)[:, None] * [[0.6, 0.0, 0.8]] if line else g.uniform(-1, 1, (k, 3))
    d = d - d.mean(0)
    w = np.array([0.3, -0.7, 0.2])
    x, v = d + 3.0, np.cross(w, d) + [1.0, 2.0, 3.0]
    got, ref = bodies(tds, x, v, np.full(k, 0.04), [{"planes": S.box_planes((3, 3, 3), (2, 2, 2))}])
    a, b = got[0], ref[0]
    assert a["count"] == b["count"] == k
    if line or k < 3:
        u = np.array([0.6, 0.0, 0.8]) if line else (d[0] / np.linalg.norm(d[0]) if k > 1 else None)
        if k > 1:  # no spin about the line itself (the FP32 positions lie within 1e-7 of it)
            want = w - (w @ u) * u
            assert np.abs((a["omega"] - (a["omega"] @ u) * u) - want).max() <= 1e-4
        else:
            assert np.abs(a["omega"]).max() == 0.0
    else:
        assert np.abs(a["omega"] - w).max() <= 1e-4
