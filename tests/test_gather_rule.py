"""Where the Gaussian fields gather and where they scatter: measured times of
both on either side of the line."""
import ctypes

import pytest

from tests.native_rules import compile_rules


@pytest.fixture(scope="module")
def pays(tmp_path_factory):
    L = compile_rules(tmp_path_factory.mktemp("rule"),
                      'extern "C" int pays(double v, double q, double n) { return gather_pays(v, q, n); }')
    L.pays.argtypes = [ctypes.c_double] * 3
    return lambda v, q, n: bool(L.pays(v, q, n))


# voxels, smoothing length in voxels, particles, us of the gather and of the scatter
MEASURED = [(120, 0.4, 20000, 318, 251), (280, 0.4, 20000, 111, 152), (64, 0.6, 20000, 668, 1202),
            (120, 0.5, 1e6, 23583, 16539), (650, 0.5, 1e6, 2399, 6693), (120, 0.3, 1e6, 22814, 5475),
            (34000, 0.3, 200000, 58, 46), (12200, 1.0, 200000, 161, 1653), (73000, 0.5, 200000, 91, 105),
            (244000, 0.5, 200000, 170, 114), (158000, 1.0, 200000, 281, 582), (940000, 1.0, 200000, 1125, 563),
            (1820000, 3.0, 200000, 11033, 12688), (21780, 0.5, 20000, 42, 47), (220000, 1.0, 20000, 254, 130),
            (176715, 2.0, 20000, 463, 609), (97336, 3.0, 1000, 450, 1823), (97336, 1.0, 1000, 113, 105),
            (97336, 0.5, 1000, 75, 42), (8700000, 2.0, 1e6, 24945, 16460)]


@pytest.mark.parametrize("voxels,q,n,gather,scatter", MEASURED)
def test_the_faster_one_is_taken(pays, voxels, q, n, gather, scatter):
    assert pays(voxels, q, n) == (gather < scatter)
