"""Warps of a solver CTA: never none, never more than the shape's, enough for a
bed's row tiles as long as the shape has them."""
import ctypes

import pytest

from tests.native_rules import compile_rules


@pytest.fixture(scope="module")
def warps(tmp_path_factory):
    L = compile_rules(tmp_path_factory.mktemp("warps"),
                      'extern "C" int warps(uint32_t n, int blocks, int most) { return solver_warps(n, blocks, most); }')
    L.warps.argtypes = [ctypes.c_uint32, ctypes.c_int, ctypes.c_int]
    return L.warps


@pytest.mark.parametrize("n", [1, 13, 14, 500, 2000, 8000, 20000, 1000000, 2 ** 31 - 2])
@pytest.mark.parametrize("blocks", [1, 2, 143, 152, 304, 456])
@pytest.mark.parametrize("most", [8, 13, 16, 24])
def test_range(warps, n, blocks, most):
    w = warps(n, blocks, most)
    assert 1 <= w <= most
    assert w == most or w * blocks >= 4 * n / 32 + 64 - blocks


def test_small_beds_leave_room(warps):
    assert warps(2000, 143, 16) == 3 and warps(8000, 152, 16) == 7 and warps(20000, 152, 16) == 16
