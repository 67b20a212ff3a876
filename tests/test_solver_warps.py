"""Warps of a solver CTA: never none, never more than the shape's, enough for a
bed's row tiles and a batch's scenes as long as the shape has them."""
import ctypes

import pytest

from tests.native_rules import compile_rules


@pytest.fixture(scope="module")
def warps(tmp_path_factory):
    L = compile_rules(tmp_path_factory.mktemp("warps"),
                      'extern "C" int warps(uint32_t n, uint32_t scenes, int blocks, int most) { '
                      'return solver_warps(n, scenes, blocks, most); }')
    L.warps.argtypes = [ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int, ctypes.c_int]
    return L.warps


@pytest.mark.parametrize("n", [1, 13, 14, 500, 2000, 8000, 20000, 1000000, 2 ** 31 - 2])
@pytest.mark.parametrize("blocks", [1, 2, 143, 152, 304, 456])
@pytest.mark.parametrize("most", [8, 13, 16, 24])
@pytest.mark.parametrize("scenes", [1, 2, 9, 4096])
def test_range(warps, n, blocks, most, scenes):
    w = warps(n, scenes, blocks, most)
    assert 1 <= w <= most
    assert w == most or w * blocks >= 4 * n / 32 + 64 - blocks
    assert 8 * w >= min(8 * most, scenes)


def test_small_beds_leave_room(warps):
    assert warps(2000, 1, 143, 16) == 3 and warps(8000, 1, 152, 16) == 7 and warps(20000, 1, 152, 16) == 16


def test_batches_keep_a_warp_for_eight_scenes(warps):
    assert warps(4000, 1000, 152, 16) == 16 and warps(640, 64, 46, 16) == 8 and warps(600, 5, 43, 16) == 4
