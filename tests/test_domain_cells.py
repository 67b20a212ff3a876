"""The broadphase's cells over any domain: their number must neither wrap nor
overflow, and the memory a scene asks for must hold them."""
import ctypes

import numpy as np
import pytest

from paper_2011_00459_gb300 import build, scenes as S

R = 0.03
CELL = float(np.float32(np.float32(np.float32(2.0 * R) * np.float32(1.025)) * np.float32(1.02)))
MAX_CELLS = 1 << 26


@pytest.fixture(scope="module")
def tds():
    build.build()
    from paper_2011_00459_gb300 import tds

    return tds


def workspace(tds, domain):
    x = np.zeros((2, 3), np.float32)
    x[1] = 0.5
    d, keep, _ = tds._make_desc(S.with_particles(S.base_params(), x, np.full(2, R, np.float32)), 0, domain)
    nb = ctypes.c_uint64()
    tds._check(tds.lib().tds_batch_workspace_bytes(ctypes.byref(d), 1, ctypes.byref(nb)))
    return nb.value


def box(*cells):
    return ((0.0, 0.0, 0.0), tuple((c - 0.5) * CELL for c in cells))


def test_a_moderate_domain(tds):
    assert workspace(tds, box(256, 256, 256)) - workspace(tds, box(1, 1, 1)) >= 8 * (256 ** 3 - 1)  # counts and starts


@pytest.mark.parametrize("cells", [(2.0 ** 22,) * 3, (2.0 ** 24, 2.0 ** 20, 2.0 ** 20), (2.0 ** 31, 2.0 ** 31, 4.0),
                                   (1e12, 1e12, 1e12), (1e30, 5.0, 5.0), (1e36, 1e36, 1e36)])
def test_a_huge_domain_gets_coarser_cells_not_fewer(tds, cells):
    """Cells 1.25 times as wide until they fit: at least half the limit for three long axes, and for one long axis
    what is left when the short ones are down to one cell."""
    got = workspace(tds, box(*cells))
    assert 8 * MAX_CELLS / 2.0 < got < 8 * MAX_CELLS + (64 << 20)


def test_no_cell_is_too_narrow_to_be_widened(tds):
    x = np.zeros((1, 3), np.float32)
    d, keep, _ = tds._make_desc(S.with_particles(S.base_params(), x, np.full(1, 1e-45, np.float32)), 0,
                                ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0)))
    nb = ctypes.c_uint64()
    tds._check(tds.lib().tds_batch_workspace_bytes(ctypes.byref(d), 1, ctypes.byref(nb)))
    assert nb.value < 8 * MAX_CELLS + (64 << 20)
