"""The cell grid's plan for extents of any size: a far particle must coarsen
the cells, never make more of them than there is memory for (extents beyond
2^31 cells, products beyond 2^64, infinities, cells too small to be widened by
a factor)."""
import ctypes
import math

import numpy as np
import pytest

from tests.native_rules import compile_rules

MAX_CELLS = 262144
F = ctypes.c_float


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    L = compile_rules(tmp_path_factory.mktemp("plan"), """
extern "C" float plan(const float *e, float cell, uint32_t max_cells, int *dims) {
  return grid_plan(e, cell, max_cells, dims);
}""")
    L.plan.restype = F
    L.plan.argtypes = [ctypes.POINTER(F), F, ctypes.c_uint32, ctypes.POINTER(ctypes.c_int)]

    def call(extent, cell, max_cells=MAX_CELLS):
        dims = (ctypes.c_int * 3)()
        got = L.plan((F * 3)(*extent), cell, max_cells, dims)
        return got, list(dims)

    return call


def narrowest(extent, cell):
    """The first cell of cell, 1.25 cell, ... whose grid fits, by exact integers."""
    cell = np.float32(cell)
    while True:
        with np.errstate(over="ignore"):
            cells = [float(np.ceil(np.float32(e) / cell)) for e in extent]
        if math.prod(c + 1 for c in cells) <= MAX_CELLS:  # (infinite when a quotient overflows)
            return float(cell), [int(c) + 1 for c in cells]
        cell = np.float32(np.float32(1.25) * cell)


@pytest.mark.parametrize("extent", [(0, 0, 0), (1.0, 2.0, 0.5), (1e3, 1e3, 1e3), (1e6, 0.1, 30.0), (1.5e8, 1.5e8, 0.2),
                                    (4e8, 4e8, 0.3), (1e12, 1e12, 1e12), (3e38, 3e38, 0.15), (3e38, 3e38, 3e38),
                                    (2.0 ** 32 * 0.0625, 2.0 ** 32 * 0.0625, 0.1), (0.0625 * (2.0 ** 22 - 1),) * 3])
def test_the_narrowest_grid_that_fits(plan, extent):
    assert plan(extent, 0.0625) == narrowest(extent, 0.0625)


INF, NAN = math.inf, math.nan


@pytest.mark.parametrize("extent", [(INF, 1.0, 1.0), (INF, INF, 0.2), (INF, INF, INF), (NAN, 1.0, 2.0), (NAN, NAN, NAN),
                                    (-INF, -INF, -INF), (-INF, 1e30, INF), (1e38, 1e38, INF)])
@pytest.mark.parametrize("cell", [0.05, 1e-45, 1e-38, 1e30, 0.0, -1.0, INF, NAN])
def test_no_extent_or_cell_overruns_the_table(plan, extent, cell):
    got, dims = plan(extent, cell)
    assert got > 0 and all(d >= 1 for d in dims) and math.prod(dims) <= MAX_CELLS
    if any(e == INF for e in extent):  # as far as cells go
        assert got == INF and dims == [1, 1, 1]


def test_cells_too_narrow_to_be_widened_by_a_factor(plan):
    got, dims = plan((1.0, 1.0, 1.0), 1e-45)  # 1.25 times the smallest denormal rounds back to it
    assert math.prod(dims) <= MAX_CELLS and 1.0 / 64 <= got <= 1.25 / 60


def test_random_extents(plan):
    g = np.random.Generator(np.random.PCG64(7))
    for _ in range(2000):
        extent = [float(np.float32(10.0 ** g.uniform(-3, 37))) for _ in range(3)]
        cell = float(np.float32(10.0 ** g.uniform(-4, 1)))
        got, dims = plan(extent, cell)
        assert all(1 <= d <= MAX_CELLS for d in dims) and math.prod(dims) <= MAX_CELLS, extent
        assert (got, dims) == narrowest(extent, cell)
