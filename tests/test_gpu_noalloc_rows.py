"""tds_find_pair_contacts_noalloc on rows of candidates around the length from
which the whole warp takes them: all particles in one cell, or crowded cells
beside sparse ones. The pairs against the same FP32 predicate over all pairs,
the order against the cells' (one cell: ascending), and the first keys of a
short output buffer."""
import numpy as np
import pytest

from tests.test_zz_no_alloc import Inputs, env  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


def all_pairs(x, r, cohesive):
    f = np.float32
    a, b = np.triu_indices(len(r), 1)
    d = x[b] - x[a]
    d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
    s = r[a] + r[b]
    R = s + f(0.025) * s if cohesive else s
    hit = d2 < R * R
    return (a[hit].astype(np.uint64) << np.uint64(32)) | b[hit].astype(np.uint64)


@pytest.mark.parametrize("m", [1, 2, 31, 32, 33, 64, 127, 128, 129, 130, 160, 161, 300, 1500])
@pytest.mark.parametrize("cohesive", [False, True])
def test_one_cell(env, m, cohesive):  # noqa: F811
    torch, tds, L = env
    g = np.random.Generator(np.random.PCG64(m))
    x = g.uniform(0.0, 0.09, (m, 3)).astype(np.float32)
    r = g.uniform(0.001, 0.02, m).astype(np.float32)
    r[0] = 0.05  # one cell covers them all: 2 * 0.05 * 1.0455 wide
    x[-1] = 0.1045, 0.1045, 0.1045
    want = all_pairs(x, r, cohesive)
    keys, count = Inputs(torch, x, r, len(want) + 8).call(torch, L, cohesive)
    assert count == len(want) and np.array_equal(np.sort(keys), want)
    near = keys[(keys & np.uint64(0xFFFFFFFF)) != m - 1]  # (the last particle lies in the next cell)
    assert np.array_equal(near, np.sort(near))


@pytest.mark.parametrize("crowds", [(33, 140, 127), (400, 3, 129)])
def test_crowded_cells_beside_sparse_ones(env, crowds):  # noqa: F811
    torch, tds, L = env
    g = np.random.Generator(np.random.PCG64(sum(crowds)))
    parts = [g.uniform(0.0, 2.0, (1500, 3))]
    for c, at in zip(crowds, ((0.3, 0.3, 0.3), (1.0, 1.9, 0.1), (1.5, 0.7, 1.2))):
        parts.append(np.array(at) + g.uniform(0.0, 0.03, (c, 3)))
    x = np.concatenate(parts).astype(np.float32)[g.permutation(1500 + sum(crowds))]
    r = g.uniform(0.01, 0.03, len(x)).astype(np.float32)
    want = all_pairs(x, r, True)
    full, count = Inputs(torch, x, r, len(want)).call(torch, L, True)
    assert count == len(want) and np.array_equal(np.sort(full), want)
    for cap in (1, len(want) // 2, len(want) - 1):
        part, count = Inputs(torch, x, r, cap).call(torch, L, True)
        assert count == len(want) and np.array_equal(part, full[:cap])
