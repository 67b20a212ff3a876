"""What a scene's workspace takes: no more than it did before row tiles and
versioned records (4571 bytes a particle of a large bed of 10 contacts each, and
256 bytes and a histogram row per array for a small one), so beds that fit a
GPU or a caller's buffer still do."""
import ctypes

import numpy as np
import pytest

from paper_2011_00459_gb300 import build, scenes as S


@pytest.mark.parametrize("n,most", [(1, 1_750_080), (2000, 10_897_728), (200000, 915_705_152), (1000000, 4_570_792_512)])
def test_workspace(n, most):
    build.build()
    from paper_2011_00459_gb300 import tds

    x, r, v, w = S.packed_block(n, 0.02, 0.03, 1)
    d, keep, _ = tds._make_desc(S.with_particles(S.base_params(), x, r, v, w), 0, None)
    nb = ctypes.c_uint64()
    tds._check(tds.lib().tds_batch_workspace_bytes(ctypes.byref(d), 1, ctypes.byref(nb)))
    assert nb.value <= most
