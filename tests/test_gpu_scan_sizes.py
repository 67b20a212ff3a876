"""Prefix sums at the sizes where their form changes: the contact search (whose
pair counts are summed over the particles) on particle numbers around one
block's share, around a tile and at the largest, against a search by distance
on the host; and an empty result."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tds():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2011_00459_gb300 import build, tds

    build.build()
    return tds


@pytest.mark.parametrize("n", [1, 2, 7, 8191, 8192, 8193, 16384, 16385, 18432, 18433, 65536])
def test_pairs_of_a_line(tds, n):
    """Spheres of radius 0.5 on a line, 0.9 apart except every third gap (1.2):
    sphere i touches the next where the gap is 0.9."""
    import torch

    gap = np.where(np.arange(n - 1) % 3 == 2, 1.2, 0.9)
    x = np.concatenate([[0.0], np.cumsum(gap)])[:n].astype(np.float32) if n < 4000 else None
    if x is None:  # folded into rows 3 apart, so that FP32 keeps the gaps
        row, col = np.arange(n) // 99, np.arange(n) % 99
        x = (np.concatenate([[0.0], np.cumsum(np.where(np.arange(98) % 3 == 2, 1.2, 0.9))])[col]).astype(np.float32)
        y, touch = (3.0 * row).astype(np.float32), (col[:-1] % 3 != 2) & (col[1:] > 0)
    else:
        y, touch = np.zeros(n, np.float32), np.arange(n - 1) % 3 != 2
    want = np.flatnonzero(touch)
    want = (want.astype(np.uint64) << np.uint64(32)) | (want + 1).astype(np.uint64)
    dev = [torch.tensor(a, device="cuda") for a in (x, y, np.zeros(n, np.float32), np.full(n, 0.5, np.float32))]
    keys = torch.full((n + 1,), -1, dtype=torch.int64, device="cuda")
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert tds.lib().tds_find_pair_contacts_noalloc(*[p(t) for t in dev], n, 0, p(keys), n, p(count), st) == 0
    m = int(count.item())
    got = keys.cpu().numpy().view(np.uint64)
    assert m == len(want)
    assert np.array_equal(np.sort(got[:m]), want)
    assert (got[m:] == np.uint64(0xFFFFFFFFFFFFFFFF)).all()
