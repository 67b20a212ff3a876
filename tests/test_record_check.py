"""The check word of the solver's versioned records, four 64-bit words (v.x,
v.y), (v.z, version), (w.x, w.y), (w.z, check): no mixture of the words of two
versions may pass for a whole record. Updates as they occur: late in a solve a
few components change by one unit in the last place, on symmetric paths several
components are equal, versions count up by one."""
import ctypes

import numpy as np
import pytest

from tests.native_rules import compile_rules

U = ctypes.c_uint32


@pytest.fixture(scope="module")
def mixtures(tmp_path_factory):
    """Mixtures of record a (the older) and b that pass for a version, of all 2^4 choices of 64-bit words, without
    those that are a or b."""
    L = compile_rules(tmp_path_factory.mktemp("check"), """
#include <string.h>
static uint32_t check(const uint32_t *q) { return record_check(check_of_version(q[3]), q[0], q[1], q[4], q[5]); }
extern "C" uint32_t mixtures(const uint32_t *a, const uint32_t *b, uint32_t count) {
  uint32_t passed = 0;
  for (uint32_t i = 0; i < count; ++i, a += 7, b += 7) {
    uint32_t A[8], B[8];
    memcpy(A, a, 28);
    memcpy(B, b, 28);
    A[7] = check(a);
    B[7] = check(b);
    for (uint32_t m = 0; m < 16u; ++m) {
      uint32_t q[8];
      for (int k = 0; k < 8; ++k) q[k] = (m >> (k / 2)) & 1u ? B[k] : A[k];
      if (memcmp(q, A, 32) && memcmp(q, B, 32)) passed += q[7] == check(q);
    }
  }
  return passed;
}""")
    L.mixtures.restype = U
    L.mixtures.argtypes = [ctypes.c_void_p, ctypes.c_void_p, U]

    def call(a, b):
        a, b = np.ascontiguousarray(a, np.uint32), np.ascontiguousarray(b, np.uint32)
        return L.mixtures(a.ctypes.data, b.ctypes.data, len(a))

    return call


def records(n, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    a = g.normal(0, 1, (n, 7)).astype(np.float32).view(np.uint32)
    a[:, 3] = g.integers(0, 40000, n)
    return g, a


def test_last_place_updates(mixtures):
    """Every set of components moved by one unit in the last place, up or
    down, with the version."""
    g, a = records(64 * 300, 1)
    b = a.copy()
    sets = np.tile(np.arange(64), 300)
    for bit, word in enumerate((0, 1, 2, 4, 5, 6)):
        on = (sets >> bit) & 1 == 1
        b[on, word] += np.where(g.random(on.sum()) < 0.5, 1, 0xFFFFFFFF).astype(np.uint32)
    b[:, 3] += 1
    assert mixtures(a, b) == 0


def test_equal_components(mixtures):
    """Components that are equal before and after (symmetric paths)."""
    g, a = records(63 * 200, 2)
    b = records(63 * 200, 3)[1]
    sets = np.tile(np.arange(1, 64), 200)
    words = (0, 1, 2, 4, 5, 6)
    for bit, word in enumerate(words):
        on = (sets >> bit) & 1 == 1
        a[on, word], b[on, word] = a[on, 0], b[on, 0]
    b[:, 3] = a[:, 3] + 1
    assert mixtures(a, b) == 0


def test_a_single_word(mixtures):
    """One component set, cleared or negated, from rest (all words zero but the version)."""
    a = np.zeros((7 * 32, 7), np.uint32)
    b = a.copy()
    for k in range(7 * 32):
        b[k, k // 32] ^= np.uint32(1 << (k % 32))
        b[k, 3] += 1
    assert mixtures(a, b) == 0
    assert mixtures(b, a) == 0


def test_unrelated_updates(mixtures):
    """Any change at all: a mixture passes with a chance of 2^-32 (expected here: 0.0002)."""
    _, a = records(50000, 4)
    _, b = records(50000, 5)
    b[:, 3] = a[:, 3] + 1
    assert mixtures(a, b) == 0
