// tds_rules.cuh -- rules on sizes and records shared by host and device code,
// in plain C++ that a host compiler takes as well (the tests call them there).
#pragma once
#include <cfloat>
#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define TDS_HD __host__ __device__ __forceinline__
#else
#define TDS_HD inline
#endif

// Cells of one size that cover an extent along one axis, or -1 for more than
// max_cells (decided before the conversion to an integer, which a far particle
// would overflow). None for an extent that is no number: no particle has a
// position there, or cell and extent are both infinite.
TDS_HD int cells_along(float extent, float cell, uint32_t max_cells) {
  const float c = ceilf(extent / cell);
  if (!(c > 0.f)) return 0;
  return c <= (float)max_cells ? (int)c : -1;
}

// The next cell size to try: 1.25 times as wide. (Every step grows: from the
// smallest normal number on, infinity is reached within 800 steps.)
TDS_HD float coarser(float cell) { return fmaxf(1.25f * cell, FLT_MIN); }

// The grid of at most max_cells cells (max_cells <= 2^20, so that the product
// of three axes fits 64 bits) over an extent, in the narrowest cells of the
// sequence cell, 1.25 cell, ... that allow it. Returns the cell size; at the
// latest infinite cells, one along each axis, fit.
TDS_HD float grid_plan(const float extent[3], float cell, uint32_t max_cells, int dims[3]) {
  if (!(cell > 0.f)) cell = 1.f;
  for (;; cell = coarser(cell)) {
    uint64_t total = 1;
    bool fits = true;
    for (int a = 0; a < 3; ++a) {
      const int c = cells_along(extent[a], cell, max_cells);
      fits &= c >= 0;
      dims[a] = c + 1;
      total *= (uint64_t)dims[a];
    }
    if (fits && total <= max_cells) return cell;
  }
}

// The check word of a solver record, four 64-bit words that each move whole:
// (v.x, v.y), (v.z, version), (w.x, w.y), (w.z, check). The second carries its
// version itself; check ties the other three to it: the version and what the
// first and third hold, each word rotated by its own amount, so that changes
// of several words by the same bits (equal components, a version and a
// velocity that both change in their last bit) do not cancel, as they would
// in a plain exclusive or. (The amounts differ by no multiple of 8: the
// rotations of equal words by 0, 8, 16 and 24 cancel for one word in 256.)
TDS_HD uint32_t rotl(uint32_t x, int r) { return (x << r) | (x >> (32 - r)); }
TDS_HD uint32_t check_of_version(uint32_t version) { return rotl(version, 22) ^ 0x5bd1e995u; }
TDS_HD uint32_t record_check(uint32_t of_version, uint32_t vx, uint32_t vy, uint32_t wx, uint32_t wy) {
  return of_version ^ vx ^ rotl(vy, 5) ^ rotl(wx, 10) ^ rotl(wy, 15);
}
