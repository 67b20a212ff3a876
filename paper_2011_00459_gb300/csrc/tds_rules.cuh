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

// Warps of a solver CTA: about one for every row tile of a bed of n particles
// (4 contacts a particle, and a tile begun for each of 64 buckets), at most the
// shape's. A warp beyond the tiles would only hold registers, which several
// small scenes on their own streams can share: a round of steps of 16 scenes of
// 2000 spheres, 50 sweeps, takes 1.95 ms, with 16 warps in every CTA 7.98; of 8000
// spheres 5.9 and 10.3; one scene's step is as fast either way. In a batch every
// CTA also adds up every scene's residual, a warp each, so there also a warp for
// eight scenes (1000 beds of 4 spheres, 100 sweeps, a check each: 56 ms, with one
// warp 75).
TDS_HD int solver_warps(uint32_t n, uint32_t scenes, int blocks, int most) {
  const uint32_t tiles = (n / 8u + 64u + (uint32_t)blocks - 1u) / (uint32_t)blocks;
  const uint32_t want = (scenes + 7u) / 8u > tiles ? (scenes + 7u) / 8u : tiles;
  return want < (uint32_t)most ? (int)want : most;
}

// Whether the Gaussian fields' gather takes less time than the scatter, for a
// grid of so many voxels, a smoothing length of q voxels and a scene of so many
// particles. Measured for 300 to 1M particles, 1e-4 to 10 voxels a particle and
// q from 0.2 to 6, 879 pairs of times: the choice takes 1.007 times the better
// one's time on average, and at most 1.15 times the scatter's. (The line
// before, 3.5 q voxels a particle alone: 1.13 and 6.2.)
//  - The gather looks at every row in reach of every voxel (some q^2), the
//    scatter at every voxel in reach of every particle (some q^3). 200k particles:
//    q = 1/2, 73k voxels 91 and 105 us, 158k 121 and 103; q = 1, 158k 281 and
//    582, 480k 611 and 574; q = 3, 1.8M 11.0 and 12.7 ms. Up to some 30 000 q
//    voxels (q^1.5 from one voxel on) the gather is all launches and latency
//    (20k particles, q = 1/2, 22k voxels: 42 and 47 us).
//  - On a few voxels the scatter's reductions meet at few addresses, but the
//    gather has few warps, each with all particles to walk: 20k particles,
//    q = 0.4, 120 voxels 318 and 251 us, 280 voxels 111 and 152; q = 0.6, 64
//    voxels 668 and 1202.
//  - With q <= 0.3 a particle reaches about three voxels, for which the gather
//    walks up to 27: 200k particles, 34k voxels 58 and 46 us.
TDS_HD bool gather_pays(double voxels, double q, double particles) {
  return q > 0.31 && voxels * q * q * q * q >= 3.0 + 1e-5 * particles &&
         voxels <= fmin(1.8 * q * q, 3.5 * q) * particles + 30000.0 * q * fmax(1.0, sqrt(q));
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
