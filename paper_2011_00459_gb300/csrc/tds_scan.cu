// tds_scan.cu -- exclusive prefix sums of uint32 counts (cell occupancy,
// contacts per particle, incidences per particle, bucket histograms), built
// from warp-shuffle scans: up to kOneBlock elements by one block in one launch
// (launches bound it there: one instead of three, 3.9 us against 9.4 for 2001
// elements), more in two phases, tile sums and then a per-tile scan whose block
// adds up the tiles before its own itself (a separate scan of the tile sums is
// a launch and a pass of one block: 2.4 to 4 us more). Those sums are quadratic
// in the tiles, from L2: with the largest grid (2^26 cells, 32768 tiles) 2 GB,
// and still a step of 2000 spheres in it takes 0.75 ms against 1.48.
#include "tds_internal.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;  // 2048 elements per block
constexpr int kOneThreads = 1024;
constexpr uint32_t kOneBlock = 2 * kOneThreads * kItems;

__device__ __forceinline__ uint32_t warp_inclusive(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// Exclusive scan of one value per thread across a block of T threads; returns
// the block total through *total.
template <int T>
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t *total) {
  __shared__ uint32_t warp_sums[T / 32 + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = warp_inclusive(v);
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t s = lane < T / 32 ? warp_sums[lane] : 0u;
    uint32_t si = warp_inclusive(s);
    if (lane < T / 32) warp_sums[lane] = si - s;
    if (lane == T / 32 - 1) warp_sums[T / 32] = si;  // total
  }
  __syncthreads();
  uint32_t excl = inc - v + warp_sums[warp];
  *total = warp_sums[T / 32];
  __syncthreads();
  return excl;
}

// A thread's kItems consecutive elements, as 16-byte accesses where the
// pointer and the range allow it (0 past the end).
__device__ __forceinline__ void load_items(const uint32_t *in, size_t base, uint32_t m, bool vec, uint32_t (&v)[kItems]) {
  if (vec && base + kItems <= m) {
    const uint4 a = *reinterpret_cast<const uint4 *>(in + base), b = *reinterpret_cast<const uint4 *>(in + base + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < kItems; ++k) v[k] = base + k < m ? in[base + k] : 0u;
  }
}
// Their exclusive prefix sums, starting at run.
__device__ __forceinline__ void store_items(uint32_t *out, size_t base, uint32_t m, bool vec, const uint32_t (&v)[kItems],
                                            uint32_t run) {
  uint32_t p[kItems];
#pragma unroll
  for (int k = 0; k < kItems; ++k) {
    p[k] = run;
    run += v[k];
  }
  if (vec && base + kItems <= m) {
    *reinterpret_cast<uint4 *>(out + base) = make_uint4(p[0], p[1], p[2], p[3]);
    *reinterpret_cast<uint4 *>(out + base + 4) = make_uint4(p[4], p[5], p[6], p[7]);
  } else {
#pragma unroll
    for (int k = 0; k < kItems; ++k)
      if (base + k < m) out[base + k] = p[k];
  }
}
__device__ __forceinline__ uint32_t sum_items(const uint32_t (&v)[kItems]) {
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kItems; ++k) s += v[k];
  return s;
}

// (in and out may be the same array: no restrict)
// (m_dev, if not null: the length, known on the device only; m is then its bound)
__global__ void __launch_bounds__(kOneThreads) k_scan_one(const uint32_t *in, uint32_t m, const uint32_t *m_dev,
                                                          uint32_t *out, bool vec) {
  if (m_dev) m = min(m, *m_dev);
  uint32_t carry = 0;
  for (uint32_t start = 0; start < m; start += kOneThreads * kItems) {
    const size_t base = start + (size_t)threadIdx.x * kItems;
    uint32_t v[kItems], total;
    load_items(in, base, m, vec, v);
    const uint32_t run = block_exclusive<kOneThreads>(sum_items(v), &total) + carry;
    store_items(out, base, m, vec, v, run);
    carry += total;
  }
  if (threadIdx.x == 0) out[m] = carry;
}

__global__ void __launch_bounds__(kThreads) k_tile_sums(const uint32_t *__restrict__ in, uint32_t m,
                                                        const uint32_t *m_dev, bool vec, uint32_t *__restrict__ sums) {
  if (m_dev) m = min(m, *m_dev);
  if (blockIdx.x > 0 && (size_t)blockIdx.x * kTile >= m) return;
  uint32_t v[kItems], total;
  load_items(in, (size_t)blockIdx.x * kTile + threadIdx.x * kItems, m, vec, v);
  (void)block_exclusive<kThreads>(sum_items(v), &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kThreads) k_tile_scan(const uint32_t *in, uint32_t m, const uint32_t *m_dev, bool vec,
                                                        const uint32_t *sums, uint32_t *out) {
  if (m_dev) m = min(m, *m_dev);
  if (blockIdx.x > 0 && (size_t)blockIdx.x * kTile >= m) return;
  const size_t base = (size_t)blockIdx.x * kTile + threadIdx.x * kItems;
  uint32_t v[kItems], before, total, mine = 0;
  load_items(in, base, m, vec, v);
  for (uint32_t t = threadIdx.x; t < blockIdx.x; t += kThreads) mine += __ldg(sums + t);  // the tiles before this one
  (void)block_exclusive<kThreads>(mine, &before);
  const uint32_t run = block_exclusive<kThreads>(sum_items(v), &total) + before;
  store_items(out, base, m, vec, v, run);
  if ((size_t)(blockIdx.x + 1) * kTile >= m && threadIdx.x == 0) out[m] = before + total;  // the last tile
}

}  // namespace

size_t tds_scan_tmp_words(uint32_t m) { return (size_t)(m + kTile - 1) / kTile + 2; }

// out[0..m] = exclusive prefix sums of in[0..m), out[m] = total. In-place
// (in == out) is allowed. tmp holds tds_scan_tmp_words(m) words.
// Returns the kernels launched.
// With m_dev, the length is *m_dev (at most m) and known on the device only.
int tds_scan_exclusive(const uint32_t *in, uint32_t *out, uint32_t m, uint32_t *tmp, cudaStream_t st,
                       const uint32_t *m_dev) {
  const bool vec = (((uintptr_t)in | (uintptr_t)out) & 15u) == 0u;
  if (m <= kOneBlock) {
    k_scan_one<<<1, kOneThreads, 0, st>>>(in, m, m_dev, out, vec);
    return 1;
  }
  const uint32_t ntiles = (m + kTile - 1) / kTile;
  k_tile_sums<<<ntiles, kThreads, 0, st>>>(in, m, m_dev, vec, tmp);
  k_tile_scan<<<ntiles, kThreads, 0, st>>>(in, m, m_dev, vec, tmp, out);
  return 2;
}
