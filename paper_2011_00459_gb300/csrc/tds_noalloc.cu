// tds_noalloc.cu -- tds_find_pair_contacts_noalloc: the particle-pair contact
// search of tds_step (sorted-cell broadphase + the bit-exact FP32 pair
// predicate) as a standalone call that allocates no memory.
//
// Some callers cannot let a library allocate device memory: a simulator
// stepping inside a fixed-rate real-time loop, where cudaMalloc/cudaFree may
// synchronize the device and stall the frame, or a host application whose
// device memory is entirely owned by its own pool allocator with a fixed
// budget. This call takes the caller's input and output buffers and keeps all
// of its intermediate arrays in one file-scope __device__ array of fixed size
// (below), which every GPU that loads the library holds until the process
// exits.
//
// Properties of the shared scratch array:
//  * Host code cannot use the array's name as a device address; the first call
//    on each device looks the address up with cudaGetSymbolAddress (with that
//    device current) and caches it. That first call should therefore come
//    before any stream capture.
//  * Every call reuses the same array and leaves its contents behind; what must
//    start at zero (the cell counters) is cleared by each call on its stream.
//  * Calls whose GPU work overlaps (on different streams, or from different
//    host threads) race on the array; serialize them on one stream.
//  * The cached address belongs to the device's primary context: after the
//    caller resets the device (cudaDeviceReset), it is stale.
//  * The order of the output keys depends only on the input: every cell's
//    particles are sorted by index, whatever its size.
#include <mutex>
#include <string>

#include "tds_internal.cuh"
#include "tds_rules.cuh"

namespace {

constexpr uint32_t kMaxN = TDS_NOALLOC_MAX_PARTICLES;
constexpr uint32_t kMaxCells = 262144u;

constexpr size_t align64(size_t w) { return (w + 63) & ~(size_t)63; }  // 256-byte regions
constexpr size_t kPlan = 0, kBounds = 16, kFinished = 24, kNBig = 25;  // (zeroed with the cell counts)
constexpr size_t kCellCount = kPlan + 64;
constexpr size_t kCellStart = kCellCount + align64(kMaxCells + 1);
constexpr size_t kPlace = kCellStart + align64(kMaxCells + 1);
constexpr size_t kCellOf = kPlace + align64(kMaxN);
constexpr size_t kPerm = kCellOf + align64(kMaxN);
constexpr size_t kSPos = kPerm + align64(kMaxN);
constexpr size_t kSId = kSPos + align64(4 * (size_t)kMaxN);
constexpr size_t kCnt = kSId + align64(kMaxN);
constexpr size_t kCStart = kCnt + align64(kMaxN + 1);
constexpr size_t kTmp = kCStart + align64(kMaxN + 1);
constexpr size_t kTotalWords = kTmp + align64(kMaxCells / 2048 + 64);

// The scratch array (about 5.3 MB).
static __device__ __align__(256) uint32_t g_noalloc_scratch[kTotalWords];

struct Plan {
  float lo[3];
  float inv;
  int gnx, gny, gnz;
  int cohesive;
};

struct View {
  uint32_t *base;
  __device__ Plan *plan() const { return reinterpret_cast<Plan *>(base + kPlan); }
  __device__ uint32_t *cell_count() const { return base + kCellCount; }
  __device__ uint32_t *cell_start() const { return base + kCellStart; }
  __device__ uint32_t *bounds() const { return base + kBounds; }
  __device__ uint32_t *finished() const { return base + kFinished; }
  __device__ uint32_t *nbig() const { return base + kNBig; }
  __device__ uint32_t *big() const { return base + kCnt; }  // (before the counts are written)
  __device__ uint32_t *place() const { return base + kPlace; }
  __device__ uint32_t *cell_of() const { return base + kCellOf; }
  __device__ uint32_t *perm() const { return base + kPerm; }
  __device__ float4 *spos() const { return reinterpret_cast<float4 *>(base + kSPos); }
  __device__ uint32_t *sid() const { return base + kSId; }
  __device__ uint32_t *cnt() const { return base + kCnt; }
  __device__ uint32_t *cstart() const { return base + kCStart; }
};

// Same FP32 pair predicate as the step (explicit round-to-nearest, this
// association, strict comparison).
__device__ __forceinline__ bool touch(float4 A, float4 B, int cohesive) {
  float dx = __fsub_rn(B.x, A.x), dy = __fsub_rn(B.y, A.y), dz = __fsub_rn(B.z, A.z);
  float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
  float rs = __fadd_rn(A.w, B.w);
  float R = cohesive ? __fadd_rn(rs, __fmul_rn(0.025f, rs)) : rs;
  return d2 < __fmul_rn(R, R);
}

__device__ __forceinline__ int axis_cell(float x, float x0, float inv, int n) {
  float t = floorf((x - x0) * inv);
  if (!(t >= 0.0f)) return 0;
  if (t >= (float)(n - 1)) return n - 1;
  return (int)t;
}

// Floats as unsigned numbers of the same order (every number's above 0, so
// that zeroed memory is below all of them).
__device__ __forceinline__ uint32_t ordered(float f) {
  const uint32_t u = __float_as_uint(f);
  return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float unordered(uint32_t u) {
  return __uint_as_float(u & 0x80000000u ? u & 0x7FFFFFFFu : ~u);
}

// Bounding box and largest radius, and a grid of at most kMaxCells cells, each
// wider than any contact reach. Every block reduces its share; the last one to
// finish makes the plan (one block for all of it took 27 us at 40 000
// particles, latency of its serial loads; 152 blocks 6).
__global__ void __launch_bounds__(256) k_plan(View v, const float *x, const float *y, const float *z, const float *r,
                                              uint32_t n, int cohesive) {
  __shared__ uint32_t sh[7];
  __shared__ bool last;
  if (threadIdx.x < 7) sh[threadIdx.x] = 0u;
  __syncthreads();
  // largest of -x, -y, -z, x, y, z, r (fmaxf passes over NaN)
  float m[7] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY, -INFINITY, -INFINITY, 0.f};
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float p[3] = {x[i], y[i], z[i]};
    for (int a = 0; a < 3; ++a) { m[a] = fmaxf(m[a], -p[a]); m[3 + a] = fmaxf(m[3 + a], p[a]); }
    m[6] = fmaxf(m[6], r[i]);
  }
  for (int q = 0; q < 7; ++q) {
    const uint32_t t = __reduce_max_sync(0xffffffffu, ordered(m[q]));
    if ((threadIdx.x & 31) == 0) atomicMax(sh + q, t);
  }
  __syncthreads();
  if (threadIdx.x < 7) atomicMax(v.bounds() + threadIdx.x, sh[threadIdx.x]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(v.finished(), 1u) == gridDim.x - 1;
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    for (int q = 0; q < 7; ++q) m[q] = unordered(*(volatile uint32_t *)(v.bounds() + q));
    for (int a = 0; a < 3; ++a) m[a] = -m[a];
    const float extent[3] = {m[3] - m[0], m[4] - m[1], m[5] - m[2]};
    int dims[3];
    const float cell = grid_plan(extent, 2.0f * m[6] * 1.025f * 1.02f, kMaxCells, dims);
    Plan *P = v.plan();
    for (int a = 0; a < 3; ++a) P->lo[a] = m[a];
    P->inv = 1.0f / cell;
    P->gnx = dims[0]; P->gny = dims[1]; P->gnz = dims[2];
    P->cohesive = cohesive;
  }
}

__global__ void k_cells(View v, const float *x, const float *y, const float *z, uint32_t n) {
  const Plan P = *v.plan();
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int cx = axis_cell(x[i], P.lo[0], P.inv, P.gnx);
    int cy = axis_cell(y[i], P.lo[1], P.inv, P.gny);
    int cz = axis_cell(z[i], P.lo[2], P.inv, P.gnz);
    uint32_t c = ((uint32_t)cz * P.gny + cy) * P.gnx + cx;
    v.cell_of()[i] = c;
    v.place()[i] = atomicAdd(v.cell_count() + c, 1u);  // its place in the cell, for now in any order
  }
}

__global__ void k_scatter(View v, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    v.perm()[v.cell_start()[v.cell_of()[i]] + v.place()[i]] = i;
}

// Reproducible order inside each cell, whatever the order of the atomic
// scatter: ascending particle index. In cells of up to kSmallCell particles
// each particle counts the smaller indexes of its cell and goes straight to
// its place; larger cells are listed for k_cell_sort_big.
constexpr uint32_t kSmallCell = 64;

__device__ __forceinline__ void put(View v, uint32_t j, uint32_t i, const float *x, const float *y, const float *z,
                                    const float *r) {
  v.spos()[j] = make_float4(x[i], y[i], z[i], r[i]);
  v.sid()[j] = i;
}

__global__ void k_place(View v, const float *x, const float *y, const float *z, const float *r, uint32_t n) {
  const uint32_t *perm = v.perm();
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    const uint32_t i = perm[j], c = v.cell_of()[i];
    const uint32_t s = v.cell_start()[c], e = v.cell_start()[c + 1];
    if (e - s > kSmallCell) {
      if (j == s) v.big()[atomicAdd(v.nbig(), 1u)] = c;
      continue;
    }
    uint32_t at = s;
    for (uint32_t k = s; k < e; ++k) at += perm[k] < i;
    put(v, at, i, x, y, z, r);
  }
}

// Cells with more than kSmallCell particles (a grid that k_plan coarsened
// because of a far outlier puts thousands of particles in one cell): one
// block per listed cell sorts its m entries in place with a bitonic network in the
// form whose every comparator puts the smaller value at the lower index
// (each merge stage starts by comparing mirrored positions of its blocks,
// then halves). Comparators that reach past m are skipped, which is the same
// as padding the sequence to a power of two with values larger than any
// index. (Walking all cells to find the large ones took 76 us at 40 000
// particles, which have none; the list 2.)
__global__ void __launch_bounds__(1024) k_cell_sort_big(View v, const float *x, const float *y, const float *z,
                                                        const float *r) {
  uint32_t *perm = v.perm();
  const uint32_t nbig = *v.nbig();
  for (uint32_t q = blockIdx.x; q < nbig; q += gridDim.x) {
    const uint32_t c = v.big()[q];
    const uint32_t s = v.cell_start()[c], e = v.cell_start()[c + 1];
    const uint32_t m = e - s;
    uint32_t *a = perm + s;
    uint32_t pow2 = 1;
    while (pow2 < m) pow2 <<= 1;
    const uint32_t half = pow2 >> 1;
    for (uint32_t k = 2; k <= pow2; k <<= 1) {
      const uint32_t hk = k >> 1;
      for (uint32_t t = threadIdx.x; t < half; t += blockDim.x) {  // mirrored pairs of each k-block
        const uint32_t blk = t / hk, o = t % hk;
        const uint32_t i = blk * k + o, j = blk * k + (k - 1u - o);
        if (j < m) {
          const uint32_t ai = a[i], aj = a[j];
          if (ai > aj) { a[i] = aj; a[j] = ai; }
        }
      }
      __syncthreads();
      for (uint32_t d = k >> 2; d > 0; d >>= 1) {  // half-cleaners at distance d
        for (uint32_t t = threadIdx.x; t < half; t += blockDim.x) {
          const uint32_t i = (t / d) * 2u * d + (t % d), j = i + d;
          if (j < m) {
            const uint32_t ai = a[i], aj = a[j];
            if (ai > aj) { a[i] = aj; a[j] = ai; }
          }
        }
        __syncthreads();
      }
    }
    for (uint32_t t = threadIdx.x; t < m; t += blockDim.x) put(v, s + t, a[t], x, y, z, r);
    __syncthreads();
  }
}

// Nine lanes a particle, one for each row of three cells around it (27 lanes
// of a warp: three particles): a row's candidates are contiguous and its pairs
// precede the next row's. One thread for all nine rows left the GPU waiting on
// a chain of loads: 20 us to count and 27 to write at 40 000 particles, against
// 12.7 and 17.4.
// Where there are cells of more than kSmallCell particles (coarsened by a far
// particle or one large radius), rows of more than kLaneRow candidates are
// taken by the whole warp, 32 candidates at a time, one row after another: with
// all particles in one cell a lane's row holds all of them and the other eight
// none. 40 001 particles and an outlier, the whole call: 7.1 ms, by lanes alone
// 31.6, by a thread a particle 11.3; an outlier along one axis, 10 km away: 1.3,
// 4.4 and 3.6. (At 128 candidates the 27 rows of a warp take about as many turns
// either way.)
constexpr uint32_t kLaneRow = 128;

struct WideRow {  // the row of the lowest lane in m, known to all lanes
  uint32_t owner, me, s, e;
  float4 A;
  __device__ __forceinline__ WideRow(unsigned m, float4 a, uint32_t id, uint32_t first, uint32_t end) {
    owner = (uint32_t)__ffs(m) - 1u;
    me = __shfl_sync(0xffffffffu, id, owner);
    s = __shfl_sync(0xffffffffu, first, owner);
    e = __shfl_sync(0xffffffffu, end, owner);
    A = make_float4(__shfl_sync(0xffffffffu, a.x, owner), __shfl_sync(0xffffffffu, a.y, owner),
                    __shfl_sync(0xffffffffu, a.z, owner), __shfl_sync(0xffffffffu, a.w, owner));
  }
  // the lanes whose candidate k is a pair of the row's particle
  __device__ __forceinline__ unsigned hits(uint32_t k, const float4 *sp, const uint32_t *sid, int cohesive) const {
    return __ballot_sync(0xffffffffu, k < e && sid[k] > me && touch(A, sp[k], cohesive));
  }
};

template <bool kWrite, bool kCrowded>
__device__ __forceinline__ void pairs(View v, const Plan P, uint32_t n, unsigned long long *keys, uint32_t cap,
                                      uint32_t *count_out) {
  const float4 *sp = v.spos();
  const uint32_t *sid = v.sid();
  if (kWrite && blockIdx.x == 0 && threadIdx.x == 0) *count_out = v.cstart()[n];
  const uint32_t lane = threadIdx.x & 31u, who = lane / 9u, row = lane % 9u;
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  for (uint32_t j0 = 3u * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); j0 < n; j0 += 3u * warps) {
    const uint32_t j = j0 + who;
    const bool on = who < 3u && j < n;
    uint32_t s = 0, e = 0, me = 0, hits = 0, found = 0;
    float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
    if (on) {
      A = sp[j];
      me = sid[j];
      const int cx = axis_cell(A.x, P.lo[0], P.inv, P.gnx);
      const int cy = axis_cell(A.y, P.lo[1], P.inv, P.gny) + (int)(row % 3u) - 1;
      const int cz = axis_cell(A.z, P.lo[2], P.inv, P.gnz) + (int)(row / 3u) - 1;
      if (cy >= 0 && cy < P.gny && cz >= 0 && cz < P.gnz) {
        const uint32_t first = ((uint32_t)cz * P.gny + cy) * P.gnx;
        s = v.cell_start()[first + max(cx - 1, 0)];
        e = v.cell_start()[first + min(cx + 1, P.gnx - 1) + 1];
      }
    }
    const uint32_t own = kCrowded && e - s > kLaneRow ? s : e;  // where the candidates the lane takes by itself end
    for (uint32_t k = s; k < own; ++k)
      if (sid[k] > me && touch(A, sp[k], P.cohesive)) {
        ++found;
        if (k - s < 32u) hits |= 1u << (k - s);
      }
    for (unsigned m = kCrowded ? __ballot_sync(0xffffffffu, own != e) : 0u; m; m &= m - 1u) {
      const WideRow r(m, A, me, s, e);
      uint32_t f = 0;
      for (uint32_t k0 = r.s; k0 < r.e; k0 += 32u) f += __popc(r.hits(k0 + lane, sp, sid, P.cohesive));
      if (lane == r.owner) found = f;
    }
    uint32_t before = 0, all = 0;  // pairs of the particle's earlier rows, of all
    for (uint32_t q = 0; q < 9u; ++q) {
      const uint32_t f = __shfl_sync(0xffffffffu, found, min(9u * who + q, 31u));
      if (q < row) before += f;
      all += f;
    }
    if (!kWrite) {
      if (on && row == 0u) v.cnt()[j] = all;
      continue;
    }
    uint32_t out = found ? v.cstart()[j] + before : 0u;
    for (unsigned m = kCrowded ? __ballot_sync(0xffffffffu, own != e) : 0u; m; m &= m - 1u) {
      const WideRow r(m, A, me, s, e);
      uint32_t at = __shfl_sync(0xffffffffu, out, r.owner);
      if (!__shfl_sync(0xffffffffu, found, r.owner)) continue;
      for (uint32_t k0 = r.s; k0 < r.e; k0 += 32u) {
        const unsigned h = r.hits(k0 + lane, sp, sid, P.cohesive);
        const uint32_t mine = at + __popc(h & ((1u << lane) - 1u));
        if ((h >> lane) & 1u && mine < cap) keys[mine] = ((unsigned long long)r.me << 32) | sid[k0 + lane];
        at += __popc(h);
      }
    }
    if (found)
      for (uint32_t k = s; k < own; ++k) {
        if (k - s < 32u ? !((hits >> (k - s)) & 1u) : (sid[k] <= me || !touch(A, sp[k], P.cohesive))) continue;
        if (out < cap) keys[out] = ((unsigned long long)me << 32) | sid[k];
        ++out;
      }
  }
}

// (16 blocks an SM: 32 registers, as many as the usual path needs)
template <bool kWrite>
__global__ void __launch_bounds__(128, 16) k_pairs(View v, uint32_t n, unsigned long long *keys, uint32_t cap,
                                                   uint32_t *count_out) {
  const Plan P = *v.plan();
  if (*v.nbig() == 0u) pairs<kWrite, false>(v, P, n, keys, cap, count_out);
  else pairs<kWrite, true>(v, P, n, keys, cap, count_out);
}

std::mutex g_mu;
uint32_t *g_base[256];  // device address of the scratch array, per device ordinal

}  // namespace

tds_status tds_set_error_message(tds_status s, const char *msg);  // tds_api.cu

extern "C" tds_status tds_find_pair_contacts_noalloc(const float *x, const float *y, const float *z,
                                                     const float *radius, uint32_t n, int32_t cohesive,
                                                     uint64_t *keys, uint32_t cap, uint32_t *count,
                                                     void *stream) {
  if (!x || !y || !z || !radius || !keys || !count)
    return tds_set_error_message(TDS_ERR_INVALID_ARG, "tds_find_pair_contacts_noalloc: NULL pointer");
  if (n == 0)
    return tds_set_error_message(TDS_ERR_INVALID_ARG, "tds_find_pair_contacts_noalloc: n must be >= 1");
  if (n > kMaxN)
    return tds_set_error_message(TDS_ERR_CAPACITY,
                                 "tds_find_pair_contacts_noalloc: n exceeds TDS_NOALLOC_MAX_PARTICLES (65536)");
  // an error left pending by an earlier call of the caller is reported, and
  // left pending, rather than blamed on this call's launches
  cudaError_t e = cudaPeekAtLastError();
  if (e != cudaSuccess)
    return tds_set_error_message(TDS_ERR_CUDA, (std::string("tds_find_pair_contacts_noalloc: a CUDA error of an "
                                                            "earlier call is pending: ") +
                                                    cudaGetErrorString(e)).c_str());
  int dev = 0;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 256)
    return tds_set_error_message(TDS_ERR_CUDA, "tds_find_pair_contacts_noalloc: cudaGetDevice failed");
  uint32_t *base;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_base[dev]) {
      void *p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p)
        return tds_set_error_message(TDS_ERR_CUDA,
                                     "tds_find_pair_contacts_noalloc: cudaGetSymbolAddress failed");
      g_base[dev] = static_cast<uint32_t *>(p);
    }
    base = g_base[dev];
  }
  cudaStream_t st = (cudaStream_t)stream;
  View v{base};
  const unsigned grid = (n + 255) / 256;
  e = cudaMemsetAsync(base, 0, sizeof(uint32_t) * (kCellCount + kMaxCells + 1), st);
  if (e != cudaSuccess)
    return tds_set_error_message(TDS_ERR_CUDA, (std::string("tds_find_pair_contacts_noalloc: cudaMemsetAsync: ") +
                                                    cudaGetErrorString(e)).c_str());
  const unsigned pair_blocks = (n + 11) / 12;  // three particles a warp, four warps a block
  k_plan<<<grid < 152 ? grid : 152, 256, 0, st>>>(v, x, y, z, radius, n, cohesive ? 1 : 0);
  k_cells<<<grid, 256, 0, st>>>(v, x, y, z, n);
  tds_scan_exclusive(base + kCellCount, base + kCellStart, kMaxCells, base + kTmp, st);
  k_scatter<<<grid, 256, 0, st>>>(v, n);
  k_place<<<grid, 256, 0, st>>>(v, x, y, z, radius, n);
  k_cell_sort_big<<<128, 1024, 0, st>>>(v, x, y, z, radius);
  k_pairs<false><<<pair_blocks, 128, 0, st>>>(v, n, nullptr, 0, nullptr);
  tds_scan_exclusive(base + kCnt, base + kCStart, n, base + kTmp, st);
  k_pairs<true><<<pair_blocks, 128, 0, st>>>(v, n, reinterpret_cast<unsigned long long *>(keys), cap, count);
  // the launches above are the only work since the pending-error check on
  // entry, so an error now is theirs
  e = cudaGetLastError();
  if (e != cudaSuccess)
    return tds_set_error_message(TDS_ERR_CUDA, (std::string("tds_find_pair_contacts_noalloc: launch: ") +
                                                    cudaGetErrorString(e)).c_str());
  return TDS_OK;
}
