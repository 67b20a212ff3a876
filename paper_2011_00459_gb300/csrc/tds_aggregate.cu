// tds_aggregate.cu -- aggregate bodies of active zones (section "Macroscale
// model", Eqs. aggregate_mass to aggregate_rot_vel): per zone the mass,
// centre of mass, velocity, inertia tensor about the centre of mass and the
// angular velocity I^+ L of the particles it contains. Two passes, as in the
// definition: (1) membership, M, sum m x, sum m v; (2) the second moments and
// angular momentum about the centre of mass. FP64 accumulation in
// registers (see LaneSums). What bounds the passes: FP64 issue (13 and 19
// operations a particle; an FP64 instruction takes 16 cycles of an SM). 1M
// particles, 8 zones: 39 and 44 us; with FP64 divisions, conversions and five
// shuffle steps and additions per component and 32 particles 146 and 185.
// k_agg_final 6.4 us against 24.
#include <cfloat>
#include <cstring>

#include "tds_internal.cuh"

namespace {

struct ZoneTable {  // the zones as a kernel argument
  tds_zone z[TDS_MAX_ZONES];
};

constexpr int kAggThreads = 256;
constexpr int kFirst = 8;   // m, m x (3), m v (3), count
constexpr int kSecond = 9;  // m dx dx^T (6: xx yy zz xy xz yz), m dx x v (3)

// First zone of the particle's scene containing p (-1: none); the FP32
// half-space test in the documented operation order.
__device__ __forceinline__ int zone_of(const tds_zone *zones, uint32_t nz, uint32_t sid, float4 p) {
  for (uint32_t z = 0; z < nz; ++z) {
    const tds_zone &Z = zones[z];
    if (Z.scene != sid) continue;
    bool in = true;
    for (uint32_t k = 0; k < Z.n_planes && in; ++k) {
      const float *q = Z.planes[k];
      const float s = __fadd_rn(__fadd_rn(__fmul_rn(q[0], p.x), __fmul_rn(q[1], p.y)), __fmul_rn(q[2], p.z));
      in = s <= q[3];
    }
    if (in) return (int)z;
  }
  return -1;
}

// An FP32 number as FP64, exactly, by integer operations: the conversion
// instruction takes an FP64 issue slot, worth 64 integer ones here. Zeros and
// denormals are scaled up first; infinities and NaN keep their exponent.
__device__ __forceinline__ double widen(float x) {
  const bool tiny = (__float_as_uint(x) & 0x7F800000u) == 0u;
  const uint32_t u = __float_as_uint(tiny ? __fmul_rn(x, 18446744073709551616.0f) : x);  // 2^64
  const uint32_t mag = u & 0x7FFFFFFFu;
  uint32_t hi = (mag >> 3) + (tiny ? (896u - 64u) << 20 : 896u << 20);
  if (mag == 0u) hi = 0u;
  if (mag >= 0x7F800000u) hi = 0x7FF00000u | ((mag & 0x7FFFFFu) >> 3);
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}

// Mass of a particle: the reciprocal of the FP32 record's 1/m. FP64 division
// costs about twenty FP64 operations, which this GPU issues at a sixty-fourth
// of the FP32 rate; Newton's iteration r <- r + r (1 - a r) doubles the correct
// digits of the FP32 reciprocal, to 2^-46 and then to the last bit. Where that
// reciprocal is no normal number (masses beyond FP32's range, an infinite or a
// zero one) the iteration has nothing to start from, and the division is taken.
__device__ __forceinline__ double mass_of(float inv_m) {
  const double a = widen(inv_m);
  const float start = __frcp_rn(inv_m);
  if (!(start >= FLT_MIN && start <= FLT_MAX)) return 1.0 / a;
  double r = widen(start);
  r = fma(r, fma(-a, r, 1.0), r);
  return fma(r, fma(-a, r, 1.0), r);
}

// Sums of K components per zone. Each warp walks its own contiguous stretch of
// slots, 32 consecutive particles per iteration (coalesced); each lane keeps
// the running sums of the zone of its last particle in registers and flushes
// them into shared memory when its zone changes (rarely: slot order is
// spatial). At the end of the stretch the lanes of one zone are added by
// shuffles first.
template <int K>
struct LaneSums {
  int cur = -1;
  double acc[K] = {};
  __device__ __forceinline__ void flush(double *sh) {
#pragma unroll
    for (int c = 0; c < K; ++c) {
      if (cur >= 0 && acc[c] != 0.0) atomicAdd(sh + cur * K + c, acc[c]);
      acc[c] = 0.0;
    }
  }
  // makes z (>= 0) the zone the sums belong to
  __device__ __forceinline__ void enter(double *sh, int z) {
    if (z != cur) {
      flush(sh);
      cur = z;
    }
  }
  __device__ __forceinline__ void finish(double *sh) {
    const unsigned full = 0xffffffffu;
    __syncwarp();
    const int z = __reduce_max_sync(full, cur);
    if (!__all_sync(full, cur == z || cur < 0)) {
      flush(sh);
      return;
    }
    // eight components: each exchange halves the components a lane holds (9
    // additions instead of 40); the lane's bits
    // 4, 3, 2 say which it ends with
    const unsigned lane = threadIdx.x & 31u;
#pragma unroll
    for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1) {
      const bool up = lane & (unsigned)o;
#pragma unroll
      for (int c = 0; c < h; ++c) {
        const double keep = up ? acc[c + h] : acc[c], send = up ? acc[c] : acc[c + h];
        acc[c] = keep + __shfl_xor_sync(full, send, o);
      }
    }
    acc[0] += __shfl_xor_sync(full, acc[0], 2);
    acc[0] += __shfl_xor_sync(full, acc[0], 1);
    const int c = (lane & 16u ? 4 : 0) + (lane & 8u ? 2 : 0) + (lane & 4u ? 1 : 0);
    if (z >= 0 && (lane & 3u) == 0u && acc[0] != 0.0) atomicAdd(sh + z * K + c, acc[0]);
#pragma unroll
    for (int q = 8; q < K; ++q) {
      double t = acc[q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(full, t, o);
      if (z >= 0 && lane == 0u && t != 0.0) atomicAdd(sh + z * K + q, t);
    }
  }
};

template <int K>
__device__ __forceinline__ void block_to_global(double *sh, double *sums, uint32_t nz) {
  __syncthreads();
  for (uint32_t q = threadIdx.x; q < nz * K; q += blockDim.x)
    if (sh[q] != 0.0) atomicAdd(sums + q, sh[q]);
}

// The stretch [lo, hi) of slots of this warp (a multiple of 32 long).
__device__ __forceinline__ void warp_stretch(uint32_t n, uint32_t &lo, uint32_t &hi) {
  const uint32_t nw = gridDim.x * (blockDim.x >> 5), w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  uint32_t per = (n + nw - 1) / nw;
  per = (per + 31u) & ~31u;
  lo = min(n, w * per);
  hi = min(n, lo + per);
}

__global__ void __launch_bounds__(kAggThreads) k_agg_first(DevPtrs d, uint32_t n,
                                                           const __grid_constant__ ZoneTable zones, uint32_t nz,
                                                           uint8_t *zone_id, double *mass, double *sums) {
  __shared__ tds_zone sz[TDS_MAX_ZONES];
  __shared__ double sh[TDS_MAX_ZONES * kFirst];
  for (uint32_t q = threadIdx.x; q < nz * sizeof(tds_zone) / 4; q += blockDim.x)
    reinterpret_cast<uint32_t *>(sz)[q] = reinterpret_cast<const uint32_t *>(zones.z)[q];
  for (uint32_t q = threadIdx.x; q < nz * kFirst; q += blockDim.x) sh[q] = 0.0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  uint32_t lo, hi;
  warp_stretch(n, lo, hi);
  LaneSums<kFirst> ls;
  for (uint32_t base = lo; base < hi; base += 32) {
    const uint32_t i = base + lane;
    if (i >= hi) continue;
    const float4 p = d.pos[i];
    const int z = p.w > 0.0f ? zone_of(sz, nz, d.sid[i], p) : -1;  // dormant slots belong to no zone
    zone_id[i] = z < 0 ? 0xFF : (uint8_t)z;
    if (z < 0) continue;
    const float4 v = d.pv[2 * (size_t)i];
    ls.enter(sh, z);
    const double m = mass_of(v.w);
    mass[i] = m;
    ls.acc[0] += m;
    ls.acc[1] = fma(m, widen(p.x), ls.acc[1]);
    ls.acc[2] = fma(m, widen(p.y), ls.acc[2]);
    ls.acc[3] = fma(m, widen(p.z), ls.acc[3]);
    ls.acc[4] = fma(m, widen(v.x), ls.acc[4]);
    ls.acc[5] = fma(m, widen(v.y), ls.acc[5]);
    ls.acc[6] = fma(m, widen(v.z), ls.acc[6]);
    ls.acc[7] += 1.0;
  }
  ls.finish(sh);
  block_to_global<kFirst>(sh, sums, nz);
}

__global__ void __launch_bounds__(kAggThreads) k_agg_second(DevPtrs d, uint32_t n, uint32_t nz,
                                                            const uint8_t *zone_id, const double *mass, const double *first,
                                                            double *sums) {
  __shared__ double com[TDS_MAX_ZONES][3];
  __shared__ double sh[TDS_MAX_ZONES * kSecond];
  for (uint32_t z = threadIdx.x; z < nz; z += blockDim.x) {
    const double M = first[z * kFirst];
    for (int a = 0; a < 3; ++a) com[z][a] = M > 0.0 ? first[z * kFirst + 1 + a] / M : 0.0;
  }
  for (uint32_t q = threadIdx.x; q < nz * kSecond; q += blockDim.x) sh[q] = 0.0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  uint32_t lo, hi;
  warp_stretch(n, lo, hi);
  LaneSums<kSecond> ls;
  for (uint32_t base = lo; base < hi; base += 32) {
    const uint32_t i = base + lane;
    const int z = i < hi ? zone_id[i] : 0xFF;
    if (z == 0xFF) continue;
    const float4 p = d.pos[i];
    const float4 v = d.pv[2 * (size_t)i];
    ls.enter(sh, z);
    const double m = mass[i];
    const double dx = widen(p.x) - com[z][0], dy = widen(p.y) - com[z][1], dz = widen(p.z) - com[z][2];
    const double vx = widen(v.x), vy = widen(v.y), vz = widen(v.z);
    const double mx = m * dx, my = m * dy, mz = m * dz;
    ls.acc[0] = fma(mx, dx, ls.acc[0]);
    ls.acc[1] = fma(my, dy, ls.acc[1]);
    ls.acc[2] = fma(mz, dz, ls.acc[2]);
    ls.acc[3] = fma(mx, dy, ls.acc[3]);
    ls.acc[4] = fma(mx, dz, ls.acc[4]);
    ls.acc[5] = fma(my, dz, ls.acc[5]);
    ls.acc[6] = fma(my, vz, fma(-mz, vy, ls.acc[6]));
    ls.acc[7] = fma(mz, vx, fma(-mx, vz, ls.acc[7]));
    ls.acc[8] = fma(mx, vy, fma(-my, vx, ls.acc[8]));
  }
  ls.finish(sh);
  block_to_global<kSecond>(sh, sums, nz);
}

// Eigen-decomposition of a symmetric 3x3 matrix by cyclic Jacobi rotations
// (Jacobi's method: zero one off-diagonal entry at a time); A becomes
// diagonal, V holds the eigenvectors as columns.
__device__ void jacobi3(double A[3][3], double V[3][3]) {
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) V[i][j] = i == j ? 1.0 : 0.0;
  for (int sweep = 0; sweep < 50; ++sweep) {
    const double off = fabs(A[0][1]) + fabs(A[0][2]) + fabs(A[1][2]);
    const double scale = fabs(A[0][0]) + fabs(A[1][1]) + fabs(A[2][2]);
    if (off <= 1e-300 || off <= 1e-17 * scale) break;
    for (int p = 0; p < 2; ++p)
      for (int q = p + 1; q < 3; ++q) {
        if (A[p][q] == 0.0) continue;
        const double theta = (A[q][q] - A[p][p]) / (2.0 * A[p][q]);
        const double tt = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
        const double c = 1.0 / sqrt(tt * tt + 1.0), s = tt * c;
        for (int k = 0; k < 3; ++k) {  // A <- A J
          const double akp = A[k][p], akq = A[k][q];
          A[k][p] = c * akp - s * akq;
          A[k][q] = s * akp + c * akq;
        }
        for (int k = 0; k < 3; ++k) {  // A <- J^T A
          const double apk = A[p][k], aqk = A[q][k];
          A[p][k] = c * apk - s * aqk;
          A[q][k] = s * apk + c * aqk;
        }
        for (int k = 0; k < 3; ++k) {  // V <- V J
          const double vkp = V[k][p], vkq = V[k][q];
          V[k][p] = c * vkp - s * vkq;
          V[k][q] = s * vkp + c * vkq;
        }
      }
  }
}

__global__ void k_agg_final(uint32_t nz, const double *first, const double *second, tds_aggregate *out) {
  const uint32_t z = blockIdx.x * blockDim.x + threadIdx.x;
  if (z >= nz) return;
  tds_aggregate o{};
  const double *F = first + z * kFirst, *S = second + z * kSecond;
  const double M = F[0];
  if (M > 0.0) {
    o.count = (uint32_t)F[7];
    o.mass = M;
    for (int a = 0; a < 3; ++a) {
      o.com[a] = F[1 + a] / M;
      o.vel[a] = F[4 + a] / M;
    }
    if (o.count == 1u) {  // one point: no extent, no spin (its centre of mass is its position to rounding only)
      out[z] = o;
      return;
    }
    // I = tr(S) 1 - S with S the second moment about the centre of mass
    const double tr = S[0] + S[1] + S[2];
    double I[3][3] = {{tr - S[0], -S[3], -S[4]}, {-S[3], tr - S[1], -S[5]}, {-S[4], -S[5], tr - S[2]}};
    o.inertia[0] = I[0][0]; o.inertia[1] = I[1][1]; o.inertia[2] = I[2][2];
    o.inertia[3] = I[0][1]; o.inertia[4] = I[0][2]; o.inertia[5] = I[1][2];
    // the momentum about the centre of mass of the velocities relative to v_A
    // equals sum m dx x v, since sum m dx = 0
    const double L[3] = {S[6], S[7], S[8]};
    // omega = I^+ L. det I = l1 l2 l3 <= lmin tr^2, so with det > 1e-10 tr^3
    // every eigenvalue is far above the pseudo-inverse's cut (1e-12 of the
    // largest) and I^+ is the inverse, I^-1 L = adj(I) L / det I; the
    // decomposition (about 20 us of dependent FP64 divisions) is for the rest.
    const double c00 = I[1][1] * I[2][2] - I[1][2] * I[1][2], c01 = I[0][2] * I[1][2] - I[0][1] * I[2][2],
                 c02 = I[0][1] * I[1][2] - I[0][2] * I[1][1], c11 = I[0][0] * I[2][2] - I[0][2] * I[0][2],
                 c12 = I[0][1] * I[0][2] - I[0][0] * I[1][2], c22 = I[0][0] * I[1][1] - I[0][1] * I[0][1];
    const double det = I[0][0] * c00 + I[0][1] * c01 + I[0][2] * c02, trI = I[0][0] + I[1][1] + I[2][2];
    if (det > 1e-10 * trI * trI * trI) {
      o.omega[0] = (c00 * L[0] + c01 * L[1] + c02 * L[2]) / det;
      o.omega[1] = (c01 * L[0] + c11 * L[1] + c12 * L[2]) / det;
      o.omega[2] = (c02 * L[0] + c12 * L[1] + c22 * L[2]) / det;
    } else {
      double V[3][3];
      jacobi3(I, V);
      const double lam[3] = {I[0][0], I[1][1], I[2][2]};
      const double lmax = fmax(fabs(lam[0]), fmax(fabs(lam[1]), fabs(lam[2])));
      for (int k = 0; k < 3; ++k) {
        if (!(fabs(lam[k]) > 1e-12 * lmax)) continue;  // pseudo-inverse: skip null directions
        const double proj = (V[0][k] * L[0] + V[1][k] * L[1] + V[2][k] * L[2]) / lam[k];
        for (int a = 0; a < 3; ++a) o.omega[a] += proj * V[a][k];
      }
    }
  }
  out[z] = o;
}

}  // namespace

int tds_launch_aggregate(const DevPtrs &d, uint32_t n, const tds_zone *zones, uint32_t nz, uint8_t *zone_id,
                         double *sums, tds_aggregate *out, cudaStream_t st) {
  double *first = sums, *second = sums + (size_t)TDS_MAX_ZONES * kFirst;
  cudaMemsetAsync(sums, 0, sizeof(double) * TDS_MAX_ZONES * (kFirst + kSecond), st);
  int sms = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // three blocks per SM (2, 3, 4: 89, 83, 87 us for both passes over
  // 1M particles; the longer a warp's stretch, the fewer reductions
  // at its end), fewer for small n so that every
  // warp has at least 128 slots
  uint32_t blocks = (n + 128u * (kAggThreads / 32) - 1) / (128u * (kAggThreads / 32));
  if (blocks < 1) blocks = 1;
  if (blocks > (uint32_t)(3 * sms)) blocks = 3 * sms;
  double *mass = reinterpret_cast<double *>(d.stage);  // of the particles in a zone (read-back scratch)
  ZoneTable table;
  std::memcpy(table.z, zones, sizeof(tds_zone) * nz);
  k_agg_first<<<blocks, kAggThreads, 0, st>>>(d, n, table, nz, zone_id, mass, first);
  k_agg_second<<<blocks, kAggThreads, 0, st>>>(d, n, nz, zone_id, mass, first, second);
  k_agg_final<<<1, TDS_MAX_ZONES, 0, st>>>(nz, first, second, out);
  return 3;
}

size_t tds_aggregate_sums_words() { return (size_t)TDS_MAX_ZONES * (kFirst + kSecond); }
