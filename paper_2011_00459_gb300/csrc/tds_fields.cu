// tds_fields.cu -- coarse-grained fields of the particles on a voxel grid
// (section "Coarse-graining", Eq. cg_velocity) and the conserved upwind
// advection of fluidized mass (Eq. advection).
#include <algorithm>
#include <cmath>

#include "tds_internal.cuh"
#include "tds_rules.cuh"

tds_status tds_set_error_message(tds_status s, const char *msg);

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int voxel_axis(float x, float o, float l0, uint32_t n) {
  const float t = floorf(__fdiv_rn(__fsub_rn(x, o), l0));
  if (!(t >= 0.0f)) return 0;
  if (t >= (float)(n - 1)) return (int)n - 1;
  return (int)t;
}

// Scatter of every particle of the grid's scene into rho and p: grids with
// more voxels than the scene has scratch for, and smooth fields on grids too
// sparsely filled for the gather.
__global__ void k_cg_scatter(DevPtrs d, uint32_t n, tds_grid g, int kernel, float R, float *rho, float *p) {
  const float vol = g.l0 * g.l0 * g.l0;
  const float inv2R2 = kernel ? 1.0f / (2.0f * R * R) : 0.0f;
  const float norm = kernel ? 1.0f / (powf(2.5066282746310002f * R, 3.0f)) : 0.0f;  // (sqrt(2 pi) R)^-3
  const float cut2 = 9.0f * R * R;
  const int reach = kernel ? (int)ceilf(3.0f * R / g.l0) + 1 : 0;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (d.sid[i] != g.scene) continue;
    const float4 x = d.pos[i];
    if (x.w == 0.0f) continue;  // dormant reserve slot
    const float4 v = d.pv[2 * (size_t)i];
    const float m = 1.0f / v.w;
    const int ci = voxel_axis(x.x, g.origin[0], g.l0, g.nx);
    const int cj = voxel_axis(x.y, g.origin[1], g.l0, g.ny);
    const int ck = voxel_axis(x.z, g.origin[2], g.l0, g.nz);
    if (kernel == 0) {
      const size_t q = ((size_t)ck * g.ny + cj) * g.nx + ci;
      const float w = m / vol;
      atomicAdd(rho + q, w);
      atomicAdd(p + 3 * q, w * v.x);
      atomicAdd(p + 3 * q + 1, w * v.y);
      atomicAdd(p + 3 * q + 2, w * v.z);
      continue;
    }
    for (int k = max(ck - reach, 0); k <= min(ck + reach, (int)g.nz - 1); ++k) {
      const float dz = g.origin[2] + ((float)k + 0.5f) * g.l0 - x.z;
      for (int j = max(cj - reach, 0); j <= min(cj + reach, (int)g.ny - 1); ++j) {
        const float dy = g.origin[1] + ((float)j + 0.5f) * g.l0 - x.y;
        for (int ii = max(ci - reach, 0); ii <= min(ci + reach, (int)g.nx - 1); ++ii) {
          const float dx = g.origin[0] + ((float)ii + 0.5f) * g.l0 - x.x;
          const float r2 = dx * dx + dy * dy + dz * dz;
          if (r2 > cut2) continue;
          const float w = m * norm * expf(-r2 * inv2R2);
          const size_t q = ((size_t)k * g.ny + j) * g.nx + ii;
          atomicAdd(rho + q, w);
          atomicAdd(p + 3 * q, w * v.x);
          atomicAdd(p + 3 * q + 1, w * v.y);
          atomicAdd(p + 3 * q + 2, w * v.z);
        }
      }
    }
  }
}

// ---- with scratch for one float4 per voxel --------------------------------------
// The voxel kernel: a particle is one 16-byte reduction into (rho, p) kept
// together, instead of four 4-byte ones into two arrays; k_cg_split then
// writes the three fields in one pass. What bounds it: L2's reductions. 1M
// particles, 161k voxels: scatter 14.9 us against 28.3, the whole call 24.6
// against 41.0.
__device__ __forceinline__ void add_cell(float4 *cell, float w, float4 v) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(cell), "f"(w), "f"(w * v.x),
               "f"(w * v.y), "f"(w * v.z)
               : "memory");
}

__global__ void __launch_bounds__(kThreads) k_cg_voxel(DevPtrs d, uint32_t n, tds_grid g, float4 *cells) {
  const float vol = g.l0 * g.l0 * g.l0;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (d.sid[i] != g.scene) continue;
    const float4 x = d.pos[i];
    if (x.w == 0.0f) continue;  // dormant reserve slot
    const float4 v = d.pv[2 * (size_t)i];
    const float m = 1.0f / v.w;
    const int ci = voxel_axis(x.x, g.origin[0], g.l0, g.nx);
    const int cj = voxel_axis(x.y, g.origin[1], g.l0, g.ny);
    const int ck = voxel_axis(x.z, g.origin[2], g.l0, g.nz);
    add_cell(cells + ((size_t)ck * g.ny + cj) * g.nx + ci, m / vol, v);
  }
}

__device__ __forceinline__ void store_voxel(size_t q, float4 c, float *rho, float *p, float *u) {
  rho[q] = c.x;
  p[3 * q] = c.y; p[3 * q + 1] = c.z; p[3 * q + 2] = c.w;
  u[3 * q] = c.x > 0.0f ? c.y / c.x : 0.0f;
  u[3 * q + 1] = c.x > 0.0f ? c.z / c.x : 0.0f;
  u[3 * q + 2] = c.x > 0.0f ? c.w / c.x : 0.0f;
}

__global__ void __launch_bounds__(kThreads) k_cg_split(uint32_t nvox, const float4 *cells, float *rho, float *p,
                                                       float *u) {
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < nvox; q += gridDim.x * blockDim.x)
    store_voxel(q, __ldg(cells + q), rho, p, u);
}

// The Gaussian kernel as a gather: the scene's particles are sorted by their
// voxel (count, scan, place), and each warp sums the particles within 3R of
// one voxel's centre in registers. What bounds it: the arithmetic of the
// (particle, voxel) pairs. A scatter adds each pair with four global
// reductions; 200k particles, R = l0, 8 particles a voxel (23M pairs): the
// gather takes 97 us (115 with sorting), the scatter 758.
struct GaussBins {
  uint32_t *count;  // per voxel, then (scanned) its first sorted particle; nvox + 1
  uint2 *at;        // per particle: voxel (~0: none), place inside it
  float4 *x, *v;    // sorted: (x, y, z, mass (sqrt(2 pi) R)^-3), (v, -)
};

// Distance along one axis to the nearest voxel centre's plane, from outside.
__device__ __forceinline__ float outside(float x, float o, float l0, uint32_t n) {
  return fmaxf(fmaxf(o + 0.5f * l0 - x, x - (o + ((float)n - 0.5f) * l0)), 0.0f);
}

// Only particles within 3R of some voxel's centre are sorted: the others would
// all lie in the border voxels, whose warps would walk them (a grid of 1000
// voxels in a bed of 1M particles, R = l0: 83 us; 3.4 ms with all sorted, 245 us
// with the scatter).
__global__ void __launch_bounds__(kThreads) k_cg_bin(DevPtrs d, uint32_t n, tds_grid g, float R, GaussBins b) {
  const float cut2 = 9.0f * R * R * 1.001f;  // (wider than the gather's own cut by more than its rounding)
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint2 at = make_uint2(~0u, 0u);
    const float4 x = d.pos[i];
    const float ox = outside(x.x, g.origin[0], g.l0, g.nx), oy = outside(x.y, g.origin[1], g.l0, g.ny),
                oz = outside(x.z, g.origin[2], g.l0, g.nz);
    if (d.sid[i] == g.scene && x.w != 0.0f && !(ox * ox + oy * oy + oz * oz > cut2)) {  // (radius 0: dormant reserve slot)
      const int ci = voxel_axis(x.x, g.origin[0], g.l0, g.nx);
      const int cj = voxel_axis(x.y, g.origin[1], g.l0, g.ny);
      const int ck = voxel_axis(x.z, g.origin[2], g.l0, g.nz);
      at.x = ((uint32_t)ck * g.ny + cj) * g.nx + ci;
      at.y = atomicAdd(b.count + at.x, 1u);
    }
    b.at[i] = at;
  }
}

__global__ void __launch_bounds__(kThreads) k_cg_place(DevPtrs d, uint32_t n, float R, GaussBins b) {
  const float norm = 1.0f / (powf(2.5066282746310002f * R, 3.0f));  // (sqrt(2 pi) R)^-3
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint2 at = b.at[i];
    if (at.x == ~0u) continue;
    const uint32_t q = b.count[at.x] + at.y;
    const float4 x = d.pos[i], v = d.pv[2 * (size_t)i];
    b.x[q] = make_float4(x.x, x.y, x.z, 1.0f / v.w * norm);
    b.v[q] = v;
  }
}

constexpr int kMaxRows = 101;  // rows of voxels across the reach along one axis (R <= 16 l0)

// 2^x by the hardware's approximation (relative error at most 2^-22, as
// expf's). The argument r2 (-log2 e / 2 R^2) is two roundings from the exact
// one, expf's -r2 (1 / 2 R^2) three; expf's own arithmetic was a quarter of the
// gather's instructions.
__device__ __forceinline__ float exp2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// A warp per voxel; its four groups of eight lanes take the rows in turn (runs
// of voxels along x, whose particles are contiguous) that can hold a particle
// within 3R, a lane per particle. The rows are taken longest first, so that
// the four in work at a time have about the same length. A row is cut to the
// voxels in reach: the particles of a voxel da rows away are at least
// (|da| - 1/2) l0 from the centre along that axis (those of a border voxel,
// which also holds what lies outside the grid, even more).
constexpr int kGatherBlocks = 6;  // per SM
__global__ void __launch_bounds__(kThreads, kGatherBlocks) k_cg_gather(tds_grid g, float R, float exponent, int reach,
                                                                       GaussBins b, uint32_t nvox, float *rho,
                                                                       float *p, float *u) {
  const float cut2 = 9.0f * R * R;
  const int span = 2 * reach + 1;
  extern __shared__ uint32_t rows[];            // span^2: dz + reach | dy + reach << 8 | voxels to either side << 16
  __shared__ uint32_t first[kMaxRows / 2 + 2];  // rows of each half width, then where they start
  for (int k = threadIdx.x; k < kMaxRows / 2 + 2; k += blockDim.x) first[k] = 0u;
  __syncthreads();
  auto half_width = [&](int k) {
    const float a = fmaxf((float)abs(k / span - reach) - 0.5f, 0.0f), c = fmaxf((float)abs(k % span - reach) - 0.5f, 0.0f);
    const float rest = 9.0f * (R / g.l0) * (R / g.l0) * 1.001f - (a * a + c * c);
    return rest < 0.0f ? -1 : min((int)floorf(sqrtf(rest) + 0.5f + 1e-3f), reach);
  };
  for (int k = threadIdx.x; k < span * span; k += blockDim.x) {
    const int hw = half_width(k);
    if (hw >= 0) atomicAdd(first + hw, 1u);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int h = reach; h >= 0; --h) {
      const uint32_t c = first[h];
      first[h] = run;
      run += c;
    }
    first[kMaxRows / 2 + 1] = run;
  }
  __syncthreads();
  const uint32_t nrow = first[kMaxRows / 2 + 1];
  for (int k = threadIdx.x; k < span * span; k += blockDim.x) {
    const int hw = half_width(k);
    if (hw >= 0) rows[atomicAdd(first + hw, 1u)] = (uint32_t)(k / span) | ((uint32_t)(k % span) << 8) | ((uint32_t)hw << 16);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const uint32_t group = (uint32_t)lane >> 3, l8 = (uint32_t)lane & 7u;
  const uint32_t warps = gridDim.x * (kThreads / 32);
  for (uint32_t q = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); q < nvox; q += warps) {
    const int i = (int)(q % g.nx), j = (int)((q / g.nx) % g.ny), k = (int)(q / (g.nx * g.ny));
    const float cx = g.origin[0] + ((float)i + 0.5f) * g.l0, cy = g.origin[1] + ((float)j + 0.5f) * g.l0,
                cz = g.origin[2] + ((float)k + 0.5f) * g.l0;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (uint32_t r = group; r < nrow; r += 4u) {
      const uint32_t w = rows[r];
      const uint32_t z = (uint32_t)(k - reach) + (w & 0xFFu), y = (uint32_t)(j - reach) + ((w >> 8) & 0xFFu);
      const int hw = (int)(w >> 16);
      if (y < g.ny && z < g.nz) {  // (negative ones wrap around)
        const uint32_t *row = b.count + (z * g.ny + y) * g.nx;
        uint32_t t = __ldg(row + max(i - hw, 0)) + l8;
        const uint32_t e = __ldg(row + min(i + hw, (int)g.nx - 1) + 1);
#pragma unroll 2
        for (; t < e; t += 8u) {
          const float4 x = __ldg(b.x + t), v = __ldg(b.v + t);
          const float dx = cx - x.x, ey = cy - x.y, ez = cz - x.z;
          const float r2 = dx * dx + ey * ey + ez * ez;
          const float m = r2 <= cut2 ? x.w * exp2_approx(r2 * exponent) : 0.0f;
          acc.x += m;
          acc.y += m * v.x;
          acc.z += m * v.y;
          acc.w += m * v.z;
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
      acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
    }
    if (lane == 0) store_voxel(q, acc, rho, p, u);
  }
}

__global__ void k_cg_velocity(size_t nvox, const float *rho, const float *p, float *u) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < nvox; q += (size_t)gridDim.x * blockDim.x) {
    const float r = rho[q];
    for (int a = 0; a < 3; ++a) u[3 * q + a] = r > 0.0f ? p[3 * q + a] / r : 0.0f;
  }
}

// Upwind flux through the face between voxels a (lower) and b (upper) along
// axis ax; both neighbours evaluate it with the same operations.
__device__ __forceinline__ float face_flux(const float *u, const float *rho, size_t a, size_t b, int ax) {
  const float uf = 0.5f * (u[3 * a + ax] + u[3 * b + ax]);
  return uf > 0.0f ? uf * rho[a] : uf * rho[b];
}

__global__ void k_advect(tds_grid g, const float *u, const float *rho, const float *src, float dt, float *out) {
  const size_t nvox = (size_t)g.nx * g.ny * g.nz;
  const size_t stride[3] = {1, g.nx, (size_t)g.nx * g.ny};
  const float c = dt / g.l0;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < nvox; q += (size_t)gridDim.x * blockDim.x) {
    const uint32_t idx[3] = {(uint32_t)(q % g.nx), (uint32_t)((q / g.nx) % g.ny), (uint32_t)(q / ((size_t)g.nx * g.ny))};
    const uint32_t dim[3] = {g.nx, g.ny, g.nz};
    float net = 0.0f;  // inflow minus outflow
    for (int ax = 0; ax < 3; ++ax) {
      if (idx[ax] > 0) net += face_flux(u, rho, q - stride[ax], q, ax);
      if (idx[ax] + 1 < dim[ax]) net -= face_flux(u, rho, q, q + stride[ax], ax);
    }
    out[q] = rho[q] + c * net + (src ? dt * src[q] : 0.0f);
  }
}

int grid_blocks(size_t n) {
  size_t b = (n + kThreads - 1) / kThreads;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  return (int)b;
}

}  // namespace

// Scratch: the impact stage's colour-order arrays (used only inside a step)
// for the voxels, the read-back staging and the broadphase's for the sorted
// particles. scratch_cells: float4 entries of the first. live: about how
// many particles lie within reach of the grid.
int tds_launch_coarse_grain(const DevPtrs &d, uint32_t n, double live, const tds_grid &g, int kernel, float R,
                            float *rho, float *p, float *u, size_t scratch_cells, cudaStream_t st) {
  const size_t nvox = (size_t)g.nx * g.ny * g.nz;
  if (kernel == 0 && nvox <= scratch_cells) {
    cudaMemsetAsync(d.p_il, 0, sizeof(float4) * nvox, st);
    k_cg_voxel<<<grid_blocks(n), kThreads, 0, st>>>(d, n, g, d.p_il);
    k_cg_split<<<grid_blocks(nvox), kThreads, 0, st>>>((uint32_t)nvox, d.p_il, rho, p, u);
    return 2;
  }
  if (kernel == 1 && nvox + 1 + tds_scan_tmp_words((uint32_t)nvox) <= 4 * scratch_cells && nvox < 0x7FFFFFFFu &&
      gather_pays((double)nvox, (double)(R / g.l0), live)) {
    GaussBins b;
    b.count = reinterpret_cast<uint32_t *>(d.p_il);
    uint32_t *tmp = b.count + nvox + 1;
    b.at = reinterpret_cast<uint2 *>(d.stage + 8 * (size_t)n);  // 10 n words in all
    b.x = reinterpret_cast<float4 *>(d.stage);
    b.v = b.x + n;
    cudaMemsetAsync(b.count, 0, sizeof(uint32_t) * (nvox + 1), st);
    k_cg_bin<<<grid_blocks(n), kThreads, 0, st>>>(d, n, g, R, b);
    const int scans = tds_scan_exclusive(b.count, b.count, (uint32_t)nvox, tmp, st);
    k_cg_place<<<grid_blocks(n), kThreads, 0, st>>>(d, n, R, b);
    const int reach = (int)floorf(3.0f * R / g.l0 + 0.5f + 1e-3f), span = 2 * reach + 1;
    k_cg_gather<<<std::min(grid_blocks(nvox * 32), 152 * kGatherBlocks), kThreads, sizeof(uint32_t) * span * span, st>>>(
        g, R, (float)(-1.4426950408889634 / (2.0 * (double)R * (double)R)), reach, b, (uint32_t)nvox, rho, p, u);
    return 3 + scans;
  }
  cudaMemsetAsync(rho, 0, sizeof(float) * nvox, st);
  cudaMemsetAsync(p, 0, sizeof(float) * 3 * nvox, st);
  k_cg_scatter<<<grid_blocks(n), kThreads, 0, st>>>(d, n, g, kernel, R, rho, p);
  k_cg_velocity<<<grid_blocks(nvox), kThreads, 0, st>>>(nvox, rho, p, u);
  return 2;
}

bool tds_grid_valid(const tds_grid *g) {
  if (!g || !(g->l0 > 0.0f) || !std::isfinite(g->l0) || g->nx == 0 || g->ny == 0 || g->nz == 0) return false;
  for (int a = 0; a < 3; ++a)
    if (!std::isfinite(g->origin[a])) return false;
  return (double)g->nx * g->ny * g->nz < 4.0e9;
}

extern "C" tds_status tds_advect_fluid(const tds_grid *grid, const float *u, const float *rho_f,
                                       const float *source, float dt, float *rho_out, void *stream) {
  if (!tds_grid_valid(grid)) return tds_set_error_message(TDS_ERR_INVALID_ARG, "invalid grid");
  if (!u || !rho_f || !rho_out) return tds_set_error_message(TDS_ERR_INVALID_ARG, "NULL field");
  if (rho_out == rho_f) return tds_set_error_message(TDS_ERR_INVALID_ARG, "rho_out must not alias rho_f");
  if (!(dt >= 0.0f) || !std::isfinite(dt)) return tds_set_error_message(TDS_ERR_INVALID_ARG, "dt must be >= 0");
  const size_t nvox = (size_t)grid->nx * grid->ny * grid->nz;
  k_advect<<<grid_blocks(nvox), kThreads, 0, (cudaStream_t)stream>>>(*grid, u, rho_f, source, dt, rho_out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return tds_set_error_message(TDS_ERR_CUDA, cudaGetErrorString(e));
  return TDS_OK;
}
