// tds_solve.cu -- the iterative PGS solve of the mesoscale MCP and the
// position update of the particle step (Algorithm 1).
//
// The MCP of the SPOOK stepper (section "Contacting rigid multibodies") is
// solved by projected Gauss-Seidel on the physical impulses, colour by
// colour: within a colour no two contacts share a particle, so all of them
// are updated in parallel and the result equals sequential Gauss-Seidel in
// colour-major order. One persistent, co-resident kernel runs the whole
// solve, each contact waiting only for the versions of its two particles
// that the order gives it (or, as an option, every colour at a grid barrier):
// first v = M^-1 (p + G^T lambda_0) from the warm-start impulses, then the
// sweeps, with residual checks where the tolerance asks for them. Per contact and
// sweep: the normal row (clamped at -f_c), the 2-D tangent rows projected on
// the Coulomb disk mu |Lambda_n|, the 3 rolling rows projected on the ball
// rbar mu_r |Lambda_n| (Eqs. signCoul1-3), each followed by
// v += M^-1 G^T dLambda. Particle velocities are read and written through L2
// because other SMs update them between colours.
#include <cstddef>

#include "tds_internal.cuh"
#include "tds_rules.cuh"

namespace {

__device__ __forceinline__ bool is_dyn(uint32_t b) { return (b & TDS_STATIC) == 0u; }


struct Side {
  float3 v, w;
  float im, iI;
};

__device__ __forceinline__ Side load_side(const DevPtrs &d, uint32_t s) {
  float4 v, w;
  ld_state(d.pv + 2 * (size_t)s, v, w);
  return Side{f3(v), f3(w), v.w, w.w};
}
__device__ __forceinline__ void store_side(const DevPtrs &d, uint32_t s, const Side &x) {
  st_state(d.pv + 2 * (size_t)s, make_float4(x.v.x, x.v.y, x.v.z, x.im),
           make_float4(x.w.x, x.w.y, x.w.z, x.iI));
}

struct Row {
  uint2 ab;
  float3 n;
  float la, lb, qn, Sn, fc, mu, rmu;
  float3 sv, sw;
  bool dyn;
};

__device__ __forceinline__ Row load_row(const DevPtrs &d, uint32_t p) {
  Row r;
  const RowTile &t = row_tile(d, p);
  const uint32_t at = p & 31u;
  r.ab = t.ab[at];
  float4 rn = t.rn[at], rq = t.rq[at];
  float2 rm = t.rm[at];
  r.n = f3(rn);
  r.la = rn.w;
  r.lb = rq.x; r.qn = rq.y; r.Sn = rq.z; r.fc = rq.w;
  r.mu = rm.x; r.rmu = rm.y;
  r.dyn = is_dyn(r.ab.y);
  if (!r.dyn) { r.sv = f3(d.p_sv[p]); r.sw = f3(d.p_sw[p]); }
  return r;
}

// Projections on the Coulomb disk / rolling ball of radius bound (a zero
// bound forces zero). All solver arithmetic below spells out its rounding
// (see the vector helpers): every launch shape of the solver computes the
// same bits. Without a branch: inside the bound the factor is 1, which leaves
// every value as it is.
__device__ __forceinline__ float shrink(float m2, float bound) {
  const float s = bound > 0.f ? __fmul_rn(bound, rsqrtf(m2)) : 0.f;
  return m2 > __fmul_rn(bound, bound) ? s : 1.f;
}
__device__ __forceinline__ void disk(float &a, float &b, float bound) {
  const float s = shrink(__fmaf_rn(b, b, __fmul_rn(a, a)), bound);
  a = __fmul_rn(a, s);
  b = __fmul_rn(b, s);
}
__device__ __forceinline__ void ball(float3 &a, float bound) { a = shrink(dot(a, a), bound) * a; }

// v += M^-1 G^T dLambda for each row group. A static side has zero inverse
// mass and inertia, so its (discarded) update is a no-op.
__device__ __forceinline__ void apply_normal(const Row &r, Side &A, Side &B, float dn) {
  const float3 P = dn * r.n;
  A.v = axpy(-A.im, P, A.v);
  B.v = axpy(B.im, P, B.v);
}
__device__ __forceinline__ void apply_tangent(const Row &r, Side &A, Side &B, float3 dt) {
  const float3 c = cross(r.n, dt);  // torque arms: +la n on a, -lb n on b
  A.v = axpy(-A.im, dt, A.v);
  A.w = axpy(-__fmul_rn(A.iI, r.la), c, A.w);
  B.v = axpy(B.im, dt, B.v);
  B.w = axpy(-__fmul_rn(B.iI, r.lb), c, B.w);
}
__device__ __forceinline__ void apply_rolling(Side &A, Side &B, float3 dr) {
  A.w = axpy(-A.iI, dr, A.w);
  B.w = axpy(B.iI, dr, B.w);
}
// v += M^-1 G^T (dn, dt(world), dr) on both sides.
__device__ __forceinline__ void apply(const Row &r, Side &A, Side &B, float dn, float3 dt, float3 dr) {
  apply_normal(r, A, B, dn);
  apply_tangent(r, A, B, dt);
  apply_rolling(A, B, dr);
}

// Relative velocity of the contact points:
// (v_b + w_b x (-lb n)) - (v_a + w_a x (la n)) = (v_b - v_a) - (lb w_b + la w_a) x n
__device__ __forceinline__ float3 slip(const Row &r, const Side &A, const Side &B) {
  return (B.v - A.v) - cross(axpy(r.la, A.w, r.lb * B.w), r.n);
}

// Diagonal entries of the three row groups: 1/m_a + 1/m_b + Sigma_n,
// 1/m_a + 1/m_b + la^2/I_a + lb^2/I_b + sigma_t, 1/I_a + 1/I_b + sigma_r.
__device__ __forceinline__ float diag_n(const Row &r, const Side &A, const Side &B) {
  return __fadd_rn(__fadd_rn(A.im, B.im), r.Sn);
}
__device__ __forceinline__ float diag_t(const Row &r, const Side &A, const Side &B, float sig_t) {
  const float rot = __fmaf_rn(__fmul_rn(r.lb, r.lb), B.iI, __fmul_rn(__fmul_rn(r.la, r.la), A.iI));
  return __fadd_rn(__fadd_rn(__fadd_rn(A.im, B.im), rot), sig_t);
}
__device__ __forceinline__ float diag_r(const Side &A, const Side &B, float sig_r) {
  return __fadd_rn(__fadd_rn(A.iI, B.iI), sig_r);
}

// What an update of a contact needs besides the velocities: the inverse
// diagonals and the tangent basis.
struct Pre {
  float iDn, iDt, iDr;
  float3 t1, t2;
};
__device__ __forceinline__ Pre prepare_update(const Row &r, const Side &A, const Side &B, float sig_t, float sig_r) {
  Pre q;
  q.iDn = __frcp_rn(diag_n(r, A, B));
  q.iDt = __frcp_rn(diag_t(r, A, B, sig_t));
  q.iDr = __frcp_rn(diag_r(A, B, sig_r));
  onb(r.n, q.t1, q.t2);
  return q;
}
// One projected Gauss-Seidel update of one contact.
__device__ __forceinline__ void pgs_update(const Row &r, const Pre &q, Side &A, Side &B, float4 &L0, float2 &L1,
                                           float sig_t, float sig_r) {
  // normal row
  const float res = __fsub_rn(__fmaf_rn(r.Sn, L0.x, dot(r.n, B.v - A.v)), r.qn);
  const float ln = fmaxf(__fmaf_rn(-res, q.iDn, L0.x), -r.fc);
  apply_normal(r, A, B, __fsub_rn(ln, L0.x));
  L0.x = ln;
  // tangent rows (Coulomb disk)
  const float3 u = slip(r, A, B);
  float y1 = __fmaf_rn(-__fmaf_rn(sig_t, L0.y, dot(q.t1, u)), q.iDt, L0.y);
  float y2 = __fmaf_rn(-__fmaf_rn(sig_t, L0.z, dot(q.t2, u)), q.iDt, L0.z);
  disk(y1, y2, __fmul_rn(r.mu, fabsf(ln)));
  apply_tangent(r, A, B, axpy(__fsub_rn(y2, L0.z), q.t2, __fsub_rn(y1, L0.y) * q.t1));
  L0.y = y1;
  L0.z = y2;
  // rolling rows (ball)
  const float3 lr = make_float3(L0.w, L1.x, L1.y);
  float3 y = axpy(-q.iDr, axpy(sig_r, lr, B.w - A.w), lr);
  ball(y, __fmul_rn(r.rmu, fabsf(ln)));
  apply_rolling(A, B, y - lr);
  L0.w = y.x;
  L1.x = y.y;
  L1.y = y.z;
}

// Contribution of one contact to the natural-map residual (Jacobi pass).
__device__ __forceinline__ void resid_terms(const Row &r, const Side &A, const Side &B, float4 L0,
                                            float2 L1, float sig_t, float sig_r, double &num,
                                            double &den) {
  const float wn = __fsub_rn(__fmaf_rn(r.Sn, L0.x, dot(r.n, B.v - A.v)), r.qn);
  const float pn = fmaxf(__fmaf_rn(-wn, __frcp_rn(diag_n(r, A, B)), L0.x), -r.fc);
  float3 t1, t2;
  onb(r.n, t1, t2);
  const float iDt = __frcp_rn(diag_t(r, A, B, sig_t));
  const float3 u = slip(r, A, B);
  float y1 = __fmaf_rn(-__fmaf_rn(sig_t, L0.y, dot(t1, u)), iDt, L0.y);
  float y2 = __fmaf_rn(-__fmaf_rn(sig_t, L0.z, dot(t2, u)), iDt, L0.z);
  disk(y1, y2, __fmul_rn(r.mu, fabsf(L0.x)));
  const float3 lr = make_float3(L0.w, L1.x, L1.y);
  float3 y = axpy(-__frcp_rn(diag_r(A, B, sig_r)), axpy(sig_r, lr, B.w - A.w), lr);
  ball(y, __fmul_rn(r.rmu, fabsf(L0.x)));
  const float e0 = __fsub_rn(L0.x, pn), e1 = __fsub_rn(L0.y, y1), e2 = __fsub_rn(L0.z, y2);
  const float3 e3 = lr - y;
  const float l2 = __fmaf_rn(L0.z, L0.z, __fmaf_rn(L0.y, L0.y, __fmul_rn(L0.x, L0.x)));
  num += (double)__fadd_rn(__fmaf_rn(e2, e2, __fmaf_rn(e1, e1, __fmul_rn(e0, e0))), dot(e3, e3));
  den += (double)__fadd_rn(l2, dot(lr, lr));
}

// Per-scene stop state of the solver (a bit per scene in shared memory).
__device__ __forceinline__ bool scene_done(const uint32_t *done, uint32_t q) {
  return (done[q >> 5] >> (q & 31u)) & 1u;
}
// The residual r of scene q at sweep it: CTA 0 keeps it as the scene's latest
// (residual, sweeps); below the tolerance the scene is marked to stop, else it
// competes for the largest residual of the scenes still sweeping (r >= 0, so
// its bits order like the values).
__device__ __forceinline__ void record_scene(const DevPtrs &d, uint32_t q, float r, float tol, uint32_t it,
                                             uint32_t *done_new, uint32_t *rmax) {
  if (blockIdx.x == 0) {
    d.scene_res[q] = r;
    d.scene_iters[q] = it;
  }
  if (tol > 0.f && r <= tol) atomicOr(done_new + (q >> 5), 1u << (q & 31u));
  else atomicMax(rmax, __float_as_uint(r));
}

__device__ __forceinline__ void load_pair(const DevPtrs &d, const Row &r, Side &A, Side &B) {
  A = load_side(d, r.ab.x);
  if (r.dyn) B = load_side(d, r.ab.y);
  else B = Side{r.sv, r.sw, 0.f, 0.f};
}

struct SolveArgs {
  uint32_t max_iters, every;
  float tol, sig_t, sig_r;
  int apply_warm;
  int sync;  // between colours: 0 grid barrier, 1 the particle records' versions alone
};

// ---------------------------------------------------------------------------
// The solver's order without barriers: versioned particle records
// ---------------------------------------------------------------------------
// Within a sweep a particle's contacts update it in colour order, one at a
// time. The contact with the k-th smallest colour among the particle's deg
// contacts (its rank) therefore reads the record that the update before it
// wrote: in pass p (pass 0: the warm start, if there is one, then the sweeps)
// exactly the version p deg + k, counting every update from 0. The record
// carries its version, so a contact waits for its two particles only, by
// reading their records until they hold the versions it needs, and hands
// them on by storing version + 1 with the new velocities. A version has one
// reader and one writer, so nothing is ever overwritten before it is read.
// All warps are co-resident and take their contacts in (pass, colour) order;
// the earliest outstanding contact needs only finished ones, so some warp
// always advances.
//
// A record is one 32-byte sector, moved by one access of four 64-bit words:
// (v.x, v.y), (v.z, version), (w.x, w.y), (w.z, check). The memory model
// promises that each of the four moves whole, not all of them together. A
// mixture of two versions passes only if the differences of the words taken
// from each cancel in the check word (record_check), a chance of 2^-32 for
// unrelated bits; beyond that the order rests on the sector moving whole, as
// it does on this hardware.
__device__ __forceinline__ uint32_t check_word(uint32_t of_version, float4 v, float3 w) {
  return record_check(of_version, __float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(w.x), __float_as_uint(w.y));
}
__device__ __forceinline__ void ld_rec(const float4 *rec, float4 &v, float4 &w) {
  asm volatile(
      "{\n .reg .b64 a, b, c, d;\n ld.relaxed.gpu.global.v4.b64 {a, b, c, d}, [%8];\n mov.b64 {%0, %1}, a;\n"
      " mov.b64 {%2, %3}, b;\n mov.b64 {%4, %5}, c;\n mov.b64 {%6, %7}, d;\n}\n"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w), "=f"(w.x), "=f"(w.y), "=f"(w.z), "=f"(w.w)
      : "l"(rec)
      : "memory");
}
__device__ __forceinline__ void st_rec(float4 *rec, float3 v, float3 w, uint32_t version) {
  const float4 a = make_float4(v.x, v.y, v.z, __uint_as_float(version));
  asm volatile(
      "{\n .reg .b64 a, b, c, d;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n mov.b64 c, {%5, %6};\n"
      " mov.b64 d, {%7, %8};\n st.relaxed.gpu.global.v4.b64 [%0], {a, b, c, d};\n}\n" ::"l"(rec),
      "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w), "f"(w.x), "f"(w.y), "f"(w.z), "f"(__uint_as_float(check_word(check_of_version(version), a, w)))
      : "memory");
}
// (without a branch, and with the version's part of the check worked out
// before the wait: 2000 spheres, 50 sweeps 0.442 ms against 0.463 with both
// compared in turn)
__device__ __forceinline__ bool is_version(float4 v, float4 w, uint32_t version, uint32_t of_version) {
  return ((__float_as_uint(v.w) ^ version) | (__float_as_uint(w.w) ^ check_word(of_version, v, f3(w)))) == 0u;
}

// v* = v + h g, and (records != 0) the solver's records at version 0.
__global__ void k_predict(DevPtrs d, StepConsts k, int records) {
  if (step_failed(d)) return;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < k.n; i += gridDim.x * blockDim.x) {
    float4 v = d.pv[2 * i];
    if (v.w != 0.0f) {  // (1/m = 0: a dormant reserve slot, no gravity)
      v.x += k.dt * k.g[0];
      v.y += k.dt * k.g[1];
      v.z += k.dt * k.g[2];
      d.pv[2 * i] = v;
    }
    if (records) st_rec(d.rec + 2 * (size_t)i, f3(v), f3(d.pv[2 * i + 1]), 0u);
  }
}

// The solver's records at version 0 from the particle state (after the impact
// stage, which changes the predicted velocities).
__global__ void k_records(DevPtrs d, uint32_t n) {
  if (step_failed(d)) return;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    st_rec(d.rec + 2 * (size_t)i, f3(d.pv[2 * i]), f3(d.pv[2 * i + 1]), 0u);
}

// CTA shapes compiled: (threads, row tiles in flight per warp, co-resident
// CTAs per SM the register budget is sized for); launch configurations choose
// one by index, the first is the default.
constexpr int kShapes[][3] = {{512, 2, 1}, {416, 1, 2}, {768, 1, 1}, {640, 2, 1}, {512, 3, 1}, {256, 1, 3}};
constexpr int kNumShapes = 6;
constexpr int kStages = 1;                           // ring stages per row tile in flight (and one in use)
constexpr uint32_t kFirstCheck = 5;                  // first residual check in adaptive mode
constexpr uint32_t kResSum = 256;                    // residual: partial sums of a large scene's chunks
constexpr uint32_t kWarpChunks = 1024;               // residual: scenes with at most this many chunks
                                                     // are added by one warp, larger ones by the CTA
// A warp's ring holds row tiles (see RowTile) with their impulses. Per contact:
// (n, la) 16 | (lb, q_n, Sigma_n, f_c) 16 | (1/m_a, 1/I_a, 1/m_b, 1/I_b) 16 |
// ab 8 | (mu, rbar mu_r) 8 | ranks and degrees 4 | impulses (n, t1, t2, r.x) 16 |
// (r.y, r.z) 8
constexpr size_t kRowBytes = 92;
constexpr size_t kOffRn = 0, kOffRq = 16, kOffIm = 32, kOffAb = 48, kOffRm = 56, kOffRk = 64, kOffLa = 68,
                 kOffLb = 84;  // x 32 contacts
static_assert(sizeof(RowTile) == 32 * kOffLa && offsetof(RowTile, ab) == 32 * kOffAb && offsetof(RowTile, rk) == 32 * kOffRk,
              "the ring's tiles are row tiles followed by impulses");
constexpr size_t kTileBytes = 32 * kRowBytes;
__host__ __device__ constexpr int ring_tiles(int per_thread) { return kStages * per_thread + 1; }
__host__ __device__ constexpr size_t pgs_smem(int threads, int per_thread) {
  return (size_t)(threads / 32) * ring_tiles(per_thread) * (kTileBytes + 8);  // + a barrier per tile
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint32_t bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for a phase of a tile's barrier (its own warp's copy, which
// completes in microseconds: the fixed limit): false, with the error latched,
// when it runs out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int32_t *err) {
  if (mbar_test(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_test(bar, parity))
    if (global_ns() - t0 > TDS_BARRIER_NS) {
      latch_error(err, DEV_ERR_BARRIER);
      return false;
    }
  return true;
}
// One lane: the row tile into shared memory, counted by the barrier.
__device__ __forceinline__ void bulk_rows(uint32_t dst, const RowTile *src, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)sizeof(RowTile))
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
      "r"((uint32_t)sizeof(RowTile)), "r"(bar)
      : "memory");
}
template <int B>
__device__ __forceinline__ void cp_async(uint32_t dst, const void *src) {
  if (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(B) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The row and both sides of contact p as the residual pass reads them (after
// a grid barrier: no update is in flight).
__device__ __forceinline__ Row settled_pair(const DevPtrs &d, uint32_t p, Side &A, Side &B) {
  Row r = load_row(d, p);
  const float4 im = row_tile(d, p).im[p & 31u];
  float4 v, w;
  ld_rec(d.rec + 2 * (size_t)r.ab.x, v, w);
  A = Side{f3(v), f3(w), im.x, im.y};
  if (r.dyn) {
    ld_rec(d.rec + 2 * (size_t)r.ab.y, v, w);
    B = Side{f3(v), f3(w), im.z, im.w};
  } else {
    B = Side{r.sv, r.sw, 0.f, 0.f};
  }
  return r;
}

// The persistent solver. The colour order is cut into row tiles of 32
// contacts, dealt out to the warps in turn. A warp runs through its tiles
// sweep after sweep without any barrier: a tile's rows arrive in a ring of
// shared memory as one bulk copy, its impulses by a copy of each lane (or both
// stay there when the ring holds all of the warp's tiles), the particle
// records of the next tile are read while this one is solved, and a contact
// waits only for the versions of its two particles. Grid barriers remain
// around residual checks.
//
// What bounds it: on beds of a few thousand tiles the chain of dependent
// updates (1.1 to 1.3 us of L2 round trips and arithmetic from one update of a
// particle to the next, a read taking about 850 cycles); on the largest beds
// the L1 data pipe (a record is one wavefront per lane and access), L2 and the
// rows' DRAM traffic about equally. Measured against the solver this replaced
// (rows staged by a TMA warp, every colour a barrier between neighbouring
// CTAs), same box, ms for 100 sweeps: 1M spheres (3.2M contacts) 8.64 against
// 12.1, 200k 2.55 against 5.05, 50k 1.59 against 3.45; 2000 spheres, 50 sweeps
// 0.44 against 1.29; 64 beds of 406k spheres in all, 50 sweeps 1.35 against
// 2.36.
//  - 16 warps an SM with 128 registers each, which read records ahead (8.63
//    ms): with 20, 24 and 26 warps (640x2, 768x1, 416x1) there are no registers
//    for it, 8.9, 10.2 and 11.7. On the batch of 64 beds 640x2 is 1 % faster
//    (1.346 against 1.364), on 2000 spheres 14 % slower.
//  - Tiles in turn rather than a stretch of slots per warp: every warp gets the
//    same number (2000 spheres 0.70 against 1.48 ms), and dependent tiles are
//    a whole colour apart.
//  - One lane polls while a record is two or more updates away: polling with
//    every lane of every waiting warp saturates L2 (50k spheres 4.42 against
//    2.69 ms).
//  - Rows by one bulk copy a tile rather than six copies of each lane: 8.57
//    against 8.77 ms at 1M, 1.61 against 1.68 at 50k.
template <int kThreads, int kPerThread, int kMinBlocks>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_pgs(DevPtrs d, SolveArgs a) {
  constexpr int kRing = ring_tiles(kPerThread);  // tiles in a warp's ring
  constexpr int kAhead = kRing - 1;              // tiles fetched ahead
  // Shapes of up to 16 warps an SM read the next tile's records ahead and work
  // this one's rows out during the wait. The others have too few registers for
  // it: with both they spilled 750 bytes a thread (416x1) and took 19.9 ms (1M
  // spheres, 100 sweeps; 768x1 and 256x1 16.0, 640x2 13.1); without, 200 bytes
  // and 11.7 ms (10.2, 10.2 and 8.9).
  constexpr bool kReadAhead = kThreads * kMinBlocks <= 512;
  if (step_failed(d)) return;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ double s_rn[kResSum], s_rd[kResSum];
  __shared__ int s_flag, s_news;
  __shared__ uint32_t s_done[TDS_MAX_SCENES / 32], s_done_new[TDS_MAX_SCENES / 32];
  __shared__ uint32_t s_rmax, s_ndone, s_ndone_check, s_next;
  __shared__ unsigned long long s_acc[2];
  const uint32_t ncol = min(d.ctr[CTR_NCOL], (uint32_t)TDS_MAX_COLOURS);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t cta_warps = blockDim.x >> 5;  // kThreads / 32, or fewer for small beds (solver_warps)
  const uint32_t nwarps = gridDim.x * cta_warps;
  if (threadIdx.x == 0) {
    s_ndone = 0;
    s_acc[0] = s_acc[1] = 0ull;
  }
  for (uint32_t w = threadIdx.x; w < TDS_MAX_SCENES / 32; w += blockDim.x) s_done[w] = 0u;
  __syncthreads();
  uint32_t gen = 0;  // grid barriers passed

  // Tiles are numbered in (colour, static?, slot) order and dealt out to the
  // warps in turn: warp w takes w, w + W, ... Every warp has the same number
  // of them, whatever the buckets' sizes, and the tiles in work at any time
  // are consecutive ones, a whole colour (a bed's width) ahead of the tiles
  // that depend on them. Each warp enters its own tiles in the table.
  uint32_t all = 0;
  for (uint32_t g = lane; g < 2 * ncol; g += 32) all += (d.bend[g] - d.bstart[g] + 31u) / 32u;
  all = __reduce_add_sync(0xffffffffu, all);
  // With up to two tiles a warp, consecutive warps lie on different SMs: the
  // tiles of one colour then share an SM's issue slots with fewer others
  // (2000 spheres 0.45 against 0.51 ms, 50k of the microscale bed 2.75 against
  // 2.91). With more, they lie on one SM and a tile finds its neighbours'
  // rows in the same part of DRAM and L2 (1M spheres 8.57 against 9.13 ms).
  const uint32_t warp = all <= 2u * nwarps ? (threadIdx.x >> 5) * gridDim.x + blockIdx.x
                                           : blockIdx.x * cta_warps + (threadIdx.x >> 5);
  uint32_t total = 0;
  for (uint32_t g0 = 0; g0 < 2 * ncol; g0 += 32) {
    const uint32_t g = g0 + lane;
    const uint32_t s = g < 2 * ncol ? d.bstart[g] : 0u, e = g < 2 * ncol ? d.bend[g] : 0u;
    const uint32_t T = (e - s + 31u) / 32u;
    uint32_t incl = T;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
      if ((int)lane >= o) incl += up;
    }
    const uint32_t base = total + incl - T;  // first tile of the bucket
    for (uint32_t t = (warp + nwarps - base % nwarps) % nwarps; t < T; t += nwarps)
      d.tiles[base + t] = make_uint2(s + 32u * t, min(32u, e - s - 32u * t) | (g << 8));
    total += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
  uint32_t ntile = warp < total ? (total - warp + nwarps - 1u) / nwarps : 0u;
  uint2 *list = d.tiles + warp;

  // (the ring's tiles stay 128-byte aligned: the barriers come after all of them)
  const uint32_t ring = smem_u32(smem) + (threadIdx.x >> 5) * (uint32_t)(kRing * kTileBytes);
  unsigned char *ring_p = smem + (size_t)(threadIdx.x >> 5) * (kRing * kTileBytes);
  const uint32_t bars = smem_u32(smem) + cta_warps * (uint32_t)(kRing * kTileBytes) + (threadIdx.x >> 5) * (kRing * 8u);
  // lane l keeps entry l of the list's current group of 32
  uint2 ent;
  uint32_t group;
  auto entry = [&](uint32_t j) {
    if ((j >> 5) != group) {  // lists of more than 32 tiles
      group = j >> 5;
      ent = 32u * group + lane < ntile ? list[(size_t)(32u * group + lane) * nwarps] : make_uint2(0u, 0u);
    }
    return make_uint2(__shfl_sync(0xffffffffu, ent.x, j & 31u), __shfl_sync(0xffffffffu, ent.y, j & 31u));
  };

  const uint32_t warm = a.apply_warm ? 1u : 0u;
  // The ring holds all of the warp's tiles: they are fetched once, and the
  // impulses live in it. Otherwise a tile is fetched again every sweep, at
  // least one tile after its impulses were stored.
  bool resident;
  uint32_t stages;
  bool dead = false;  // this warp's wait gave up (the error is latched)
  uint32_t it = 0;
  uint32_t fetch, fst, st;        // next tile to fetch, its ring stage, the current tile's stage
  uint32_t fetched, taken;        // tiles fetched, and waited for, since the ring was started
  uint32_t tst, tparity;          // the next tile to wait for: its stage, its barrier's phase
  uint32_t first_of[kAhead + 1];  // first contact of the current tile and the ones fetched after it
  auto fetch_next = [&](bool on) {
    if (on) {
      const uint32_t p0 = entry(fetch).x, stage = ring + fst * (uint32_t)kTileBytes;
      first_of[kAhead] = p0;
      __syncwarp();  // every lane has read what the stage held
      if (lane == 0) bulk_rows(stage, &row_tile(d, p0), bars + 8u * fst);
      cp_async<16>(stage + kOffLa * 32 + 16 * lane, d.p_la + p0 + lane);
      cp_async<8>(stage + kOffLb * 32 + 8 * lane, d.p_lb + p0 + lane);
      if (++fetch == ntile) fetch = 0;
      if (++fst == stages) fst = 0;
      ++fetched;
    }
    cp_commit();
  };
  // every tile fetched is waited for in turn (a stage's barrier completes a
  // phase per tile); resident tiles once
  auto take_rows = [&](uint32_t upto) {
    bool ok = true;
    while (taken < min(upto, fetched) && ok) {
      ok = __all_sync(0xffffffffu, mbar_wait(bars + 8u * tst, tparity, d.err));
      ++taken;
      if (++tst == stages) {
        tst = 0;
        tparity ^= 1u;
      }
    }
    return ok;
  };
  // before the CTA gives up its shared memory: all copies into it have landed
  auto drain = [&] {
    cp_wait<0>();
    while (taken < fetched) (void)take_rows(fetched);  // (a wait that runs out counts as taken)
  };
  // The records of a tile are read one tile ahead: whether they hold the
  // versions it needs is looked at when its turn comes, and only those that
  // did not are read again.
  float4 nva, nwa, nvb, nwb;
  nva = nwa = nvb = nwb = make_float4(0.f, 0.f, 0.f, 0.f);
  auto load_sides = [&](const unsigned char *stage, uint32_t p) {  // p: the lane's contact
    const uint2 ab = reinterpret_cast<const uint2 *>(stage + kOffAb * 32)[lane];
    if (ab.x == ~0u) return;
    ld_rec(d.rec + 2 * (size_t)ab.x, nva, nwa);
    if (is_dyn(ab.y)) {
      ld_rec(d.rec + 2 * (size_t)ab.y, nvb, nwb);
    } else {
      nvb = __ldg(d.p_sv + p);
      nwb = __ldg(d.p_sw + p);
    }
  };
  // (Re)starts the ring at the list's first tile; no copy is in flight.
  auto start_ring = [&] {
    if (lane == 0) {
      for (int k = 0; k < kRing; ++k) mbar_init(bars + 8u * k);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    resident = ntile <= (uint32_t)kRing;
    stages = resident ? ntile : (uint32_t)kRing;
    ent = lane < ntile ? list[(size_t)lane * nwarps] : make_uint2(0u, 0u);
    group = 0;
    fetch = fst = st = fetched = taken = tst = tparity = 0;
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      fetch_next(ntile > 0 && (!resident || k < (int)ntile));
      first_of[k] = first_of[kAhead];
    }
    dead = !take_rows(1);
    if (kReadAhead && ntile > 0 && !dead) load_sides(ring_p, entry(0).x + lane);
  };
  start_ring();

  // residual checks: every `every` sweeps, or (every == 0) where the decay
  // seen so far says the tolerance will be met (see below)
  uint32_t next_check = a.every ? a.every : kFirstCheck;
  float resid = -1.f, prev_res = -1.f;
  uint32_t prev_it = 0;
  uint32_t passes = 0;  // passes done (warm start and sweeps)
  bool done = a.max_iters == 0 && !warm;
  while (!done) {
    const bool warm_pass = passes < warm;
    uint32_t col = 0;
    for (uint32_t j = 0; j < ntile && !dead; ++j) {
      if (!a.sync)  // grid barrier after every colour
        for (const uint32_t c = entry(j).y >> 9; col < c; ++col)
          if (!grid_barrier(d.bar, d.err, gen, d.wait_ns)) {
            drain();
            return;
          }
      fetch_next(!resident || fetched < ntile);
      cp_wait<kAhead>();  // this tile's impulses are here
      dead = !take_rows(resident ? ntile : taken + 1u);  // and the next tile's rows
      if (dead) break;
      unsigned char *stage = ring_p + st * kTileBytes;
      if (++st == stages) st = 0;
      const uint32_t p = (resident ? entry(j).x : first_of[0]) + lane;
      const uint32_t p_next = (resident ? entry(j + 1 == ntile ? 0 : j + 1).x : first_of[1]) + lane;
#pragma unroll
      for (int k = 0; k < kAhead; ++k) first_of[k] = first_of[k + 1];
      const float4 *s_rn = reinterpret_cast<const float4 *>(stage + kOffRn * 32) + lane;
      const float4 *s_rq = reinterpret_cast<const float4 *>(stage + kOffRq * 32) + lane;
      const float4 *s_im = reinterpret_cast<const float4 *>(stage + kOffIm * 32) + lane;
      const uint2 ab = reinterpret_cast<const uint2 *>(stage + kOffAb * 32)[lane];
      const uint32_t rk = reinterpret_cast<const uint32_t *>(stage + kOffRk * 32)[lane];
      const bool live = rk != 0u;  // (0: padding, or a contact of a stopped scene)
      const bool dyn = is_dyn(ab.y);
      float4 *rec_a = d.rec + 2 * (size_t)ab.x, *rec_b = d.rec + 2 * (size_t)ab.y;
      if (!kReadAhead) {
        nva = nwa = nvb = nwb = make_float4(0.f, 0.f, 0.f, 0.f);  // (nothing is carried over)
        load_sides(stage, p);
      }
      float4 va = nva, wa = nwa, vb = nvb, wb = nwb;
      if (kReadAhead && ntile > 1) load_sides(ring_p + st * kTileBytes, p_next);
      uint32_t want_a = 0, want_b = 0, chk_a = 0, chk_b = 0;  // versions, and their parts of the check words
      bool need_a = live, need_b = live && dyn;
      Row r;
      float4 im, L0;
      float2 L1;
      Pre pre;
      if (live) {
        want_a = passes * ((rk >> 8) & 0xFFu) + (rk & 0xFFu);
        want_b = passes * (rk >> 24) + ((rk >> 16) & 0xFFu);
        chk_a = check_of_version(want_a);
        chk_b = check_of_version(want_b);
        asm volatile("" : "+r"(chk_a), "+r"(chk_b));  // (here, not after the wait)
      }
      auto read_row = [&] {
        const float4 rn = *s_rn, rq = *s_rq;
        im = *s_im;
        r.n = f3(rn); r.la = rn.w;
        r.lb = rq.x; r.qn = rq.y; r.Sn = rq.z; r.fc = rq.w;
        const float2 rm = reinterpret_cast<const float2 *>(stage + kOffRm * 32)[lane];
        r.mu = rm.x; r.rmu = rm.y;
        L0 = reinterpret_cast<const float4 *>(stage + kOffLa * 32)[lane];
        L1 = reinterpret_cast<const float2 *>(stage + kOffLb * 32)[lane];
        Side A, B;
        A.im = im.x; A.iI = im.y; B.im = im.z; B.iI = im.w;
        pre = prepare_update(r, A, B, a.sig_t, a.sig_r);
      };
      if (kReadAhead && live) {
        // computed while the records are on their way (the empty asm keeps it here)
        read_row();
        asm volatile("" : "+f"(pre.iDn), "+f"(pre.iDt), "+f"(pre.iDr), "+f"(pre.t1.x), "+f"(pre.t1.y), "+f"(pre.t1.z),
                     "+f"(pre.t2.x), "+f"(pre.t2.y), "+f"(pre.t2.z)::"memory");
      }
      // Wait for the versions the tile needs (bounded, as every wait). Every
      // lane that needs one reads again; while some record has two or more
      // updates to come, only the lane with the most of them polls.
      need_a &= !is_version(va, wa, want_a, chk_a);
      need_b &= !is_version(vb, wb, want_b, chk_b);
      if (__any_sync(0xffffffffu, need_a || need_b)) {
        unsigned long long t0 = 0;
        uint32_t lead = 32u;  // the polling lane; 32: every lane reads
        for (unsigned spins = 0;; ++spins) {
          if (lead == 32u || lane == lead) {
            if (need_a) ld_rec(rec_a, va, wa);
            if (need_b) ld_rec(rec_b, vb, wb);
          }
          uint32_t behind = 0;
          if (need_a) {
            need_a = !is_version(va, wa, want_a, chk_a);
            if (need_a) behind = max(1u, want_a - __float_as_uint(va.w));
          }
          if (need_b) {
            need_b = !is_version(vb, wb, want_b, chk_b);
            if (need_b) behind = max(max(behind, 1u), want_b - __float_as_uint(vb.w));
          }
          if (!__any_sync(0xffffffffu, behind != 0u)) break;
          if (lead == 32u) {
            const uint32_t worst = __reduce_max_sync(0xffffffffu, (min(behind, 0xFFFFFu) << 5) | lane);
            if (worst >= 64u) lead = worst & 31u;
          } else if (__shfl_sync(0xffffffffu, behind, lead) < 2u) {
            lead = 32u;
          }
          if ((spins & 15u) == 15u) {
            const unsigned long long t = global_ns();
            if (t0 == 0) t0 = t;
            else if (t - t0 > d.wait_ns) latch_error(d.err, DEV_ERR_BARRIER);
            dead = __any_sync(0xffffffffu, *(volatile int32_t *)d.err != 0);
            if (dead) break;
          }
        }
      }
      if (live && !dead) {
        if (!kReadAhead) read_row();
        float4 &s_la = reinterpret_cast<float4 *>(stage + kOffLa * 32)[lane];
        float2 &s_lb = reinterpret_cast<float2 *>(stage + kOffLb * 32)[lane];
        Side A{f3(va), f3(wa), im.x, im.y}, B{f3(vb), f3(wb), im.z, im.w};
        if (warm_pass) {  // v = M^-1 (p + G^T lambda_0)
          if (!(L0.x == 0.f && L0.y == 0.f && L0.z == 0.f && L0.w == 0.f && L1.x == 0.f && L1.y == 0.f))
            apply(r, A, B, L0.x, L0.y * pre.t1 + L0.z * pre.t2, make_float3(L0.w, L1.x, L1.y));
        } else {
          pgs_update(r, pre, A, B, L0, L1, a.sig_t, a.sig_r);
        }
        st_rec(rec_a, A.v, A.w, want_a + 1u);
        if (dyn) st_rec(rec_b, B.v, B.w, want_b + 1u);
        if (!warm_pass) {
          d.p_la[p] = L0;
          d.p_lb[p] = L1;
          if (resident) {
            s_la = L0;
            s_lb = L1;
          }
        }
      }
      if (kReadAhead && ntile == 1) load_sides(stage, p);
    }
    if (!a.sync)
      for (; col < ncol; ++col)
        if (!grid_barrier(d.bar, d.err, gen, d.wait_ns)) {
          drain();
          return;
        }
    ++passes;
    if (!warm_pass) ++it;
    else if (!dead) {
      done = a.max_iters == 0;
      continue;
    }
    // (a warp whose wait gave up goes straight to the barrier, which sees the
    // error in every CTA and ends the launch)
    if (dead || it == a.max_iters || (a.tol > 0.f && it == next_check)) {
      // the residual reads every contact: all updates of this sweep first
      if (!grid_barrier(d.bar, d.err, gen, d.wait_ns)) {
        drain();
        return;
      }
      // Every scene has its own residual, summed in an order that neither the
      // launch shape nor the other scenes of a batch change: its chunks (its
      // contacts of one bucket, at most TDS_RES_CHUNK of them, consecutive in
      // the colour order) are each added by one warp (lane l takes l, l + 32,
      // ..., then a fixed shuffle tree); then every CTA adds each scene's
      // chunk sums the same way, so all CTAs take the same stop decisions
      // from the same values. A scene that met the tolerance stops sweeping
      // and keeps the residual of that check.
      const uint32_t nchunk = d.ctr[CTR_NCHUNK];
      for (uint32_t ch = warp; ch < nchunk; ch += nwarps) {
        const uint4 cd = __ldcg(d.chunk + ch);
        if (scene_done(s_done, cd.z)) continue;
        double cn = 0.0, cdn = 0.0;
        for (uint32_t q = lane; q < cd.y; q += 32u) {
          const uint32_t p = cd.x + q;
          Side A, B;
          const Row r = settled_pair(d, p, A, B);
          resid_terms(r, A, B, __ldcg(d.p_la + p), __ldcg(d.p_lb + p), a.sig_t, a.sig_r, cn, cdn);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          cn += __shfl_down_sync(0xffffffffu, cn, o);
          cdn += __shfl_down_sync(0xffffffffu, cdn, o);
        }
        if (lane == 0) {
          __stcg(d.dres + 2 * ch, cn);
          __stcg(d.dres + 2 * ch + 1, cdn);
        }
      }
      if (!grid_barrier(d.bar, d.err, gen, d.wait_ns)) {
        drain();
        return;
      }
      const uint32_t S = d.nscenes;
      for (uint32_t w = threadIdx.x; w < (S + 31u) / 32u; w += blockDim.x) s_done_new[w] = 0u;
      if (threadIdx.x == 0) s_rmax = 0u;
      __syncthreads();
      // scenes with many chunks: the whole CTA adds them (fixed strides, fixed tree)
      for (uint32_t q = 0; q < S; ++q) {
        const uint32_t c0 = __ldcg(d.scq_chunk + (size_t)q * TDS_NBUCKETS);
        const uint32_t c1 = __ldcg(d.scq_chunk + (size_t)(q + 1) * TDS_NBUCKETS);
        if (c1 - c0 <= kWarpChunks || scene_done(s_done, q)) continue;
        for (uint32_t t = threadIdx.x; t < kResSum; t += blockDim.x) {
          double n0 = 0.0, n1 = 0.0, d0 = 0.0, d1 = 0.0;
          uint32_t ch = c0 + t;
          for (; ch + kResSum < c1; ch += 2u * kResSum) {
            const double2 u = __ldcg(reinterpret_cast<const double2 *>(d.dres) + ch);
            const double2 v = __ldcg(reinterpret_cast<const double2 *>(d.dres) + ch + kResSum);
            n0 += u.x; d0 += u.y;
            n1 += v.x; d1 += v.y;
          }
          if (ch < c1) {
            const double2 u = __ldcg(reinterpret_cast<const double2 *>(d.dres) + ch);
            n0 += u.x; d0 += u.y;
          }
          s_rn[t] = n0 + n1;
          s_rd[t] = d0 + d1;
        }
        __syncthreads();
        for (uint32_t h = kResSum / 2u; h > 0u; h >>= 1) {
          for (uint32_t t = threadIdx.x; t < h; t += blockDim.x) {
            s_rn[t] += s_rn[t + h];
            s_rd[t] += s_rd[t + h];
          }
          __syncthreads();
        }
        if (threadIdx.x == 0)
          record_scene(d, q, (float)(sqrt(s_rn[0]) / fmax(sqrt(s_rd[0]), 1e-12)), a.tol, it, s_done_new, &s_rmax);
        __syncthreads();
      }
      // the other scenes: one warp each (lane strides, fixed shuffle tree)
      for (uint32_t q = threadIdx.x >> 5; q < S; q += blockDim.x >> 5) {
        const uint32_t c0 = __ldcg(d.scq_chunk + (size_t)q * TDS_NBUCKETS);
        const uint32_t c1 = __ldcg(d.scq_chunk + (size_t)(q + 1) * TDS_NBUCKETS);
        if (c1 - c0 > kWarpChunks || scene_done(s_done, q)) continue;
        double tn = 0.0, td = 0.0;
        for (uint32_t ch = c0 + lane; ch < c1; ch += 32u) {
          const double2 u = __ldcg(reinterpret_cast<const double2 *>(d.dres) + ch);
          tn += u.x;
          td += u.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          tn += __shfl_down_sync(0xffffffffu, tn, o);
          td += __shfl_down_sync(0xffffffffu, td, o);
        }
        if (lane == 0) record_scene(d, q, (float)(sqrt(tn) / fmax(sqrt(td), 1e-12)), a.tol, it, s_done_new, &s_rmax);
      }
      __syncthreads();
      if (threadIdx.x == 0) s_ndone_check = 0u;
      __syncthreads();
      for (uint32_t w = threadIdx.x; w < (S + 31u) / 32u; w += blockDim.x) {
        s_done[w] |= s_done_new[w];
        atomicAdd(&s_ndone_check, (uint32_t)__popc(s_done[w]));
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        s_news = s_ndone_check != s_ndone;
        s_ndone = s_ndone_check;
        // the largest residual of the scenes still sweeping (0 when all stopped)
        resid = __uint_as_float(s_rmax);
        s_flag = a.tol > 0.f && s_ndone == S;
        // next check: a fixed period, or the sweep where the geometric decay
        // of that residual between the last two checks reaches the tolerance
        // (at least 2 and at most 64 sweeps on); every CTA computes the same
        // value from the same residuals
        uint32_t gap = a.every;
        if (a.every == 0) {
          gap = kFirstCheck;
          if (prev_res > 0.f && resid < prev_res && resid > a.tol) {
            const double rate = log((double)resid / (double)prev_res) / (double)(it - prev_it);
            const double need = ceil(log((double)a.tol / (double)resid) / rate);
            gap = (uint32_t)fmin(64.0, fmax(2.0, need));
          }
          prev_res = resid;
          prev_it = it;
        }
        s_next = it + gap;
      }
      __syncthreads();
      next_check = s_next;
      done = s_flag || it == a.max_iters;
      if (s_news && !done) {
        // Tiles whose scenes have all stopped leave the list, and a stopped
        // scene's contacts in the tiles that stay lose their ranks (they then
        // count as padding): the last sweeps of a batch cost what its
        // unfinished beds cost. A tile's contacts are in owner order, so its
        // scenes are the ones from its first contact's to its last one's; 32
        // tiles at a time, a lane each.
        // 256 beds to the 1e-4 residual (cap 2000 sweeps): 156 against 253 ms a step.
        cp_wait<0>();
        dead = !take_rows(fetched);
        if (dead) continue;
        uint32_t kept = 0;
        for (uint32_t j0 = 0; j0 < ntile; j0 += 32u) {
          uint2 e = make_uint2(0u, 0u);
          bool keep = false, mixed = false;
          if (j0 + lane < ntile) {
            e = list[(size_t)(j0 + lane) * nwarps];
            const uint2 *ab = row_tile(d, e.x).ab;
            const uint32_t q1 = __ldcg(d.sid + __ldcg(ab + (e.y & 0xFFu) - 1u).x);
            for (uint32_t q = __ldcg(d.sid + __ldcg(ab).x); q <= q1; ++q) {
              const bool off = scene_done(s_done, q);
              keep |= !off;
              mixed |= off;
            }
          }
          const uint32_t keeps = __ballot_sync(0xffffffffu, keep);
          if (keep) list[(size_t)(kept + __popc(keeps & ((1u << lane) - 1u))) * nwarps] = e;
          kept += __popc(keeps);
          for (uint32_t m = __ballot_sync(0xffffffffu, keep && mixed); m; m &= m - 1u) {
            RowTile &t = row_tile(d, __shfl_sync(0xffffffffu, e.x, __ffs(m) - 1));
            const uint32_t i = __ldcg(t.ab + lane).x;
            if (i != ~0u && scene_done(s_done, __ldcg(d.sid + i))) t.rk[lane] = 0u;
          }
        }
        asm volatile("fence.proxy.async;" ::: "memory");  // the bulk copies read the ranks
        __syncwarp();
        ntile = kept;
        if (lane == 0)
          for (int k = 0; k < kRing; ++k) mbar_inval(bars + 8u * k);
        start_ring();
      }
    }
  }
  drain();
  if (blockIdx.x == 0) {
    // statistics: the sweeps done (the most any scene did), the largest final
    // residual, and per scene its sweeps x its contacts (the solver's work)
    __syncthreads();
    const uint32_t S = d.nscenes;
    if (it == 0u)
      for (uint32_t q = threadIdx.x; q < S; q += blockDim.x) {
        d.scene_iters[q] = 0u;
        d.scene_res[q] = -1.f;
      }
    __syncthreads();
    if (threadIdx.x == 0) s_rmax = 0u;
    __syncthreads();
    unsigned long long pp = 0ull, sc = 0ull;
    for (uint32_t q = threadIdx.x; q < S; q += blockDim.x) {
      const unsigned long long iq = d.scene_iters[q];
      for (uint32_t b = 0; b < 2u * ncol; ++b) {
        const unsigned long long c = d.scq_cnt[(size_t)q * TDS_NBUCKETS + b];
        if (b & 1u) sc += iq * c;
        else pp += iq * c;
      }
      const float r = d.scene_res[q];
      if (r > 0.f) atomicMax(&s_rmax, __float_as_uint(r));
    }
    if (pp) atomicAdd(&s_acc[0], pp);
    if (sc) atomicAdd(&s_acc[1], sc);
    __syncthreads();
    if (threadIdx.x == 0) {
      d.ctr[CTR_ITERS] = it;
      d.fscal[FS_RESID] = it == 0u ? -1.f : __uint_as_float(s_rmax);
      d.acc[ACC_SWEEP_PP] += s_acc[0];
      d.acc[ACC_SWEEP_ST] += s_acc[1];
      d.acc[ACC_CONTACTS] += d.ctr[CTR_NC];
      d.acc[ACC_STEPS] += 1;
    }
  }
}

// Impact stage (the Newton impact law): a rigid velocity-level solve on the
// predicted velocities v* before the main solve. Pass 0 classifies every
// contact by its approach speed at the start of the step, -G_n v_n (G_n v* for
// a particle pair; G_n v* + h n.g against a static surface, which does not
// fall), sets the normal target e * approach for impacts and 0 otherwise, and
// zeroes the stage's impulses; with no impact the kernel stops there. Then
// `iters` colour sweeps of the main solve's update on rows with no compliance
// (Sigma_n = 0), that target as q_n and no cohesion; finally every contact's
// q_n takes the post-impact normal velocity: q_n += Upsilon (G_n v+ - G_n v*).
struct ImpactArgs {
  float e, vimp, h, g[3], ups, sig_t, sig_r;
  uint32_t iters;
};

constexpr int kImpactThreads = 512;
__global__ void __launch_bounds__(kImpactThreads) k_impact(DevPtrs d, ImpactArgs a) {
  if (step_failed(d)) return;
  __shared__ uint32_t s_count;
  const uint32_t ncol = min(d.ctr[CTR_NCOL], (uint32_t)TDS_MAX_COLOURS);
  const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  uint32_t gen = 0;
  if (threadIdx.x == 0) s_count = 0;
  __syncthreads();
  uint32_t mine = 0;
  for (uint32_t col = 0; col < ncol; ++col)
    for (int part = 0; part < 2; ++part)
      for (uint32_t p = d.bstart[2 * col + part] + tid; p < d.bend[2 * col + part]; p += stride) {
        const Row r = load_row(d, p);
        Side A, B;
        load_pair(d, r, A, B);
        const float gv = dot(r.n, B.v - A.v);
        const float gvn = r.dyn ? gv : gv + a.h * (r.n.x * a.g[0] + r.n.y * a.g[1] + r.n.z * a.g[2]);
        const bool hit = -gvn > a.vimp;
        mine += hit;
        d.p_il[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        d.p_il2[p] = make_float4(0.f, 0.f, gv, hit ? a.e * -gvn : 0.f);
      }
  if (mine) atomicAdd(&s_count, mine);
  __syncthreads();
  if (threadIdx.x == 0 && s_count) atomicAdd(d.ctr + CTR_IMPACTS, s_count);
  if (!grid_barrier(d.bar, d.err, gen, d.wait_ns)) return;
  if (*(volatile uint32_t *)(d.ctr + CTR_IMPACTS) == 0) return;  // the same value in every CTA
  for (uint32_t it = 0; it < a.iters; ++it)
    for (uint32_t col = 0; col < ncol; ++col) {
      for (int part = 0; part < 2; ++part)
        for (uint32_t p = d.bstart[2 * col + part] + tid; p < d.bend[2 * col + part]; p += stride) {
          Row r = load_row(d, p);
          const float4 t = d.p_il2[p];
          r.Sn = 0.f;
          r.fc = 0.f;
          r.qn = t.w;
          float4 L0 = d.p_il[p];
          float2 L1 = make_float2(t.x, t.y);
          Side A, B;
          load_pair(d, r, A, B);
          pgs_update(r, prepare_update(r, A, B, a.sig_t, a.sig_r), A, B, L0, L1, a.sig_t, a.sig_r);
          store_side(d, r.ab.x, A);
          if (r.dyn) store_side(d, r.ab.y, B);
          d.p_il[p] = L0;
          d.p_il2[p] = make_float4(L1.x, L1.y, t.z, t.w);
        }
      if (!grid_barrier(d.bar, d.err, gen, d.wait_ns)) return;
    }
  for (uint32_t col = 0; col < ncol; ++col)
    for (int part = 0; part < 2; ++part)
      for (uint32_t p = d.bstart[2 * col + part] + tid; p < d.bend[2 * col + part]; p += stride) {
        const Row r = load_row(d, p);
        Side A, B;
        load_pair(d, r, A, B);
        row_tile(d, p).rq[p & 31u].y = r.qn + a.ups * (dot(r.n, B.v - A.v) - d.p_il2[p].z);
      }
}

// Colour order -> owner order warm-start memory: (key's other side,
// impulses with the tangent in world coordinates).
__global__ void k_writeback(DevPtrs d) {
  if (step_failed(d)) return;
  const uint32_t np = d.ctr[CTR_PADDED];
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
    uint32_t c = d.order[p];
    if (c == 0xFFFFFFFFu) continue;  // padding slot
    float4 L0 = d.p_la[p];
    float2 L1 = d.p_lb[p];
    float3 n = f3(row_tile(d, p).rn[p & 31u]), t1, t2;
    onb(n, t1, t2);
    float3 tw = L0.y * t1 + L0.z * t2;
    d.prev_other[1][c] = (uint32_t)(d.c_key[c] & 0xFFFFFFFFull);
    d.prev_l0[1][c] = make_float4(L0.x, tw.x, tw.y, tw.z);
    d.prev_l1[1][c] = make_float4(L0.w, L1.x, L1.y, __uint_as_float((uint32_t)d.colour[c]));  // + its colour
    if (d.targ) {  // training targets of the learned warm start (final impulses in the slip frame)
      const float4 sw = d.sdirw[c];
      const float3 s = f3(sw);
      d.targ[3 * (size_t)c] = L0.x / sw.w;
      d.targ[3 * (size_t)c + 1] = dot(tw, s) / sw.w;
      d.targ[3 * (size_t)c + 2] = dot(tw, cross(n, s)) / sw.w;
    }
  }
}

__global__ void k_integrate(DevPtrs d, StepConsts k, uint32_t cap) {
  if (step_failed(d)) return;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < k.n; i += gridDim.x * blockDim.x) {
    // the range of the particle's own contacts in the warm-start memory
    const uint32_t me = d.pid[i], s = min(d.cstart[i], cap), e = min(d.cstart[i + 1], cap);
    d.prev_first[1][me] = s;
    d.prev_cnt[1][me] = e - s;
    // the solved velocities come back from the solver's records
    const float im = d.pv[2 * i].w, iI = d.pv[2 * i + 1].w;
    float4 p = d.pos[i], v = d.rec[2 * (size_t)i], w = d.rec[2 * (size_t)i + 1];
    d.pv[2 * i] = make_float4(v.x, v.y, v.z, im);
    d.pv[2 * i + 1] = make_float4(w.x, w.y, w.z, iI);
    p.x += k.dt * v.x;
    p.y += k.dt * v.y;
    p.z += k.dt * v.z;
    d.pos[i] = p;
    if (!(isfinite(p.x) && isfinite(p.y) && isfinite(p.z) && isfinite(v.x) && isfinite(v.y) &&
          isfinite(v.z) && isfinite(w.x) && isfinite(w.y) && isfinite(w.z)))
      latch_error(d.err, DEV_ERR_NONFINITE);
  }
}

// Soil-on-tool force and torque about the tool origin: sum over tool
// contacts of (Lambda_n n + Lambda_t) / dt at the contact point, plus the
// rolling impulse / dt. Only the static buckets hold tool contacts (all
// contacts: 98 us on the 1M bed). A single scene's result is reproducible:
// fixed block partition and fixed-order sums, the blocks' added by the last one
// to finish. A batch's scenes are added by FP64 atomics in any order, which the
// rounding to FP32 hides but for ties.

// Sums of six values per thread over a block of 256 threads, in threads 0 to 5.
__device__ __forceinline__ double block_sum6(const double (&v)[6], double (*sh)[6]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    double t = v[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) sh[warp][q] = t;
  }
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 6)
    for (int w = 0; w < 8; ++w) t += sh[w][threadIdx.x];
  __syncthreads();
  return t;
}

__global__ void __launch_bounds__(256) k_tool(DevPtrs d, StepConsts k) {
  if (step_failed(d)) return;
  __shared__ double sh[8][6];
  __shared__ bool last;
  __shared__ uint32_t first[TDS_MAX_COLOURS + 1], start[TDS_MAX_COLOURS];  // static contacts before a colour's, its range
  const uint32_t ncol = min(d.ctr[CTR_NCOL], (uint32_t)TDS_MAX_COLOURS);
  for (uint32_t c = threadIdx.x; c < ncol; c += blockDim.x) {
    start[c] = d.bstart[2 * c + 1];
    first[c + 1] = d.bend[2 * c + 1] - start[c];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    first[0] = 0u;
    for (uint32_t c = 0; c < ncol; ++c) first[c + 1] += first[c];
  }
  __syncthreads();
  double acc[6] = {0, 0, 0, 0, 0, 0};
  uint32_t col = 0;
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < first[ncol]; t += gridDim.x * blockDim.x) {
    while (t >= first[col + 1]) ++col;
    const uint32_t p = start[col] + (t - first[col]);
    const RowTile &row = row_tile(d, p);
    const uint2 ab = row.ab[p & 31u];
    const uint32_t sid = d.sid[ab.x];
    const SceneGeo &G = k.geo[sid];
    if ((ab.y & ~TDS_STATIC) < 1u + G.nwall) continue;
    const float4 rn = row.rn[p & 31u], L0 = d.p_la[p];
    const float2 L1 = d.p_lb[p];
    float3 n = f3(rn), t1, t2;
    onb(n, t1, t2);
    float3 F = (1.0f / k.dt) * (L0.x * n + L0.y * t1 + L0.z * t2);
    float3 xc = f3(d.pos[ab.x]) + rn.w * n;
    float3 arm = xc - make_float3(G.tp[0], G.tp[1], G.tp[2]);
    float3 T = cross(arm, F) + (1.0f / k.dt) * make_float3(L0.w, L1.x, L1.y);
    if (k.nscenes > 1) {  // batches: per-scene accumulators
      double *dst = d.tool_acc + 6 * (size_t)sid;
      atomicAdd(dst + 0, (double)F.x); atomicAdd(dst + 1, (double)F.y); atomicAdd(dst + 2, (double)F.z);
      atomicAdd(dst + 3, (double)T.x); atomicAdd(dst + 4, (double)T.y); atomicAdd(dst + 5, (double)T.z);
      continue;
    }
    acc[0] += F.x; acc[1] += F.y; acc[2] += F.z;
    acc[3] += T.x; acc[4] += T.y; acc[5] += T.z;
  }
  if (k.nscenes == 1) {
    const double s = block_sum6(acc, sh);
    if (threadIdx.x < 6) __stcg(d.dpart + 6 * blockIdx.x + threadIdx.x, s);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(d.ctr + CTR_TICKET, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) d.ctr[CTR_TICKET] = 0u;  // for the next step
  if (k.nscenes == 1) {
#pragma unroll
    for (int q = 0; q < 6; ++q) acc[q] = threadIdx.x < TDS_TOOL_BLOCKS ? __ldcg(d.dpart + 6 * threadIdx.x + q) : 0.0;
    const double s = block_sum6(acc, sh);
    if (threadIdx.x < 6) d.tool_out[threadIdx.x] = (float)s;
    return;
  }
  for (uint32_t q = threadIdx.x; q < 6 * k.nscenes; q += blockDim.x) {
    d.tool_out[q] = (float)__ldcg(d.tool_acc + q);
    d.tool_acc[q] = 0.0;
  }
}

// slot order -> particle-id order staging: x y z vx vy vz wx wy wz r. On large
// beds first each id's slot and then the records gathered by id: whole sectors
// read and coalesced writes (1M particles 27 us in two launches against 72 of
// ten scattered 4-byte writes a particle); up to kStageScatter particles one
// launch that scatters (whole calls on settled beds, scattered and gathered:
// 32k particles 56 and 58 us, 65k 64 and 66, 131k 87 and 80, 262k 112 and 109,
// 1M 280 and 268). A scene that has not been stepped has its slots in id order:
// the scatter's writes are coalesced, and it is one launch (1M: 243 and 253).
constexpr uint32_t kStageScatter = 65536;

__global__ void k_slots(DevPtrs d, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    d.slot_of_pid[d.pid[i]] = i;
}
template <bool kGather>
__global__ void k_stage(DevPtrs d, uint32_t n) {
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const uint32_t i = kGather ? d.slot_of_pid[t] : t, id = kGather ? t : d.pid[t];
    float4 p = d.pos[i], v = d.pv[2 * i], w = d.pv[2 * i + 1];
    d.stage[0 * (size_t)n + id] = p.x; d.stage[1 * (size_t)n + id] = p.y;
    d.stage[2 * (size_t)n + id] = p.z; d.stage[3 * (size_t)n + id] = v.x;
    d.stage[4 * (size_t)n + id] = v.y; d.stage[5 * (size_t)n + id] = v.z;
    d.stage[6 * (size_t)n + id] = w.x; d.stage[7 * (size_t)n + id] = w.y;
    d.stage[8 * (size_t)n + id] = w.z; d.stage[9 * (size_t)n + id] = p.w;
  }
}

}  // namespace

static inline unsigned grid_for(uint32_t n, unsigned threads, unsigned maxb = 152 * 16) {
  unsigned b = (unsigned)((n + threads - 1) / threads);
  if (b == 0) b = 1;
  return b < maxb ? b : maxb;
}

int tds_launch_predict(const DevPtrs &d, const StepConsts &k, int records, cudaStream_t st) {
  k_predict<<<grid_for(k.n, 256), 256, 0, st>>>(d, k, records);
  return 1;
}
int tds_launch_records(const DevPtrs &d, uint32_t n, cudaStream_t st) {
  k_records<<<grid_for(n, 256), 256, 0, st>>>(d, n);
  return 1;
}

// The compiled solver kernels, by shape index.
using PgsKernel = void (*)(DevPtrs, SolveArgs);
template <int I>
constexpr PgsKernel pgs_kernel() {
  return k_pgs<kShapes[I][0], kShapes[I][1], kShapes[I][2]>;
}
const PgsKernel kPgsKernels[kNumShapes] = {pgs_kernel<0>(), pgs_kernel<1>(), pgs_kernel<2>(), pgs_kernel<3>(),
                                           pgs_kernel<4>(), pgs_kernel<5>()};
int g_pgs_occupancy[kNumShapes];  // co-resident CTAs per SM of each shape (tds_pgs_setup)

int tds_pgs_shapes() { return kNumShapes; }
void tds_pgs_shape(int i, int *threads, int *per_thread) {
  *threads = kShapes[i][0];
  *per_thread = kShapes[i][1];
}

cudaError_t tds_launch_pgs(const DevPtrs &d, const StepConsts &k, uint32_t max_iters, float tol,
                           uint32_t every, int apply_warm, int blocks, int sync, int shape, cudaStream_t st) {
  SolveArgs a{max_iters, every, tol, k.sig_t, k.sig_r, apply_warm, sync};
  cudaMemsetAsync(d.bar, 0, 2 * sizeof(uint32_t), st);
  DevPtrs dd = d;
  void *args[] = {&dd, &a};
  const int T = 32 * solver_warps(k.n, k.nscenes, blocks, kShapes[shape][0] / 32);
  return cudaLaunchCooperativeKernel((const void *)kPgsKernels[shape], dim3(blocks), dim3(T), args,
                                     pgs_smem(T, kShapes[shape][1]), st);
}

cudaError_t tds_launch_impact(const DevPtrs &d, const StepConsts &k, float e, float vimp, uint32_t iters,
                              int blocks, cudaStream_t st) {
  ImpactArgs a{e, vimp, k.dt, {k.g[0], k.g[1], k.g[2]}, k.ups, k.sig_t, k.sig_r, iters};
  cudaMemsetAsync(d.bar, 0, 2 * sizeof(uint32_t), st);
  cudaMemsetAsync(d.ctr + CTR_IMPACTS, 0, sizeof(uint32_t), st);
  DevPtrs dd = d;
  void *args[] = {&dd, &a};
  return cudaLaunchCooperativeKernel((const void *)k_impact, dim3(blocks), dim3(kImpactThreads), args, 0, st);
}

// Opt the solver into its shared-memory stages; returns the co-resident
// blocks per SM for the cooperative launch.
int tds_pgs_setup() {
  int occ_min = 0;
  for (int i = 0; i < kNumShapes; ++i) {
    const int T = kShapes[i][0];
    const size_t smem = pgs_smem(T, kShapes[i][1]);
    if (cudaFuncSetAttribute((const void *)kPgsKernels[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess)
      return 0;
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void *)kPgsKernels[i], T, smem) != cudaSuccess)
      return 0;
    g_pgs_occupancy[i] = occ;
    occ_min = i == 0 ? occ : (occ < occ_min ? occ : occ_min);
  }
  return occ_min;
}

// Co-resident CTAs per SM of compiled shape i (after tds_pgs_setup).
int tds_pgs_occupancy(int i) { return g_pgs_occupancy[i]; }

// Co-resident CTAs per SM of the impact stage (0: none, or the query failed).
int tds_impact_occupancy() {
  int occ = 0;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void *)k_impact, kImpactThreads, 0) == cudaSuccess ? occ : 0;
}

int tds_launch_finish(const DevPtrs &d, const StepConsts &k, uint32_t cap, cudaStream_t st) {
  k_writeback<<<grid_for(cap, 256), 256, 0, st>>>(d);
  k_tool<<<TDS_TOOL_BLOCKS, 256, 0, st>>>(d, k);
  k_integrate<<<grid_for(k.n, 256), 256, 0, st>>>(d, k, cap);
  return 3;
}

void tds_launch_stage(const DevPtrs &d, uint32_t n, bool id_order, cudaStream_t st) {
  if (id_order || n <= kStageScatter) {
    k_stage<false><<<grid_for(n, 256), 256, 0, st>>>(d, n);
    return;
  }
  k_slots<<<grid_for(n, 256), 256, 0, st>>>(d, n);
  k_stage<true><<<grid_for(n, 256), 256, 0, st>>>(d, n);
}

