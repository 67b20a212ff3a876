// tds_colour.cu -- greedy colouring of the contact graph and the stable
// re-ordering of the contact rows into colour order.
//
// Two contacts are adjacent when they share a dynamic particle (static
// surfaces never couple contacts). Every contact gets the smallest colour not
// used by an adjacent contact of higher priority, priority being the
// SplitMix64 hash of its key. This is exactly sequential greedy colouring in
// decreasing priority order; on the GPU it is computed Jones-Plassmann style
// by a persistent kernel that walks the priority DAG in rounds: a contact is
// coloured as soon as all its higher-priority neighbours are, then releases
// its lower-priority neighbours. Contacts of one colour touch disjoint
// particles, so a colour is one parallel Gauss-Seidel step.
#include "tds_internal.cuh"

namespace {

__device__ __forceinline__ bool is_dyn(uint32_t b) { return (b & TDS_STATIC) == 0u; }

// Incidence entries carry the contact id and the high word of its priority,
// so walking a neighbourhood needs no dependent loads to compare priorities
// (counted, with each contact's place, when the rows were written).
__global__ void k_inc_fill(DevPtrs d) {
  const uint32_t nc = d.ctr[CTR_NC];
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    uint2 ab = d.c_ab[c];
    uint32_t hi = (uint32_t)(d.prio[c] >> 32);
    d.inc_ent[d.inc_start[ab.x] + d.frontier0[c]] = make_uint2(c, hi);
    if (is_dyn(ab.y)) d.inc_ent[d.inc_start[ab.y] + d.frontier1[c]] = make_uint2(c, hi);
  }
}

// Is neighbour entry e of higher priority than contact c (priority pc)?
// The high words decide unless they tie; then the full priorities do.
__device__ __forceinline__ bool higher(const DevPtrs &d, uint2 e, unsigned long long pc) {
  uint32_t hc = (uint32_t)(pc >> 32);
  if (e.y != hc) return e.y > hc;
  return d.prio[e.x] > pc;
}

constexpr int kBatch = 8;

// A slot in a frontier list for each calling lane: one atomic per group of
// converged lanes instead of one per lane (the frontier counter is a single
// address that every released contact would otherwise hit).
__device__ __forceinline__ uint32_t frontier_slot(uint32_t *counter) {
  const unsigned mask = __activemask();
  const unsigned lane = threadIdx.x & 31u;
  const int leader = __ffs(mask) - 1;
  uint32_t base = 0;
  if ((int)lane == leader) base = atomicAdd(counter, (uint32_t)__popc(mask));
  base = __shfl_sync(mask, base, leader);
  return base + (uint32_t)__popc(mask & ((1u << lane) - 1u));
}

// wait[c] = number of uncoloured neighbours of higher priority; sources
// start round 0. A full colouring starts with every contact uncoloured; an
// incremental one (see incremental_colouring) with the colours the
// narrowphase kept, which also enter the colour count.
__global__ void k_colour_init(DevPtrs d) {
  const uint32_t nc = d.ctr[CTR_NC];
  const bool inc = incremental_colouring(d);
  __shared__ uint32_t s_maxcol;
  if (threadIdx.x == 0) s_maxcol = 0;
  __syncthreads();
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    if (inc) {
      const uint32_t kept = d.colour[c];
      if (kept != TDS_NO_COLOUR) {
        atomicMax(&s_maxcol, kept + 1u);
        continue;
      }
    }
    uint2 ab = d.c_ab[c];
    unsigned long long pc = d.prio[c];
    int32_t w = 0;
    uint32_t ends[2] = {ab.x, ab.y};
    for (int k = 0; k < 2; ++k) {
      if (!is_dyn(ends[k])) continue;
      const uint32_t s = d.inc_start[ends[k]], e = d.inc_start[ends[k] + 1];
      for (uint32_t m0 = s; m0 < e; m0 += kBatch) {
        uint2 ent[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; ++q) ent[q] = m0 + q < e ? d.inc_ent[m0 + q] : make_uint2(c, 0u);
#pragma unroll
        for (int q = 0; q < kBatch; ++q)
          w += (ent[q].x != c && higher(d, ent[q], pc) && (!inc || d.colour[ent[q].x] == TDS_NO_COLOUR)) ? 1 : 0;
      }
    }
    d.wait[c] = w;
    if (!inc) d.colour[c] = TDS_NO_COLOUR;
    if (w == 0) {
      const uint32_t q = frontier_slot(d.ctr + CTR_FCOUNT);
      if (q < nc) d.frontier0[q] = c;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_maxcol) atomicMax(d.ctr + CTR_NCOL, s_maxcol);
}

// Persistent, co-resident launch: one round per grid barrier. A round colours
// every contact whose higher-priority neighbours are all coloured, then
// releases its lower-priority neighbours into the next round's frontier.
__global__ void k_colour_rounds(DevPtrs d) {
  const uint32_t stride = gridDim.x * blockDim.x;
  const uint32_t nc = d.ctr[CTR_NC];
  const bool inc = incremental_colouring(d);
  __shared__ uint32_t s_maxcol;
  if (threadIdx.x == 0) s_maxcol = 0;
  __syncthreads();
  uint32_t round = 0, gen = 0;
  for (;; ++round) {
    uint32_t *cur = (round & 1) ? d.frontier1 : d.frontier0;
    uint32_t *nxt = (round & 1) ? d.frontier0 : d.frontier1;
    volatile uint32_t *fc = d.ctr + CTR_FCOUNT;
    const uint32_t ncur = min(fc[round % 3], nc);
    uint32_t *push = d.ctr + CTR_FCOUNT + (round + 1) % 3;
    if (blockIdx.x == 0 && threadIdx.x == 0) d.ctr[CTR_FCOUNT + (round + 2) % 3] = 0u;
    for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < ncur; idx += stride) {
      const uint32_t c = __ldcg(cur + idx);
      const uint2 ab = d.c_ab[c];
      const unsigned long long pc = d.prio[c];
      unsigned long long used0 = 0ull, used1 = 0ull;
      const uint32_t ends[2] = {ab.x, ab.y};
      // colours of the higher-priority neighbours (all coloured already)
      for (int k = 0; k < 2; ++k) {
        if (!is_dyn(ends[k])) continue;
        const uint32_t s = d.inc_start[ends[k]], e = d.inc_start[ends[k] + 1];
        for (uint32_t m0 = s; m0 < e; m0 += kBatch) {
          uint2 ent[kBatch];
          uint32_t col[kBatch];
#pragma unroll
          for (int q = 0; q < kBatch; ++q) ent[q] = m0 + q < e ? d.inc_ent[m0 + q] : make_uint2(c, 0u);
#pragma unroll
          // a full colouring reads its higher-priority neighbours (all
          // coloured by now); an incremental one also the kept colours of
          // lower priority (its uncoloured neighbours read as no colour)
          for (int q = 0; q < kBatch; ++q)
            col[q] = (ent[q].x != c && (inc || higher(d, ent[q], pc))) ? (uint32_t)__ldcg(d.colour + ent[q].x) : 0xFFu;
#pragma unroll
          for (int q = 0; q < kBatch; ++q) {
            if (col[q] < 64) used0 |= 1ull << col[q];
            else if (col[q] < 128) used1 |= 1ull << (col[q] - 64);
          }
        }
      }
      uint32_t col;
      if (~used0) col = __ffsll((long long)~used0) - 1;
      else if (~used1) col = 64 + __ffsll((long long)~used1) - 1;
      else { col = TDS_MAX_COLOURS - 1; latch_error(d.err, DEV_ERR_CAPACITY); }
      __stcg(d.colour + c, (uint8_t)col);
      atomicMax(&s_maxcol, col + 1);
      // release the lower-priority neighbours (they read this colour in a
      // later round, after the grid barrier has published it)
      for (int k = 0; k < 2; ++k) {
        if (!is_dyn(ends[k])) continue;
        const uint32_t s = d.inc_start[ends[k]], e = d.inc_start[ends[k] + 1];
        for (uint32_t m0 = s; m0 < e; m0 += kBatch) {
          uint2 ent[kBatch];
          int32_t old[kBatch];
#pragma unroll
          for (int q = 0; q < kBatch; ++q) ent[q] = m0 + q < e ? d.inc_ent[m0 + q] : make_uint2(c, 0u);
#pragma unroll
          // (an incremental colouring releases only uncoloured neighbours:
          // a kept contact waits for nothing)
          for (int q = 0; q < kBatch; ++q)
            old[q] = (ent[q].x != c && !higher(d, ent[q], pc) &&
                      (!inc || __ldcg(d.colour + ent[q].x) == TDS_NO_COLOUR))
                         ? atomicSub(d.wait + ent[q].x, 1)
                         : 0;
#pragma unroll
          for (int q = 0; q < kBatch; ++q)
            if (old[q] == 1) {
              const uint32_t slot = frontier_slot(push);
              if (slot < nc) nxt[slot] = ent[q].x;
            }
        }
      }
    }
    if (!grid_barrier(d.bar, d.err, gen, d.wait_ns)) return;
    if (fc[(round + 1) % 3] == 0u || round > nc) break;
  }
  __syncthreads();
  if (threadIdx.x == 0) atomicMax(d.ctr + CTR_NCOL, s_maxcol);
  if (blockIdx.x == 0 && threadIdx.x == 0) d.ctr[CTR_ROUNDS] = round + 1;
}

// The colours of every particle's contacts as bits (a contact left without a
// colour, only after a latched error, counts as the last one).
__global__ void k_colour_masks(DevPtrs d, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t s = d.inc_start[i], e = d.inc_start[i + 1];
    unsigned long long lo = 0ull, hi = 0ull;
    for (uint32_t m0 = s; m0 < e; m0 += kBatch) {
      uint32_t col[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) col[q] = m0 + q < e ? (uint32_t)d.colour[d.inc_ent[m0 + q].x] : 0x100u;
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        if (col[q] == 0x100u) continue;
        const uint32_t b = min(col[q], (uint32_t)TDS_MAX_COLOURS - 1u);
        if (b < 64u) lo |= 1ull << b;
        else hi |= 1ull << (b - 64u);
      }
    }
    d.cmask[i] = make_ulonglong2(lo, hi);
  }
}

// Of a contact of colour col at a particle with these colours: how many of the
// particle's contacts come before it in a sweep (its rank), and how many there
// are (the degree).
__device__ __forceinline__ uint32_t rank_degree(ulonglong2 m, uint32_t col) {
  const uint32_t nlo = __popcll(m.x), nhi = __popcll(m.y);
  const uint32_t rank = col < 64u ? __popcll(m.x & ((1ull << col) - 1ull))
                                  : nlo + __popcll(m.y & ((1ull << (col - 64u)) - 1ull));
  return rank | ((nlo + nhi) << 8);
}

// ---- stable counting sort of contacts by bucket = 2 colour + static? ------
// Colours are < TDS_MAX_COLOURS once the colouring finished; a contact left
// uncoloured (only after a latched error) is clamped into the last bucket.
__device__ __forceinline__ uint32_t bucket_of(const DevPtrs &d, uint32_t c) {
  uint32_t col = d.colour[c];
  if (col >= TDS_MAX_COLOURS) col = TDS_MAX_COLOURS - 1;
  return 2u * col + (is_dyn(d.c_ab[c].y) ? 0u : 1u);
}

// Only the buckets and tiles in use are counted and scanned: the histogram is
// (buckets 0 .. 2 colours) x (tiles of the contacts there are), its length in
// CTR_HIST (all 256 buckets of the whole capacity are 50 times that).
constexpr int kBucketThreads = 1024;

__device__ __forceinline__ uint32_t used_buckets(const DevPtrs &d) {
  return 2u * min(d.ctr[CTR_NCOL], (uint32_t)TDS_MAX_COLOURS);
}
__device__ __forceinline__ uint32_t used_tiles(uint32_t nc) { return (nc + TDS_TILE - 1u) / TDS_TILE; }

__global__ void __launch_bounds__(kBucketThreads) k_bucket_hist(DevPtrs d) {
  __shared__ uint32_t hist[TDS_NBUCKETS];
  const uint32_t nc = d.ctr[CTR_NC], nt = used_tiles(nc), nb = used_buckets(d);
  if (blockIdx.x == 0 && threadIdx.x == 0) d.ctr[CTR_HIST] = nb * nt;
  if (blockIdx.x >= nt) return;
  for (uint32_t b = threadIdx.x; b < TDS_NBUCKETS; b += blockDim.x) hist[b] = 0;
  __syncthreads();
  const uint32_t base = blockIdx.x * TDS_TILE, lane = threadIdx.x & 31u;
  for (uint32_t k = threadIdx.x; k < TDS_TILE; k += blockDim.x) {
    const uint32_t c = base + k;
    uint32_t bk = 0xFFFFFFFFu;
    if (c < nc) {
      if (d.colour[c] >= TDS_MAX_COLOURS) latch_error(d.err, DEV_ERR_CAPACITY);
      bk = bucket_of(d, c);
    }
    const uint32_t peers = __match_any_sync(0xffffffffu, bk);  // one addition per bucket and warp
    if (bk != 0xFFFFFFFFu && (peers & ((1u << lane) - 1u)) == 0u) atomicAdd(hist + bk, (uint32_t)__popc(peers));
  }
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < nb; b += blockDim.x) d.tile_hist[b * nt + blockIdx.x] = hist[b];
}

// Exclusive prefix sum of one value per thread over a block of T threads;
// *total receives the sum.
template <int T>
__device__ __forceinline__ uint32_t block_prefix(uint32_t v, uint32_t *total) {
  __shared__ uint32_t sums[T / 32 + 1];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t up = __shfl_up_sync(0xffffffffu, inc, o);
    if ((int)lane >= o) inc += up;
  }
  if (lane == 31u) sums[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t s = lane < T / 32 ? sums[lane] : 0u;
    uint32_t si = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, si, o);
      if ((int)lane >= o) si += up;
    }
    if (lane < T / 32) sums[lane] = si - s;
    if (lane == T / 32 - 1) sums[T / 32] = si;
  }
  __syncthreads();
  const uint32_t r = inc - v + sums[warp];
  *total = sums[T / 32];
  __syncthreads();
  return r;
}

// Residual chunks. Inside a bucket the contacts keep the owner order, which
// is scene-major (slots are sorted by cell, cells by scene), so each scene's
// contacts of a bucket form one range; its start is the bucket's start plus
// the contacts of the earlier scenes. Each range is cut into chunks of at
// most TDS_RES_CHUNK contacts, numbered scene-major (scene, bucket, piece):
// a scene's chunks are consecutive, and they are the same chunks whether the
// scene is stepped alone or in a batch.
__device__ __forceinline__ uint32_t pieces(uint32_t cnt) { return (cnt + TDS_RES_CHUNK - 1u) / TDS_RES_CHUNK; }
// (thread t of n writes every n-th of them)
__device__ __forceinline__ void write_chunks(const DevPtrs &d, uint32_t first, uint32_t start, uint32_t cnt, uint32_t q,
                                             uint32_t t, uint32_t n) {
  for (uint32_t k = t; k * TDS_RES_CHUNK < cnt; k += n)
    d.chunk[first + k] = make_uint4(start + k * TDS_RES_CHUNK, min(TDS_RES_CHUNK, cnt - k * TDS_RES_CHUNK), q, 0u);
}

// Bucket ranges in the padded colour order: every bucket starts at a multiple
// of 32 contacts (a row tile); padding slots carry order == 0xFFFFFFFF and a
// row whose ab is all ones, and are never solved. For a single scene also its
// residual chunks. One block, a thread per bucket (one thread for all of them:
// 110 us against 4).
__global__ void __launch_bounds__(TDS_NBUCKETS) k_bucket_starts(DevPtrs d) {
  const uint32_t nc = d.ctr[CTR_NC], nt = used_tiles(nc), nb = used_buckets(d), b = threadIdx.x;
  const uint32_t u0 = b < nb && nt ? d.tile_off[b * nt] : nc, u1 = b + 1u < nb && nt ? d.tile_off[(b + 1u) * nt] : nc;
  const uint32_t cnt = u1 - u0, padded = (cnt + 31u) & ~31u;
  uint32_t total;
  const uint32_t start = block_prefix<TDS_NBUCKETS>(padded, &total);
  d.bstart[b] = start;
  d.bend[b] = start + cnt;
  d.bpad[b] = start - u0;
  for (uint32_t p = start + cnt; p < start + padded; ++p) {
    d.order[p] = 0xFFFFFFFFu;
    row_tile(d, p).ab[p & 31u] = make_uint2(~0u, ~0u);
    row_tile(d, p).rk[p & 31u] = 0u;
  }
  if (b == 0u) {
    d.bstart[TDS_NBUCKETS] = total;
    d.ctr[CTR_PADDED] = total;
  }
  if (d.nscenes == 1u) {
    d.scq_cnt[b] = cnt;
    uint32_t nchunk;
    const uint32_t first = block_prefix<TDS_NBUCKETS>(pieces(cnt), &nchunk);
    __shared__ uint32_t s_first[TDS_NBUCKETS], s_start[TDS_NBUCKETS], s_cnt[TDS_NBUCKETS];
    s_first[b] = first;
    s_start[b] = start;
    s_cnt[b] = cnt;
    d.scq_chunk[b] = first;
    if (b == 0u) {
      d.scq_chunk[TDS_NBUCKETS] = nchunk;
      d.ctr[CTR_NCHUNK] = nchunk;
    }
    __syncthreads();
    for (uint32_t g = 0; g < nb; ++g) write_chunks(d, s_first[g], s_start[g], s_cnt[g], 0u, b, TDS_NBUCKETS);
  }
}

// Scatter every contact's rows to its colour-order position: tile offset of
// its bucket + rank among equal buckets earlier in the tile (warp match +
// per-warp counts), so the order inside a bucket is the owner order.
__global__ void __launch_bounds__(kBucketThreads) k_bucket_scatter(DevPtrs d) {
  constexpr uint32_t W = kBucketThreads / 32;  // warps per block
  __shared__ uint32_t base[TDS_NBUCKETS];
  __shared__ uint32_t wcnt[W][TDS_NBUCKETS + 1];
  const uint32_t nc = d.ctr[CTR_NC], nt = used_tiles(nc), nb = used_buckets(d);
  if (blockIdx.x >= nt) return;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  for (uint32_t b = threadIdx.x; b < nb; b += blockDim.x) base[b] = d.tile_off[b * nt + blockIdx.x] + d.bpad[b];
  for (uint32_t chunk = 0; chunk < TDS_TILE; chunk += kBucketThreads) {
    for (uint32_t b = lane; b < nb; b += 32u) wcnt[warp][b] = 0;
    __syncwarp();
    const uint32_t c = blockIdx.x * TDS_TILE + chunk + threadIdx.x;
    uint32_t bk = c < nc ? bucket_of(d, c) : 0xFFFFFFFFu;
    const bool live = bk < nb;  // (a colouring that gave up leaves contacts outside the counted buckets: the step has failed)
    if (!live) bk = 0xFFFFFFFFu;
    const uint32_t peers = __match_any_sync(0xffffffffu, bk);
    const uint32_t rank_in_warp = __popc(peers & ((1u << lane) - 1u));
    if (live && rank_in_warp == 0) wcnt[warp][bk] = __popc(peers);
    __syncthreads();
    // per bucket, the warps' places: a warp per bucket, a lane per warp of the block
    for (uint32_t b = warp; b < nb; b += W) {
      const uint32_t v = wcnt[lane][b];
      uint32_t inc = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, inc, o);
        if ((int)lane >= o) inc += up;
      }
      const uint32_t at = base[b];
      wcnt[lane][b] = at + inc - v;
      __syncwarp();
      if (lane == 31u) base[b] = at + inc;
    }
    __syncthreads();
    if (live) {
      const uint32_t p = wcnt[warp][bk] + rank_in_warp;
      const uint2 ab = d.c_ab[c];
      d.order[p] = c;
      uint32_t rk = rank_degree(d.cmask[ab.x], bk >> 1);
      float4 im = make_float4(d.pv[2 * (size_t)ab.x].w, d.pv[2 * (size_t)ab.x + 1].w, 0.f, 0.f);
      if (is_dyn(ab.y)) {
        rk |= rank_degree(d.cmask[ab.y], bk >> 1) << 16;
        im.z = d.pv[2 * (size_t)ab.y].w;
        im.w = d.pv[2 * (size_t)ab.y + 1].w;
      }
      RowTile &row = row_tile(d, p);
      const uint32_t at = p & 31u;
      row.rn[at] = d.c_rn[c];
      row.rq[at] = d.c_rq[c];
      row.im[at] = im;
      row.ab[at] = ab;
      row.rm[at] = d.c_rm[c];
      row.rk[at] = rk;
      if (bk & 1u) { d.p_sv[p] = d.c_sv[c]; d.p_sw[p] = d.c_sw[c]; }
      d.p_la[p] = d.c_la[c];
      d.p_lb[p] = d.c_lb[c];
    }
    if (d.nscenes > 1) {  // contacts per (scene, bucket); a warp's contacts are nearly always one scene's
      const uint32_t q = live ? d.sid[d.c_ab[c].x] : 0xFFFFFFFFu;
      const uint32_t same = __match_any_sync(0xffffffffu, q) & peers;
      if (live && (same & ((1u << lane) - 1u)) == 0u)
        atomicAdd(d.scq_cnt + (size_t)q * TDS_NBUCKETS + bk, (uint32_t)__popc(same));
    }
    __syncthreads();
  }
}

// The residual chunks of a batch, over its scenes and the buckets in use. One block.
__global__ void __launch_bounds__(1024) k_scene_chunks(DevPtrs d) {
  constexpr uint32_t NB = TDS_NBUCKETS;
  const uint32_t S = d.nscenes, nb = used_buckets(d), lane = threadIdx.x & 31u;
  // a warp per bucket: the scenes' starts in it
  for (uint32_t b = threadIdx.x >> 5; b < nb; b += 32u) {
    uint32_t run = d.bstart[b];
    for (uint32_t q0 = 0; q0 < S; q0 += 32u) {
      const uint32_t q = q0 + lane;
      const uint32_t v = q < S ? d.scq_cnt[(size_t)q * NB + b] : 0u;
      uint32_t inc = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, inc, o);
        if ((int)lane >= o) inc += up;
      }
      if (q < S) d.scq_start[(size_t)q * NB + b] = run + inc - v;
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
  }
  __syncthreads();
  // number the pieces scene-major
  uint32_t carry = 0;
  for (uint32_t e0 = 0; e0 < S * nb; e0 += blockDim.x) {
    const uint32_t e = e0 + threadIdx.x, q = e / max(nb, 1u), b = e - q * nb;
    const size_t at = (size_t)q * NB + b;
    const uint32_t cnt = e < S * nb ? d.scq_cnt[at] : 0u;
    uint32_t total;
    const uint32_t first = carry + block_prefix<1024>(pieces(cnt), &total);
    if (e < S * nb) {
      if (b == 0u) d.scq_chunk[at] = first;  // (only the scenes' first chunks are asked for)
      write_chunks(d, first, d.scq_start[at], cnt, q, 0u, 1u);
    }
    carry += total;
  }
  if (nb == 0u)
    for (uint32_t q = threadIdx.x; q < S; q += blockDim.x) d.scq_chunk[(size_t)q * NB] = 0u;
  if (threadIdx.x == 0) {
    d.scq_chunk[(size_t)S * NB] = carry;
    d.ctr[CTR_NCHUNK] = carry;
  }
}

}  // namespace

int tds_launch_colouring(const DevPtrs &d, uint32_t n, uint32_t cap, int coop_blocks,
                         int coop_threads, cudaStream_t st) {
  int scans = 0;
  unsigned gc = (cap + 255) / 256;
  if (gc > 152 * 16) gc = 152 * 16;
  if (gc == 0) gc = 1;
  scans += tds_scan_exclusive(d.inc_cnt, d.inc_start, n, d.scan_tmp, st);
  k_inc_fill<<<gc, 256, 0, st>>>(d);
  cudaMemsetAsync(d.ctr + CTR_FCOUNT, 0, 3 * sizeof(uint32_t), st);
  cudaMemsetAsync(d.ctr + CTR_NCOL, 0, sizeof(uint32_t), st);
  k_colour_init<<<gc, 256, 0, st>>>(d);
  cudaMemsetAsync(d.bar, 0, 2 * sizeof(uint32_t), st);
  DevPtrs dd = d;
  void *args[] = {&dd};
  cudaLaunchCooperativeKernel((const void *)k_colour_rounds, dim3(coop_blocks), dim3(coop_threads),
                              args, 0, st);
  k_colour_masks<<<(n + 255) / 256 < 152 * 16 ? (n + 255) / 256 : 152 * 16, 256, 0, st>>>(d, n);
  return 4 + scans;
}

// Contact rows (and initial impulses) into the padded colour order.
int tds_launch_bucketing(const DevPtrs &d, uint32_t cap, cudaStream_t st) {
  int scans = 0;
  k_bucket_hist<<<d.ntiles, kBucketThreads, 0, st>>>(d);
  scans += tds_scan_exclusive(d.tile_hist, d.tile_off, TDS_NBUCKETS * d.ntiles, d.scan_tmp, st, d.ctr + CTR_HIST);
  k_bucket_starts<<<1, TDS_NBUCKETS, 0, st>>>(d);
  if (d.nscenes > 1) cudaMemsetAsync(d.scq_cnt, 0, sizeof(uint32_t) * (size_t)d.nscenes * TDS_NBUCKETS, st);
  k_bucket_scatter<<<d.ntiles, kBucketThreads, 0, st>>>(d);
  if (d.nscenes > 1) k_scene_chunks<<<1, 1024, 0, st>>>(d);
  return 3 + (d.nscenes > 1) + scans;
}

const void *tds_colour_kernel() { return (const void *)k_colour_rounds; }
