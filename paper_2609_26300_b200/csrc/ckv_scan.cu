// Summary scan: one streaming pass over every block summary (Eq. 8-9 and the compensation sums
// of Eq. 12), as a persistent, bulk-copy-pipelined, tensor-core kernel.
//
// For every block b and query head g of a unit the pass computes
//   zbar_{g,b}        = q_g . kbar_b * scale                      (block-mean logit, Sec. 4.1)
//   sigma_hat^2_{g,b} = scale^2 sum_t w_{g,t} Dbar_{b,t}         (Eq. 8 with 1/d = scale^2, w_{g,t} = sum_{i in G_t} q_{g,i}^2)
//   l_{g,b}           = log|b| + zbar + sigma_hat^2 / 2           (log of the numerator of Eq. 9)
// and stores, in log2 units, e^l sigma_hat^2 for the selection kernel and |b| e^{zbar} for the attention kernel
// (4 bytes each per head and block), together with partials of the normaliser of Eq. 9.  In the same pass it accumulates the mean-compensation terms of Eq. 12 over ALL blocks,
// sum_b |b| e^{zbar} vbar_b  and  sum_b |b| e^{zbar},  as online-softmax partials; the terms of the
// blocks that end up selected are taken out again by the attention kernel.  That way kbar, Dbar and
// vbar are each read from HBM exactly once per decode step.
//
// The two contractions are the GQA-grouped Kbar Q^T and Vbar^T W tiles, on mma.sync.m16n8k16 (bf16 in, fp32
// accumulate): 16 blocks (then 16 coordinates) are the M dimension, the heads the N dimension (ckv_mma.cuh).  The
// summaries are stored as split bf16 pairs (hi + lo), so x * y is hi * y + lo * y with no conversion instructions; the
// weights w = |b| e^{zbar - m} are split the same way.
//
// Schedule: the launch has two kinds of CTAs.  The first few ("tail" CTAs, one warp per unit) take the LAST block
// of every sequence -- the only block a decode step can change -- and, in a fused step, first append the step's new
// token to it (page write + block summary); see scan_tail.  All other blocks of all units are cut into tiles of
// 32 consecutive blocks; the tiles, in (unit, position) order, are split into one contiguous range per scan CTA,
// one scan CTA per remaining SM.  A producer thread streams the CTA's tiles into a ring of shared-memory stages
// with cp.async.bulk (two 16 KB copies and the variances per tile), completion on mbarriers.  Each of the seven
// consumer warps takes every seventh half tile (16 blocks) on its own and visits only the tiles that hold one of
// its parts -- there is no CTA-wide barrier in the loop -- with a per-warp running maximum that is only raised
// when exceeded by a slack.  The query rows and variance weights of the CTA's units are staged in shared memory
// while the first fills are in flight, so a warp that moves on to another unit sets up from there.  A warp writes one
// partial per unit its CTA touched; partial (scan CTA c, warp w, unit u) lives in entry (c + 2 u) * 7 + w, unique
// because the (c, u) pairs that occur form a monotone staircase; the entry behind a unit's last one is free and
// takes the last block's partial, so a unit's partials are one contiguous run (unit_scan_entries).
//
// Lengths in a fused step: every CTA reads the lengths as they were before the append and works with them plus
// one; a counter of CTAs that are done reading decides who stores the new lengths (lens_arrive), so the kernels
// that follow in the stream see them in place and nobody waits on anybody inside the launch.
#include <algorithm>
#include <mutex>

#include "ckv_internal.cuh"
#include "ckv_pipe.cuh"
#include "ckv_mma.cuh"
#include "ckv_blockstats.cuh"
#include "ckv_scanpart.cuh"

namespace {

using namespace ckv_pipe;

constexpr int kMaxStages = 8;
constexpr int kConsumerWarps = CKV_SCAN_WARPS;
constexpr int kThreads = kConsumerWarps * 32 + 32;   // plus the producer warp
constexpr int kMaxSeqs = 1024;      // sequence lengths are staged in shared memory up to this many sequences

struct UnitInfo { int N, X, tiles; };   // X: the blocks the scan CTAs cover (in tail mode all but the sequence's last one)

// s_len holds the clamped lengths (after this step's append, if any) of the first kMaxSeqs sequences, staged once
// per CTA; longer batches never come with an append and read the device array
__device__ __forceinline__ int seq_len_of(const CkvDev &P, const int *s_len, const int *seq_lens, int s) {
  return s < kMaxSeqs ? s_len[s] : max(min(seq_lens[s], P.max_blocks * P.bs), 0);
}
__device__ __forceinline__ UnitInfo unit_info(const CkvDev &P, const int *s_len, const int *seq_lens, int u) {
  UnitInfo ui;
  ui.N = seq_len_of(P, s_len, seq_lens, ckv_div_hkv(P, u));
  ui.X = ckv_scan_blocks(P, ui.N);
  ui.tiles = (ui.X + P.scan_tile - 1) >> P.lg_tile;
  return ui;
}

__device__ __forceinline__ int seq_tiles(const int *s_len, const int *seq_lens, const CkvDev &P, int i) {
  return (ckv_scan_blocks(P, seq_len_of(P, s_len, seq_lens, i)) + P.scan_tile - 1) >> P.lg_tile;
}

constexpr int kLenCounter = CKV_LEN_COUNTER_WORD;   // counts the CTAs which have read the lengths

// Length hand-over of a fused step.  Every CTA of the launch works with the lengths as they were before the
// append (plus one); a CTA calls this once it will not read the length array again, and the last one to call
// stores the new lengths, so that the kernels that follow find them in place.  Nobody waits: it is a counter.
// whole_cta: called by all threads of the CTA (which then share the stores), else by one thread.
__device__ __noinline__ void lens_arrive(int *counter, const int *seq_lens, int *seq_lens_out, int batch, int cap,
                                         int n_ctas, bool whole_cta) {
  if (whole_cta) {
    __shared__ int s_is_last;
    __syncthreads();
    if (threadIdx.x == 0) {
      s_is_last = atomicAdd(counter, 1) == n_ctas - 1;
      if (s_is_last) *counter = 0;   // ready for the next launch
    }
    __syncthreads();
    if (!s_is_last) return;
    for (int i = threadIdx.x; i < batch; i += blockDim.x) {
      const int raw = seq_lens[i];
      if (raw >= 0 && raw < cap) seq_lens_out[i] = raw + 1;
    }
  } else {
    if (atomicAdd(counter, 1) != n_ctas - 1) return;
    *counter = 0;
    for (int i0 = 0; i0 < batch; i0 += 8) {   // loads of a group first: the arrays are one and the same
      int raw[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) raw[k] = i0 + k < batch ? seq_lens[i0 + k] : -1;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (raw[k] >= 0 && raw[k] < cap) seq_lens_out[i0 + k] = raw[k] + 1;
    }
  }
}

// Tail CTAs of the scan launch: one warp per unit.  With a new token (fused step) the warp first stores the
// token's key and value rows into their page and recomputes the summary of the block they land in, with the
// routine the stand-alone append uses.  Then, new token or not, it does for the unit's LAST block what the scan
// CTAs do for all the others -- the block's two per-head terms and its mean-compensation partial -- reading the
// summary as stored.  The last block is the only one a step can change, so the scan CTAs depend on nothing this
// warp writes and the append costs the step no time of its own.
//
// Deliberately not inlined, and with the kernel's parameter block passed BY VALUE: inlined, its code doubled the
// kernel's size and the scan CTAs stalled on instruction fetch (the launch went from 55 to 68 us); handed a
// reference, the compiler moves the parameter block to local memory for every CTA, scan loop included.
template <int G, typename QT>
__device__ __noinline__ void scan_tail(const CkvDev P, const QT *q, const int *seq_lens, int *s_len,
                                       int len_mine, int units, int nscan, const CkvNewToken fresh, int n_tail,
                                       float *smem_f, int smem_bytes) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, hw = lane >> 4, li = lane & 15;
  const int batch = ckv_div_hkv(P, units), cap = P.max_blocks * P.bs;
  const bool append = fresh.k_new != nullptr;
  const bool lo_half = P.row_elems == CKV_ROW_ELEMS;
  const bool by_mass = (P.variant & CKV_VARIANT_RANK_BY_MASS) != 0;
  QT *k_pool = reinterpret_cast<QT *>(fresh.k_pool), *v_pool = reinterpret_cast<QT *>(fresh.v_pool);
  const QT *k_new = reinterpret_cast<const QT *>(fresh.k_new), *v_new = reinterpret_cast<const QT *>(fresh.v_new);
  float *sq = smem_f + warp * CKV_D;
  constexpr int PIECES = (int)(CKV_D * sizeof(QT) / 16);   // 16-byte pieces of a row: lanes 0-15 hold K, 16-31 hold V
  constexpr int PP = PIECES / 16;
  const int u_first = (int)blockIdx.x * 8 + warp;
  // the new row of the warp's first unit does not depend on the lengths: it is requested together with them
  uint4 piece[PP];
  // the unit's G query rows are read head by head in a rolled loop further down (this routine's time is the fetch
  // of its own instructions, executed once per launch: a short loop beats unrolled code); the L2 is asked for them
  // now, while nothing depends on them
  if (u_first < units && lane < G)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(q + ((size_t)u_first * G + lane) * CKV_D) : "memory");
  if (append && u_first < units) {
    const uint4 *src = reinterpret_cast<const uint4 *>((lane < 16 ? k_new : v_new) + (size_t)u_first * CKV_D);
#pragma unroll
    for (int k = 0; k < PP; ++k) piece[k] = src[li + 16 * k];
  }
  auto eff_len = [&](int raw) { return max(min(raw + ((append && raw >= 0 && raw < cap) ? 1 : 0), cap), 0); };
  if (tid < batch) s_len[tid] = eff_len(len_mine);
  for (int i = tid + kThreads; i < batch && i < kMaxSeqs; i += kThreads) s_len[i] = eff_len(seq_lens[i]);
  __syncthreads();
  auto len_of = [&](int i) { return seq_len_of(P, s_len, seq_lens, i); };

  // The length before the append, from the staged (already incremented and clamped) one; the device array is only
  // asked where that is ambiguous (an empty or exactly full sequence).
  auto raw_len = [&](int sq_idx) {
    const int eff = len_of(sq_idx);
    return (eff > 0 && eff < cap && sq_idx < kMaxSeqs) ? eff - 1 : seq_lens[sq_idx];
  };
#pragma unroll 1
  for (int u = u_first; u < units; u += n_tail * 8) {
    const int s = ckv_div_hkv(P, u), h = u - s * P.Hkv;
    const int *pt_row = fresh.page_table + (size_t)s * P.max_pages_per_seq;
    const int raw = append ? raw_len(s) : -1;
    const bool room = raw >= 0 && raw < cap;
    int phys = -1;
    // the page of the new token is asked for first, and the unit's place among the scan partials (which depends on
    // the lengths only) is worked out while that entry is on its way
    if (append && room) phys = pt_row[raw / CKV_PAGE];
    int first = 0, count = 0;
    unit_scan_entries(P, len_of, units, u, nscan, lane, first, count);
    if (append) {
      if (!room) {
        if (lane == 0) atomicOr(P.status, CKV_DEV_SEQ_FULL);
      } else {
        const int slot = raw % CKV_PAGE;
        const int b = raw >> P.lg_bs, cnt = raw + 1 - b * P.bs;
        if (phys >= 0 && phys < P.num_pages) {
          if (u != u_first) {
            const uint4 *src = reinterpret_cast<const uint4 *>((lane < 16 ? k_new : v_new) + (size_t)u * CKV_D);
#pragma unroll
            for (int k = 0; k < PP; ++k) piece[k] = src[li + 16 * k];
          }
          uint4 *dst = reinterpret_cast<uint4 *>((lane < 16 ? k_pool : v_pool) +
                                                 (((size_t)phys * P.Hkv + h) * CKV_PAGE + slot) * CKV_D);
#pragma unroll
          for (int k = 0; k < PP; ++k) dst[li + 16 * k] = piece[k];
        }
        __syncwarp();
        const size_t row = (size_t)u * P.max_blocks + b;
        // rows staged in this warp's slice of the (otherwise unused) ring memory when it is large enough
        constexpr int kStageBytes = 2 * CKV_PAGE * CKV_D * (int)sizeof(QT);
        if (smem_bytes >= 8 * CKV_D * 4 + 8 * kStageBytes)
          block_stats_warp_staged<QT>(P, k_pool, v_pool, pt_row, h, b, cnt,
                                      reinterpret_cast<unsigned char *>(smem_f + 8 * CKV_D) + (size_t)warp * kStageBytes, sq,
                                      P.kmean + row * P.row_elems, P.dbar + row * P.r, P.vmean + row * P.row_elems, lane);
        else
          block_stats_warp<QT, true>(P, k_pool, v_pool, pt_row, h, b, cnt, sq, P.kmean + row * P.row_elems,
                                      P.dbar + row * P.r, P.vmean + row * P.row_elems, lane);
      }
    }
    const int N = len_of(s);
    if (N == 0) continue;   // warp-uniform
    const int b = ((N + P.bs - 1) >> P.lg_bs) - 1, cnt = N - b * P.bs;
    const size_t row = (size_t)u * P.max_blocks + b;
    __syncwarp();
    float kx[8], vx[8], dx[8];   // this lane's 8 coordinates of kbar, vbar and of the variance of their group
    load_split8<false>(P.kmean + row * P.row_elems, li, b, kx, lo_half);
    load_split8<false>(P.vmean + row * P.row_elems, li, b, vx, lo_half && !P.vhi);   // as the scan CTAs read it
    if (P.r == CKV_D) {
      load_split8<false>(reinterpret_cast<const __nv_bfloat16 *>(P.dbar + row * CKV_D), li, b, dx);
    } else {
      // group of coordinate c: c / (128 / r), or ((c mod 64) / (64 / r)) in the half-split layout; r is a power of two
      const float *drow = P.dbar + row * P.r;
      const int sh = 31 - __clz(CKV_D / P.r);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int c = 8 * li + i;
        dx[i] = drow[P.glayout == 0 ? c >> sh : (c & (CKV_D / 2 - 1)) >> (sh - 1)];
      }
    }
    float *part = P.comp_part + (size_t)(first + count - 1) * G * CKV_PART_STRIDE;
    const float logc = logf((float)cnt);
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      float qx[8];   // this lane's 8 coordinates of query row u G + g
      load8<false>(q + ((size_t)u * G + g) * CKV_D + 8 * li, qx);
      float d = 0.f, sg = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        d = fmaf(qx[i], kx[i], d);
        const float qs = qx[i] * P.scale;
        sg = fmaf(qs * qs, dx[i], sg);   // Eq. 8: the squared logit scale is its 1/d
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        d += __shfl_xor_sync(0xffffffffu, d, o);
        sg += __shfl_xor_sync(0xffffffffu, sg, o);
      }
      sg = fmaxf(sg, 0.f);
      const float zbar = d * P.scale;
      const float ell = logc + zbar + P.half_var * sg;
      const float zl2 = (zbar + logc) * kLog2e;
      float *pg = part + g * CKV_PART_STRIDE;
      if (lane == 0) {
        const size_t o = ((size_t)u * G + g) * P.max_blocks + b;
        P.lu[o] = fmaf(ell, kLog2e, by_mass ? 0.f : __log2f(sg));
        P.lz[o] = zl2;
        pg[0] = zl2; pg[1] = 1.f; pg[2] = fast_exp2(P.half_var * kLog2e * sg);   // maximum, weight 1, e^{l - m}
      }
      if (hw == 1) {   // weight 1 times the mean value
        *reinterpret_cast<float4 *>(pg + 4 + 8 * li) = make_float4(vx[0], vx[1], vx[2], vx[3]);
        *reinterpret_cast<float4 *>(pg + 8 + 8 * li) = make_float4(vx[4], vx[5], vx[6], vx[7]);
      }
    }
  }
}

// RD: one variance group per coordinate (r = d).  The variance rows then have the mean rows' layout and
// sigma^2 = sum_i (scale q_i)^2 Dbar_i is a third tensor-core product, with the squared queries as the A operand.
// HS: the mean rows hold hi halves only (bf16 summaries, 256-byte rows); every product with a lo plane drops out.
// VH: full-precision rows in memory, but only the hi halves of the mean VALUES are brought in: one tensor copy per
// tile takes the first 256 bytes of each 512-byte row, and the value product is that of HS (Sec. 3.1: the
// compensation term is an average over many blocks; its rounding, at most half a bf16 step per block and of varying sign, is within that of the
// bf16 output).
template <int G, typename QT, bool RD, bool HS, bool VH>
__global__ void __launch_bounds__(kThreads, 1)
ckv_scan_kernel(CkvDev P, const QT *q, const int *seq_lens, int units, int stages, CkvNewToken fresh,
                int n_tail, const __grid_constant__ CUtensorMap tm_v) {
  constexpr bool QS = QSplit<QT>::value;   // fp32 queries are split into hi + lo like the summaries
  static_assert(!(VH && (HS || RD)), "VH is a variant of the full-precision layout with four variance groups");
  constexpr int kRowBytes = HS ? CKV_D * 2 : CKV_ROW_ELEMS * 2;   // bytes of one mean-key row in a stage
  constexpr int kRowBytesV = (HS || VH) ? CKV_D * 2 : CKV_ROW_ELEMS * 2;   // ... of one mean-value row
  constexpr int TB = ScanTile<HS || VH>::TB;
  extern __shared__ __align__(128) unsigned char stage_mem[];
  __shared__ __align__(8) uint64_t full_bar[2][kMaxStages], empty_bar[kMaxStages];
  __shared__ __align__(512) unsigned char s_zero_row[512];   // what mean-value rows past a unit's last block are read as
  __shared__ int s_u0, s_tl0, s_count, s_ulast, s_abort, s_issued;
  __shared__ int s_len[kMaxSeqs];
  // Query rows and variance weights of the first kStagedUnits units of this CTA's range (a CTA's range rarely
  // spans more than two), staged by the consumer warps while the first fills are on their way: a warp that moves
  // on to another unit then sets up from shared memory instead of paying a round trip to global memory.
  constexpr int kStagedUnits = 4;
  constexpr int kQStride = CKV_D + 8;   // (eight rows' matrix loads hit eight bank groups)
  __shared__ __align__(16) __nv_bfloat16 s_q[kStagedUnits][G][kQStride];
  __shared__ float s_w[kStagedUnits][G][4];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool r4 = P.r == 4;          // the default: the variance projection is four FMAs on one 16-byte read
  const bool dbar_bulk = P.r >= 4;   // smaller rows cannot keep the 16-byte alignment bulk copies need
  constexpr int kParts = TB / 16;    // 16-block parts of a tile, each worked on by one consumer warp
  const int stage_bytes = TB * (kRowBytes + kRowBytesV) + (dbar_bulk ? TB * P.r * 4 : 0);
  // per-warp w_{g,t} table for r != 4, behind the ring
  float *sw_all = reinterpret_cast<float *>(stage_mem + (size_t)stages * stage_bytes);

  // the sequence lengths are requested first; the ring is cleared while they are on their way
  const int batch = ckv_div_hkv(P, units);
  const bool append = fresh.k_new != nullptr;
  const int cap = P.max_blocks * P.bs;
  // length the step works on: one more than stored when a token is being appended (a full sequence keeps its length)
  auto eff_len = [&](int raw) { return max(min(raw + ((append && raw >= 0 && raw < cap) ? 1 : 0), cap), 0); };
  pdl_wait();
  const int len_mine = tid < batch ? seq_lens[tid] : 0;
  if ((int)blockIdx.x < n_tail) {
    // ---------------- tail CTAs: the new token and the last block of every unit ----------------
    scan_tail<G, QT>(P, q, seq_lens, s_len, len_mine, units, (int)gridDim.x - n_tail, fresh, n_tail,
                     reinterpret_cast<float *>(stage_mem), stages * stage_bytes);
    if (append) lens_arrive(P.status + kLenCounter, seq_lens, fresh.seq_lens, batch, cap, (int)gridDim.x, /*whole_cta=*/true);
    return;
  }
  const int bid = (int)blockIdx.x - n_tail, nscan = (int)gridDim.x - n_tail;   // this CTA among the scan CTAs
  // rows of a stage past a unit's last block are never copied and the ring is never cleared: the products over
  // blocks read such mean-value rows from a row of zeros instead (a stale NaN pattern times a zero weight would
  // poison the accumulators); everywhere else a block is an output column, and those columns are discarded
  if (tid < 32) reinterpret_cast<uint4 *>(s_zero_row)[tid] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {   // also done while the lengths are on their way: the barriers of the ring
    for (int st = 0; st < stages; ++st) { mbar_init(&full_bar[0][st], 1); mbar_init(&full_bar[1][st], 1); mbar_init(&empty_bar[st], kParts); }
    fence_barrier_init();
  }
  if (tid < batch) s_len[tid] = eff_len(len_mine);
  for (int i = tid + kThreads; i < batch && i < kMaxSeqs; i += kThreads) s_len[i] = eff_len(seq_lens[i]);
  __syncthreads();
  if (tid == 0) {
    // this CTA's range of the tiles (a step has fewer than 2^24 tiles, checked at creation: ckv_udiv24)
    unsigned T = 0;
    for (int i = 0; i < batch; ++i) T += (unsigned)seq_tiles(s_len, seq_lens, P, i) * (unsigned)P.Hkv;
    const unsigned tpc = ckv_udiv24(T + (unsigned)nscan - 1u, (unsigned)nscan);
    const unsigned first = (unsigned)bid * tpc;
    const unsigned cnt = first >= T ? 0u : min(T - first, tpc);
    int u0 = 0, tl0 = 0, ulast = 0;
    if (cnt > 0) {
      unsigned accum = 0;
      bool have_first = false;
      for (int i = 0; i < batch; ++i) {
        const unsigned t = (unsigned)seq_tiles(s_len, seq_lens, P, i);
        if (t > 0) {
          if (!have_first && first < accum + t * (unsigned)P.Hkv) {
            const unsigned off = first - accum;
            const unsigned oq = ckv_udiv24(off, t);
            u0 = i * P.Hkv + (int)oq; tl0 = (int)(off - oq * t);
            have_first = true;
          }
          if (first + cnt - 1u < accum + t * (unsigned)P.Hkv) {
            ulast = i * P.Hkv + (int)ckv_udiv24(first + cnt - 1u - accum, t);
            break;
          }
        }
        accum += t * (unsigned)P.Hkv;
      }
    }
    s_u0 = u0; s_tl0 = tl0; s_ulast = ulast; s_count = (int)cnt; s_abort = 0; s_issued = 0;
  }
  __syncthreads();
  const int count = s_count;
  // Every length this CTA needs is in shared memory now: one thread says so (the last CTA of the grid to say it
  // stores the new lengths).  It is a spare lane of the producer warp, in the same if/else as the producer, so
  // that nobody waits for its round trip.
  if (count == 0) {   // uniform: this CTA has no tiles
    if (append && tid == kThreads - 1) lens_arrive(P.status + kLenCounter, seq_lens, fresh.seq_lens, batch, cap, (int)gridDim.x, false);
    return;
  }

  if (warp == kConsumerWarps) {
    // ---------------- producer: one thread streams the CTA's tiles into the ring ----------------
    if (lane == 0) {
      int u = s_u0, tl = s_tl0, st = 0;
      uint32_t phase = 0;            // parity of the empty-barrier phase the next refill of stage `st` waits for
      uint32_t round = 0;            // times the ring has wrapped: fill `it` uses the full barrier [round & 1][st]
      UnitInfo ui = unit_info(P, s_len, seq_lens, u);
      for (int it = 0; it < count; ++it) {
        if (it >= stages && !mbar_wait(&empty_bar[st], phase, P.spin_limit)) {
          atomicOr(P.status, CKV_DEV_TIMEOUT);
          *(volatile int *)&s_abort = 1;
        }
        if (*(volatile int *)&s_abort) break;
        const int b0 = tl * TB;
        const int nb = min(TB, ui.X - b0);
        const size_t row = (size_t)u * P.max_blocks + b0;
        unsigned char *sk = stage_mem + (size_t)st * stage_bytes;
        unsigned char *sv = sk + TB * kRowBytes;
        const uint32_t kbytes = (uint32_t)nb * kRowBytes;
        const uint32_t dbytes = dbar_bulk ? (uint32_t)nb * P.r * 4 : 0;
        uint64_t *fb = &full_bar[round & 1][st];
        const uint32_t vbytes = VH ? (uint32_t)TB * kRowBytesV : kbytes;   // a tensor copy always delivers its whole box
        mbar_arrive_expect_tx(fb, kbytes + vbytes + dbytes);
        const uint32_t lo = smem_u32(stage_mem), hi = lo + (uint32_t)stages * stage_bytes;
        bool ok = nb >= 1 && u < units && row + nb <= (size_t)units * P.max_blocks;
        // test hook (ckv_debug_set): one fill is announced but never issued, so that the waits on it run out
        const bool skip = (P.debug & CKV_DEBUG_SKIP_FILL) != 0 && it == 0 && bid == 0;
        if (!skip) {
          ok = ok && bulk_g2s_checked(sk, P.kmean + row * P.row_elems, kbytes, fb, lo, hi);
          if constexpr (VH) {
            // rows [row, row + TB) of the mean-values region, first 256 bytes of each (rows past the unit's blocks are
            // never read; rows past the region's end arrive as zeros)
            const uint32_t dv = smem_u32(sv);
            const bool fits = (dv & 127u) == 0 && dv >= lo && dv + vbytes <= hi;
            if (ok && fits) tensor_g2s(dv, &tm_v, 0, (int)row, fb);
            ok = ok && fits;
          } else {
            ok = ok && bulk_g2s_checked(sv, P.vmean + row * P.row_elems, kbytes, fb, lo, hi);
          }
          if (dbar_bulk) ok = ok && bulk_g2s_checked(sv + TB * kRowBytesV, P.dbar + row * P.r, dbytes, fb, lo, hi);
          *(volatile int *)&s_issued = it + 1;
        }
        if (!ok) atomicOr(P.status, CKV_DEV_BAD_COPY);
        if (++st == stages) { st = 0; ++round; if (it >= stages) phase ^= 1; }
        if (++tl == ui.tiles) {
          tl = 0;
          do { ++u; } while (u < units && (ui = unit_info(P, s_len, seq_lens, u)).tiles == 0);
        }
      }
    } else if (append && lane == 31) {
      lens_arrive(P.status + kLenCounter, seq_lens, fresh.seq_lens, batch, cap, (int)gridDim.x, false);
    }
  } else {
    // ---------------- consumer warps: half tile j = warp, warp + 8, ... of the CTA's range ----------------
    using T = HeadTile<G>;   // which heads a lane works on
    const bool staged = !QS && !RD && P.r == 4;   // bf16 queries, four variance groups: the staged setup below
    if (staged) {
      constexpr int kPieces = G * CKV_D * 2 / 16;   // 16-byte pieces of a unit's G query rows
      for (int idx = tid; idx < kStagedUnits * kPieces; idx += kConsumerWarps * 32) {
        const int k = idx / kPieces, pc = idx % kPieces, uu = s_u0 + k;
        if (uu <= s_ulast && uu < units) {
          const int s2 = ckv_div_hkv(P, uu), h2 = uu - s2 * P.Hkv;
          const uint4 *src = reinterpret_cast<const uint4 *>(q + ((size_t)s2 * P.Hq + h2 * G) * CKV_D);
          *reinterpret_cast<uint4 *>(&s_q[k][pc >> 4][8 * (pc & 15)]) = src[pc];
        }
      }
      named_barrier(1, kConsumerWarps * 32);
      // w_{g,t} of Eq. 8: sums of squared query coordinates per variance group, times the squared logit scale
      for (int idx = tid; idx < kStagedUnits * G * 4; idx += kConsumerWarps * 32) {
        const int k = idx / (G * 4), g = (idx / 4) % G, t = idx % 4;
        if (s_u0 + k <= s_ulast) {
          float w = 0.f;
#pragma unroll
          for (int i = 0; i < CKV_D / 4; i += 8) {   // the group's 32 coordinates: one run, or two runs of 16
            const int c = P.glayout == 0 ? 32 * t + i : (i < 16 ? 16 * t + i : CKV_D / 2 + 16 * t + (i - 16));
            float x[8];
            load8<false>(&s_q[k][g][c], x);
#pragma unroll
            for (int j = 0; j < 8; ++j) w = fmaf(x[j], x[j], w);
          }
          s_w[k][g][t] = w * (P.scale * P.scale);
        }
      }
      named_barrier(1, kConsumerWarps * 32);
    }
    ScanUnit<G, QT, RD> w;
    w.reset();
    float *sw = sw_all + (size_t)warp * P.r * G;   // [t][g], r != 4 only
    const ScanPartCfg cfg{P.scale, P.half_var, logf((float)P.bs), P.r, P.max_blocks,
                          (P.variant & CKV_VARIANT_RANK_BY_MASS) != 0, r4};
    float log_last = 0.f;   // log of the token count of the unit's last block, when the scan CTAs cover it
    const int ulast = s_ulast;
    int u = s_u0, tl = s_tl0, cur = -1, next_empty = s_u0;
    UnitInfo ui = unit_info(P, s_len, seq_lens, u);
    float *lu = nullptr, *lz = nullptr;
    const float *db = nullptr;
    bool aborted = false;

    auto write_partial = [&](int unit_id, bool real) {
      float *part = P.comp_part + ((size_t)(bid + 2 * unit_id) * kConsumerWarps + warp) * G * CKV_PART_STRIDE;
      if (!real) {
        if (lane < G) {
          part[lane * CKV_PART_STRIDE] = -CUDART_INF_F;
          part[lane * CKV_PART_STRIDE + 1] = 0.f;
          part[lane * CKV_PART_STRIDE + 2] = 0.f;
        }
        return;
      }
      w.fold(lane, [&](int g, int c, float v) { part[g * CKV_PART_STRIDE + 4 + c] = v; });
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float l = T::sum_rows(w.l[e]), lp = T::sum_rows(w.lp[e]);
        if (T::owns(lane, e)) {
          float *pg = part + T::head(lane, e) * CKV_PART_STRIDE;
          pg[0] = w.m[e]; pg[1] = l; pg[2] = lp;
        }
      }
    };
    // units of this CTA's range that this warp never worked on still need an (empty) partial
    auto fill_empty_upto = [&](int upto) {
      for (; next_empty < upto; ++next_empty)
        if (unit_info(P, s_len, seq_lens, next_empty).tiles > 0) write_partial(next_empty, false);
    };

    // Part j = kParts * tile + part-of-tile belongs to warp j % W, and a warp visits only the tiles that hold one
    // of its parts: it waits for the tile's fill, works on its part and releases the stage; a stage is refilled
    // once the kParts owners of its parts have released it.  A warp's next part is at most W parts (four tiles)
    // ahead, and fill f is only issued after fill f - stages has landed and been released, so the stage a warp
    // waits on is at most two fills behind the one it wants.  A parity wait can only tell a fill from the one
    // before it, hence the two sets of full barriers used by alternate rounds of the ring: together they tell four
    // consecutive fills of a stage apart.
    int it_at = 0;   // tile the (u, tl) walk stands at
    uint32_t round = 0;   // the tile's place in the ring, kept by stepping (a division per visit would be two dozen instructions)
    int st = 0;
    for (int pidx = warp; pidx < kParts * count; pidx += kConsumerWarps) {
      const int it = pidx / kParts;
      int half = pidx - it * kParts;
      st += it - it_at;
      while (st >= stages) { st -= stages; ++round; }
      for (; it_at < it; ++it_at) {
        if (++tl == ui.tiles) {
          tl = 0;
          do { ++u; } while (u < units && (ui = unit_info(P, s_len, seq_lens, u)).tiles == 0);
        }
      }
      // a wait that runs out marks the step invalid (`aborted`); the walk still runs to the end
      if (!aborted) {
        bool fail = *(volatile int *)&s_abort != 0;
        if (!fail && !mbar_wait(&full_bar[round & 1][st], (round >> 1) & 1, P.spin_limit)) {
          atomicOr(P.status, CKV_DEV_TIMEOUT);
          *(volatile int *)&s_abort = 1;
          fail = true;
        }
        aborted = __any_sync(0xffffffffu, fail);
      }
      if (half >= 0) {
      if (u != cur) {
        if (cur >= 0) { write_partial(cur, true); next_empty = cur + 1; }
        fill_empty_upto(u);
        // per-unit setup: query fragments, variance weights, fresh accumulators
        const int s = ckv_div_hkv(P, u), h = u - s * P.Hkv;
        const QT *qrow = q + ((size_t)s * P.Hq + h * G) * CKV_D;
        const int uk = u - s_u0;
        const bool from_smem = staged && uk < kStagedUnits;
        if (from_smem) {
          if constexpr (!QS) w.load_queries(lane, P.scale, smem_u32(&s_q[uk][0][0]), kQStride * 2, smem_u32(s_zero_row));
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int t = 0; t < 4; ++t) w.wown[e][t] = T::head(lane, e) < G ? s_w[uk][T::head(lane, e) & (G - 1)][t] : 0.f;
        } else {
          w.set_queries(lane, P.scale, [&](int g, int c) {
            return make_float2(to_float(qrow[(size_t)g * CKV_D + c]), to_float(qrow[(size_t)g * CKV_D + c + 1]));
          });
        }
        if (from_smem) {
          // set up above
        } else if (RD) {
          // nothing to tabulate: the weights are the squared queries held above
        } else if (r4) {
          // w_{g,t} for this lane's heads: every lane that works on a head sums all 128 coordinates (once per unit)
#pragma unroll 1
          for (int e = 0; e < 2; ++e) {
            float wsum[4] = {0.f, 0.f, 0.f, 0.f};
            const QT *qrow_e = qrow + (size_t)(T::head(lane, e) & (G - 1)) * CKV_D;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
              float x[8];
              load8<false>(qrow_e + 8 * c, x);
              float s8 = 0.f;
#pragma unroll
              for (int i = 0; i < 8; ++i) s8 = fmaf(x[i], x[i], s8);
              // an aligned run of 8 coordinates lies in one group for r = 4 (groups are runs of 32 or 16)
              const int t = P.glayout == 0 ? (8 * c) / 32 : ((8 * c) % 64) / 16;
              wsum[0] += t == 0 ? s8 : 0.f; wsum[1] += t == 1 ? s8 : 0.f;
              wsum[2] += t == 2 ? s8 : 0.f; wsum[3] += t == 3 ? s8 : 0.f;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {   // Eq. 8's 1/d is the squared logit scale
              if (e == 0) w.wown[0][t] = wsum[t] * (P.scale * P.scale); else w.wown[1][t] = wsum[t] * (P.scale * P.scale);
            }
          }
        } else {
          __syncwarp();
          for (int idx = lane; idx < P.r * G; idx += 32) {
            const int t = idx / G, g = idx % G;
            const QT *qg = q + ((size_t)s * P.Hq + h * G + g) * CKV_D;
            float ws = 0.f;
            for (int i = 0; i < CKV_D; ++i)
              if (group_of(i, P.r, P.glayout) == t) { const float x = to_float(qg[i]); ws = fmaf(x, x, ws); }
            sw[idx] = ws * (P.scale * P.scale);
          }
          __syncwarp();
        }
        w.reset();
        log_last = logf((float)(ui.N - (ui.X - 1) * P.bs));
        const size_t row0 = (size_t)u * P.max_blocks;
        lu = P.lu + row0 * G;   // [head][block] within the unit
        lz = P.lz + row0 * G;
        db = P.dbar + row0 * P.r;
        cur = u;
      }
      const int b0 = tl * TB;
      const int nb = min(TB, ui.X - b0);
      const int rb = half * 16;          // first row of this warp's half tile
      if (!aborted && rb < nb) {
        const uint32_t sk = smem_u32(stage_mem + (size_t)st * stage_bytes);
        const uint32_t sv = sk + TB * kRowBytes;
        const float *sd = reinterpret_cast<const float *>(stage_mem + (size_t)st * stage_bytes + TB * (kRowBytes + kRowBytesV));

        scan_part<G, QT, RD, HS, VH>(
            w, cfg, sk, sv, (RD || r4 || dbar_bulk) ? sd : nullptr, smem_u32(s_zero_row), sw, db, lane, rb, nb, b0,
            P.tail ? -1 : ui.X - 1, log_last,   // in tail mode every block here is full
            [&](int g, int blk, float x, float y) {
              const size_t o = (size_t)g * P.max_blocks + blk;
              lu[o] = x;
              lz[o] = y;
            });
      }
      }   // own part
      __syncwarp();
      if (lane == 0 && !aborted) mbar_arrive(&empty_bar[st]);
    }
    if (cur >= 0) { write_partial(cur, true); next_empty = cur + 1; }
    fill_empty_upto(ulast + 1);
  }
  __syncthreads();
  if (s_abort && tid == 0) {
    // leave no bulk copy in flight into this CTA's shared memory: wait (bounded) for every issued fill
    // (a completed phase is seen as complete again, so waiting on consumed stages returns at once)
    const int issued = s_issued;
    for (int it = max(issued - stages, 0); it < issued; ++it)
      mbar_wait(&full_bar[(it / stages) & 1][it % stages], ((it / stages) >> 1) & 1, P.spin_limit);
  }
}

struct ScanCfg { int stages; size_t smem; };

ScanCfg scan_cfg(const CkvDev &P, int G) {
  const size_t TB = (size_t)P.scan_tile;
  const size_t krow = (size_t)P.row_elems * 2, vrow = P.vhi ? (size_t)CKV_D * 2 : krow;
  const size_t stage_bytes = TB * (krow + vrow) + (P.r >= 4 ? TB * P.r * 4 : 0);
  const size_t sw_bytes = (P.r == 4 || P.r == CKV_D) ? 0 : (size_t)kConsumerWarps * P.r * G * 4;   // weight table of the generic path
  // 227 KB per CTA, less the kernel's static shared memory (lengths, barriers, the row of zeros: under 6 KB; staged
  // query rows and variance weights: 4 units x G x 288 bytes) and a reserve
  const size_t stat = 6 * 1024 + (size_t)4 * G * (CKV_D * 2 + 32);
  const size_t budget = 227 * 1024 - stat - 1024 - sw_bytes;
  int stages = (int)(budget / stage_bytes);
  if (stages > kMaxStages) stages = kMaxStages;
  // A consumer warp's next part is at most kConsumerWarps parts ahead of its last one; the ring protocol needs
  // that distance, in tiles, to be no more than the number of stages (see the consumer loop).
  const int parts = (int)TB / 16;
  const int need = (kConsumerWarps + parts - 1) / parts;
  if (stages < need) stages = 0;   // refused by the launcher (no layout reaches this on a 227 KB part)
  return ScanCfg{stages, stages * stage_bytes + sw_bytes};
}

template <int G, typename QT>
cudaError_t launch_gt(ckv_ctx *c, const void *q, const int *seq_lens, int units, int grid, const CkvNewToken &fresh,
                      int n_tail, cudaStream_t st) {
  const ScanCfg cfg = scan_cfg(c->dev, G);
  if (cfg.stages == 0) return cudaErrorInvalidConfiguration;
  if (c->dev.r == CKV_D)
    return ckv_launch_pdl(ckv_scan_kernel<G, QT, true, false, false>, dim3(grid), dim3(kThreads), cfg.smem, st, 0, c->dev, (const QT *)q, seq_lens, units, cfg.stages, fresh, n_tail, c->tm_vhi);
  else if (c->dev.row_elems == CKV_D) {
    if constexpr (!QSplit<QT>::value)   // bf16 summaries come with bf16 pages and queries only
      return ckv_launch_pdl(ckv_scan_kernel<G, QT, false, true, false>, dim3(grid), dim3(kThreads), cfg.smem, st, 0, c->dev, (const QT *)q, seq_lens, units, cfg.stages, fresh, n_tail, c->tm_vhi);
    else
      return cudaErrorInvalidValue;
  } else if (c->dev.vhi) {
    if constexpr (!QSplit<QT>::value)
      return ckv_launch_pdl(ckv_scan_kernel<G, QT, false, false, true>, dim3(grid), dim3(kThreads), cfg.smem, st, 0, c->dev, (const QT *)q, seq_lens, units, cfg.stages, fresh, n_tail, c->tm_vhi);
    else
      return cudaErrorInvalidValue;
  } else
    return ckv_launch_pdl(ckv_scan_kernel<G, QT, false, false, false>, dim3(grid), dim3(kThreads), cfg.smem, st, 0, c->dev, (const QT *)q, seq_lens, units, cfg.stages, fresh, n_tail, c->tm_vhi);
}

template <int G>
cudaError_t launch_g(ckv_ctx *c, const void *q, const int *seq_lens, int units, int grid, const CkvNewToken &fresh,
                     int n_tail, cudaStream_t st) {
  if (c->layout.kv_dtype == CKV_BF16) return launch_gt<G, __nv_bfloat16>(c, q, seq_lens, units, grid, fresh, n_tail, st);
  return launch_gt<G, float>(c, q, seq_lens, units, grid, fresh, n_tail, st);
}

template <int G, typename QT>
cudaError_t configure_gt(const ckv_ctx *c) {
  const int smem = (int)scan_cfg(c->dev, G).smem;
  if (c->dev.r == CKV_D)
    return cudaFuncSetAttribute(ckv_scan_kernel<G, QT, true, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (c->dev.row_elems == CKV_D) {
    if constexpr (!QSplit<QT>::value)
      return cudaFuncSetAttribute(ckv_scan_kernel<G, QT, false, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return cudaErrorInvalidValue;
  }
  if (c->dev.vhi) {
    if constexpr (!QSplit<QT>::value)
      return cudaFuncSetAttribute(ckv_scan_kernel<G, QT, false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return cudaErrorInvalidValue;
  }
  return cudaFuncSetAttribute(ckv_scan_kernel<G, QT, false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

// The mean-values region as the copy engine sees it with vhi: a matrix of bf16 rows, [units * max_blocks][128] at a pitch
// of 512 bytes (the hi halves of the stored rows), copied in boxes of CKV_SCAN_TILE_HS rows.  Host-side arithmetic only;
// the encoder is the driver's, looked up once through the runtime.
cudaError_t make_vhi_map(ckv_ctx *c) {
  using encode_fn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                 const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static std::mutex mtx;
  static encode_fn encode = nullptr;
  {
    std::lock_guard<std::mutex> lock(mtx);
    if (encode == nullptr) {
      void *fn = nullptr;
      cudaDriverEntryPointQueryResult qres = cudaDriverEntryPointSymbolNotFound;
      const cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
      if (e != cudaSuccess) return e;
      if (qres != cudaDriverEntryPointSuccess || fn == nullptr) return cudaErrorSymbolNotFound;
      encode = reinterpret_cast<encode_fn>(fn);
    }
  }
  const CkvDev &P = c->dev;
  if (((uintptr_t)P.vmean & 15u) != 0) return cudaErrorMisalignedAddress;
  const cuuint64_t dims[2] = {(cuuint64_t)CKV_D, (cuuint64_t)c->layout.max_batch * P.Hkv * P.max_blocks};
  const cuuint64_t strides[1] = {(cuuint64_t)CKV_ROW_ELEMS * 2};   // bytes between rows
  const cuuint32_t box[2] = {CKV_D, CKV_SCAN_TILE_HS};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode(&c->tm_vhi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)P.vmean, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int G>
cudaError_t configure_g(ckv_ctx *c) {
  if (c->dev.vhi) {
    const cudaError_t e = make_vhi_map(c);
    if (e != cudaSuccess) return e;
  }
  if (c->layout.kv_dtype == CKV_BF16) return configure_gt<G, __nv_bfloat16>(c);
  return configure_gt<G, float>(c);
}

}  // namespace

// Opt in to the dynamic shared memory this context's scan instantiation needs, on the current device.
cudaError_t ckv_configure_scan(ckv_ctx *c) {
  switch (c->dev.G) {
    case 1: return configure_g<1>(c);
    case 2: return configure_g<2>(c);
    case 4: return configure_g<4>(c);
    case 8: return configure_g<8>(c);
  }
  return cudaErrorInvalidValue;
}

namespace {
// Tail CTAs of a launch: 8 warps each, one unit per warp and round.  One round is the goal: a warp's work is a chain
// of three or four dependent cache misses, each of which costs several microseconds once the scan CTAs have
// saturated DRAM (two rounds for 32 units made the whole step 7 us slower than one).
int tail_ctas(const ckv_ctx *c, int batch) {
  if (!c->dev.tail) return 0;
  const int units = batch * c->dev.Hkv;
  const int one_round = (units + 7) / 8;
  if (one_round <= 16) return std::max(1, one_round);
  return std::min((units + 15) / 16, std::max(16, c->sm_count / 4));   // many units: two rounds, at most a quarter of the SMs
}
}  // namespace

// Scan CTAs of a step: one persistent CTA per SM the tail CTAs leave free, never more CTAs than tiles.
int ckv_scan_grid(const ckv_ctx *c, int batch, int max_len) {
  const CkvDev &P = c->dev;
  const int xmax = std::max((max_len + P.bs - 1) / P.bs - P.tail, 0);   // in tail mode the last block is the tail CTAs'
  const long long tiles = (long long)batch * P.Hkv * ((xmax + P.scan_tile - 1) / P.scan_tile);
  long long grid = c->sm_count - tail_ctas(c, batch);
  if (grid > CKV_MAX_SCAN_CTAS) grid = CKV_MAX_SCAN_CTAS;
  if (grid > tiles) grid = tiles;
  return (int)(grid < 1 ? 1 : grid);
}

// Tail mode pays when the scan is long enough to hide the tail CTAs.  A tail warp's work is a chain of dependent
// cache misses behind the scan's traffic plus a few thousand instructions run once by a single warp: measured from
// launch, a round of tail work ends after 15 - 20 us without a new token and after 20 - 25 us with one (45 us before
// the routine's cold instructions were trimmed), whereas the scan streams about 5 MB per microsecond.  Below that
// size the scan CTAs cover every block and the append is a launch of its own, whose warps all run at once.
bool ckv_scan_wants_tail(const ckv_ctx *c, int batch, int max_len) {
  if (batch > kMaxSeqs || c->tail_mode == CKV_TAIL_OFF) return false;   // the lengths must fit the staging array
  if (c->tail_mode == CKV_TAIL_ON) return true;
  const CkvDev &P = c->dev;
  const int units = batch * P.Hkv;
  const int one_round = (units + 7) / 8;
  const int n_tail = one_round <= 16 ? std::max(1, one_round) : std::min((units + 15) / 16, std::max(16, c->sm_count / 4));
  const int rounds = (units + 8 * n_tail - 1) / (8 * n_tail);
  const double blocks = (double)units * ((max_len + P.bs - 1) / P.bs);
  const double bytes = blocks * (P.row_elems * 2.0 + (P.vhi ? CKV_D * 2.0 : P.row_elems * 2.0) + 4.0 * P.r);   // what the scan reads
  // scan microseconds: bandwidth-bound at about 5 MB/us, or issue-bound at about 6000 blocks/us (bf16 summaries).
  // A round of tail work with a new token ends 20 - 25 us after launch; measured crossover at 128K, 8 KV heads: three
  // sequences (scan about 30 us) gain a microsecond from tail mode, two (about 20 us) lose four.
  const double scan_us = std::max(bytes / 5.0e6, blocks / 6.0e3);
  return scan_us >= 30.0 * rounds;
}

cudaError_t ckv_launch_scan(ckv_ctx *c, const void *q, const int *seq_lens, int batch, int max_len,
                            const CkvNewToken *fresh_in, int *grid_out, cudaStream_t st) {
  const CkvDev &P = c->dev;
  const int units = batch * P.Hkv;
  const int n_scan = ckv_scan_grid(c, batch, max_len), n_tail = tail_ctas(c, batch);
  const int grid = n_tail + n_scan;
  CkvNewToken fresh = {};
  if (fresh_in != nullptr) {
    if (!P.tail || batch > kMaxSeqs) return cudaErrorInvalidValue;   // the new token is the tail CTAs' job
    fresh = *fresh_in;
  }
  *grid_out = n_scan;
  c->launches++;
  switch (P.G) {
    case 1: return launch_g<1>(c, q, seq_lens, units, grid, fresh, n_tail, st);
    case 2: return launch_g<2>(c, q, seq_lens, units, grid, fresh, n_tail, st);
    case 4: return launch_g<4>(c, q, seq_lens, units, grid, fresh, n_tail, st);
    case 8: return launch_g<8>(c, q, seq_lens, units, grid, fresh, n_tail, st);
  }
  return cudaErrorInvalidValue;
}
