// One decode step (append, scan, selection, attention, merge: Eq. 8-12) in ONE launch: a thread-block cluster per unit.
//
// A step of a few sequences is bound by latency, not by bytes: as four launches (append, scan, select, attention) the
// 32K single-sequence step spends 28 us in kernels that move 17 MB and 7 us between them, every stage paying its own
// launch, its own cold start and a trip of its results through global memory.  The units of a step are independent, so
// one cluster can take a unit from the new token to the output row: its CTAs share out the unit's blocks, exchange the
// little that crosses blocks (normalisers, block scores, partial outputs) through distributed shared memory, and
// nothing waits for another unit.  A cluster barrier costs 0.1 us here, a launch about 2 us.
//
// CTA `rank` of the cluster owns a contiguous range of the unit's blocks (all but the last one), in 16-block parts:
//   1. scan: a producer warp streams the range's summaries into a ring of shared-memory stages (its lanes issue the first
//      round, one of them the rest, and the first tile, at a guess, before the length is known), eight warps work on
//      parts (scan_part, shared with the persistent scan kernel); the score terms stay in shared memory.  Meanwhile two
//      warps of the last CTA append the new token, redo the last block's summary and compute its terms.
//   2. every CTA sends its normaliser partials (M_g, L_g) to all, then the block scores of its own range: every CTA holds
//      all scores of the unit.  Both exchanges are asynchronous stores counted on an mbarrier of the receiver: a cluster
//      barrier with release semantics would wait for the scan's stores to global memory as well (1.4 us instead of 0.6).
//   3. selection, redundantly in every CTA, a thread's scores in registers throughout: a histogram over the scores' bit
//      patterns relative to an upper bound of them (64 bins per octave, 32 octaves), the exact cut by ranking the one bin that
//      holds it (digit by digit when that bin is crowded or the cut lies below the histogram), a word of bits per thread for
//      its blocks that are in, and their ids in position order from a prefix sum.  All CTAs get the same list without another
//      exchange.  32 units of 8192 blocks: 4.2 us from the scores to the ids (6.2 with two passes over shared memory and a bit
//      map put together by shuffles and atomics), 8 units of 2048: 2.6 (3.2).
//   4. exact attention over the CTA's share of the list, a warp per page, into the SAME accumulators that hold the
//      compensation sums of step 1 (both are online-softmax sums over the same heads); the selected blocks' mean terms
//      are taken out through the tokens' weights, or with bf16 summaries as one more product over the stored rows.
//   5. the CTA's partial is reduced over its warps and sent to the CTAs that reduce it over the cluster; output.
//
// The cluster size follows from what the device can hold at once (the number of co-resident clusters by size is asked
// of the driver when a context is created): the largest size for which all units run in one wave.  72 SMs already
// stream at the full HBM rate (206 MB: 6.28 TB/s with 72, 96, 120 or 148 CTAs alike), so 8 units in clusters of 10 lose
// nothing against 148 CTAs.
#include <algorithm>
#include <mutex>

#include "ckv_internal.cuh"
#include "ckv_pipe.cuh"
#include "ckv_mma.cuh"
#include "ckv_cluster.cuh"
#include "ckv_blockstats.cuh"
#include "ckv_scanpart.cuh"
#include "ckv_attnpage.cuh"

namespace {

using namespace ckv_pipe;
using bf16 = __nv_bfloat16;

constexpr int kWarps = 8;                       // warps that work on parts and pages
constexpr int kWork = kWarps * 32;              // ... and their threads
constexpr int kProducerWarp = kWarps, kTailWarp = kWarps + 1, kValueWarp = kWarps + 2;
constexpr int kThreads = (kWarps + 3) * 32;
constexpr int kClusterCap = CKV_STEP_MAX_CLUSTER;
constexpr int kStagesCap = 6;
constexpr int kMinRing = 3;                     // ring stages that the score terms have to leave room for
constexpr int kScoresCap = 9216;                // blocks of a unit whose scores every CTA can hold (147K tokens in 16-token blocks; the bit
                                                // map and the memory would take 16384, longer units have not been tried)
constexpr int kBins = 2048;                     // score histogram: 32 octaves below the largest possible score, 64 bins each
constexpr int kBinShift = 17;                   // ... a bin is a score's bit pattern without its low 17 bits
constexpr int kIdMask = (1 << (31 - kBinShift)) - 1;   // block ids beside those 17 bits in one word
static_assert(kScoresCap <= kIdMask + 1, "block ids fit");
constexpr int kKeyGroups = kScoresCap / 4 / kWork;   // four scores each, as a thread holds them for the selection (a whole number: none of a thread's lies past the array)
static_assert(kKeyGroups * 4 * kWork == kScoresCap && kKeyGroups % 2 == 1, "see the selection");
constexpr int kMapWords = 2 * kWork;            // selection bit map: two words per working thread, enough for kScoresCap blocks
constexpr int kSelCap = 512;                    // selected blocks the id list holds (unless every block is selected)
constexpr int kOwnMost = 2800, kSeqCtas = 24;   // blocks a CTA may own where a sequence gets few CTAs (see ckv_unit_step_plan)
constexpr long long kIdleMost = 80000000;   // bytes: selected keys and values times the share of SMs without a CTA (see ckv_unit_step_plan)
constexpr int kCandCap = kWork;                 // blocks of the cut's bin that are ranked directly, one per thread
// shared memory once the ring is drained
constexpr int kOffHist = kScoresCap * 4;
constexpr int kOffMap = kOffHist + (kBins + 32) * 4;          // (cleared together with the histogram)
constexpr int kOffIds = kOffMap + kMapWords * 4;
constexpr int kOffCand = kOffIds + kSelCap * 4;
constexpr int kOffPages = (kOffCand + kCandCap * 4 + 127) / 128 * 128;
constexpr int kAfterScan = kOffPages + kWarps * 2 * kPageBytes;
constexpr int kRecvStride = 36;                 // floats of one (head, 32 coordinates) partial: values, maximum, weight sum
constexpr int kSmemCta = 227 * 1024;            // shared memory a CTA can have, static and dynamic
constexpr int kDynMost = kSmemCta - 20 * 1024;  // dynamic shared memory, at most (see ckv_configure_unit_step)

// One more in a shared-memory counter.
__device__ __forceinline__ void red_shared_inc(uint32_t addr) { asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr) : "memory"); }

__device__ __forceinline__ void work_barrier() { named_barrier(1, kWork); }

// Exclusive prefix sum of one int per working thread (one barrier; s_wt is not to be reused before the next one).
__device__ __forceinline__ int work_exclusive_scan(int v, int *s_wt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) s_wt[warp] = inc;
  work_barrier();
  int before = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) before += w < warp ? s_wt[w] : 0;
  return before + inc - v;
}
// The cut when the bin that holds it is crowded (many equal or nearly equal scores) or lies below the histogram: the
// kr-th largest ranked key from its digits of 11, 10 and 10 bits, a histogram each, then the equal keys with the lowest
// ids.  Marks what is taken in the map.  All of a unit's scores being equal is the usual reason to come here (8192 equal
// scores: 31.4 us a step, 44.8 with a bisection over the keys' bits).  res: two ints of shared memory.
__device__ __noinline__ void take_by_digits(int X, int kr, const uint32_t *keys, int rank_lo, int rank_n, int *hist, uint32_t *map,
                                            int *s_wt, int *res) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t cut = 0, known = 0;
  int need = kr;
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {
    const int bins = pass == 0 ? kBins : kBins / 2, per = bins / kWork, shift = 20 - 10 * pass;
    for (int i = tid; i < bins / 4; i += kWork) reinterpret_cast<int4 *>(hist)[i] = make_int4(0, 0, 0, 0);
    work_barrier();
#pragma unroll 2
    for (int i = tid; i < (X + 3) / 4; i += kWork) {
      const uint4 k4 = reinterpret_cast<const uint4 *>(keys)[i];
      const uint32_t k[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool in = (unsigned)(4 * i + j - rank_lo) < (unsigned)rank_n && (k[j] & known) == cut;
        atomicAdd(&hist[in ? (k[j] >> shift) & (uint32_t)(bins - 1) : kBins + lane], 1);   // no branch: the rest goes aside
      }
    }
    work_barrier();
    const int top = bins - 1 - tid * per;   // this thread's bins, largest digit first
    int sum = 0;
    for (int j = 0; j < per; ++j) sum += hist[top - j];
    int before = work_exclusive_scan(sum, s_wt);
    if (before < need && before + sum >= need) {
      int j = 0;
      while (before + hist[top - j] < need) before += hist[top - j++];
      res[0] = top - j;
      res[1] = before;
    }
    work_barrier();
    cut |= (uint32_t)res[0] << shift;
    known |= (uint32_t)(bins - 1) << shift;
    need -= res[1];
  }
  work_barrier();
  uint32_t *equal = reinterpret_cast<uint32_t *>(hist);   // bit map of the keys at the cut
  for (int i = (X + 31) / 32 + tid; i < kMapWords; i += kWork) equal[i] = 0;
#pragma unroll 4
  for (int i = warp; i < (X + 31) / 32; i += kWarps) {
    const int b = 32 * i + lane;
    const bool ranked = (unsigned)(b - rank_lo) < (unsigned)rank_n;
    const uint32_t k = keys[min(b, X - 1)];
    const uint32_t above = __ballot_sync(0xffffffffu, ranked && k > cut), at = __ballot_sync(0xffffffffu, ranked && k == cut);
    if (lane == 0) { map[i] |= above; equal[i] = at; }
  }
  work_barrier();
  const uint2 e = reinterpret_cast<const uint2 *>(equal)[tid];
  unsigned long long m = (unsigned long long)e.y << 32 | e.x;
  const int n = __popcll(m), before = work_exclusive_scan(n, s_wt), take = min(max(need - before, 0), n);
  for (int i = take; i < n; ++i) m ^= 1ull << (63 - __clzll((long long)m));   // the highest ids are left
  map[2 * tid] |= (uint32_t)m;
  map[2 * tid + 1] |= (uint32_t)(m >> 32);
}

// What the tail warps' routines take from the kernel's parameters, in shared memory: as arguments by value the two structs
// are copied to the stack (two hundred bytes of stores and loads at the start of the tail's chain).
struct TailArgs { CkvDev P; CkvNewToken fresh; };

// Whether the last block of a sequence of N tokens is shared by two warps: a new token, and one page.
__device__ __forceinline__ bool tail_is_split(const CkvDev &P, bool append, int N) {
  return append && N - ((((N + P.bs - 1) >> P.lg_bs) - 1) << P.lg_bs) <= CKV_PAGE;
}
// The length a step works on, after its append: no longer than the cache, nor than the shared arrays were sized for.
__device__ __forceinline__ int step_length(int raw, bool append, int cap, int most) {
  return min(max(min(raw + ((append && raw >= 0 && raw < cap) ? 1 : 0), cap), 0), most);
}
// The page of position `raw`: lane l of `guess` holds the entry l pages before hi_page, the last one under the host's bound.
__device__ __forceinline__ int tail_page(int guess, const int *pt_row, int hi_page, int raw) {
  const int back = hi_page - raw / CKV_PAGE;
  const int phys = __shfl_sync(0xffffffffu, guess, back & 31);
  return (unsigned)back <= 31u ? phys : pt_row[raw / CKV_PAGE];
}
// The mean value of the last block, weight 1, into the partials of heads g0, g0 + step, ...
template <int G>
__device__ __forceinline__ void tail_store_value(float *tail_part, const float (&x)[8], bool mine, int g0, int step, int li) {
  if (!mine) return;
#pragma unroll
  for (int g = g0; g < G; g += step) {
    *reinterpret_cast<float4 *>(tail_part + g * CKV_PART_STRIDE + 4 + 8 * li) = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4 *>(tail_part + g * CKV_PART_STRIDE + 8 + 8 * li) = make_float4(x[4], x[5], x[6], x[7]);
  }
}

// The last CTA's tail warp: the new token (if there is one) goes into its page and the last block's summary is redone
// with the append's own routine; then, new token or not, the last block's two per-head terms and its compensation
// partial, with plain FMAs, from the summary as stored (a fresh one is taken from the registers it was stored from).
// The cluster waits for this warp, whose time is one chain of dependent loads and cold code: so the routine is entered, and
// its addresses worked out, ahead of the wait for the launch before; every load that depends on nothing is requested first
// (the page-table entry among them: tail_page); the new row is put among the page's other rows in registers instead of being
// read back; a block of one page leaves its value rows to a second warp (tail_values) and its heads to both half warps; and
// the sums of all heads share one tree of shuffles.  us a step of one unit of 4K tokens: 13.0 with one warp that starts when
// the length is known, half its lanes idle at the heads and the two structs as arguments by value; 12.2 with two warps and
// the structs in shared memory; 11.3 entered early.  (Inlined into the kernel the routine is no slower, but the step of 32
// units at 128K then takes 54.7 us instead of 51.5.)
template <int G>
__device__ __noinline__ int tail_block(const TailArgs *args, const bf16 *q_rows, const int *page_table, const int *seq_lens, int unit,
                                       int most, int hi_page, float *sq, float *tail_u, float *tail_part, float4 *norm) {
  const CkvDev P = args->P;
  const CkvNewToken fresh = args->fresh;
  const int lane = threadIdx.x & 31, hw = lane >> 4, li = lane & 15;
  const int s = ckv_div_hkv(P, unit), h = unit - s * P.Hkv;
  const int cap = P.max_blocks * P.bs;
  const bool lo_half = P.row_elems == CKV_ROW_ELEMS;
  const bool by_mass = (P.variant & CKV_VARIANT_RANK_BY_MASS) != 0;
  const int *pt_row = page_table + (size_t)s * P.max_pages_per_seq;
  const bool any = fresh.k_new != nullptr;
  const bf16 *k_new = reinterpret_cast<const bf16 *>(fresh.k_new) + (size_t)unit * CKV_D, *v_new = reinterpret_cast<const bf16 *>(fresh.v_new) + (size_t)unit * CKV_D;
  constexpr int GH = G >= 2 ? G / 2 : 1;   // heads of a half warp
  const int g0 = G >= 2 ? hw * GH : 0;
  pdl_wait();
  const int raw = seq_lens[s], page_guess = any && hi_page >= lane ? pt_row[hi_page - lane] : -1;
  uint4 kn = make_uint4(0u, 0u, 0u, 0u), vn;   // this lane's eight coordinates of the new rows
  if (any) kn = reinterpret_cast<const uint4 *>(k_new)[li];
  uint4 qr[GH];    // ... and of the queries
#pragma unroll
  for (int g = 0; g < GH; ++g) qr[g] = reinterpret_cast<const uint4 *>(q_rows + (size_t)(g0 + g) * CKV_D)[li];
  named_arrive(3, kThreads);   // nothing here needs what the others set up, and the cluster will wait for this warp
  const int N = step_length(raw, any, cap, most);
  if (N == 0) return raw;
  const bool append = any && raw + 1 == N;   // (past the host's bound: see append_past_bound)
  const int phys = append ? tail_page(page_guess, pt_row, hi_page, raw) : -1;
  const int b = ((N + P.bs - 1) >> P.lg_bs) - 1, cnt = N - b * P.bs;
  const bool split = tail_is_split(P, append, N);
  vn = kn;
  if (append && !split) vn = reinterpret_cast<const uint4 *>(v_new)[li];
  const size_t row = (size_t)unit * P.max_blocks + b;
  __nv_bfloat16 *kmean_row = P.kmean + row * P.row_elems, *vmean_row = P.vmean + row * P.row_elems;
  float *dbar_row = P.dbar + row * P.r;
  BlockRow br;
  if (append) {
    bf16 *kp = reinterpret_cast<bf16 *>(fresh.k_pool), *vp = reinterpret_cast<bf16 *>(fresh.v_pool);
    const bool ok = phys >= 0 && phys < P.num_pages;
    const size_t base = ok ? ((size_t)phys * P.Hkv + h) * CKV_PAGE * CKV_D + 8 * li : 0;
    const size_t at = base + (size_t)(raw % CKV_PAGE) * CKV_D;
    if (split) {   // the token's page is all there is of its block
      uint4 kraw[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int t = hw + 2 * j;
        kraw[j] = kn;
        if (ok && t < cnt - 1) kraw[j] = *reinterpret_cast<const uint4 *>(kp + base + (size_t)t * CKV_D);
      }
      if (ok && hw == 0) *reinterpret_cast<uint4 *>(kp + at) = kn;
      float km[8], none[8], ssq[8];
      block_stats_rows16<false, true, false>(kraw, kraw, ok, cnt, lane, km, none, ssq);
      block_stats_finish<true, false>(P, b, (float)cnt, km, none, ssq, sq, kmean_row, dbar_row, vmean_row, lane, !ok, &br);
    } else {
      if (ok) *reinterpret_cast<uint4 *>((hw == 0 ? kp : vp) + at) = hw == 0 ? kn : vn;
      __syncwarp();
      block_stats_warp<bf16, true>(P, kp, vp, pt_row, h, b, cnt, sq, kmean_row, dbar_row, vmean_row, lane, &br);
    }
  } else {   // the summary as stored: lower half warp the mean key, upper the mean value (as the scan reads it)
    if (fresh.k_new != nullptr && raw >= cap && lane == 0) atomicOr(P.status, CKV_DEV_SEQ_FULL);
    load_split8<false>(hw == 0 ? kmean_row : vmean_row, li, b, br.x, lo_half && !(hw == 1 && P.vhi));
    if (P.r == CKV_D) {
      load_split8<false>(reinterpret_cast<const bf16 *>(dbar_row), li, b, br.dvar);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) br.dvar[i] = dbar_row[group_of(8 * li + i, P.r, P.glayout)];
    }
  }
  if (!split) {   // the upper half warp parts with the mean value and takes the mean key, too
    tail_store_value<G>(tail_part, br.x, hw == 1, 0, 1, li);
#pragma unroll
    for (int i = 0; i < 8; ++i) br.x[i] = __shfl_sync(0xffffffffu, br.x[i], li);
  }
  // sums over the 16 lanes of a half warp: d, then sigma^2, of its heads
  float v[2 * GH];
#pragma unroll
  for (int g = 0; g < GH; ++g) {
    float qx[8];
    bf16x8_to_float(qr[g], qx);
    v[g] = v[GH + g] = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      v[g] = fmaf(qx[i], br.x[i], v[g]);
      const float qs = qx[i] * P.scale;
      v[GH + g] = fmaf(qs * qs, br.dvar[i], v[GH + g]);   // Eq. 8: the squared logit scale is its 1/d
    }
  }
  reduce16<2 * GH, 1>(v, li);   // half-warp lane i now holds sum i / (8 / GH)
  const int from = (G >= 2 ? (lane / GH) * 16 : 0) + (lane % GH) * (8 / GH);   // (lanes past G: any)
  const float d = __shfl_sync(0xffffffffu, v[0], from & 31);
  const float sg = fmaxf(__shfl_sync(0xffffffffu, v[0], (from + 8) & 31), 0.f);
  if (lane < G) {
    const float zbar = d * P.scale, logc = logf((float)cnt), zl2 = (zbar + logc) * kLog2e;
    const float u = fmaf(logc + zbar + P.half_var * sg, kLog2e, by_mass ? 0.f : __log2f(sg));
    tail_u[lane] = u;
    P.lz[((size_t)unit * G + lane) * P.max_blocks + b] = zl2;
    norm[lane] = make_float4(zl2, fast_exp2(P.half_var * kLog2e * sg), u, 0.f);
    tail_part[lane * CKV_PART_STRIDE] = zl2;
    tail_part[lane * CKV_PART_STRIDE + 1] = 1.f;
  }
  return raw;
}

// The value rows of a last block that tail_block shares with a second warp: new row into its page, mean value, partial.
template <int G>
__device__ __noinline__ int tail_values(const TailArgs *args, const int *page_table, const int *seq_lens, int unit, int most, int hi_page, float *tail_part) {
  const CkvDev P = args->P;
  const CkvNewToken fresh = args->fresh;
  const int lane = threadIdx.x & 31, hw = lane >> 4, li = lane & 15;
  const int s = ckv_div_hkv(P, unit), h = unit - s * P.Hkv;
  const int *pt_row = page_table + (size_t)s * P.max_pages_per_seq;
  const bool any = fresh.k_new != nullptr;
  pdl_wait();
  const int raw = seq_lens[s], page_guess = any && hi_page >= lane ? pt_row[hi_page - lane] : -1;
  uint4 vn = make_uint4(0u, 0u, 0u, 0u);
  if (any) vn = reinterpret_cast<const uint4 *>(reinterpret_cast<const bf16 *>(fresh.v_new) + (size_t)unit * CKV_D)[li];
  named_arrive(3, kThreads);
  const int N = step_length(raw, any, P.max_blocks * P.bs, most);
  if (!any || N == 0 || raw + 1 != N || !tail_is_split(P, true, N)) return raw;
  const int phys = tail_page(page_guess, pt_row, hi_page, raw);
  const int b = ((N + P.bs - 1) >> P.lg_bs) - 1, cnt = N - b * P.bs;
  bf16 *vp = reinterpret_cast<bf16 *>(fresh.v_pool);
  const bool ok = phys >= 0 && phys < P.num_pages;
  const size_t base = ok ? ((size_t)phys * P.Hkv + h) * CKV_PAGE * CKV_D + 8 * li : 0;
  uint4 vraw[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int t = hw + 2 * j;
    vraw[j] = vn;
    if (ok && t < cnt - 1) vraw[j] = *reinterpret_cast<const uint4 *>(vp + base + (size_t)t * CKV_D);
  }
  if (ok && hw == 0) *reinterpret_cast<uint4 *>(vp + base + (size_t)(raw % CKV_PAGE) * CKV_D) = vn;
  float none[8], vs[8], none2[8];
  block_stats_rows16<false, false, true>(vraw, vraw, ok, cnt, lane, none, vs, none2);
  BlockRow br;
  block_stats_finish<false, true>(P, b, (float)cnt, none, vs, none2, nullptr, nullptr, nullptr,
                                  P.vmean + ((size_t)unit * P.max_blocks + b) * P.row_elems, lane, false, &br);
  tail_store_value<G>(tail_part, br.x, true, hw, 2, li);
  return raw;
}

// The append of a sequence that has outgrown the host's bound: the token lands in a block that the step does not look at,
// whose summary is kept up to date all the same.
__device__ __noinline__ void append_past_bound(const CkvDev P, const int *page_table, const CkvNewToken fresh, int unit, int raw, float *sq) {
  const int lane = threadIdx.x & 31, hw = lane >> 4, li = lane & 15;
  const int s = ckv_div_hkv(P, unit), h = unit - s * P.Hkv;
  const int *pt_row = page_table + (size_t)s * P.max_pages_per_seq;
  bf16 *kp = reinterpret_cast<bf16 *>(fresh.k_pool), *vp = reinterpret_cast<bf16 *>(fresh.v_pool);
  const int phys = pt_row[raw / CKV_PAGE], b = raw >> P.lg_bs;
  if (phys >= 0 && phys < P.num_pages) {
    const bf16 *src = reinterpret_cast<const bf16 *>(hw == 0 ? fresh.k_new : fresh.v_new) + (size_t)unit * CKV_D + 8 * li;
    bf16 *dst = (hw == 0 ? kp : vp) + (((size_t)phys * P.Hkv + h) * CKV_PAGE + raw % CKV_PAGE) * CKV_D + 8 * li;
    *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(src);
  }
  __syncwarp();
  const size_t row = (size_t)unit * P.max_blocks + b;
  block_stats_warp<bf16, true>(P, kp, vp, pt_row, h, b, raw + 1 - b * P.bs, sq, P.kmean + row * P.row_elems, P.dbar + row * P.r,
                                P.vmean + row * P.row_elems, lane);
}

// The last cluster to have read the lengths stores the new ones (nobody waits: it is a counter).
__device__ __noinline__ void store_lens(int *counter, int *seq_lens, int batch, int cap, int n_clusters) {
  if (atomicAdd(counter, 1) != n_clusters - 1) return;
  *counter = 0;
  for (int i = 0; i < batch; ++i) {
    const int raw = seq_lens[i];
    if (raw >= 0 && raw < cap) seq_lens[i] = raw + 1;
  }
}

template <int G, bool RD, bool HS, bool VH>
__global__ void __launch_bounds__(kThreads, 1)
ckv_unit_step_kernel(const __grid_constant__ CkvDev P, const bf16 *q, const int *seq_lens, const bf16 *k_pool, const bf16 *v_pool,
                     const int *page_table, const __grid_constant__ CkvNewToken fresh, int kcap, CkvStepPlan plan, int batch,
                     int *__restrict__ sel_ids, int *__restrict__ sel_cnt, bf16 *__restrict__ out, float *__restrict__ lse,
                     CkvHostDone done, const __grid_constant__ CUtensorMap tm_v) {
  constexpr int kRowBytesK = HS ? CKV_D * 2 : CKV_ROW_ELEMS * 2;
  constexpr int kRowBytesV = (HS || VH) ? CKV_D * 2 : CKV_ROW_ELEMS * 2;
  constexpr int TB = ScanTile<HS || VH>::TB;
  constexpr int kParts = TB / 16;              // parts of a tile
  constexpr int kSkip = kWarps / kParts;       // a warp works on every kSkip-th tile
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full_bar[2][kStagesCap], empty_bar[kStagesCap];
  __shared__ __align__(8) uint64_t s_xbar[4];                 // what the cluster's CTAs send: normalisers, scores, partial outputs; global stores done
  __shared__ __align__(512) unsigned char s_zero_row[512];
  constexpr int kQStride = CKV_D + 8;                         // 17 pieces of 16 bytes: the matrix loads of eight rows hit eight bank groups
  __shared__ __align__(16) bf16 s_q[G][kQStride];
  __shared__ float s_w[G * 64];                               // variance weights [t][g], r < d
  __shared__ __align__(16) float4 s_wn[kWarps + 1][G];        // (maximum m, sum of e^{l - m}, largest score term) per warp, then of the last block
  __shared__ __align__(16) float4 s_norm[kClusterCap][G];     // ... per CTA of the cluster
  __shared__ float s_tail_u[G];
  __shared__ __align__(16) float s_tail_part[G][CKV_PART_STRIDE];
  __shared__ __align__(16) float s_recv[(4 * G + kClusterCap) * kRecvStride];
  __shared__ float s_sq[CKV_D];
  __shared__ TailArgs s_tail;
  __shared__ int s_digit, s_before, s_nc, s_ncand, s_wt[3][kWarps], s_abort, s_issued;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  using T = HeadTile<G>;       // which heads a lane works on
  const int C = (int)cluster_size(), rank = (int)cluster_rank();
  const int unit = blockIdx.y, s = ckv_div_hkv(P, unit), h = unit - s * P.Hkv;
  const bool append = fresh.k_new != nullptr;
  const int cap = P.max_blocks * P.bs;
  auto div_c = [&](int x) { return C == 1 ? x : (int)__umulhi((unsigned)x, plan.c_magic); };   // x / C, 0 <= x < 2^32 / C
  float log_bs = logf((float)P.bs);
  asm volatile("" : "+f"(log_bs));   // (here, ahead of the wait for the launch before, and not where it is used)
  if (tid == kProducerWarp * 32) {
    for (int st = 0; st < plan.stages; ++st) { mbar_init(&full_bar[0][st], 1); mbar_init(&full_bar[1][st], 1); mbar_init(&empty_bar[st], kParts); }
    for (int i = 0; i < 3; ++i) mbar_init(&s_xbar[i], 1);
    mbar_init(&s_xbar[3], C);
    fence_barrier_init();
    const int n_items = (4 * G - rank + C - 1) / C;   // partial outputs this CTA reduces (see the merge)
    mbar_arrive_expect_tx(&s_xbar[0], (uint32_t)(C * G * 16));
    mbar_arrive_expect_tx(&s_xbar[2], (uint32_t)(n_items * C * (32 * 4 + 8)));
    s_abort = 0; s_issued = 0; s_digit = -1; s_ncand = 0;
  }
  if (warp == kProducerWarp) __syncwarp();   // its other lanes arm these barriers, too
  if (warp >= kTailWarp) {
    const int i = tid - kTailWarp * 32;
    static_assert(sizeof(CkvDev) % 4 == 0 && sizeof(CkvDev) <= 256 && sizeof(CkvNewToken) % 4 == 0 && sizeof(CkvNewToken) <= 256, "a word per thread");
    if (i < (int)sizeof(CkvDev) / 4) reinterpret_cast<int *>(&s_tail.P)[i] = reinterpret_cast<const int *>(&P)[i];
    if (i < (int)sizeof(CkvNewToken) / 4) reinterpret_cast<int *>(&s_tail.fresh)[i] = reinterpret_cast<const int *>(&fresh)[i];
    named_barrier(4, 64);
  }
  if (warp == kValueWarp) reinterpret_cast<uint4 *>(s_zero_row)[lane] = make_uint4(0u, 0u, 0u, 0u);
  cluster_arrive_release();   // "this CTA runs, its barriers are set up"
  pdl_trigger();              // the next launch of the stream may set itself up ...
  const size_t row0 = (size_t)unit * P.max_blocks;
  const bool dbar_bulk = P.r >= 4;
  const int stage_bytes = TB * (kRowBytesK + kRowBytesV) + (dbar_bulk ? TB * P.r * 4 : 0);
  // test hook (ckv_debug_set): one fill is announced but never issued, so that the waits on it run out
  auto withheld = [&](int f) { return (P.debug & CKV_DEBUG_SKIP_FILL) != 0 && f == 0 && rank == 0 && unit == 0; };
  // fill `f` of the ring: nb blocks from block b on into stage `st`, counted on full barrier `fb`
  auto fill = [&](int f, int b, int nb, int st, uint64_t *fb) {
    const size_t row = row0 + b;
    unsigned char *sk = smem + (size_t)st * stage_bytes;
    unsigned char *sv = sk + TB * kRowBytesK;
    const uint32_t kbytes = (uint32_t)nb * kRowBytesK;
    const uint32_t vbytes = VH ? (uint32_t)TB * kRowBytesV : (uint32_t)nb * kRowBytesV;   // a tensor copy always delivers its whole box
    const uint32_t dbytes = dbar_bulk ? (uint32_t)nb * P.r * 4 : 0;
    mbar_arrive_expect_tx(fb, kbytes + vbytes + dbytes);
    const uint32_t lo = smem_u32(smem), hi = lo + (uint32_t)plan.stages * stage_bytes;
    bool ok = nb >= 1 && b + nb <= P.max_blocks;
    if (!withheld(f)) {
      ok = ok && bulk_g2s_checked(sk, P.kmean + row * P.row_elems, kbytes, fb, lo, hi);
      if constexpr (VH) {
        // rows [row, row + TB) of the mean-values region, first 256 bytes of each (rows past the range are never read)
        const uint32_t dv = smem_u32(sv);
        const bool fits = (dv & 127u) == 0 && dv >= lo && dv + vbytes <= hi;
        if (ok && fits) tensor_g2s(dv, &tm_v, 0, (int)row, fb);
        ok = ok && fits;
      } else {
        ok = ok && bulk_g2s_checked(sv, P.vmean + row * P.row_elems, vbytes, fb, lo, hi);
      }
      if (dbar_bulk) ok = ok && bulk_g2s_checked(sv + TB * kRowBytesV, P.dbar + row * P.r, dbytes, fb, lo, hi);
    }
    if (!ok) atomicOr(P.status, CKV_DEV_BAD_COPY);
  };
  // Ahead of the length, the tile that a sequence as long as the host's bound would have the CTA begin with is copied.  A
  // sequence that puts the CTA's range elsewhere leaves it unused: which blocks a CTA works on, and with them the last bits of
  // the results, depend on the length and not on the bound.  (Bounds of 128K over lengths of 1.6K to 100K: against ranges laid
  // out by the bound, whose copies are all used, 0 to 0.25 us a step, 0.6 with four sequences of 64K; 72 units of 8.4K to 9.2K
  // tokens with r = d, where every second CTA's copy goes unused, 20.3 -> 20.6.)  With this copy ahead
  // of the length, the others issued by the producer's lanes and the queries' fragments loaded as matrices, a CTA starts on
  // its first part 1.2 us after the length is known instead of 2.0 (a step of 8 units at 32K 15.4 -> 14.8 us, 16 units with
  // r = d at 88K 40.5 -> 39.6, 32 units at 128K 52.6 -> 51.5).
  const int b_early = rank * plan.early_parts * 16;
  const int n_early = max(min(min(TB, plan.early_parts * 16), plan.max_blocks - b_early), 0);
  // The launch ahead of this one is waited for in each of the three branches: nobody touches anything before that.  The tail
  // routines set up all they can ahead of it.  Only the working warps wait for the queries' staging: the producer wants the
  // length alone (queries in host memory take 3 us to arrive).
  const int *pt_row = page_table + (size_t)s * P.max_pages_per_seq;
  const int most_len = plan.max_blocks * P.bs;
  int raw;
  if (warp >= kTailWarp && rank == C - 1) {
    raw = warp == kTailWarp ? tail_block<G>(&s_tail, q + (size_t)unit * G * CKV_D, page_table, seq_lens, unit, most_len, plan.hi_page, s_sq,
                                            s_tail_u, &s_tail_part[0][0], s_wn[kWarps])
                            : tail_values<G>(&s_tail, page_table, seq_lens, unit, most_len, plan.hi_page, &s_tail_part[0][0]);
  } else {
    pdl_wait();
    if (tid == kProducerWarp * 32 && n_early > 0) fill(0, b_early, n_early, 0, &full_bar[0][0]);
    raw = seq_lens[s];
    if (tid < G * 16) *reinterpret_cast<uint4 *>(&s_q[tid >> 4][8 * (tid & 15)]) = reinterpret_cast<const uint4 *>(q + (size_t)unit * G * CKV_D)[tid];
    if (warp < kWarps) named_barrier(3, kThreads);
    else named_arrive(3, kThreads);
  }
  // the length the step works on; of a sequence longer than the host's bound, what the shared arrays were sized for
  const int N_all = max(min(raw + ((append && raw >= 0 && raw < cap) ? 1 : 0), cap), 0);
  const int N = min(N_all, most_len);
  if (N < N_all && rank == 0 && tid == 0) atomicOr(P.status, CKV_DEV_BAD_BOUND);
  const int X = (N + P.bs - 1) >> P.lg_bs, Xs = max(X - 1, 0);
  // what the CTA owns: `own` blocks from b_lo on
  const int n_parts = (Xs + 15) >> 4, ppc = div_c(n_parts + C - 1);
  const int b_lo = min(rank * ppc, n_parts) * 16;
  const int own = max(min(min(b_lo + ppc * 16, Xs) - b_lo, plan.own_cap), 0);
  const int tiles = (own + TB - 1) / TB;
  auto tile_len = [&](int it) { return min(TB, own - it * TB); };
  // The early copy is the first tile, or fill 0 of the ring is nobody's and tile `it` is fill it + 1.
  const int skew = n_early > 0 && !(own > 0 && b_lo == b_early && tile_len(0) <= n_early) ? 1 : 0, n_fills = tiles + skew;
  // score terms of the CTA's own blocks, [g][us] (eight more than the range holds: a tile's eight rows x four heads then
  // fall into 32 different banks)
  float *ub = reinterpret_cast<float *>(smem + plan.u_off);
  const int us = plan.own_cap + 8;

  ScanUnit<G, bf16, RD> w;
  w.reset();
  if (warp == kProducerWarp) {
    // ---------------- producer: its lanes issue the first round of fills, one thread refills the ring ----------------
    auto fill_tile = [&](int f, int st, uint64_t *fb) { const int it = f - skew; fill(f, b_lo + it * TB, tile_len(it), st, fb); };
    const int first_fills = min(n_fills, plan.stages);
    if (lane >= (n_early > 0 ? 1 : 0) && lane < first_fills) fill_tile(lane, lane, &full_bar[0][lane]);
    __syncwarp();
    if (lane == 0) {
      mbar_arrive_expect_tx(&s_xbar[1], (uint32_t)(X * 4));
      *(volatile int *)&s_issued = first_fills;
      if (skew != 0) {   // nobody else waits for this copy or releases its stage
        if (!mbar_wait(&full_bar[0][0], 0, P.spin_limit)) {
          atomicOr(P.status, CKV_DEV_TIMEOUT);
          *(volatile int *)&s_abort = 1;
        }
        for (int i = 0; i < kParts; ++i) mbar_arrive(&empty_bar[0]);
      }
      int st = 0;
      uint32_t phase = 0, round = 1;
      for (int f = plan.stages; f < n_fills; ++f) {
        if (!mbar_wait(&empty_bar[st], phase, P.spin_limit)) {
          atomicOr(P.status, CKV_DEV_TIMEOUT);
          *(volatile int *)&s_abort = 1;
        }
        if (*(volatile int *)&s_abort) break;
        fill_tile(f, st, &full_bar[round & 1][st]);
        *(volatile int *)&s_issued = f + 1;
        if (++st == plan.stages) { st = 0; ++round; phase ^= 1; }
      }
    } else {
      // the other lanes ask the L2 for this CTA's share of the page-table row: the attention's lookups are then short
      const int lines = (X * P.ppb + 31) / 32, per = (lines + C - 1) / C;
      for (int i = rank * per + lane - 1; i < min((rank + 1) * per, lines); i += 31)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(pt_row + 32 * i) : "memory");
    }
  } else if (warp >= kTailWarp) {
    if (warp == kTailWarp && rank == C - 1 && append && raw >= N && raw < cap) append_past_bound(P, page_table, fresh, unit, raw, s_sq);
    if (warp == kTailWarp && (rank != C - 1 || N == 0) && lane < G) s_wn[kWarps][lane] = make_float4(-CUDART_INF_F, 0.f, -CUDART_INF_F, 0.f);
    if (warp == kTailWarp && append && raw < 0 && rank == C - 1 && lane == 0) atomicOr(P.status, CKV_DEV_SEQ_FULL);   // no place for the token
  } else {
    // ---------------- working warps: parts of 16 blocks ----------------
    if (!RD) {
      // w_{g,t} of Eq. 8 times the squared logit scale, summed in coordinate order as the scan kernel sums the weights it
      // stages (those of a CTA's later units it sums in runs of eight): scores that differ in the last bit can swap blocks
      // at the cut.  (The first tile's data is still on its way.)
      const int lg_r = __ffs(P.r) - 1, gs = CKV_D >> lg_r, run = P.glayout == 0 ? gs : gs >> 1;
      for (int i = tid; i < P.r * G; i += kWork) {
        const int g = i & (G - 1), t = i / G;
        float a = 0.f;
        if (run >= 8) {
#pragma unroll 2
          for (int k = 0; k < gs; k += 8) {
            float x[8];
            bf16x8_to_float(*reinterpret_cast<const uint4 *>(&s_q[g][t * run + (k < run ? k : CKV_D / 2 + k - run)]), x);
#pragma unroll
            for (int j = 0; j < 8; ++j) a = fmaf(x[j], x[j], a);
          }
        } else {
          for (int k = 0; k < gs; ++k) {
            const float x = __bfloat162float(s_q[g][t * run + (k < run ? k : CKV_D / 2 + k - run)]);
            a = fmaf(x, x, a);
          }
        }
        s_w[i] = a * (P.scale * P.scale);
      }
    }
    w.load_queries(lane, P.scale, smem_u32(&s_q[0][0]), kQStride * 2, smem_u32(s_zero_row));
    if (!RD) work_barrier();
    if (!RD && P.r == 4) {
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int t = 0; t < 4; ++t) w.wown[e][t] = T::head(lane, e) < G ? s_w[t * G + T::head(lane, e)] : 0.f;
    }
    const ScanPartCfg cfg{P.scale, P.half_var, log_bs, P.r, P.max_blocks, (P.variant & CKV_VARIANT_RANK_BY_MASS) != 0, P.r == 4};
    float *lz = P.lz + row0 * G;
    const int part = warp % kParts;
    // A warp visits every kSkip-th tile.  A fill is only issued once the one plan.stages before it was released, and
    // kSkip <= plan.stages (checked by the launcher): alternate rounds of the ring use two sets of full barriers, which
    // together tell the fills a parity wait could confuse apart (see the scan kernel).
    int st = 0, at = 0;
    uint32_t round = 0;
    bool aborted = false;
    float umax[2] = {-CUDART_INF_F, -CUDART_INF_F};   // largest score terms this lane has seen, of its heads
    for (int it = warp / kParts; it < tiles; it += kSkip) {
      st += it + skew - at;
      at = it + skew;
      while (st >= plan.stages) { st -= plan.stages; ++round; }
      if (!aborted) {
        bool fail = *(volatile int *)&s_abort != 0;
        if (!fail && !mbar_wait(&full_bar[round & 1][st], (round >> 1) & 1, P.spin_limit)) {
          atomicOr(P.status, CKV_DEV_TIMEOUT);
          *(volatile int *)&s_abort = 1;
          fail = true;
        }
        aborted = __any_sync(0xffffffffu, fail);
      }
      const int nb = tile_len(it), rb = part * 16, tb0 = b_lo + it * TB;
      if (!aborted && rb < nb) {
        const uint32_t sk = smem_u32(smem + (size_t)st * stage_bytes);
        const float *sd = reinterpret_cast<const float *>(smem + (size_t)st * stage_bytes + TB * (kRowBytesK + kRowBytesV));
        scan_part<G, bf16, RD, HS, VH>(
            w, cfg, sk, sk + TB * kRowBytesK, (RD || dbar_bulk) ? sd : nullptr, smem_u32(s_zero_row), s_w, P.dbar + row0 * P.r,
            lane, rb, nb, tb0, -1, 0.f,
            [&](int g, int blk, float x, float y) {
              ub[g * us + (blk - b_lo)] = x;
              lz[(size_t)g * P.max_blocks + blk] = y;
              if (g & 1) umax[1] = fmaxf(umax[1], x); else umax[0] = fmaxf(umax[0], x);
            });
      }
      __syncwarp();
      if (lane == 0 && !aborted) mbar_arrive(&empty_bar[st]);
    }
    // this warp's normaliser partial
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float lp = T::sum_rows(w.lp[e]), um = T::max_rows(umax[e]);
      if (T::owns(lane, e)) s_wn[warp][T::head(lane, e)] = make_float4(w.m[e], lp, um, 0.f);
    }
  }
  __syncwarp();
  cluster_wait();    // every CTA of the cluster has started
  __syncthreads();
  if (s_abort) {     // leave no copy in flight into memory that is about to be reused: wait (bounded) for every issued fill
    if (tid == 0)
      for (int it = max(s_issued - plan.stages, 0); it < s_issued; ++it)
        if (!withheld(it)) mbar_wait(&full_bar[(it / plan.stages) & 1][it % plan.stages], ((it / plan.stages) >> 1) & 1);
    __syncthreads();
  }

  // ---- normalisers of Eq. 9 over the whole unit ----
  if (warp < G) {   // the CTA's own: warp g for head g, every lane the whole sum
    float4 e[kWarps + 1];
#pragma unroll
    for (int i = 0; i <= kWarps; ++i) e[i] = s_wn[i][warp];
    const float mine = s_wn[min(lane, kWarps)][warp].x;
    float m = e[0].x, l = 0.f, u = e[0].z;
#pragma unroll
    for (int i = 1; i <= kWarps; ++i) { m = fmaxf(m, e[i].x); u = fmaxf(u, e[i].z); }
    // One weight a lane, handed round, here and in the merges below: what is weighted may be as large as fp32 allows, so a
    // weight below 2^-126 counts, and exp2f with its steps for such results is a few instructions once instead of per entry.
    // The code between the phases is run once a launch and its length is its time (us a step of one unit of 4K tokens, of 8 of
    // 32K, of 32 of 128K: 10.7, 12.9, 47.9 this way; 11.1, 13.3, 48.2 with exp2f for every entry).
    const float sc = exp2_diff(mine, m);
#pragma unroll
    for (int i = 0; i <= kWarps; ++i) l = fmaf(e[i].y, __shfl_sync(0xffffffffu, sc, i), l);
    if (lane < C) {
      const uint32_t x0 = smem_u32(&s_xbar[0]), there = cluster_map(x0, lane);   // the CTAs' shared memories are congruent windows
      st_async_u32x4(there + (smem_u32(&s_norm[rank][warp]) - x0), __float_as_uint(m), __float_as_uint(l), __float_as_uint(u), 0u, there);
    }
  }
  if (warp >= kWarps) {   // meanwhile: histogram and bit map start at zero (the ring is drained)
    int4 *hist = reinterpret_cast<int4 *>(smem + kOffHist);
    for (int i = tid - kWork; i < (kBins + 32 + kMapWords) / 4; i += kThreads - kWork) hist[i] = make_int4(0, 0, 0, 0);
    if (warp == kTailWarp) {
      // What this CTA's scan and tail warps wrote to global memory and others of the cluster will read (mean-term weights,
      // the new token's rows) is released by this warp for all of them: the wait for those stores is off the critical path.
      __threadfence();
      if (lane < C) mbar_arrive_cluster(cluster_map(smem_u32(&s_xbar[3]), lane));
    }
  }
  auto wait_x = [&](int i) {
    if (mbar_wait_cluster(&s_xbar[i], 0, P.spin_limit)) return true;
    atomicOr(P.status, CKV_DEV_TIMEOUT);
    *(volatile int *)&s_abort = 1;
    return false;
  };
  const bool normed = wait_x(0);   // false: a CTA of the cluster may still be scanning, its ring in use and the lengths unread
  const bool counts = append && rank == 0 && tid == kTailWarp * 32;
  if (counts && normed) store_lens(P.status + CKV_LEN_COUNTER_WORD, fresh.seq_lens, batch, cap, (int)gridDim.y);   // all CTAs of this cluster have read them
  float Mg[G], iL[G], bound = 0.f;   // every warp by itself: 32 / G lanes per head.  bound: no block scores more
  {
    constexpr int LPH = 32 / G, EPL = (kClusterCap + LPH - 1) / LPH;
    const int g = lane / LPH, k0 = lane % LPH;
    float4 e[EPL];
    float m = -CUDART_INF_F, l = 0.f, u = -CUDART_INF_F;
#pragma unroll
    for (int i = 0; i < EPL; ++i) {
      const int k = k0 + i * LPH;
      e[i] = k < C ? s_norm[k < kClusterCap ? k : 0][g] : make_float4(-CUDART_INF_F, 0.f, -CUDART_INF_F, 0.f);
      m = fmaxf(m, e[i].x);
      u = fmaxf(u, e[i].z);
    }
#pragma unroll
    for (int o = LPH / 2; o > 0; o >>= 1) {
      m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      u = fmaxf(u, __shfl_xor_sync(0xffffffffu, u, o));
    }
#pragma unroll
    for (int i = 0; i < EPL; ++i) l = fmaf(e[i].y, exp2_diff(e[i].x, m), l);
#pragma unroll
    for (int o = LPH / 2; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    const float il = 1.0f / l, b = fast_exp2(u - m) * il;
#pragma unroll
    for (int i = 0; i < G; ++i) {
      Mg[i] = __shfl_sync(0xffffffffu, m, i * LPH);
      iL[i] = __shfl_sync(0xffffffffu, il, i * LPH);
      bound += __shfl_sync(0xffffffffu, b, i * LPH);
    }
  }

  // ---- scores of the CTA's own blocks (Eq. 10), to every CTA of the cluster ----
  const int n_recent = min(P.recent, X);
  const int rank_lo = P.sink, rank_n = max(X - n_recent - P.sink, 0);   // blocks [rank_lo, rank_lo + rank_n) are ranked, the others mandatory
  uint32_t *keys = reinterpret_cast<uint32_t *>(smem);   // the unit's scores; their bit patterns are ordered like the scores
  // No score is larger, with room for the bound's and the scores' roundings; the senders hold themselves to it, too, because
  // the histogram's addresses rely on it.
  const uint32_t most = __float_as_uint(fminf(bound, 3.0e38f)) + (1u << 10);
  if (!normed) {
    // nothing is sent into a CTA that may not be ready for it: its wait for the scores runs out, too
  } else if (warp < kWarps) {
    bool nonfinite = false;
    const uint32_t xbar1 = smem_u32(&s_xbar[1]);
    for (int i = 4 * tid; i < own; i += 4 * kWork) {
      float sc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float4 u = *reinterpret_cast<const float4 *>(ub + g * us + i);
        sc[0] = fmaf(fast_exp2(u.x - Mg[g]), iL[g], sc[0]); sc[1] = fmaf(fast_exp2(u.y - Mg[g]), iL[g], sc[1]);
        sc[2] = fmaf(fast_exp2(u.z - Mg[g]), iL[g], sc[2]); sc[3] = fmaf(fast_exp2(u.w - Mg[g]), iL[g], sc[3]);
      }
      uint32_t k[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool real = i + j < own;
        if (real && (!(sc[j] >= 0.f) || sc[j] > 3.0e38f)) { nonfinite = true; sc[j] = 0.f; }
        k[j] = min(__float_as_uint(sc[j]), most);
      }
      const uint32_t dst = smem_u32(keys + b_lo + i);
      if (i + 4 <= own) {
        for (int c = 0; c < C; ++c) {
          const uint32_t there = cluster_map(xbar1, c);   // the CTAs' shared memories are congruent windows
          st_async_u32x4(there + (dst - xbar1), k[0], k[1], k[2], k[3], there);
        }
      } else {   // the end of the unit's range: what follows belongs to somebody else
        for (int c = 0; c < C; ++c)
#pragma unroll
          for (int j = 0; j < 3; ++j)
            if (i + j < own) st_async_u32(cluster_map(dst + 4 * j, c), k[j], cluster_map(smem_u32(&s_xbar[1]), c));
      }
    }
    if (nonfinite) atomicOr(P.status, CKV_DEV_NONFINITE);
  } else if (warp == kTailWarp && rank == C - 1 && N > 0) {   // the last block
    float sc = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) sc = fmaf(fast_exp2(s_tail_u[g] - Mg[g]), iL[g], sc);
    if (!(sc >= 0.f) || sc > 3.0e38f) { if (lane == 0) atomicOr(P.status, CKV_DEV_NONFINITE); sc = 0.f; }
    if (lane < C) st_async_u32(cluster_map(smem_u32(keys + Xs), lane), min(__float_as_uint(sc), most), cluster_map(smem_u32(&s_xbar[1]), lane));
  }
  // While the scores are on their way: a thread will keep those of 4 nj blocks in a row, s0 .. s0 + 4 nj - 1, in registers for
  // both passes of the selection.  nj is 2 or odd, so that a warp's 16-byte reads fall into different banks (two of them,
  // with 2), and 9 at most.  A thread's part of the selection is a word of bits; the mandatory blocks are in.
  const int nj0 = (int)((unsigned)(X + 4 * kWork - 1) / (4 * kWork)), nj = nj0 > 2 ? nj0 | 1 : max(nj0, 1), s0 = 4 * nj * tid;
  auto below = [](int n) { return n >= 64 ? ~0ull : (1ull << max(n, 0)) - 1ull; };   // bits 0 .. n - 1
  unsigned long long here = below(min(4 * nj, X - s0));
  unsigned long long rk = here & below(rank_lo + rank_n - s0) & ~below(rank_lo - s0);
  float lg_bs = log2f((float)P.bs), lg_last = log2f((float)max(N - Xs * P.bs, 1));   // the attention's
  const int K = min(kcap, X);
  const bool all = X <= kcap;          // every block is selected: the step is dense attention
  // ... and the attention's share of the selected pages
  const int n_pages = all ? (N + CKV_PAGE - 1) / CKV_PAGE : K * P.ppb, share = div_c(n_pages + C - 1);
  int p0 = min(rank * share, n_pages), n_mine = max((min(p0 + share, n_pages) - p0 - warp + kWarps - 1) / kWarps, 0);
  asm volatile("" : "+l"(here), "+l"(rk), "+f"(lg_bs), "+f"(lg_last), "+r"(p0), "+r"(n_mine));   // (here, and not where they are used)
  wait_x(1);
  // (the histogram is clear, too.)  A CTA one of whose waits ran out has scores that never came: it selects nothing and
  // contributes an empty partial, so that the others get what they wait for.
  const bool dead = __syncthreads_or(*(volatile int *)&s_abort) != 0;

  // ---- selection (Eq. 11), the same in every CTA ----
  int *ids = reinterpret_cast<int *>(smem + kOffIds);
  if (warp >= kWarps && !dead) {   // the idle warps leave the range's scores where ckv_copy_scores() finds them
    float *scores = P.scores + row0;
    for (int i = tid - kWork; i < own; i += kThreads - kWork) scores[b_lo + i] = __uint_as_float(keys[b_lo + i]);
    if (rank == C - 1 && N > 0 && tid == kWork) scores[Xs] = __uint_as_float(keys[Xs]);
  }
  if (warp < kWarps) {
    int *gids = sel_ids + (size_t)unit * kcap;
    if (dead) {
      if (rank == 0) {
        for (int i = tid; i < kcap; i += kWork) gids[i] = -1;
        if (tid == 0) sel_cnt[unit] = 0;
      }
    } else if (all) {
      if (rank == 0) {
        for (int b = tid; b < kcap; b += kWork) gids[b] = b < X ? b : -1;
        if (tid == 0) sel_cnt[unit] = X;
      }
    } else {
      const int Kr = K - (X - rank_n);   // blocks to rank in (the host guarantees K >= sink + recent when K < X)
      uint32_t *map = reinterpret_cast<uint32_t *>(smem + kOffMap);   // blocks found by id (clear so far)
      unsigned long long sel = here & ~rk;
      if (Kr > 0) {
        int *hist = reinterpret_cast<int *>(smem + kOffHist);
        const uint4 *keys4 = reinterpret_cast<const uint4 *>(keys);
        const uint32_t top = most >> kBinShift;   // bin 0
        uint32_t key[kKeyGroups][4];
#pragma unroll
        for (int j = 0; j < kKeyGroups; ++j) {
          if (j >= nj) break;
          const uint4 k4 = keys4[tid * nj + j];
          key[j][0] = k4.x; key[j][1] = k4.y; key[j][2] = k4.z; key[j][3] = k4.w;
        }
        {
          // a bin's address falls with the score; what lies below the last bin or is not ranked goes aside, without a branch
          const uint32_t h_top = smem_u32(hist) + 4 * top, aside = smem_u32(hist + kBins + lane);
          const bool whole = __all_sync(0xffffffffu, rk == below(4 * nj));
#pragma unroll
          for (int j = 0; j < kKeyGroups; ++j) {
            if (j >= nj) break;
            uint32_t at[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) at[e] = min(h_top - (key[j][e] >> (kBinShift - 2) & ~3u), aside);
            if (!whole) {
#pragma unroll
              for (int e = 0; e < 4; ++e) at[e] = (rk >> (4 * j + e) & 1) != 0 ? at[e] : aside;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) red_shared_inc(at[e]);
          }
        }
        work_barrier();
        constexpr int BPT = kBins / kWork;   // bins per thread, largest scores first
        int c[BPT], csum = 0;
#pragma unroll
        for (int j = 0; j < BPT; j += 4) {
          const int4 x = reinterpret_cast<const int4 *>(hist)[(tid * BPT + j) / 4];
          c[j] = x.x; c[j + 1] = x.y; c[j + 2] = x.z; c[j + 3] = x.w;
          csum += (x.x + x.y) + (x.z + x.w);
        }
        int before = work_exclusive_scan(csum, s_wt[0]);
        if (before < Kr && before + csum >= Kr) {
#pragma unroll
          for (int j = 0; j < BPT; ++j) {
            if (before < Kr && before + c[j] >= Kr) { s_digit = tid * BPT + j; s_before = before; s_nc = c[j]; before = Kr; }
            else before += c[j];
          }
        }
        work_barrier();
        const int digit = s_digit, nc = s_nc;
        if (digit >= 0 && nc <= kCandCap) {
          // higher bins are taken whole; the cut's bin is ranked by (score descending, id ascending): what tells its blocks
          // apart, the scores' low bits and the ids, fits one word
          uint32_t *cand = reinterpret_cast<uint32_t *>(smem + kOffCand);
          const int take = Kr - s_before;
          // sign bits of (threshold - 1 - score), shifted into words: 1 where the score reaches the threshold
          // (unsigned: words past the unit's scores hold anything, their bits are masked)
          const uint32_t lo1 = ((top - (uint32_t)digit) << kBinShift) - 1u;
          const uint32_t hi1 = digit == 0 ? 0x7fffffffu : ((top - (uint32_t)digit + 1u) << kBinShift) - 1u;
          uint32_t ge_hi[2] = {0, 0}, ge_lo[2] = {0, 0};
#pragma unroll
          for (int j = kKeyGroups - 1; j >= 0; --j) {
            if (j < nj) {
#pragma unroll
              for (int e = 3; e >= 0; --e) {
                ge_hi[j >> 3] = __funnelshift_l(hi1 - key[j][e], ge_hi[j >> 3], 1);
                ge_lo[j >> 3] = __funnelshift_l(lo1 - key[j][e], ge_lo[j >> 3], 1);
              }
            }
          }
          const unsigned long long above = rk & ((unsigned long long)ge_hi[1] << 32 | ge_hi[0]);
          unsigned long long at = rk & ~above & ((unsigned long long)ge_lo[1] << 32 | ge_lo[0]);
          sel |= above;
          if (tid >= nc && tid < nc + 3) cand[tid] = 0;   // the last group of four is filled up
          while (at != 0) {
            const int b = s0 + __ffsll((long long)at) - 1;
            at &= at - 1;
            const int slot = atomicAdd(&s_ncand, 1);
            if (slot < kCandCap) cand[slot] = keys[b] << (32 - kBinShift) >> 1 | (uint32_t)(kIdMask - b);
          }
          work_barrier();
          if (tid < nc) {
            const uint32_t mine = cand[tid];
            int place = 0;
#pragma unroll 2
            for (int j = 0; j < nc; j += 4) {
              const uint4 k = *reinterpret_cast<const uint4 *>(cand + j);
              place += (k.x > mine ? 1 : 0) + (k.y > mine ? 1 : 0) + (k.z > mine ? 1 : 0) + (k.w > mine ? 1 : 0);
            }
            const int b = kIdMask - (int)(mine & kIdMask);
            if (place < take) atomicOr(&map[b >> 5], 1u << (b & 31));
          }
        } else {
          take_by_digits(X, Kr, keys, rank_lo, rank_n, hist, map, s_wt[1], s_wt[2]);
        }
      }
      work_barrier();
      // ids in position order
      {
        const uint32_t *m = map + (s0 >> 5);
        const uint32_t m0 = m[0], m1 = m[1], m2 = m[2];
        sel |= here & ((unsigned long long)__funnelshift_r(m1, m2, s0 & 31) << 32 | __funnelshift_r(m0, m1, s0 & 31));
      }
      int pos = work_exclusive_scan(__popcll(sel), s_wt[1]);
      for (; sel != 0; ++pos) {
        const int b = s0 + __ffsll((long long)sel) - 1;
        sel &= sel - 1;
        if (pos < K) {
          ids[pos] = b;
          if (rank == 0) gids[pos] = b;
        }
      }
      if (rank == 0) {
        for (int i = K + tid; i < kcap; i += kWork) gids[i] = -1;
        if (tid == 0) sel_cnt[unit] = K;
      }
      work_barrier();
    }
  }
  const int nsel = K;
  if (warp < kWarps) {
    wait_x(3);       // acquires what the other CTAs of the cluster released
    // ---- exact attention over the CTA's share of the selected pages ----
    const bool comp = nsel < X && !dead && !(P.variant & CKV_VARIANT_DROP);
    if (!comp) w.reset();   // nothing is compensated: the scan's sums are not wanted
    if (dead) n_mine = 0;
    const int pshift = P.ppb == 1 ? 0 : (P.ppb == 2 ? 1 : 2);
    const float *lz = P.lz + row0 * G;
    const float sl2 = P.scale * kLog2e;
    const uint32_t buf0 = smem_u32(smem + kOffPages) + warp * 2 * kPageBytes;
    const bool rows_rm = HS && comp;   // one more item per 16 pages: the mean-value rows of their blocks
    bool bad = false;
    struct Page { int phys, ntok, blk; };
    Page mine{-1, 0, -1};
    auto lookup = [&](int n) {         // lane l looks the warp's page n + l up: 32 pages cost one round trip
      mine = Page{-1, 0, -1};
      if (n + lane < n_mine) {
        const int i = p0 + warp + kWarps * (n + lane);
        const int blk = all ? i >> pshift : ids[i >> pshift];
        const int page = all ? i : (blk << pshift) + (i & (P.ppb - 1));
        mine.blk = (i & (P.ppb - 1)) == 0 ? blk : ~blk;   // complemented on the block's later pages
        mine.ntok = (unsigned)blk < (unsigned)X ? max(min(CKV_PAGE, N - page * CKV_PAGE), 0) : 0;
        if (mine.ntok > 0) {
          mine.phys = pt_row[page];
          if (mine.phys < 0 || mine.phys >= P.num_pages) {   // skipped: nothing is added, and no mean row taken off
            mine.phys = -1;
            mine.blk = mine.blk < 0 ? mine.blk : ~mine.blk;
            bad = true;
          }
        }
      }
    };
    // items: pages 0 .. 15, [rows], pages 16 .. 31, [rows], ...; the last group may be short
    const int n_items = n_mine + (rows_rm ? (n_mine + 15) / 16 : 0);
    // ntok > 0: a page; 0: nothing; -1: rows.  A page's z is kept as loaded and lowered by lb where it is used: with the
    // subtraction beside the load the warp waited for it, page after page (selections of 32K tokens, 80 units: 326 us a
    // step then, 290 now).
    struct Item { int ntok; float lb, z[HS ? T::NR : 1][2]; };
    int gpos = 0, page_n = 0;
    auto issue = [&](int buf) -> Item {
      Item it;
      it.ntok = 0;
      it.lb = 0.f;
      it.z[0][0] = it.z[0][1] = -CUDART_INF_F;
      const uint32_t kb = buf0 + buf * kPageBytes;
      const bool rows = rows_rm && (gpos == 16 || page_n == n_mine);
      if (!rows) {
        if ((page_n & 31) == 0) lookup(page_n);
        const int phys = __shfl_sync(0xffffffffu, mine.phys, page_n & 31);
        const int ntok = __shfl_sync(0xffffffffu, mine.ntok, page_n & 31);
        const int bx = __shfl_sync(0xffffffffu, mine.blk, page_n & 31);
        if (phys >= 0) {
          const size_t src = ((size_t)phys * P.Hkv + h) * (CKV_PAGE * CKV_D);
          issue_page(kb, kb + kTileBytes, k_pool + src, v_pool + src, ntok, lane);
          it.ntok = ntok;
          if (!HS && comp) {   // log2 of e^{zbar} of the page's block for this lane's heads
            const int blk = bx < 0 ? ~bx : bx;
            it.lb = blk == Xs ? lg_last : lg_bs;
#pragma unroll
            for (int e = 0; e < 2; ++e)
              if (T::head(lane, e) < G) it.z[0][e] = __ldcg(lz + (size_t)T::head(lane, e) * P.max_blocks + blk);
          }
        }
        ++page_n; ++gpos;
      } else if constexpr (HS) {
        // mean-value rows of the group's blocks (row j: the group's page j, if it is its block's first), as a value tile
        const int first = page_n - gpos;
        it.ntok = -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int idx = lane + 32 * k, row = idx >> 4, c = idx & 15;
          const int blk = __shfl_sync(0xffffffffu, mine.blk, (first + row) & 31);
          const bool real = row < gpos && blk >= 0;
          const bf16 *src = P.vmean + (row0 + (real ? blk : 0)) * P.row_elems + 8 * swz_chunk(c, real ? blk : 0);
          cp_async16(kb + kTileBytes + (uint32_t)(row * kRowBytes + ((c ^ (row & 7)) << 4)), src, real);
        }
#pragma unroll
        for (int k = 0; k < T::NR; ++k) {
          const int row = T::row(lane, k);
          const int blk = __shfl_sync(0xffffffffu, mine.blk, (first + row) & 31);
#pragma unroll
          for (int e = 0; e < 2; ++e)
            it.z[HS ? k : 0][e] = (T::head(lane, e) < G && row < gpos && blk >= 0) ? __ldcg(lz + (size_t)T::head(lane, e) * P.max_blocks + blk) : -CUDART_INF_F;
        }
        gpos = 0;
      }
      return it;
    };
    Item cur;
    cur.ntok = 0;
    if (n_items > 0) cur = issue(0);
    cp_async_commit();
    for (int n = 0, buf = 0; n < n_items; ++n, buf ^= 1) {
      Item nxt;
      nxt.ntok = 0;
      if (n + 1 < n_items) nxt = issue(buf ^ 1);
      cp_async_commit();
      cp_async_wait<1>();
      __syncwarp();
      const uint32_t kb = buf0 + buf * kPageBytes;
      if (cur.ntok > 0) {
        const float lzt[2] = {HS ? -CUDART_INF_F : cur.z[0][0] - cur.lb, HS ? -CUDART_INF_F : cur.z[0][1] - cur.lb};
        attn_page<G>(kb, kb + kTileBytes, w.qa, cur.ntok, lane, sl2, lzt, w);
      } else if constexpr (HS) {
        if (cur.ntok < 0) {
          attn_raise<G>(cur.z, w);
          float x[T::NR][2];
#pragma unroll
          for (int k = 0; k < T::NR; ++k)
#pragma unroll
            for (int e = 0; e < 2; ++e) {   // the negated weights
              x[k][e] = cur.z[k][e] == -CUDART_INF_F ? 0.f : -fast_exp2(cur.z[k][e] - w.m[e]);
              w.l[e] += x[k][e];
            }
          attn_pv<G>(kb + kTileBytes, x, lane, w);
        }
      }
      __syncwarp();
      cur = nxt;
    }
    cp_async_wait<0>();
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(P.status, CKV_DEV_BAD_PAGE);

    // ---- the CTA's partial: its warps (each with its own running maximum) and the last block's mean term ----
    float *wpart = reinterpret_cast<float *>(smem + kOffPages) + (size_t)warp * (2 * kPageBytes / 4);
    __syncwarp();
    w.fold(lane, [&](int g, int c, float v) { wpart[g * CKV_PART_STRIDE + 4 + c] = v; });
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float l = T::sum_rows(w.l[e]);
      if (T::owns(lane, e)) { wpart[T::head(lane, e) * CKV_PART_STRIDE] = w.m[e]; wpart[T::head(lane, e) * CKV_PART_STRIDE + 1] = l; }
    }
    const bool with_tail = comp && rank == C - 1;
    auto entry = [&](int e) { return e < kWarps ? reinterpret_cast<const float *>(smem + kOffPages) + (size_t)e * (2 * kPageBytes / 4) : &s_tail_part[0][0]; };
    work_barrier();
    // thread t: four coordinates of one head over all entries.  Item i = (head, 32 coordinates) is reduced over the
    // cluster by CTA i mod C, into slot i / C.
    for (int idx = tid; idx < G * CKV_D / 4; idx += kWork) {
      const int g = idx / (CKV_D / 4), c = 4 * (idx % (CKV_D / 4));
      float2 ml[kWarps + 1];
      float4 x[kWarps + 1];
      float mine = *(entry(min(lane, kWarps)) + g * CKV_PART_STRIDE);   // a warp works on one head
#pragma unroll
      for (int e = 0; e <= kWarps; ++e) {
        const float *p = entry(e) + g * CKV_PART_STRIDE;
        ml[e] = *reinterpret_cast<const float2 *>(p);
        x[e] = *reinterpret_cast<const float4 *>(p + 4 + c);
      }
      if (!with_tail) {
        ml[kWarps].x = -CUDART_INF_F;
        if (lane >= kWarps) mine = -CUDART_INF_F;
      }
      float M = ml[0].x;
#pragma unroll
      for (int e = 1; e <= kWarps; ++e) M = fmaxf(M, ml[e].x);
      const float sc_mine = exp2_diff(mine, M);
      float den = 0.f;
      float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int e = 0; e <= kWarps; ++e) {
        const float sc = __shfl_sync(0xffffffffu, sc_mine, e);
        if (sc != 0.f) {   // an entry that holds nothing may hold any bits
          den = fmaf(ml[e].y, sc, den);
          num.x = fmaf(x[e].x, sc, num.x); num.y = fmaf(x[e].y, sc, num.y);
          num.z = fmaf(x[e].z, sc, num.z); num.w = fmaf(x[e].w, sc, num.w);
        }
      }
      const int item = 4 * g + (c >> 5), slot = div_c(item);
      const uint32_t to = (uint32_t)(item - slot * C);
      const uint32_t ent = smem_u32(s_recv) + (uint32_t)((slot * C + rank) * kRecvStride) * 4u;
      const uint32_t bar = cluster_map(smem_u32(&s_xbar[2]), to);
      st_async_u32x4(cluster_map(ent + (c & 31) * 4, to), __float_as_uint(num.x), __float_as_uint(num.y), __float_as_uint(num.z),
                     __float_as_uint(num.w), bar);
      if ((c & 31) == 0) st_async_f32x2(cluster_map(ent + 128, to), M, den, bar);
    }
    // ---- the outputs this CTA reduces over the cluster: a warp per item ----
    if (4 * G > rank) wait_x(2);
    for (int slot = warp; slot * C + rank < 4 * G; slot += kWarps) {
      const int item = slot * C + rank, g = item >> 2, c = (item & 3) * 32 + lane;
      const float *e0 = s_recv + (size_t)slot * C * kRecvStride;
      const float mine = e0[min(lane, C - 1) * kRecvStride + 32];
      const float M = warp_max(mine);
      float den = 0.f, o = 0.f;
      // eight entries at a time, those past the last with a weight of zero: a loop with a remainder, like any other code here,
      // costs its length (24 units of 100K with bf16 summaries 27.2 us a step that way, 26.7 this way)
      const float sc_mine = lane < C ? exp2_diff(mine, M) : 0.f;
      for (int e = 0; e < C; e += 8)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float *p = e0 + min(e + j, C - 1) * kRecvStride;
          const float sc = __shfl_sync(0xffffffffu, sc_mine, e + j);
          den = fmaf(p[33], sc, den);
          o = fmaf(p[lane], sc, o);
        }
      out[((size_t)unit * G + g) * CKV_D + c] = __float2bfloat16_rn(N > 0 ? o / den : 0.f);   // an empty sequence: zero
      if (lse != nullptr && (item & 3) == 0 && lane == 0) lse[(size_t)unit * G + g] = N > 0 ? (M + log2f(den)) * kLn2 : -CUDART_INF_F;
    }
  }
  if (done.flag != nullptr) {   // the results are in the caller's host buffers: the last CTA to say so stores the word
    __syncthreads();
    if (tid == 0) {
      __threadfence();   // the CTA's results before its count ...
      if (atomicAdd(done.ctas, 1) == (int)(gridDim.x * gridDim.y) - 1) {
        __threadfence_system();   // ... and all that were counted before the word, as the host sees it
        *done.ctas = 0;
        const int e = *done.count + 1;   // counted on the device, call after call
        *done.count = e;
        *(volatile int *)done.flag = e;
      }
    }
  }
  __syncwarp();
  cluster_arrive_relaxed();   // nobody leaves while somebody may still send to it
  cluster_wait();
  if (counts && !normed) store_lens(P.status + CKV_LEN_COUNTER_WORD, fresh.seq_lens, batch, cap, (int)gridDim.y);
}

// The instantiation a context's layout uses.
template <int G> const void *kernel_g(const CkvDev &P) {
  if (P.r == CKV_D) return (const void *)ckv_unit_step_kernel<G, true, false, false>;
  if (P.row_elems == CKV_D) return (const void *)ckv_unit_step_kernel<G, false, true, false>;
  if (P.vhi) return (const void *)ckv_unit_step_kernel<G, false, false, true>;
  return (const void *)ckv_unit_step_kernel<G, false, false, false>;
}
const void *kernel_of(const CkvDev &P) {
  switch (P.G) {
    case 1: return kernel_g<1>(P);
    case 2: return kernel_g<2>(P);
    case 4: return kernel_g<4>(P);
    case 8: return kernel_g<8>(P);
  }
  return nullptr;
}

cudaLaunchConfig_t launch_config(int C, int units, size_t smem, cudaStream_t st, cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C, units);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

// Attributes of the context's instantiation, and how many clusters of each size the device holds at once (every CTA
// takes an SM for itself, so the answer depends on the device alone: asked once per device).
cudaError_t ckv_configure_unit_step(ckv_ctx *c) {
  for (int i = 0; i <= CKV_STEP_MAX_CLUSTER; ++i) c->step_clusters[i] = 0;
  if (c->layout.kv_dtype != CKV_BF16) return cudaSuccess;
  const void *k = kernel_of(c->dev);
  if (k == nullptr) return cudaErrorInvalidValue;
  // What the static arrays leave: all of kDynMost today, with groups of eight to the byte; a field more in the structs that
  // are copied into shared memory makes the ring a little smaller, and no context fails.
  cudaFuncAttributes fa = {};
  cudaError_t e = cudaFuncGetAttributes(&fa, k);
  if (e != cudaSuccess) return e;
  c->step_smem = std::min(kDynMost, (kSmemCta - (int)fa.sharedSizeBytes) / 1024 * 1024);
  if (c->step_smem < kAfterScan) return cudaSuccess;   // the step stays with its separate launches
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, c->step_smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  int dev = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  constexpr int kMaxDev = 64;
  static std::mutex mtx;
  static int table[kMaxDev][CKV_STEP_MAX_CLUSTER + 1];
  static bool known[kMaxDev];
  if (dev < 0 || dev >= kMaxDev) return cudaSuccess;   // no table: the step stays with its separate launches
  std::lock_guard<std::mutex> lock(mtx);
  if (!known[dev]) {
    for (int C = 1; C <= CKV_STEP_MAX_CLUSTER; ++C) {
      cudaLaunchAttribute attr[1];
      cudaLaunchConfig_t cfg = launch_config(C, 1, kAfterScan, nullptr, attr);
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
      table[dev][C] = n;
    }
    known[dev] = true;
  }
  for (int C = 1; C <= CKV_STEP_MAX_CLUSTER; ++C) c->step_clusters[C] = table[dev][C];
  return cudaSuccess;
}

// Whether a step of this size runs as one launch, and how.  All figures: one launch / the faster form of the separate
// launches, us per step, sixteen steps replayed back to back, pages in random order, budgets of 2K tokens where nothing is
// said.  11.3 / 20.1 (one head, 4K, 256 tokens), 12.3 / 25.3 (8 units, 32K, 1K tokens), 16.4 / 29.4 (8 units, 128K, 32-token
// blocks, 4K tokens), 29.5 / 39.0 (24 units, 100K, bf16 summaries), 36.4 / 47.7 (16 units, 88K, r = d), 47.6 / 64.1 (32 units,
// 128K), 56.8 / 77.3 (72 units, 64K), 63.7 / 74.6 (128 units, 32K).
// What stays with the separate launches, and why:
//   * fp32 pages (the attention is on bf16 tensor cores) and an explicit ckv_set_tail_mode, which asks for them;
//   * caches under CKV_STEP_MIN_TOKENS.  Not a crossover -- one launch is ahead there too (one sequence of 1600 tokens 11.8 /
//     21.4, 16 of them 21.1 / 30.4) -- but the size below which the documented two-call arrangement (append, scan, select,
//     attention as launches of their own) is kept;
//   * more units than CTAs run at once: a last wave that is nearly empty costs a whole wave (192 units, one CTA each: 8K 73.8 /
//     76.1, 16K 89.7 / 89.7, 32K 117.6 / 113.5; 256 units, whose last wave is not, 16K 96.3 / 108.0);
//   * more than kOwnMost blocks a CTA where a sequence gets fewer than kSeqCtas of them.  The host knows the longest
//     sequence only: alone among short ones, its few CTAs are all that works.  128 units of the default layout, all
//     long, then lengths of a quarter and up, then one long and 15 of 1K: 32K 63.5 / 74.7, 55.7 / 66.7, 48.4 / 40.0; 40K 71.3 /
//     84.1, 62.6 / 71.3, 54.0 / 41.1; 56K 86.8 / 101.1, 77.3 / 84.9, 66.2 / 43.8; one head a group, 130K 152 / 172, 133 / 131,
//     114 / 51.  From 45K a CTA on the uneven batch loses a third and more, against a gain of a tenth that is gone at 130K.
//     (24 CTAs a sequence, 128K: 57.7 / 76.7, 52.0 / 66.3, 44.6 / 38.4: no line.  Groups other than 4 and 128: one launch is
//     ahead either way, 77.6 / 148, 68.4 / 196, 66.6 / 102 at 32K with 16 of them.);
//   * large selections where the clusters leave SMs idle (selected bytes x idle share from kIdleMost on): the attention is most
//     of such a step, and a launch of its own keeps the whole chip at it.  64-token blocks, with the product: 80 units (68
//     SMs idle) 4K tokens of 32K 51.6 / 56.7 / 77 MB, 8K of 16K 82.4 / 76.0 / 154, 32K of 40K 286 / 221 / 616; 104 units 8K of
//     16K 90.7 / 93.3 / 130; 128 units 8K of 16K 98.5 / 107.0 / 72, 16K of 40K 184.7 / 192.9 / 145.  (The line is from before
//     the step got faster; by these figures it costs 3 to 4 % between 80 MB and 150.)  Not where the
//     attention's own clusters fill more than nine tenths of their places, two a SM, and no longer pack: 72 units in
//     clusters of 4 (288 CTAs), 32K of 40K 193 / 259;
//   * more selected blocks or scores than the shared arrays hold, or score terms that leave no room for the ring: one CTA
//     per unit with eight heads beyond about 30K tokens.  There the persistent scan's even split of the tiles is worth
//     more (a long sequence of a ragged batch is one CTA's work here), and its three launches are kept.
bool ckv_unit_step_plan(const ckv_ctx *c, int batch, int max_len, int kcap, CkvStepPlan *plan) {
  const CkvDev &P = c->dev;
  if (c->layout.kv_dtype != CKV_BF16 || c->tail_mode != CKV_TAIL_AUTO || max_len < CKV_STEP_MIN_TOKENS) return false;
  const int units = batch * P.Hkv, xmax = (max_len + P.bs - 1) / P.bs;
  if (xmax > kScoresCap || (kcap < xmax && kcap > kSelCap)) return false;
  int C = 0;
  for (int k = CKV_STEP_MAX_CLUSTER; k >= 1 && C == 0; --k)
    if (c->step_clusters[k] >= units) C = k;
  if (C == 0) return false;
  if (kcap < xmax) {
    const int sms = c->sm_count, splits = std::min(std::max(2 * sms / units, 1), 8);   // as ckv_launch_attn splits it
    const long long selected = (long long)units * kcap * P.bs * (2 * CKV_D * 2), idle = std::max(sms - C * units, 0);
    if (selected * idle >= kIdleMost * sms && splits * units * 10 <= 2 * sms * 9) return false;
  }
  const int skip = kWarps / (P.scan_tile / 16);
  const size_t krow = (size_t)P.row_elems * 2, vrow = (P.vhi || P.row_elems == CKV_D) ? (size_t)CKV_D * 2 : krow;
  const size_t stage = (size_t)P.scan_tile * (krow + vrow) + (P.r >= 4 ? (size_t)P.scan_tile * P.r * 4 : 0);
  auto blocks_per_cta = [C](int x) { const int parts = (std::max(x - 1, 0) + 15) / 16; return 16 * std::max((parts + C - 1) / C, 1); };
  auto term_bytes = [&P](int own) { return (size_t)(own + 8) * P.G * sizeof(float); };
  plan->own_cap = blocks_per_cta(xmax);
  plan->early_parts = plan->own_cap / 16;
  plan->hi_page = std::min((max_len - 1) / CKV_PAGE, P.max_pages_per_seq - 1);
  if (plan->own_cap > kOwnMost && P.Hkv * C < kSeqCtas && (P.r == 4 || P.r == CKV_D)) return false;
  if (term_bytes(plan->own_cap) + (size_t)std::max(kMinRing, skip) * stage > (size_t)c->step_smem) return false;
  const int tiles = (plan->own_cap + P.scan_tile - 1) / P.scan_tile;
  plan->stages = std::min({kStagesCap, (int)(((size_t)c->step_smem - term_bytes(plan->own_cap)) / stage), std::max(tiles, skip)});
  plan->u_off = (int)(plan->stages * stage);
  plan->max_blocks = xmax;
  // Where the arrays can be sized for the cache's capacity beside the same ring, they are: a bound that turns out too small
  // (a captured step replayed once too often) then costs nothing.
  const int full = blocks_per_cta(P.max_blocks);
  if (P.max_blocks <= kScoresCap && (kcap >= P.max_blocks || kcap <= kSelCap) && plan->u_off + term_bytes(full) <= (size_t)c->step_smem) {
    plan->own_cap = full;
    plan->max_blocks = P.max_blocks;
  }
  plan->smem = (int)std::max(plan->u_off + term_bytes(plan->own_cap), (size_t)kAfterScan);
  plan->cluster = C;
  plan->c_magic = C > 1 ? (unsigned)(0x100000000ull / (unsigned)C) + 1u : 0u;
  return true;
}

cudaError_t ckv_launch_unit_step(ckv_ctx *c, const CkvStepPlan &plan, const void *q, const void *k_pool, const void *v_pool,
                                 const int *page_table, const int *seq_lens, const CkvNewToken *fresh_in, int batch, int kcap,
                                 int *sel_ids, int *sel_cnt, void *out, float *lse, const CkvHostDone &done_in, cudaStream_t st) {
  CkvHostDone done = done_in;
  CkvNewToken fresh = {};
  if (fresh_in != nullptr) fresh = *fresh_in;
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = launch_config(plan.cluster, batch * c->dev.Hkv, plan.smem, st, attr);
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  CkvStepPlan p = plan;
  void *args[] = {&c->dev, &q, &seq_lens, &k_pool, &v_pool, &page_table, &fresh, &kcap, &p, &batch, &sel_ids, &sel_cnt, &out, &lse, &done, &c->tm_vhi};
  c->launches++;
  return cudaLaunchKernelExC(&cfg, kernel_of(c->dev), args);
}
