// The scan's work on 16 blocks of a unit by one warp (Eq. 8-9 and the compensation sums of Eq. 12), shared by the
// persistent scan kernel and by the one-launch step: block-mean logits and grouped variances on tensor cores, the two
// per-(head, block) terms the later stages read, the running maximum, and the weighted sum of the mean values.
#ifndef CKV_SCANPART_CUH_
#define CKV_SCANPART_CUH_
#include "ckv_internal.cuh"
#include "ckv_attnpage.cuh"
#include "ckv_mma.cuh"
#include "ckv_pipe.cuh"

template <bool WIDE> struct ScanTile { static constexpr int TB = WIDE ? CKV_SCAN_TILE_HS : CKV_SCAN_TILE; };   // blocks per tile

// One box of a tensor map from global to shared memory (x: first element of the row, y: first row); completion is
// counted on `bar` in bytes -- always the whole box, rows past the tensor's end arriving as zeros.
__device__ __forceinline__ void tensor_g2s(uint32_t dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
               "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(ckv_pipe::smem_u32(bar))
               : "memory");
}

template <typename QT> struct QSplit { static constexpr bool value = false; };
template <> struct QSplit<float> { static constexpr bool value = true; };

// What a warp holds of the unit it works on.
template <int G, typename QT, bool RD>
struct ScanUnit : HeadAcc<G> {
  using T = HeadTile<G>;
  static constexpr bool QS = QSplit<QT>::value;        // fp32 queries are split into hi + lo like the summaries
  static constexpr bool QB = QS && !T::PAIR;           // ... as a second operand where columns 4..7 cannot take the lo halves
  uint32_t qa[8][2], qb[QB ? 8 : 1][2];                // B fragments of the unit's queries, per 16-coordinate step
  uint32_t qs[RD ? 8 : 1][2], qs2[RD ? 8 : 1][2];      // (scale q)^2 as hi and lo halves, same fragment positions
  float wown[2][4];                                    // variance weights of this lane's heads (r = 4)
  float lp[2];                                         // sum of e^{l - m}

  __device__ __forceinline__ void reset() {
    HeadAcc<G>::reset();
    lp[0] = lp[1] = 0.f;
  }
  // Query fragments; row(head, c): coordinates c, c + 1 of a head as floats.
  template <class F>
  __device__ __forceinline__ void set_queries(int lane, float scale, F row) {
    const int h = T::col_head(lane), qd = lane & 3;
    const bool hv = h < G, low = T::PAIR && lane >= 16;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const float2 x = hv ? row(h, 16 * ks + 8 * hh + 2 * qd) : make_float2(0.f, 0.f);
        const uint32_t xh = pack_bf16(x.x, x.y);
        if constexpr (QS) {
          const uint32_t xl = pack_bf16(x.x - __uint_as_float(xh << 16), x.y - __uint_as_float(xh & 0xffff0000u));
          qa[ks][hh] = low ? xl : xh;
          if constexpr (QB) qb[QB ? ks : 0][hh] = xl;
        } else {
          qa[ks][hh] = xh;
        }
        if constexpr (RD) {
          const float s0 = (x.x * scale) * (x.x * scale), s1 = (x.y * scale) * (x.y * scale);
          const uint32_t sh = pack_bf16(s0, s1);
          const uint32_t sl = pack_bf16(s0 - __uint_as_float(sh << 16), s1 - __uint_as_float(sh & 0xffff0000u));
          qs[RD ? ks : 0][hh] = sh;
          qs2[RD ? ks : 0][hh] = sl;
        }
      }
  }
  // The same from bf16 rows in shared memory `stride` bytes apart (an odd multiple of 16, so that eight rows fall into
  // different banks), four matrix loads in all; zero_row: what heads past G are read as.
  __device__ __forceinline__ void load_queries(int lane, float scale, uint32_t rows, uint32_t stride, uint32_t zero_row) {
    static_assert(!QS, "bf16 queries");
    // lane roles: matrix lane / 8 -> eight coordinates, row lane % 8 -> column of the product
    const int col = lane & 7, head = T::PAIR ? col & 3 : col;
    const uint32_t at = (head < G ? rows + (uint32_t)head * stride : zero_row) + (uint32_t)((lane >> 3) << 4);
#pragma unroll
    for (int ks = 0; ks < 8; ks += 2) {
      uint32_t r[4];
      ldmatrix_x4(r, at + 32u * ks);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        qa[ks + (i >> 1)][i & 1] = r[i];
        if constexpr (RD) {
          const float x0 = __uint_as_float(r[i] << 16) * scale, x1 = __uint_as_float(r[i] & 0xffff0000u) * scale;
          const float s0 = x0 * x0, s1 = x1 * x1;
          const uint32_t sh = pack_bf16(s0, s1);
          qs[RD ? ks + (i >> 1) : 0][i & 1] = sh;
          qs2[RD ? ks + (i >> 1) : 0][i & 1] = pack_bf16(s0 - __uint_as_float(sh << 16), s1 - __uint_as_float(sh & 0xffff0000u));
        }
      }
    }
  }
};

// Parameters of a part that do not change between a warp's parts.
struct ScanPartCfg {
  float scale, half_var, log_bs;
  int r, max_blocks;
  bool by_mass, r4;
};

// One part: rows rb .. rb + 15 of the tile whose first block is b0 and which holds nb blocks.  sk / sv / sd: the tile's
// mean keys, mean values and variances in shared memory; zero_row: 512 bytes of zeros, 128-byte aligned (what mean-value rows past nb are
// read as: a stale NaN pattern times a zero weight would poison the accumulators; elsewhere a block is an output column,
// and those columns are discarded).  b_partial: the block that may hold fewer than block_size tokens (-1: none), with
// log_partial the log of its token count.  sw: variance weights [t][g] for r not 4 or d; dbar_row0: the unit's variance
// rows in global memory when the tile does not carry them (sd null).
// store(head, block, u, z): log2 of a block's score term and of its mean-term weight, for one head.
// RD: one variance group per coordinate (r = d): sigma^2 = sum_i (scale q_i)^2 Dbar_i is a third tensor-core product.
// HS: the mean rows hold hi halves only.  VH: only the mean VALUES' hi halves were brought in.
template <int G, typename QT, bool RD, bool HS, bool VH, class Store>
__device__ __forceinline__ void scan_part(ScanUnit<G, QT, RD> &w, const ScanPartCfg &cfg, uint32_t sk, uint32_t sv,
                                          const float *sd, uint32_t zero_row, const float *sw, const float *dbar_row0,
                                          int lane, int rb, int nb, int b0, int b_partial, float log_partial, Store store) {
  constexpr int kRowBytes = HS ? CKV_D * 2 : CKV_ROW_ELEMS * 2;            // bytes of one mean-key row in a stage
  constexpr int kRowBytesV = (HS || VH) ? CKV_D * 2 : CKV_ROW_ELEMS * 2;   // ... of one mean-value row
  constexpr int TB = ScanTile<HS || VH>::TB;
  using T = HeadTile<G>;

  // ---- Z = Kbar Q^T: 16 blocks x heads, hi and lo planes of the mean keys into one sum ----
  // four accumulation chains (hi / lo plane x even / odd 16-coordinate step): the products of a chain depend on one
  // another, and a warp has little else to issue while it waits for them
  float z[4] = {0.f, 0.f, 0.f, 0.f}, z2[4] = {0.f, 0.f, 0.f, 0.f}, zl[4] = {0.f, 0.f, 0.f, 0.f}, zl2_[4] = {0.f, 0.f, 0.f, 0.f};
  // ldmatrix lane roles: matrix lane / 8 -> (row half, coordinate chunk parity), row lane % 8
  const int kr = rb + ((lane >> 3) & 1) * 8 + (lane & 7);
  const uint32_t kx = ((lane >> 4) ^ (lane & 7)) << 4;   // chunk parity and row swizzle (rb is a multiple of 8)
  {
    const uint32_t rowaddr = (sk + kr * kRowBytes) | kx;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      const uint32_t at = swz_at(rowaddr, ks);
      uint32_t ah[4], al[4];
      ldmatrix_x4(ah, at);
      mma_16816((ks & 1) ? z2 : z, ah, w.qa[ks][0], w.qa[ks][1]);
      if (!HS) {
        ldmatrix_x4(al, at + 256);
        mma_16816((ks & 1) ? zl2_ : zl, al, w.qa[ks][0], w.qa[ks][1]);
      }
      if constexpr (ScanUnit<G, QT, RD>::QB) mma_16816((ks & 1) ? zl2_ : zl, ah, w.qb[ks][0], w.qb[ks][1]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] = (z[i] + z2[i]) + (zl[i] + zl2_[i]);
    if constexpr (QSplit<QT>::value && T::PAIR) T::add_copies(z);   // columns 4..7: the queries' lo halves
  }
  float sgm[T::NR][2];
  if constexpr (RD) {   // sigma^2 for the same tile: (qs_hi + qs_lo) (D_hi + D_lo) without the lo lo term
    float g[4] = {0.f, 0.f, 0.f, 0.f}, g2[4] = {0.f, 0.f, 0.f, 0.f};
    const uint32_t rowaddr = (sv + TB * kRowBytes + kr * kRowBytes) | kx;
#pragma unroll
    for (int ks = 0; ks < 8; ks += 2) {   // the order of the chains is part of the result: scores that differ in the last bit
      uint32_t dh[2][4], dl[2][4];        // can swap blocks at the cut
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const uint32_t at = swz_at(rowaddr, ks + j);
        ldmatrix_x4(dh[j], at);
        ldmatrix_x4(dl[j], at + 256);
        mma_16816(g, dh[j], w.qs[RD ? ks + j : 0][0], w.qs[RD ? ks + j : 0][1]);
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) mma_16816(g2, dh[j], w.qs2[RD ? ks + j : 0][0], w.qs2[RD ? ks + j : 0][1]);
#pragma unroll
      for (int j = 0; j < 2; ++j) mma_16816(g2, dl[j], w.qs[RD ? ks + j : 0][0], w.qs[RD ? ks + j : 0][1]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) g[i] += g2[i];
    T::pick(g, lane, sgm);
  }

  // ---- per (block, head): variance projection, l, running maximum, compensation weight ----
  float zin[T::NR][2], zw[T::NR][2], sig[T::NR][2], wt[T::NR][2];
  T::pick(z, lane, zin);
#pragma unroll
  for (int k = 0; k < T::NR; ++k) {
    const int r = rb + T::row(lane, k), b = b0 + r;
    const bool real = r < nb;
    const float logc = b == b_partial ? log_partial : cfg.log_bs;
    float4 dv = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool r4 = VH || cfg.r4;   // VH comes with four variance groups only
    if (!RD && r4 && real) dv = *reinterpret_cast<const float4 *>(sd + r * 4);
    // r not 4 or d: both heads' sums from one reading of the row, four variances at a time (the 16 rows of a part lie in the
    // same banks when r >= 32; one by one and once per head, a step of 128 units of 48K took 564 us with r = 64, now 350)
    float sgr[2] = {0.f, 0.f};
    if (!RD && !r4 && real) {
      const float *swh[2] = {sw + (T::head(lane, 0) & (G - 1)), sw + (T::head(lane, 1) & (G - 1))};
      if (sd != nullptr) {
        for (int t = 0; t < cfg.r; t += 4) {
          const float4 d4 = *reinterpret_cast<const float4 *>(sd + r * cfg.r + t);
          const float d[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) sgr[e] = fmaf(swh[e][(t + j) * G], d[j], sgr[e]);
        }
      } else {
        for (int t = 0; t < cfg.r; ++t) {
          const float d = dbar_row0[(size_t)b * cfg.r + t];
#pragma unroll
          for (int e = 0; e < 2; ++e) sgr[e] = fmaf(swh[e][t * G], d, sgr[e]);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int head = T::head(lane, e);
      const bool val = real && head < G;
      float sg = 0.f;
      if (val) {
        if constexpr (RD) {
          sg = fmaxf(sgm[k][e], 0.f);
        } else if (r4) {
          sg = fmaf(w.wown[e][0], dv.x, fmaf(w.wown[e][1], dv.y, fmaf(w.wown[e][2], dv.z, w.wown[e][3] * dv.w)));
        } else {
          sg = sgr[e];
        }
      }
      sig[k][e] = sg;
      const float zbar = zin[k][e] * cfg.scale;
      const float ell = logc + zbar + cfg.half_var * sg;
      zw[k][e] = val ? (zbar + logc) * kLog2e : -CUDART_INF_F;   // log2 of |b| e^{zbar}
      // what the later stages read, both in log2 units: the head's term of the block score, e^l sigma^2 (e^l alone
      // when blocks are ranked by mass), and the block's mean-compensation weight |b| e^{zbar}
      if (val) store(head, b, fmaf(ell, kLog2e, cfg.by_mass ? 0.f : __log2f(sg)), zw[k][e]);
    }
  }
  {   // the running maximum is only raised when exceeded by a slack
    const float m0 = w.m[0], m1 = w.m[1];
    attn_raise<G>(zw, w);
    if (w.m[0] != m0) w.lp[0] *= exp2_diff(m0, w.m[0]);
    if (w.m[1] != m1) w.lp[1] *= exp2_diff(m1, w.m[1]);
  }
#pragma unroll
  for (int k = 0; k < T::NR; ++k)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      wt[k][e] = zw[k][e] == -CUDART_INF_F ? 0.f : fast_exp2(zw[k][e] - w.m[e]);
      w.l[e] += wt[k][e];
      w.lp[e] = fmaf(wt[k][e], fast_exp2(cfg.half_var * kLog2e * sig[k][e]), w.lp[e]);   // e^{l - m} = e^{zbar + log|b| - m} e^{sigma^2/2}
    }

  // ---- acc += Vbar^T W: 128 coordinates x heads, k = this part's 16 blocks ----
  {
    uint32_t b[T::NR][2];
    T::weights(wt, lane, b);
    // ldmatrix.trans lane roles: matrix lane / 8 -> (coordinate chunk parity, row half), row lane % 8
    const int r = rb + (lane >> 4) * 8 + (lane & 7);
    // rows past the last block: the row of zeros, which is as long as a stored row
    const uint32_t rowaddr = (r < nb ? sv + r * kRowBytesV : zero_row) | ((((lane >> 3) & 1) ^ (lane & 7)) << 4);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const uint32_t at = swz_at(rowaddr, t);
      uint32_t vh[4];
      ldmatrix_x4_trans(vh, at);
      mma_16816(w.acc[t], vh, b[0][0], b[0][1]);
      if constexpr (!T::PAIR) mma_16816(w.acc[t], vh, b[T::NR - 1][0], b[T::NR - 1][1]);
      if constexpr (!HS && !VH) {
        uint32_t vl[4];
        ldmatrix_x4_trans(vl, at + 256);
        mma_16816(w.acc[t], vl, b[0][0], b[0][1]);
      }
    }
  }
}

#endif  // CKV_SCANPART_CUH_
