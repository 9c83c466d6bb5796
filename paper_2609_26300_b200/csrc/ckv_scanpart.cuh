// The scan's work on 16 blocks of a unit by one warp (Eq. 8-9 and the compensation sums of Eq. 12), shared by the
// persistent scan kernel and by the one-launch step: block-mean logits and grouped variances on tensor cores, the two
// per-(head, block) terms the later stages read, the running maximum, and the weighted sum of the mean values.
#ifndef CKV_SCANPART_CUH_
#define CKV_SCANPART_CUH_
#include "ckv_internal.cuh"
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

// What a warp holds of the unit it works on.  Rows (heads) of the fragments: head = lane / 4 < G, zero otherwise.
template <int G, typename QT, bool RD>
struct ScanUnit {
  static constexpr bool QS = QSplit<QT>::value;      // fp32 queries are split into hi + lo like the summaries
  uint32_t qa[8][2], qb[QS ? 8 : 1][2];              // A fragments of the unit's queries (rows 0..7), per 16-coordinate step
  uint32_t qsh[RD ? 8 : 1][2], qsl[RD ? 8 : 1][2];   // (scale q)^2 as hi and lo halves, same fragment positions
  float acc[16][2];                                  // W Vbar accumulator: head `head`, coordinates 8 t + 2 qd + {0, 1}
  float wown[4];                                     // variance weights of this lane's head (r = 4)
  float m_ref, l_acc, lp_acc;                        // running maximum, sum of weights, sum of e^{l - m}

  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int t = 0; t < 16; ++t) { acc[t][0] = 0.f; acc[t][1] = 0.f; }
    m_ref = -CUDART_INF_F; l_acc = 0.f; lp_acc = 0.f;
  }
};

// Parameters of a part that do not change between a warp's parts.
struct ScanPartCfg {
  float scale, half_var, log_bs;
  int r, max_blocks;
  bool by_mass, r4;
};

// One part: rows rb .. rb + 15 of the tile whose first block is b0 and which holds nb blocks.  sk / sv / sd: the tile's
// mean keys, mean values and variances in shared memory; zero_row: 512 bytes of zeros (what mean-value rows past nb are
// read as: a stale NaN pattern times a zero weight would poison the accumulators; elsewhere a block is an output column,
// and those columns are discarded).  b_partial: the block that may hold fewer than block_size tokens (-1: none), with
// log_partial the log of its token count.  sw: variance weights [t][g] for r not 4 or d; dbar_row0: the unit's variance
// rows in global memory when the tile does not carry them (sd null).
// store(head, block, u0, u1, z0, z1, v0, v1): log2 of the score terms and of the mean-term weights of blocks `block` and
// `block` + 1 for one head; v0 / v1: whether they exist.
// RD: one variance group per coordinate (r = d): sigma^2 = sum_i (scale q_i)^2 Dbar_i is a third tensor-core product.
// HS: the mean rows hold hi halves only.  VH: only the mean VALUES' hi halves were brought in.
template <int G, typename QT, bool RD, bool HS, bool VH, class Store>
__device__ __forceinline__ void scan_part(ScanUnit<G, QT, RD> &w, const ScanPartCfg &cfg, uint32_t sk, uint32_t sv,
                                          const float *sd, uint32_t zero_row, const float *sw, const float *dbar_row0,
                                          int lane, int rb, int nb, int b0, int b_partial, float log_partial, Store store) {
  constexpr bool QS = QSplit<QT>::value;
  constexpr int kRowBytes = HS ? CKV_D * 2 : CKV_ROW_ELEMS * 2;            // bytes of one mean-key row in a stage
  constexpr int kRowBytesV = (HS || VH) ? CKV_D * 2 : CKV_ROW_ELEMS * 2;   // ... of one mean-value row
  constexpr int TB = ScanTile<HS || VH>::TB;
  constexpr bool SP = (G <= 4) && !RD;   // the per-(head, block) arithmetic is shared between the half warps
  constexpr int NE = SP ? 1 : 2;         // n-tiles a lane works on there
  const int head = lane >> 2, qd = lane & 3;   // this thread's accumulator row (head) and column pair
  const int hsel = lane >> 4;                  // ... and which n-tile: the lower half warp the first, the upper the second
  const int ehead = SP ? (head & 3) : head;
  const bool ehv = ehead < G;

  // ---- Z^T = Q Kbar^T: heads x 16 blocks (two n-tiles of 8 blocks), hi and lo planes into one accumulator ----
  // four accumulation chains per n-tile (hi / lo plane x even / odd 16-coordinate step): the products of a chain
  // depend on one another, and a warp has little else to issue while it waits for them
  float z[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, zlo[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  float z2[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, zlo2[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  {
    // ldmatrix lane roles: matrix lane / 8 -> 8-coordinate chunk, row lane % 8
    const int lrow = lane & 7, lmat = lane >> 3;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int r = rb + nt * 8 + lrow;
      const uint32_t rowaddr = sk + r * kRowBytes;
#pragma unroll
      for (int j = 0; j < 4; ++j) {   // two 16-coordinate steps per ldmatrix.x4
        const uint32_t coff = (uint32_t)swz_chunk(4 * j + lmat, r) * 16;
        uint32_t bh[4], bl[4];
        ldmatrix_x4(bh, rowaddr + coff);
        mma_rows8(z[nt][0], z[nt][1], w.qa[2 * j][0], w.qa[2 * j][1], bh[0], bh[1]);
        mma_rows8(z2[nt][0], z2[nt][1], w.qa[2 * j + 1][0], w.qa[2 * j + 1][1], bh[2], bh[3]);
        if (!HS) {
          ldmatrix_x4(bl, rowaddr + 256 + coff);
          mma_rows8(zlo[nt][0], zlo[nt][1], w.qa[2 * j][0], w.qa[2 * j][1], bl[0], bl[1]);
          mma_rows8(zlo2[nt][0], zlo2[nt][1], w.qa[2 * j + 1][0], w.qa[2 * j + 1][1], bl[2], bl[3]);
        }
        if (QS) {
          mma_rows8(zlo[nt][0], zlo[nt][1], w.qb[QS ? 2 * j : 0][0], w.qb[QS ? 2 * j : 0][1], bh[0], bh[1]);
          mma_rows8(zlo[nt][0], zlo[nt][1], w.qb[QS ? 2 * j + 1 : 0][0], w.qb[QS ? 2 * j + 1 : 0][1], bh[2], bh[3]);
        }
      }
      z[nt][0] = (z[nt][0] + z2[nt][0]) + (zlo[nt][0] + zlo2[nt][0]);
      z[nt][1] = (z[nt][1] + z2[nt][1]) + (zlo[nt][1] + zlo2[nt][1]);
    }
  }
  float sgm[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  if (RD) {   // sigma^2 for the same heads x blocks tile: (qs_hi + qs_lo) (D_hi + D_lo) without the lo lo term
    float sg2[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
    const uint32_t sdr = sv + TB * kRowBytes;
    const int lrow = lane & 7, lmat = lane >> 3;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int r = rb + nt * 8 + lrow;
      const uint32_t rowaddr = sdr + r * kRowBytes;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t coff = (uint32_t)swz_chunk(4 * j + lmat, r) * 16;
        uint32_t dh[4], dl[4];
        ldmatrix_x4(dh, rowaddr + coff);
        ldmatrix_x4(dl, rowaddr + 256 + coff);
        mma_rows8(sgm[nt][0], sgm[nt][1], w.qsh[RD ? 2 * j : 0][0], w.qsh[RD ? 2 * j : 0][1], dh[0], dh[1]);
        mma_rows8(sgm[nt][0], sgm[nt][1], w.qsh[RD ? 2 * j + 1 : 0][0], w.qsh[RD ? 2 * j + 1 : 0][1], dh[2], dh[3]);
        mma_rows8(sg2[nt][0], sg2[nt][1], w.qsl[RD ? 2 * j : 0][0], w.qsl[RD ? 2 * j : 0][1], dh[0], dh[1]);
        mma_rows8(sg2[nt][0], sg2[nt][1], w.qsl[RD ? 2 * j + 1 : 0][0], w.qsl[RD ? 2 * j + 1 : 0][1], dh[2], dh[3]);
        mma_rows8(sg2[nt][0], sg2[nt][1], w.qsh[RD ? 2 * j : 0][0], w.qsh[RD ? 2 * j : 0][1], dl[0], dl[1]);
        mma_rows8(sg2[nt][0], sg2[nt][1], w.qsh[RD ? 2 * j + 1 : 0][0], w.qsh[RD ? 2 * j + 1 : 0][1], dl[2], dl[3]);
      }
      sgm[nt][0] += sg2[nt][0]; sgm[nt][1] += sg2[nt][1];
    }
  }

  // ---- per (head, block): variance projection, l, running maximum, compensation weight ----
  // The products leave this part's 16 blocks x G heads in the lanes of rows 0..G-1 (four values per lane).
  // With G <= 4 those are lanes 0-15 only, so the upper half warp takes over the second n-tile: every lane
  // then works on one n-tile's pair of blocks (half the dependent chain), and the weights travel back to
  // the lower lanes, which hold the A operand of the next product.
  float zin[NE][2];
  if constexpr (SP) {
    const float t0 = __shfl_sync(0xffffffffu, z[1][0], lane & 15), t1 = __shfl_sync(0xffffffffu, z[1][1], lane & 15);
    zin[0][0] = hsel ? t0 : z[0][0];
    zin[0][1] = hsel ? t1 : z[0][1];
  } else {
#pragma unroll
    for (int k = 0; k < NE; ++k) { zin[k][0] = z[k][0]; zin[k][1] = z[k][1]; }
  }
  float zl2[NE][2], sig[NE][2], wt[NE][2];
  bool val[NE][2];
  float tmax = -CUDART_INF_F;
#pragma unroll
  for (int k = 0; k < NE; ++k) {
    const int nt = SP ? hsel : k;
    const int r0 = rb + nt * 8 + 2 * qd;     // this thread's two blocks of the n-tile: rows r0, r0 + 1
    float ell[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int r = r0 + e, b = b0 + r;
      val[k][e] = ehv && r < nb;
      float sg = 0.f;
      if (val[k][e]) {
        if (RD) {
          sg = fmaxf(sgm[RD ? k : 0][e], 0.f);
        } else if (cfg.r4) {
          const float4 dv = *reinterpret_cast<const float4 *>(sd + r * 4);
          sg = fmaf(w.wown[0], dv.x, fmaf(w.wown[1], dv.y, fmaf(w.wown[2], dv.z, w.wown[3] * dv.w)));
        } else {
          for (int t = 0; t < cfg.r; ++t) {
            const float dv = sd != nullptr ? sd[r * cfg.r + t] : __ldg(dbar_row0 + (size_t)b * cfg.r + t);
            sg = fmaf(sw[t * G + ehead], dv, sg);
          }
        }
      }
      sig[k][e] = sg;
      const float zbar = zin[k][e] * cfg.scale;
      const float logc = b == b_partial ? log_partial : cfg.log_bs;
      ell[e] = logc + zbar + cfg.half_var * sg;
      zl2[k][e] = val[k][e] ? (zbar + logc) * kLog2e : -CUDART_INF_F;   // log2 of |b| e^{zbar}
      tmax = fmaxf(tmax, zl2[k][e]);
    }
    // what the later stages read, both in log2 units: the head's term of the block score, e^l sigma^2 (e^l
    // alone when blocks are ranked by mass), and the block's mean-compensation weight |b| e^{zbar}
    const float u0 = fmaf(ell[0], kLog2e, cfg.by_mass ? 0.f : __log2f(sig[k][0]));
    const float u1 = fmaf(ell[1], kLog2e, cfg.by_mass ? 0.f : __log2f(sig[k][1]));
    store(ehead, b0 + r0, u0, u1, zl2[k][0], zl2[k][1], val[k][0], val[k][1]);
  }
  tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 1));
  tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 2));
  if (SP) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 16));
  if (tmax > w.m_ref + CKV_RESCALE_SLACK) {   // the running maximum is only raised when exceeded by a slack
    const float sc = exp2_diff(w.m_ref, tmax);
    w.m_ref = tmax;
    w.l_acc *= sc; w.lp_acc *= sc;
#pragma unroll
    for (int t = 0; t < 16; ++t) { w.acc[t][0] *= sc; w.acc[t][1] *= sc; }
  }
  uint32_t whm[NE], wlm[NE];
#pragma unroll
  for (int k = 0; k < NE; ++k) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      wt[k][e] = val[k][e] ? fast_exp2(zl2[k][e] - w.m_ref) : 0.f;
      w.l_acc += wt[k][e];
      w.lp_acc = fmaf(wt[k][e], fast_exp2(cfg.half_var * kLog2e * sig[k][e]), w.lp_acc);   // e^{l - m} = e^{zbar + log|b| - m} e^{sigma^2/2}
    }
    whm[k] = pack_bf16(wt[k][0], wt[k][1]);
    wlm[k] = pack_bf16(wt[k][0] - bf16_round(wt[k][0]), wt[k][1] - bf16_round(wt[k][1]));
  }
  uint32_t wh[2], wl[2];   // A fragments of the weights: k = blocks 2 qd + {0, 1} (+ 8), hi and lo halves
  if constexpr (SP) {
    // rows 0..3 (lanes 0-15) get their second n-tile from the lane 16 above; rows 4..7 carry zero weights
    const uint32_t oh = __shfl_sync(0xffffffffu, whm[0], (lane & 15) + 16);
    const uint32_t ol = __shfl_sync(0xffffffffu, wlm[0], (lane & 15) + 16);
    wh[0] = hsel ? 0u : whm[0]; wl[0] = hsel ? 0u : wlm[0];
    wh[1] = hsel ? 0u : oh;     wl[1] = hsel ? 0u : ol;
  } else {
#pragma unroll
    for (int k = 0; k < NE; ++k) { wh[k] = whm[k]; wl[k] = wlm[k]; }
  }

  // ---- acc += W Vbar: heads x 128 coordinates, k = this part's 16 blocks ----
  {
    // ldmatrix.trans lane roles: matrix lane / 8 -> (block half, coordinate chunk parity), row lane % 8
    const int r = rb + ((lane >> 3) & 1) * 8 + (lane & 7);
    const bool real = r < nb;   // rows past the last block: zeros
    const uint32_t rowaddr = real ? sv + r * kRowBytesV : zero_row;
    const int cpar = lane >> 4;
#pragma unroll
    for (int t2 = 0; t2 < 8; ++t2) {   // two 8-coordinate n-tiles per ldmatrix.x4
      const uint32_t coff = real ? (uint32_t)swz_chunk(2 * t2 + cpar, r) * 16 : 0u;
      uint32_t vh[4], vl[4];
      ldmatrix_x4_trans(vh, rowaddr + coff);
      mma_rows8(w.acc[2 * t2][0], w.acc[2 * t2][1], wh[0], wh[1], vh[0], vh[1]);
      mma_rows8(w.acc[2 * t2][0], w.acc[2 * t2][1], wl[0], wl[1], vh[0], vh[1]);
      mma_rows8(w.acc[2 * t2 + 1][0], w.acc[2 * t2 + 1][1], wh[0], wh[1], vh[2], vh[3]);
      mma_rows8(w.acc[2 * t2 + 1][0], w.acc[2 * t2 + 1][1], wl[0], wl[1], vh[2], vh[3]);
      if (!HS && !VH) {
        ldmatrix_x4_trans(vl, rowaddr + (real ? 256u : 0u) + coff);
        mma_rows8(w.acc[2 * t2][0], w.acc[2 * t2][1], wh[0], wh[1], vl[0], vl[1]);
        mma_rows8(w.acc[2 * t2 + 1][0], w.acc[2 * t2 + 1][1], wh[0], wh[1], vl[2], vl[3]);
      }
    }
  }
}

#endif  // CKV_SCANPART_CUH_
