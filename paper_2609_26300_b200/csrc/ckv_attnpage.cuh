// One cache page (16 tokens, bf16) through the tensor cores by one warp: asynchronous copies into XOR-swizzled shared
// memory tiles, logits, softmax weights and the weighted sum of the value rows.  Shared by the attention kernel and by
// the one-launch step.
#ifndef CKV_ATTNPAGE_CUH_
#define CKV_ATTNPAGE_CUH_
#include "ckv_internal.cuh"
#include "ckv_mma.cuh"

constexpr int kTileBytes = CKV_PAGE * CKV_D * 2;      // one head's K (or V) page in bf16: 4 KB
constexpr int kPageBytes = 2 * kTileBytes;            // K tile | V tile
constexpr int kRowBytes = CKV_D * 2;                  // 256

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
  // valid == false copies nothing and zero-fills the 16 bytes
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }


// Start the copies of one page (k, v: its first row): 256 16-byte pieces per tile, 8 per lane; piece c of row r lands at
// chunk c ^ (r & 7) of the row, so that the matrix loads below are conflict-free; rows at or past ntok are zero-filled.
__device__ __forceinline__ void issue_page(uint32_t kb, uint32_t vb, const __nv_bfloat16 *k, const __nv_bfloat16 *v, int ntok, int lane) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int idx = lane + 32 * i, row = idx >> 4, c = idx & 15;
    const uint32_t off = (uint32_t)(row * kRowBytes + ((c ^ (row & 7)) << 4));
    const bool valid = row < ntok;
    const size_t so = (size_t)(valid ? row : 0) * CKV_D + 8 * c;
    cp_async16(kb + off, k + so, valid);
    cp_async16(vb + off, v + so, valid);
  }
}

// O += P V for one tile of 16 value rows at vb (swizzled by row): A fragments of the weights as bf16 hi and lo halves.
__device__ __forceinline__ void attn_pv(uint32_t vb, const uint32_t (&ph)[2], const uint32_t (&pl)[2], int lane, float (&acc)[16][2]) {
  const int r = ((lane >> 3) & 1) * 8 + (lane & 7);
  const uint32_t rowaddr = vb + r * kRowBytes;
  const int cpar = lane >> 4;
#pragma unroll
  for (int t2 = 0; t2 < 8; ++t2) {   // two 8-coordinate n-tiles per ldmatrix.x4
    uint32_t v[4];
    ldmatrix_x4_trans(v, rowaddr + (uint32_t)(((2 * t2 + cpar) ^ (r & 7)) << 4));
    mma_rows8(acc[2 * t2][0], acc[2 * t2][1], ph[0], ph[1], v[0], v[1]);
    mma_rows8(acc[2 * t2][0], acc[2 * t2][1], pl[0], pl[1], v[0], v[1]);
    mma_rows8(acc[2 * t2 + 1][0], acc[2 * t2 + 1][1], ph[0], ph[1], v[2], v[3]);
    mma_rows8(acc[2 * t2 + 1][0], acc[2 * t2 + 1][1], pl[0], pl[1], v[2], v[3]);
  }
}

// The running maximum is raised to tmax when that exceeds it by the slack, and what was accumulated is rescaled.
__device__ __forceinline__ void attn_raise(float tmax, float &m_ref, float &l_acc, float (&acc)[16][2]) {
  if (tmax > m_ref + CKV_RESCALE_SLACK) {
    const float sc = exp2_diff(m_ref, tmax);
    m_ref = tmax;
    l_acc *= sc;
#pragma unroll
    for (int t = 0; t < 16; ++t) { acc[t][0] *= sc; acc[t][1] *= sc; }
  }
}

// One page: S^T = Q K^T, P = 2^(S^T - m) - 2^(lzt - m) (lzt: log2 of what is taken off every token's weight, -inf for
// nothing), O += P V.  sl2: logit scale in log2 units.  hv: this lane's head exists.  SHARED: the lanes 16 above hold
// partial sums of the same heads (G <= 4) and follow their running maximum.
template <bool SHARED>
__device__ __forceinline__ void attn_page(uint32_t kb, uint32_t vb, const uint32_t (&qa)[8][2], int ntok, bool hv, int lane,
                                          float sl2, float lzt, float (&acc)[16][2], float &m_ref, float &l_acc) {
  const int qd = lane & 3;
  // ---- S^T = Q K^T: heads x 16 tokens (two n-tiles of 8 tokens) ----
  float sv[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, sv2[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  {
    const int lrow = lane & 7, lmat = lane >> 3;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int r = nt * 8 + lrow;
      const uint32_t rowaddr = kb + r * kRowBytes;
#pragma unroll
      for (int j = 0; j < 4; ++j) {   // two 16-coordinate steps per ldmatrix.x4
        uint32_t b[4];
        ldmatrix_x4(b, rowaddr + (uint32_t)(((4 * j + lmat) ^ (r & 7)) << 4));
        mma_rows8(sv[nt][0], sv[nt][1], qa[2 * j][0], qa[2 * j][1], b[0], b[1]);
        mma_rows8(sv2[nt][0], sv2[nt][1], qa[2 * j + 1][0], qa[2 * j + 1][1], b[2], b[3]);
      }
      sv[nt][0] += sv2[nt][0]; sv[nt][1] += sv2[nt][1];
    }
  }
  // ---- softmax weights for this thread's head and its four tokens ----
  float tmax = lzt;
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const bool ok = hv && nt * 8 + 2 * qd + e < ntok;
      sv[nt][e] = ok ? sv[nt][e] * sl2 : -CUDART_INF_F;
      tmax = fmaxf(tmax, sv[nt][e]);
    }
  tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 1));
  tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 2));
  if (SHARED) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 16));
  attn_raise(tmax, m_ref, l_acc, acc);
  const float wtok = lzt == -CUDART_INF_F ? 0.f : fast_exp2(lzt - m_ref);
  uint32_t ph[2], pl[2];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
    float p[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      p[e] = sv[nt][e] == -CUDART_INF_F ? 0.f : fast_exp2(sv[nt][e] - m_ref) - wtok;
      l_acc += p[e];
    }
    ph[nt] = pack_bf16(p[0], p[1]);
    pl[nt] = pack_bf16(p[0] - bf16_round(p[0]), p[1] - bf16_round(p[1]));
  }
  attn_pv(vb, ph, pl, lane, acc);
}

#endif  // CKV_ATTNPAGE_CUH_
