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
// A lane's rows lane / 16 + 2 i differ in their swizzle by an XOR with 2 i.
__device__ __forceinline__ void issue_page(uint32_t kb, uint32_t vb, const __nv_bfloat16 *k, const __nv_bfloat16 *v, int ntok, int lane) {
  const int r0 = lane >> 4, c = lane & 15;
  const uint32_t at = (uint32_t)(r0 * kRowBytes + ((c ^ r0) << 4));
  const __nv_bfloat16 *ks = k + r0 * CKV_D + 8 * c, *vs = v + r0 * CKV_D + 8 * c;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t off = (at ^ (uint32_t)(((2 * i) & 7) << 4)) + (uint32_t)(2 * i * kRowBytes);
    const bool valid = r0 + 2 * i < ntok;   // (a copy of no bytes fills with zeros; its source is not read)
    cp_async16(kb + off, ks + 2 * i * CKV_D, valid);
    cp_async16(vb + off, vs + 2 * i * CKV_D, valid);
  }
}

// O += rows^T W for the tile of 16 value rows at vb (swizzled by row): the lane's weights x (HeadTile).
template <int G>
__device__ __forceinline__ void attn_pv(uint32_t vb, const float (&x)[HeadTile<G>::NR][2], int lane, HeadAcc<G> &w) {
  uint32_t b[HeadTile<G>::NR][2];
  HeadTile<G>::weights(x, lane, b);
  // ldmatrix.trans lane roles: matrix lane / 8 -> (coordinate chunk parity, row half), row lane % 8
  const uint32_t rowaddr = (vb + ((lane >> 4) * 8 + (lane & 7)) * kRowBytes) | ((((lane >> 3) & 1) ^ (lane & 7)) << 4);
#pragma unroll
  for (int t = 0; t < 8; ++t) {   // 16 coordinates
    uint32_t a[4];
    ldmatrix_x4_trans(a, swz_at(rowaddr, t));
    mma_16816(w.acc[t], a, b[0][0], b[0][1]);
    if constexpr (!HeadTile<G>::PAIR) mma_16816(w.acc[t], a, b[1][0], b[1][1]);
  }
}

// The running maxima are raised to those of z (the lane's values) where these exceed them by the slack.  One vote in the
// usual case that nothing does.
template <int G, int N>
__device__ __forceinline__ void attn_raise(const float (&z)[N][2], HeadAcc<G> &w) {
  float mx[2] = {z[0][0], z[0][1]};
#pragma unroll
  for (int k = 1; k < N; ++k) { mx[0] = fmaxf(mx[0], z[k][0]); mx[1] = fmaxf(mx[1], z[k][1]); }
  if (!__any_sync(0xffffffffu, mx[0] > w.m[0] + CKV_RESCALE_SLACK || mx[1] > w.m[1] + CKV_RESCALE_SLACK)) return;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const float t = HeadTile<G>::max_rows(mx[e]);
    if (t > w.m[e] + CKV_RESCALE_SLACK) {
      w.rescale(e, exp2_diff(w.m[e], t));
      w.m[e] = t;
    }
  }
}

// One page: logits L = K q^T, weights 2^(L - m) - 2^(lzt - m) (lzt: log2 of what is taken off every token's weight, per
// head of the lane, -inf for nothing), O += V^T W.  qa: the queries' B fragments; sl2: logit scale in log2 units.
template <int G>
__device__ __forceinline__ void attn_page(uint32_t kb, uint32_t vb, const uint32_t (&qa)[8][2], int ntok, int lane, float sl2,
                                          const float (&lzt)[2], HeadAcc<G> &w) {
  using T = HeadTile<G>;
  float z[4] = {0.f, 0.f, 0.f, 0.f}, z2[4] = {0.f, 0.f, 0.f, 0.f};   // two chains: the products of one depend on one another
  {
    // ldmatrix lane roles: matrix lane / 8 -> (row half, coordinate chunk parity), row lane % 8
    const uint32_t rowaddr = (kb + (((lane >> 3) & 1) * 8 + (lane & 7)) * kRowBytes) | (((lane >> 4) ^ (lane & 7)) << 4);
#pragma unroll
    for (int ks = 0; ks < 8; ks += 2) {
      uint32_t a[4], a2[4];
      ldmatrix_x4(a, swz_at(rowaddr, ks));
      ldmatrix_x4(a2, swz_at(rowaddr, ks + 1));
      mma_16816(z, a, qa[ks][0], qa[ks][1]);
      mma_16816(z2, a2, qa[ks + 1][0], qa[ks + 1][1]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] += z2[i];
  }
  float s[T::NR + 1][2], x[T::NR][2];
  {
    float v[T::NR][2];
    T::pick(z, lane, v);
#pragma unroll
    for (int k = 0; k < T::NR; ++k)
#pragma unroll
      for (int e = 0; e < 2; ++e)
        s[k][e] = T::row(lane, k) < ntok && T::head(lane, e) < G ? v[k][e] * sl2 : -CUDART_INF_F;
    s[T::NR][0] = lzt[0]; s[T::NR][1] = lzt[1];
  }
  attn_raise<G>(s, w);
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const float off = lzt[e] == -CUDART_INF_F ? 0.f : fast_exp2(lzt[e] - w.m[e]);
#pragma unroll
    for (int k = 0; k < T::NR; ++k) {
      x[k][e] = s[k][e] == -CUDART_INF_F ? 0.f : fast_exp2(s[k][e] - w.m[e]) - off;
      w.l[e] += x[k][e];
    }
  }
  attn_pv<G>(vb, x, lane, w);
}

#endif  // CKV_ATTNPAGE_CUH_
