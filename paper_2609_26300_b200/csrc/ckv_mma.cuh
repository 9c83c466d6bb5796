// Warp-level tensor-core tiles (mma.sync m16n8k16 bf16 -> fp32, ldmatrix, movmatrix) shared by the summary scan, the
// attention kernel and the one-launch step.
//
// A tile is 16 rows of the cache (16 blocks' mean rows, or the 16 tokens of a page) against the G <= 8 query heads of a
// unit.  The cache rows are the M dimension and the heads the N dimension of both products:
//   logits  L [16 rows x 8 columns]         = rows [16 x 128] * queries^T [128 x 8]        8 mma
//   output  O [128 coordinates x 8 columns] += rows^T [128 x 16] * weights [16 x 8]        8 mma
// With the heads as M rows, half or more of every instruction's rows were padding (16 and 32 instructions) and the warps'
// work, not DRAM, bounded the scans; us per step before and after the change of sides: 8 units at 32K 20.3 / 17.4, 32 units
// at 128K 63.9 / 56.1, 24 units with bf16 summaries 45.8 / 32.2, 16 units with r = d 65.4 / 60.0; dense pass 331 / 320.
// Columns: with G = 8 column c is head c.  With G <= 4 columns 0..3 are heads 0..3 and columns 4..7 carry the same heads
// once more: the weights' bf16 remainders w - bf16(w) in the second product, so that high and low halves share one
// instruction; in the first product a copy of the queries, so that every lane finds the logits it works on in its own
// registers.  A lane works on two heads of one row (G <= 4) or of two rows (G = 8): see HeadTile.
#pragma once

#include <cuda_bf16.h>
#include <math_constants.h>
#include <stdint.h>

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr) : "memory");
}
// Transpose of an 8x8 matrix of 16-bit values held across the warp (lane: row lane / 4, columns 2 (lane % 4) + {0, 1}).
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}
// Address of the 16-byte chunk 2 j + parity of a row whose chunks are XORed by (row & 7): `base` is the row's address
// (a multiple of 128) with (parity ^ row & 7) * 16 in its low bits, so that one XOR per chunk of a half row is enough.
__device__ __forceinline__ uint32_t swz_at(uint32_t base, int j) { return (base ^ (32u * (j & 3))) + 128u * (j >> 2); }
// D (16x8) += A (16x16) B (16x8)
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// {lo, hi} as a bf16 pair, lo in the lower half
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&v);
}

// Which (row, head) pairs of a tile a lane works on: rows row(lane, k), k < NR, heads head(lane, 0) and head(lane, 1)
// (beyond G: the lane's values are padding).  `copy` lanes hold the same heads as the lane two below, for other rows.
template <int G>
struct HeadTile {
  static constexpr bool PAIR = G <= 4;        // columns 4..7 repeat the heads
  static constexpr int NR = PAIR ? 1 : 2;
  __device__ static __forceinline__ bool copy(int lane) { return PAIR && (lane & 2) != 0; }
  __device__ static __forceinline__ int row(int lane, int k) { return (lane >> 2) + (PAIR ? 4 * (lane & 2) : 8 * k); }
  __device__ static __forceinline__ int head(int lane, int e) { return (PAIR ? 2 * (lane & 1) : 2 * (lane & 3)) + e; }
  // head of the lane's column in a B fragment (queries)
  __device__ static __forceinline__ int col_head(int lane) { return PAIR ? (lane >> 2) & 3 : lane >> 2; }

  // the lane's logits out of a product's accumulator
  __device__ static __forceinline__ void pick(const float (&z)[4], int lane, float (&v)[NR][2]) {
    if constexpr (PAIR) {
      v[0][0] = copy(lane) ? z[2] : z[0];
      v[0][1] = copy(lane) ? z[3] : z[1];
    } else {
      v[0][0] = z[0]; v[0][1] = z[1]; v[NR - 1][0] = z[2]; v[NR - 1][1] = z[3];
    }
  }
  // sum of the two column sets (where they carry high and low halves of one operand); G <= 4
  __device__ static __forceinline__ void add_copies(float (&z)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] += __shfl_xor_sync(0xffffffffu, z[i], 2);
  }
  // reductions over the lanes that work on the same heads
  __device__ static __forceinline__ float max_rows(float x) {
    x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 4));
    x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 8));
    x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 16));
    return PAIR ? fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2)) : x;
  }
  __device__ static __forceinline__ float sum_rows(float x) {
    x += __shfl_xor_sync(0xffffffffu, x, 4);
    x += __shfl_xor_sync(0xffffffffu, x, 8);
    x += __shfl_xor_sync(0xffffffffu, x, 16);
    return PAIR ? x + __shfl_xor_sync(0xffffffffu, x, 2) : x;
  }
  // whether this lane speaks for head(lane, e) of the unit (one lane per head does)
  __device__ static __forceinline__ bool owns(int lane, int e) { return (lane >> 2) == 0 && !copy(lane) && head(lane, e) < G; }

  // The lane's weights as B fragments of the second product, high and low bf16 halves: b[0] (and b[1], G = 8).
  __device__ static __forceinline__ void weights(const float (&x)[NR][2], int lane, uint32_t (&b)[NR][2]) {
    if constexpr (PAIR) {
      const uint32_t h = pack_bf16(x[0][0], x[0][1]);
      const uint32_t l = pack_bf16(x[0][0] - __uint_as_float(h << 16), x[0][1] - __uint_as_float(h & 0xffff0000u));
      // rows 0..7 sit in the lower lanes of a quad, rows 8..15 in the upper ones; columns 4..7 take the low halves
      const bool up = copy(lane);
      const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? h : l, 2);
      b[0][0] = movmatrix_trans(up ? got : h);
      b[0][1] = movmatrix_trans(up ? l : got);
    } else {
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        const uint32_t h = pack_bf16(x[k][0], x[k][1]);
        const uint32_t l = pack_bf16(x[k][0] - __uint_as_float(h << 16), x[k][1] - __uint_as_float(h & 0xffff0000u));
        b[0][k] = movmatrix_trans(h);
        b[NR - 1][k] = movmatrix_trans(l);
      }
    }
  }
};

// Online-softmax state of a warp: acc[t]: coordinates 16 t + lane / 4 (+ 8), columns 2 (lane % 4) + {0, 1}; running maxima
// (log2) and weight sums of the lane's two heads.
template <int G>
struct HeadAcc {
  using T = HeadTile<G>;
  float acc[8][4];
  float m[2], l[2];
  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int t = 0; t < 8; ++t)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[t][i] = 0.f;
    m[0] = m[1] = -CUDART_INF_F;
    l[0] = l[1] = 0.f;
  }
  __device__ __forceinline__ void rescale(int e, float sc) {
    l[e] *= sc;
#pragma unroll
    for (int t = 0; t < 8; ++t) { acc[t][e] *= sc; acc[t][2 + e] *= sc; }
  }
  // Calls f(head, coordinate, value) for the lane's share of the complete sums.
  template <class F>
  __device__ __forceinline__ void fold(int lane, F f) const {
    const int r = lane >> 2;
    if constexpr (T::PAIR) {   // high-half and low-half columns are added; each lane of the pair keeps one row half
      const bool up = T::copy(lane);
#pragma unroll
      for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float got = __shfl_xor_sync(0xffffffffu, up ? acc[t][e] : acc[t][2 + e], 2);
          const float v = (up ? acc[t][2 + e] : acc[t][e]) + got;
          if (T::head(lane, e) < G) f(T::head(lane, e), 16 * t + r + (up ? 8 : 0), v);
        }
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i) f(T::head(lane, i & 1), 16 * t + r + 8 * (i >> 1), acc[t][i]);
    }
  }
};
