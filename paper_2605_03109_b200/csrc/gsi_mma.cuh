// Contractions of a few tokens on mma.sync (m16n8k16): 16 rows of a bf16 (or split fp32) matrix as
// the A operand, eight tokens as the B operand, fp32 operands as three exact bf16 terms.  Shared by
// the calls that run as one launch (gsi_fused.cu, gsi_cluster.cu).
#pragma once

#include "gsi_common.cuh"

namespace gsi {
namespace mma16 {

__device__ __forceinline__ void mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                    uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// A pair of fp32 values -> their hi, mid and lo bf16 terms, packed in pairs.
__device__ __forceinline__ void split3_pair(float a, float b, uint32_t (&t)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    t[i] = pack2(a, b);
    a -= __uint_as_float(t[i] << 16);
    b -= __uint_as_float(t[i] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ void split3_x8(const float (&v)[8], uint4 (&t)[3]) {
  uint32_t w[4][3];
#pragma unroll
  for (int i = 0; i < 4; ++i) split3_pair(v[2 * i], v[2 * i + 1], w[i]);
#pragma unroll
  for (int q = 0; q < 3; ++q) t[q] = make_uint4(w[0][q], w[1][q], w[2][q], w[3][q]);
}

// Operand, per column (token) a run of `stride` bytes: for every step (32 of the contraction) and
// term 64 bytes, the elements in order.  A stride of 64 modulo 128 bytes makes the reads (eight
// columns x four lane quarters of 16 bytes) free of bank conflicts.
__host__ __device__ __forceinline__ int op_stride(int steps) { return steps * 192 + ((steps & 1) ? 0 : 64); }
// Byte offset of elements j, j + 1 (j even) of term q within a column.
__device__ __forceinline__ int op_pair(int j, int q) { return ((j >> 5) * 3 + q) * 64 + (j & 31) * 2; }
__device__ __forceinline__ void op_store_pair(unsigned char* column, int j, uint32_t hi, uint32_t mid, uint32_t lo) {
  *reinterpret_cast<uint32_t*>(column + op_pair(j, 0)) = hi;
  *reinterpret_cast<uint32_t*>(column + op_pair(j, 1)) = mid;
  *reinterpret_cast<uint32_t*>(column + op_pair(j, 2)) = lo;
}
// ... of a column of `len` elements in global memory; the last pair brings the zeros past the end.
__device__ __forceinline__ void terms_store_pair(unsigned char* column, int j, int len, const uint32_t (&t)[3]) {
  op_store_pair(column, j, t[0], t[1], t[2]);
  if (j + 2 == len)
    for (j += 2; j & 31; j += 2) op_store_pair(column, j, 0u, 0u, 0u);
}

template <int NB>
__device__ __forceinline__ void clear(float (&v)[NB][4]) {
#pragma unroll
  for (int nb = 0; nb < NB; ++nb)
#pragma unroll
    for (int i = 0; i < 4; ++i) v[nb][i] = 0.f;
}

// sum[nb] += rows g and g + 8 (p0, p1: this lane's pointers to element 8 t of each row, null when
// the row does not exist) x columns 8 nb .. 8 nb + 7 over steps s0, s0 + ds, .. < s1.  `op`: the
// operand from step op0 on, NC columns; K: length of the contraction.  The tensor core's own accumulation
// truncates (a chain of 48 instructions is 2e-6 off, ten times an FMA chain), so the products of
// the leading terms start from zero in every step and are added in fp32; those of the lower
// terms, 2^-8 of the value, go through one accumulator of their own (low).
template <int NB, bool AF32, bool kStream, int U = (AF32 || NB >= 4 ? 2 : 4)>   // U: steps in flight
__device__ __forceinline__ void dot_steps(const void* p0, const void* p1, int K, int s0, int ds, int s1,
                                          const unsigned char* op, int stride, int op0, int NC, float (&low)[NB][4],
                                          float (&sum)[NB][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  constexpr int kTerms = AF32 ? 3 : 1;
#pragma unroll 1
  for (int sb = s0; sb < s1; sb += U * ds) {
    uint4 a[U][2][AF32 ? 2 : 1];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int s = sb + u * ds;
      const bool in = s < s1 && s * 32 + t * 8 < K;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const void* p = h ? p1 : p0;
        a[u][h][0] = make_uint4(0u, 0u, 0u, 0u);
        if constexpr (AF32) a[u][h][1] = make_uint4(0u, 0u, 0u, 0u);
        if (in && p) {
          if constexpr (AF32) {
            const uint4* q = static_cast<const uint4*>(p) + (size_t)s * 8;
            a[u][h][0] = __ldg(q);
            a[u][h][1] = __ldg(q + 1);
          } else {
            const uint4* q = static_cast<const uint4*>(p) + (size_t)s * 4;
            a[u][h][0] = kStream ? ld_stream(q) : __ldg(q);
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int s = sb + u * ds;
      if (s >= s1) break;   // warp-uniform
      uint4 at[2][kTerms];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if constexpr (AF32) {
          float v[8];
          const uint4 lo = a[u][h][0], hi = a[u][h][1];
          v[0] = __uint_as_float(lo.x); v[1] = __uint_as_float(lo.y);
          v[2] = __uint_as_float(lo.z); v[3] = __uint_as_float(lo.w);
          v[4] = __uint_as_float(hi.x); v[5] = __uint_as_float(hi.y);
          v[6] = __uint_as_float(hi.z); v[7] = __uint_as_float(hi.w);
          split3_x8(v, at[h]);
        } else {
          at[h][0] = a[u][h][0];
        }
      }
#pragma unroll
      for (int nb = 0; nb < NB; ++nb) {
        float hi[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          uint4 b = make_uint4(0u, 0u, 0u, 0u);
          if (nb * 8 + g < NC)
            b = *reinterpret_cast<const uint4*>(op + (nb * 8 + g) * stride + ((s - op0) * 3 + q) * 64 + t * 16);
#pragma unroll
          for (int r = 0; r < kTerms; ++r) {
            float(&to)[4] = (q == 0 && r == 0) ? hi : low[nb];
            mma(to, at[0][r].x, at[1][r].x, at[0][r].y, at[1][r].y, b.x, b.y);
            mma(to, at[0][r].z, at[1][r].z, at[0][r].w, at[1][r].w, b.z, b.w);
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) sum[nb][i] += hi[i];
      }
    }
  }
}
template <int NB>
__device__ __forceinline__ void add_low(const float (&low)[NB][4], float (&sum)[NB][4]) {
#pragma unroll
  for (int nb = 0; nb < NB; ++nb)
#pragma unroll
    for (int i = 0; i < 4; ++i) sum[nb][i] += low[nb][i];
}

}  // namespace mma16
}  // namespace gsi
