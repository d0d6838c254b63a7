// Words that carry their own validity between the CTAs of one cooperative launch: 64 bits, an
// fp32 value in the lower half and the number of the call that wrote it in the upper half,
// written and read whole.  A reader that sees this call's number has the value: one L2 round
// trip, no fence, no counter, nothing to clear between calls.  Every wait is bounded.
#pragma once

#include "gsi_common.cuh"

namespace gsi {
namespace exchange {

constexpr int kCols = 32;              // columns of c per CTA in the projection: 64-byte pieces of a basis row
constexpr unsigned kSpinF = 1u << 20;

__device__ __forceinline__ void put(unsigned long long* p, float v, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p),
               "l"(((unsigned long long)tag << 32) | __float_as_uint(v))
               : "memory");
}
__device__ __forceinline__ unsigned long long get(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool is(unsigned long long w, unsigned tag) { return (unsigned)(w >> 32) == tag; }
__device__ __forceinline__ float val(unsigned long long w) { return __uint_as_float((unsigned)w); }

// `count` words p[i * stride] in order, eight in flight; false when a wait ran out.
template <typename F>
__device__ __forceinline__ bool gather(const unsigned long long* p, size_t stride, int count, unsigned tag, F&& take) {
  for (int i0 = 0; i0 < count; i0 += 8) {
    unsigned long long w[8];
    for (unsigned it = 0;; ++it) {
      bool all = true;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i0 + u < count) w[u] = get(p + (size_t)(i0 + u) * stride);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i0 + u < count) all = all && is(w[u], tag);
      if (all) break;
      if (it > kSpinF) return false;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + u < count) take(i0 + u, val(w[u]));
  }
  return true;
}

// Sum of `count` words by one warp in double (lane l: words l, l + 32, ...; fixed order).
__device__ __forceinline__ bool warp_gather_sum(const unsigned long long* p, size_t stride, int count, unsigned tag,
                                                double& sum) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  const int mine = count > lane ? (count - lane + 31) / 32 : 0;
  const bool ok = gather(p + (size_t)lane * stride, 32 * stride, mine, tag, [&](int, float v) { s += (double)v; });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  sum = s;
  return __all_sync(0xffffffffu, ok);
}

// The words of a handle of B tokens: partial c [slab][token][k], partial ||x||^2 [slab][token],
// partial ||r||^2 [cta][token], c [token][k], r [token][d].
struct Words {
  unsigned long long *c, *x2, *r2, *cf, *r;
};
__device__ __forceinline__ Words words_of(const GroupParams& g) {
  Words w;
  w.c = g.fused_words;
  w.x2 = w.c + (size_t)kFusedMaxGrid * g.B * kCols;
  w.r2 = w.x2 + (size_t)kFusedMaxGrid * g.B;
  w.cf = w.r2 + (size_t)kFusedMaxGrid * g.B;
  w.r = w.cf + (size_t)g.B * g.k;
  return w;
}

}  // namespace exchange

// SMs of the current device, as CTAs of a cooperative launch; 0 on error.
int fused_grid();
// Slabs of basis rows for the projection: slabs x column blocks over the grid, at least 32 rows each.
int fused_slabs(int d, int k, int grid);

}  // namespace gsi
