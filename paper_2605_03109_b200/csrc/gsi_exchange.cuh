// Words that carry their own validity between the CTAs of one cooperative launch: 64 bits, an
// fp32 value in the lower half and the tag of the call that wrote it in the upper half,
// written and read whole.  A reader that sees this call's tag has the value: one L2 round
// trip, no fence, no counter, nothing to clear between calls.  Every wait is bounded.
#pragma once

#include "gsi_common.cuh"

namespace gsi {
namespace exchange {

constexpr int kCols = 32;              // columns of c per CTA in the projection: 64-byte pieces of a basis row

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
// Orders this thread's accesses, and what it has learned of others', for the whole GPU (__threadfence()
// is sequentially consistent on top of that, which nothing here needs).
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ bool is(unsigned long long w, unsigned tag) { return (unsigned)(w >> 32) == tag; }
__device__ __forceinline__ float val(unsigned long long w) { return __uint_as_float((unsigned)w); }

// Wider words: 96 bits of payload and the call's tag, written and read as one 128-bit access.
struct Word128 {
  uint32_t a, b, c, tag;
};
__device__ __forceinline__ void put128(Word128* p, uint32_t a, uint32_t b, uint32_t c, unsigned tag) {
  asm volatile("{\n .reg .b128 v;\n mov.b128 v, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], v;\n}" ::"l"(p),
               "l"(((unsigned long long)b << 32) | a), "l"(((unsigned long long)tag << 32) | c)
               : "memory");
}
__device__ __forceinline__ Word128 get128(const Word128* p) {
  unsigned long long lo, hi;
  asm volatile("{\n .reg .b128 v;\n ld.relaxed.gpu.global.b128 v, [%2];\n mov.b128 {%0, %1}, v;\n}"
               : "=l"(lo), "=l"(hi)
               : "l"(p)
               : "memory");
  Word128 w;
  w.a = (uint32_t)lo;
  w.b = (uint32_t)(lo >> 32);
  w.c = (uint32_t)hi;
  w.tag = (uint32_t)(hi >> 32);
  return w;
}

// Words at(0) .. at(count - 1), four in flight; false when a wait ran out (`limit` polls).
template <typename P, typename F>
__device__ __forceinline__ bool gather128(P&& at, int count, unsigned tag, unsigned limit, F&& take) {
  for (int i0 = 0; i0 < count; i0 += 4) {
    Word128 w[4];
    for (unsigned it = 1;; ++it) {
      bool all = true;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < count) w[u] = get128(at(i0 + u));
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < count) all = all && w[u].tag == tag;
      if (all) break;
      if (it >= limit) return false;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u < count) take(i0 + u, w[u]);
  }
  return true;
}

// `count` words p[i * stride] in order, kIn in flight; false when a wait ran out.
template <int kIn = 8, typename F>
__device__ __forceinline__ bool gather(const unsigned long long* p, size_t stride, int count, unsigned tag,
                                       unsigned limit, F&& take) {
  for (int i0 = 0; i0 < count; i0 += kIn) {
    unsigned long long w[kIn];
    for (unsigned it = 1;; ++it) {
      bool all = true;
#pragma unroll
      for (int u = 0; u < kIn; ++u)
        if (i0 + u < count) w[u] = get(p + (size_t)(i0 + u) * stride);
#pragma unroll
      for (int u = 0; u < kIn; ++u)
        if (i0 + u < count) all = all && is(w[u], tag);
      if (all) break;
      if (it >= limit) return false;
    }
#pragma unroll
    for (int u = 0; u < kIn; ++u)
      if (i0 + u < count) take(i0 + u, val(w[u]));
  }
  return true;
}

// Sum of `count` words by one warp in double (lane l: words l, l + 32, ...; fixed order).
__device__ __forceinline__ bool warp_gather_sum(const unsigned long long* p, size_t stride, int count, unsigned tag,
                                                unsigned limit, double& sum) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  const int mine = count > lane ? (count - lane + 31) / 32 : 0;
  const bool ok = gather(p + (size_t)lane * stride, 32 * stride, mine, tag, limit, [&](int, float v) { s += (double)v; });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  sum = s;
  return __all_sync(0xffffffffu, ok);
}

// The first of a launch's four tags, and a CTA's leave.  The CTAs of a launch add kTickets to the
// counter between them (block 0 what the others leave of it), each when it has done with its waits, so
// its multiple of kTickets changes when the last one leaves: they all read the same launch number
// whenever they begin, whatever the size of the grid, and a launch whose waits ran out, in part
// before its last CTA had begun, shares no tag with the next.
constexpr unsigned kTickets = 1024;
static_assert(2 * kFusedMaxGrid <= (int)kTickets, "more for block 0 than for all others");
__device__ __forceinline__ unsigned first_tag(const unsigned long long* counter) {
  return (unsigned)(*counter / kTickets) * 4u + 1u;
}
__device__ __forceinline__ void leave_launch(unsigned long long* counter) {   // one thread, behind a barrier
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(counter),
               "l"(blockIdx.x == 0 ? (unsigned long long)(kTickets - (gridDim.x - 1)) : 1ull)
               : "memory");
}
// Gates and rho of a forward call are block 0's to write, but a CTA that gave up writes its report over
// them, and that has to stay.  Block 0 leaves behind what it wrote; the CTA waits, itself not yet gone,
// until block 0 has left, and for what block 0 wrote before to land (kLanding cycles, ten microseconds; a
// release by block 0 would order the two, at 0.2 to 0.3 us in every call: 13.58 -> 13.84, 12.86 -> 13.15).
constexpr int kReportPolls = 1 << 20;   // about a second
constexpr int kLanding = 20000;
__device__ __forceinline__ bool block0_left(const unsigned long long* counter) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(counter) : "memory");
  return v % kTickets >= kTickets / 2;
}
__device__ __forceinline__ void let_land() {
  for (const long long t0 = clock64(); clock64() - t0 < kLanding;) {}
}
// What a call that gave up leaves instead of gates and rho; every thread of the CTA, which leaves.
__device__ __forceinline__ void report_give_up(const GroupParams& g, const IoRef& io, int n_tokens) {
  const long long at = (long long)io_slot(io) * io.log_step_stride;
  for (int t = threadIdx.x; t < n_tokens; t += blockDim.x) {
    io.gate[at + t] = 1;
    (io.rho ? io.rho + at : g.rho_scratch)[t] = __int_as_float(0x7fc00000);
  }
  __syncthreads();
  if (threadIdx.x == 0) leave_launch(g.tickets);
}

// The exchange area of a handle (or of the allocation-free entry point).  A location holds words
// of one kind only, so a stale payload is never taken for a tag.  What every CTA reads in
// bulk only when some token is gated (rb) is plain memory: the warp that sends a CTA's norm words
// fences between learning that the CTA's rows are written and the words, a reader fences between the
// words and rb, and a warp that passes a decision on does both; a barrier of its own for c, with its fences, took 6 us where the words take 2.
// Every CTA starts a bulk read at another place: 148 readers in step at one place get 13 KB per
// microsecond and SM, spread out 50.
struct Area {
  unsigned long long* c;      // partial c [slab][token][k]
  Word128* norm;              // [cta][token]: ||r||^2 and ||x||^2 of the CTA's rows
  Word128* gate;              // [token]: rho, fired
  Word128* cf;                // [token][k / 2]: two coefficients as three bf16 terms each
  unsigned char* rb;          // r as three bf16 terms, in operand order: [token][term_bytes(d)]
  unsigned long long *ext_r, *ext_x2, *ext_r2;   // basis extension: [d], [slab], [cta] of pass 1
  Word128* ext_r2d;           // ... [cta] of pass 2, a double each
};
// Operand bytes of one column: 192 for every 32 elements (zeros past the end).
__host__ __device__ __forceinline__ int term_bytes(int n) { return (n + 31) / 32 * 192; }
__device__ __forceinline__ Area area_of(const GroupParams& g) {
  Area w;
  w.c = g.fused_words;
  w.norm = reinterpret_cast<Word128*>(w.c + (size_t)kFusedMaxGrid * g.area_B * kCols);
  w.gate = w.norm + (size_t)kFusedMaxGrid * g.area_B;
  w.cf = w.gate + g.area_B;
  w.rb = reinterpret_cast<unsigned char*>(w.cf + (size_t)g.area_B * (g.area_k / 2));
  w.ext_x2 = reinterpret_cast<unsigned long long*>(w.rb + (size_t)g.area_B * term_bytes(g.area_d));
  w.ext_r2 = w.ext_x2 + kFusedMaxGrid;
  w.ext_r2d = reinterpret_cast<Word128*>(w.ext_r2 + kFusedMaxGrid);
  w.ext_r = w.ext_r2 + 3 * kFusedMaxGrid;
  return w;
}

}  // namespace exchange

// Id of the current context, which is never used again; 0 when it cannot be told.
unsigned long long context_id();
// CTAs of a cooperative launch: the SMs of the current context (a green context has fewer than its
// device); 0 on error.
int fused_grid();
// launch(grid) with that many, or with fewer where the stream's SMs are fewer still: the kernels run on
// any grid, and what the launches that waited for nobody took is taken.
template <typename F>
cudaError_t launch_resident(F&& launch) {
  const int most = fused_grid();
  if (!most) return cudaErrorInvalidDevice;
  cudaError_t e = cudaErrorCooperativeLaunchTooLarge;
  for (int grid = most; grid >= 1 && e == cudaErrorCooperativeLaunchTooLarge; grid /= 2) {
    e = launch(grid);
    if (e == cudaErrorCooperativeLaunchTooLarge) (void)cudaGetLastError();
  }
  return e;
}
// Slabs of basis rows for the projection: slabs x column blocks over the grid, at least 32 rows each.
int fused_slabs(int d, int k, int grid);

}  // namespace gsi
