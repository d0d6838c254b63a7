// One call of any supported shape as ONE launch: Algorithm 1 with two grid-wide exchanges inside a
// cooperative kernel (every CTA resident).  It serves the calls that do not fit clusters of their own
// (gsi_cluster.cu): wide bases, many tokens, contexts with few SMs.
//
//   A   partial c of a slab of basis rows x 32 columns per CTA              (line 1)
//   x1  the partials are added in a fixed order: by every CTA for itself in calls of one or two
//       tokens, else each coefficient by one CTA, which passes its terms on to all
//   B   r of its rows of the basis, then y = W_P c of its image rows        (lines 2, 5)
//   x2  every CTA gathers all partial norms and takes the gate decision     (lines 3-4, Eq. (3.3))
//   C   gated tokens: y += W r over its rows of W                           (Eq. (3.2))
//
// All contractions run on mma.sync (m16n8k16) with 16 rows of the matrix, straight from global
// memory, as the A operand and eight tokens as the B operand; the fp32 operands x, c and r (and an
// fp32 basis) enter as three bf16 terms (hi + mid + lo = the fp32 value), so products are exact
// and sums are fp32.  A lane's 16 bytes of a row hold eight neighbours of the contraction; they
// serve two instructions with the contraction index permuted alike in both operands.
//
// What bounds it: a few MB and a chain of latencies; tcgen05 with its tensor-memory round trip
// per 16-row unit would add to that chain.  Time per call, one after the other on a stream, against
// the five launches of the per-stage kernels before: one token at 768 x 64 -> 3072 27.3 -> 12.3 us
// (of which the kernel 10.3; the rest is the caller's side), at 4096 x 256 -> 28672, nothing gated,
// 43.0 -> 15.8 us; 21 tokens at 3000 x 200 -> 1576 90 -> 27 us; 16 tokens, fp32 basis, 768 x 128 ->
// 2304 50 -> 21 us.
//
// The exchanges are words that carry the call's tag (gsi_exchange.cuh): a release / acquire
// barrier would cost two L2 round trips and a fence where these cost one.  Every token's sums run
// in an order that depends on the shape and the grid alone: results are reproducible, and a token's
// are the same in a call of any size that runs here as a whole (not where W r is left to the
// contraction, leave_from).
// Every wait is bounded; a CTA whose wait ran out sets GSI_ERR_TIMEOUT, leaves NaN and returns.
#include <cuda.h>

#include <type_traits>

#include "gsi_exchange.cuh"
#include "gsi_mma.cuh"

namespace gsi {

namespace {

using namespace exchange;
using namespace mma16;

constexpr int kT = 512, kW = kT / 32;
constexpr int kTileRows = 16 * kW;     // rows of a basis slab (and of W) per pass: 16 per warp
constexpr int kPitch = 80;             // bytes between the staged 64-byte pieces: conflict-free ldmatrix
constexpr int kDirectTokens = 2;       // calls of so few tokens gather the slabs' partials themselves
constexpr int kDecideTokens = 4;       // calls of so few tokens decide the gates on every CTA
constexpr int kTermsHoldOff = 900;     // cycles before the first look at the coefficients added elsewhere
constexpr int kTermsHoldOffFrom = 1024;   // ... in calls of so many coefficients
constexpr int kGateHoldOff = 600;      // cycles before the first look at the decisions taken elsewhere
constexpr int kSegs = 8;               // the slabs' partials are added in eight runs, these by a tree
constexpr int kSlots = 16;             // 16-row units of the basis whose norms wait in shared memory
// dynamic shared memory: operand terms (phase A: the slab), then partial sums
constexpr int kOpBytes = 131072, kAuxBytes = 32768;
constexpr int kSmemFused = kOpBytes + kAuxBytes;

// `units` 16-byte units of NC operand columns from global to shared memory, all copies in flight.
template <typename F>
__device__ __forceinline__ void copy_columns(unsigned char* op, int stride, int units, int NC, F&& column) {
  const int all = units * NC;
  int f = (int)((long long)all * blockIdx.x / gridDim.x) + (int)threadIdx.x;   // (no two CTAs at the same place at a time)
  for (int i = threadIdx.x; i < all; i += kT, f += kT) {
    if (f >= all) f -= all;
    const int c = f / units, u = f - c * units;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(op + c * stride + u * 16);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(column(c) + u * 16) : "memory");
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// y += W r for the fired tokens, 8 NB at a time.  A warp owns 16 of this CTA's rows of W and every
// ks-th step of the contraction (narrow maps: several warps share 16 rows and their sums meet in
// shared memory); r comes in operand form, as much of the width at a time as fits.
template <int NB>
__device__ __forceinline__ void stream_w(const GroupParams& g, const IoRef& io, const unsigned char* rb,
                                         const int* s_fired, unsigned char* smem, int o0, int o1) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lg = lane >> 2, lt = lane & 3;
  const int d = g.d, n_fired = s_fired[0], steps = (d + 31) / 32;
  unsigned char* op = smem;
  float* part = reinterpret_cast<float*>(smem + kOpBytes);   // [warp][16 rows][8 NB]
  static_assert(kW * 16 * 8 * NB * 4 <= kAuxBytes, "partial sums of the warps");
  for (int f0 = 0; f0 < n_fired; f0 += 8 * NB) {
    const int NC = min(8 * NB, n_fired - f0);
    const int span = min(steps, (kOpBytes / NC - 64) / 192);   // steps whose operand fits
    const int stride = op_stride(span);
    for (int b0 = o0; b0 < o1; b0 += kTileRows) {
      const int rows = min(kTileRows, o1 - b0), tiles = (rows + 15) / 16;
      int ks = 1;
      while (2 * ks * tiles <= kW) ks *= 2;
      const int tile = warp / ks, kq = warp % ks;
      const bool active = tile < tiles;
      const void* p[2] = {nullptr, nullptr};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = b0 + tile * 16 + lg + 8 * h;
        if (active && row < o1) {
          int j = 0;
          while (j + 1 < g.n_maps && row >= g.off[j + 1]) ++j;
          p[h] = g.W[j] + (size_t)(row - g.off[j]) * d + lt * 8;
        }
      }
      float low[NB][4], sum[NB][4];
      clear<NB>(low);
      clear<NB>(sum);
      for (int s0 = 0; s0 < steps; s0 += span) {
        const int s1 = min(steps, s0 + span);
        if (s0 > 0 || b0 == o0 || span < steps) {
          __syncthreads();   // the operand before is read
          copy_columns(op, stride, (s1 - s0) * 12, NC,
                       [&](int c) { return rb + (size_t)s_fired[1 + f0 + c] * term_bytes(d) + s0 * 192; });
          __syncthreads();
        }
        // step s belongs to warp s % ks (ks a power of two)
        if (active) dot_steps<NB, false, true>(p[0], p[1], d, s0 + ((kq - s0) & (ks - 1)), ks, s1, op, stride, s0,
                                                NC, low, sum);
      }
      add_low<NB>(low, sum);
      auto add = [&](int tile_, int r16, int col, float v) {
        const int row = b0 + tile_ * 16 + r16;
        if (row < o1 && col < NC) io.y[(size_t)s_fired[1 + f0 + col] * g.O + row] += v;
      };
      if (ks == 1) {
        if (active) {
#pragma unroll
          for (int nb = 0; nb < NB; ++nb)
#pragma unroll
            for (int i = 0; i < 4; ++i) add(tile, lg + 8 * (i >> 1), nb * 8 + 2 * lt + (i & 1), sum[nb][i]);
        }
      } else {
        if (active) {
#pragma unroll
          for (int nb = 0; nb < NB; ++nb)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              part[(warp * 16 + lg + 8 * (i >> 1)) * 8 * NB + nb * 8 + 2 * lt + (i & 1)] = sum[nb][i];
        }
        __syncthreads();
        for (int i = tid; i < tiles * 16 * 8 * NB; i += kT) {
          const int col = i % (8 * NB), r = i / (8 * NB);
          float v = 0.f;
          for (int q = 0; q < ks; ++q) v += part[(((r >> 4) * ks + q) * 16 + (r & 15)) * 8 * NB + col];
          add(r >> 4, r & 15, col, v);
        }
        __syncthreads();
      }
    }
  }
}

// NB: eight-token blocks at a time in the projection.  kDirect: a build for calls of up to
// kDirectTokens tokens (what the others need would cost it registers: 3 us at one token).  leave_from > 0: with that many gated tokens or
// more W r is left to the tensor-core contraction that follows (r goes to g.r, the gated tokens to
// g.fired).  False when a wait ran out (for every thread of the CTA).
template <int NB, bool PF32, bool kDirect>
__device__ __forceinline__ bool forward_fused(const GroupParams& g, const IoRef& io, int n_tokens, int n_slabs,
                                              int leave_from) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float2 s_unit[kSlots][GSI_MAX_TOKENS];    // ||r||^2, ||x||^2 of a 16-row unit of the basis
  __shared__ float2 s_run[GSI_MAX_TOKENS];             // ... of the units before
  __shared__ float s_rho[GSI_MAX_TOKENS];
  __shared__ bool s_fast[GSI_MAX_TOKENS];
  __shared__ int s_fired[GSI_MAX_TOKENS + 1];
  __shared__ int s_done;
  constexpr int kTerms = PF32 ? 3 : 1, kTok = 8 * NB;
  float* s_aux = reinterpret_cast<float*>(smem + kOpBytes);
  unsigned char* op = smem;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lg = lane >> 2, lt = lane & 3;
  const int G = gridDim.x, cta = blockIdx.x;
  const int d = g.d, k = g.k, n = n_tokens;
  const unsigned tag = first_tag(g.tickets);
  const Area words = area_of(g);
  unsigned long long* cw = words.c;
  const int slot = io_slot(io);
  const float* x = io.x + (long long)slot * io.x_step_stride;
  const int o0 = (int)((long long)g.O * cta / G), o1 = (int)((long long)g.O * (cta + 1) / G);
  const int p0 = (int)((long long)(d / 2) * cta / G) * 2, p1 = (int)((long long)(d / 2) * (cta + 1) / G) * 2;

  if (tid == 0) s_done = 0;
  if (tid == 0 && o1 > o0) {   // the image rows are asked into the L2 while c is on its way
    const char* p = reinterpret_cast<const char*>(g.WP + (size_t)o0 * k);
    const size_t bytes = (size_t)(o1 - o0) * k * 2;
    for (size_t at = 0; at < bytes; at += 32768)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p + at),
                   "r"((unsigned)min((size_t)32768, bytes - at))
                   : "memory");
  }

  // ---- A: D[column of P][token] += P^T x over the slab; 256 rows staged at a time, 16 per warp
  const int n_cb = (k + kCols - 1) / kCols;
  // (a small grid may have fewer CTAs than column blocks; the direct build is not launched there: the loop costs it 0.7 us)
  int part = cta;
  if (part < n_slabs * n_cb) do {
    const int slab = part / n_cb, cb = part % n_cb;
    const int r0 = (int)((long long)d * slab / n_slabs), r1 = (int)((long long)d * (slab + 1) / n_slabs);
    for (int tb = 0; tb < n; tb += kTok) {
      float acc[2][NB][4];
      clear<NB>(acc[0]);
      clear<NB>(acc[1]);
      for (int rb = r0; rb < r1; rb += kTileRows) {
        // this warp's rows of x: token 8 nb + lg, rows 2 lt, 2 lt + 1, + 8, + 9
        const int row = rb + 16 * warp + 2 * lt;
        float xv[NB][4];
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) {
          const int t = tb + nb * 8 + lg;
          const float* xp = x + (size_t)t * d + row;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int off = (i & 1) + 8 * (i >> 1);
            xv[nb][i] = (t < n && row + off < r1) ? __ldg(xp + off) : 0.f;
          }
        }
        if (rb > r0) __syncthreads();
        for (int i = tid; i < kTileRows * 4; i += kT) {   // 16 bytes (fp32: 32) of a row each
          const int r = i >> 2, c8 = i & 3, col = cb * kCols + c8 * 8;
          const bool in = rb + r < r1 && col < k;
          if constexpr (PF32) {
            float v[8] = {};
            uint4 tm[3];
            if (in) load8<true>(g.P, ((size_t)(rb + r) * k + col) / 8, v);
            split3_x8(v, tm);
#pragma unroll
            for (int q = 0; q < 3; ++q)
              *reinterpret_cast<uint4*>(smem + (size_t)(q * kTileRows + r) * kPitch + c8 * 16) = tm[q];
          } else {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (in) v = __ldg(reinterpret_cast<const uint4*>(g.P) + ((size_t)(rb + r) * k + col) / 8);
            *reinterpret_cast<uint4*>(smem + (size_t)r * kPitch + c8 * 16) = v;
          }
        }
        __syncthreads();
        if (rb + 16 * warp < r1) {
          uint32_t xt[NB][2][3];
#pragma unroll
          for (int nb = 0; nb < NB; ++nb)
#pragma unroll
            for (int h = 0; h < 2; ++h) split3_pair(xv[nb][2 * h], xv[nb][2 * h + 1], xt[nb][h]);
          // 8 x 8 blocks of the tile, transposed by the load: rows (k) 0-7 | 8-15 by columns (m) 0-7 | 8-15
          const int tr = 16 * warp + (lane & 7) + ((lane >> 4) << 3), tc = ((lane >> 3) & 1) * 16;
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            uint32_t a[kTerms][4];
#pragma unroll
            for (int r = 0; r < kTerms; ++r)
              asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                           : "=r"(a[r][0]), "=r"(a[r][1]), "=r"(a[r][2]), "=r"(a[r][3])
                           : "r"((uint32_t)__cvta_generic_to_shared(smem + (size_t)(r * kTileRows + tr) * kPitch +
                                                                    m * 32 + tc)));
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) {
              float hi[4] = {0.f, 0.f, 0.f, 0.f}, low[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
              for (int r = 0; r < kTerms; ++r)
#pragma unroll
                for (int q = 0; q < 3; ++q)
                  mma((q == 0 && r == 0) ? hi : low, a[r][0], a[r][1], a[r][2], a[r][3], xt[nb][0][q], xt[nb][1][q]);
#pragma unroll
              for (int i = 0; i < 4; ++i) acc[m][nb][i] += hi[i] + low[i];
            }
          }
        }
      }
      // over the warps: 16 tokens at a time
#pragma unroll
      for (int nq = 0; nq < NB; nq += 2) {
        if (tb + nq * 8 >= n) break;
        constexpr int kPair = NB > 1 ? 2 : 1;
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
          for (int h = 0; h < kPair; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              s_aux[(warp * 16 + h * 8 + 2 * lt + (i & 1)) * kCols + m * 16 + lg + 8 * (i >> 1)] = acc[m][nq + h][i];
        __syncthreads();
        {
          const int tt = tid / kCols, j = cb * kCols + tid % kCols, t = tb + nq * 8 + tt;
          if (tt < kPair * 8 && t < n && j < k) {
            float s = 0.f;
#pragma unroll
            for (int w = 0; w < kW; ++w) s += s_aux[(w * 16 + tt) * kCols + tid % kCols];
            put(cw + ((size_t)slab * n + t) * k + j, s, tag);
          }
        }
        __syncthreads();
      }
      __syncthreads();
    }
    part += G;
  } while (!kDirect && part < n_slabs * n_cb);

  // ---- x1.  Coefficient i (= token * k + column) summed over the slabs by Q adjacent lanes: each
  // adds kSegs / Q runs of slabs in order, the runs are added by a tree: the same sums for every Q
  bool ok = true;
  auto slab_sum = [&](int i, bool live, auto lanes) -> float {
    constexpr int Q = decltype(lanes)::value, R = kSegs / Q;
    float run[R];
    int end[R];   // of the runs, from the first slab of this lane on
    const int q = tid % Q, a = n_slabs * (q * R) / kSegs;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      run[r] = 0.f;
      end[r] = n_slabs * (q * R + r + 1) / kSegs - a;
    }
    if (live)
      ok = gather<Q == 2 ? 12 : 4>(cw + (size_t)a * n * k + i, (size_t)n * k, end[R - 1], tag, g.spin_limit, [&](int u, float v) {
#pragma unroll
             for (int r = 0; r < R; ++r)
               if (u < end[r] && (r == 0 || u >= end[r - 1])) run[r] += v;
           }) && ok;
#pragma unroll
    for (int h = 1; h < R; h *= 2)
#pragma unroll
      for (int r = 0; r < R; r += 2 * h) run[r] += run[r + h];
    float s = run[0];
#pragma unroll
    for (int o = 1; o < Q; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  auto timed_out = [&](bool good) -> bool {   // the same answer for every thread
    if (!__syncthreads_or(!good)) return false;
    if (tid == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
    return true;
  };
  if constexpr (!kDirect) {
    const int i0 = (int)((long long)n * (k / 2) * cta / G) * 2, i1 = (int)((long long)n * (k / 2) * (cta + 1) / G) * 2;
    for (int ib = i0; ib < i1; ib += kT / 8) {
      const int i = ib + tid / 8;
      const float s = slab_sum(i, i < i1, std::integral_constant<int, 8>());
      const float nx = __shfl_down_sync(0xffffffffu, s, 8);
      if (i < i1 && tid % 16 == 0) {   // (i0, i1 and ib are even)
        uint32_t t[3];
        split3_pair(s, nx, t);
        put128(words.cf + (i >> 1), t[0], t[1], t[2], tag);
      }
    }
  }

  // ---- x1 (end) and B, as many tokens at a time as have their c in shared memory
  const int ksteps = (k + 31) / 32, stride = op_stride(ksteps);
  const int pt = (p1 - p0 + 15) / 16, ot = (o1 - o0 + 15) / 16;   // units of 16 rows
  const int per_block = min(n, max(8, kOpBytes / stride / 8 * 8));
  for (int tb = 0; tb < n; tb += per_block) {
    const int NC = min(per_block, n - tb), ncb = (NC + 7) / 8;
    if (tb > 0) __syncthreads();
    if (tid < NC) s_run[tid] = make_float2(0.f, 0.f);
    const int tail = ksteps * 16 - k / 2;   // pairs of the operand beyond k
    for (int i = tid; i < tail * NC; i += kT) op_store_pair(op + (i / tail) * stride, k + 2 * (i % tail), 0u, 0u, 0u);
    if constexpr (kDirect) {
      for (int ib = 0; ib < NC * k; ib += kT / 2) {
        const int i = ib + tid / 2;
        const float s = slab_sum(tb * k + i, i < NC * k, std::integral_constant<int, 2>());
        const float nx = __shfl_down_sync(0xffffffffu, s, 2);
        if (i < NC * k && tid % 4 == 0) {
          uint32_t t[3];
          split3_pair(s, nx, t);
          const int c = i >= k ? 1 : 0;
          op_store_pair(op + c * stride, i - c * k, t[0], t[1], t[2]);
        }
      }
    } else {
      const int half = k / 2, all = NC * half, mine = all > tid ? (all - tid + kT - 1) / kT : 0;
      const int rot = (int)((long long)all * cta / G) + tid;   // (no two CTAs at the same place at a time)
      auto place = [&](int u) {
        const int f = rot + u * kT;
        return f < all ? f : f - all;
      };
      // (looks ahead of the words hold up the CTAs that still add theirs: 21 tokens 26.4 -> 24.6 us; three
      // tokens at k = 64, whose words are few, would lose 0.7 of 14)
      if (n * k >= kTermsHoldOffFrom)
        for (const long long t0 = clock64(); clock64() - t0 < kTermsHoldOff;) {}
      ok = gather128([&](int u) { return words.cf + (size_t)tb * half + place(u); }, mine, tag, g.spin_limit,
                     [&](int u, const Word128& w) {
                       const int f = place(u), c = f / half;
                       op_store_pair(op + c * stride, 2 * (f - c * half), w.a, w.b, w.c);
                     }) && ok;
    }
    if (timed_out(ok)) return false;
    // basis rows: a unit x eight tokens per warp.  The units' norms wait in shared memory and are
    // added in order by the warp that hands in last; it sends them off while the image rows run.
    for (int uc = 0; uc == 0 || uc < pt; uc += kSlots) {
      const int nu = min(kSlots, pt - uc);
      for (int it = warp; it < nu * ncb; it += kW) {
        const int u = it / ncb, nb = it - u * ncb, t = tb + nb * 8 + 2 * lt;
        const int row = p0 + 16 * (uc + u) + lg;
        const void* pr[2];
        float low[1][4], sum[1][4], xv[4];
        clear<1>(low);
        clear<1>(sum);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          xv[i] = (t + (i & 1) < tb + NC && row + 8 * (i >> 1) < p1) ? __ldg(x + (size_t)(t + (i & 1)) * d + row + 8 * (i >> 1)) : 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h)
          pr[h] = row + 8 * h < p1 ? static_cast<const char*>(g.P) + ((size_t)(row + 8 * h) * k + lt * 8) * (PF32 ? 4 : 2)
                                   : nullptr;
        dot_steps<1, PF32, false>(pr[0], pr[1], k, 0, 1, ksteps, op + nb * 8 * stride, stride, 0, NC - nb * 8, low, sum);
        add_low<1>(low, sum);
        float sr[2] = {0.f, 0.f}, sx[2] = {0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int tt = t + (i & 1), r = row + 8 * (i >> 1);
          const bool live = tt < tb + NC && r < p1;
          const float rv = live ? xv[i] - sum[0][i] : 0.f;
          // two rows of a token are written together (p0 is even) by the lane of the even row
          const float nx = __shfl_down_sync(0xffffffffu, rv, 4);
          if (live && !(lg & 1)) {
            uint32_t w[3];
            split3_pair(rv, nx, w);
            terms_store_pair(words.rb + (size_t)tt * term_bytes(d), r, d, w);
          }
          if (live && leave_from) g.r[(size_t)tt * d + r] = rv;
          sr[i & 1] = fmaf(rv, rv, sr[i & 1]);
          sx[i & 1] = fmaf(xv[i], xv[i], sx[i & 1]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) {
            sr[i] += __shfl_xor_sync(0xffffffffu, sr[i], o);
            sx[i] += __shfl_xor_sync(0xffffffffu, sx[i], o);
          }
          if (lg == 0) s_unit[u][nb * 8 + 2 * lt + i] = make_float2(sr[i], sx[i]);
        }
      }
      auto add_units = [&](int t) -> float2 {
        float2 v = s_run[t];
        for (int u = 0; u < nu; ++u) {
          v.x += s_unit[u][t].x;
          v.y += s_unit[u][t].y;
        }
        return v;
      };
      if (uc + nu >= pt) {
        __syncwarp();
        int before = 0;
        if (lane == 0) {
          __threadfence_block();
          before = atomicAdd(&s_done, 1);
          __threadfence_block();
        }
        before = __shfl_sync(0xffffffffu, before, 0);
        __syncwarp();
        if (before == kW - 1) {
          fence_gpu();   // the CTA's r, which this warp now knows to be written, before the word that announces it
          for (int t = lane; t < NC; t += 32) {
            const float2 v = add_units(t);
            put128(words.norm + (size_t)cta * n + tb + t, __float_as_uint(v.x), __float_as_uint(v.y), 0u, tag);
          }
          if (lane == 0) s_done = 0;
        }
      } else {
        __syncthreads();
        if (tid < NC) s_run[tid] = add_units(tid);
        __syncthreads();
      }
    }
    // image rows (the last warps, which have no basis rows in small calls, go first)
    for (int it = kW - 1 - warp; it < ot * ncb; it += kW) {
      const int u = it / ncb, nb = it - u * ncb, row = o0 + 16 * u + lg;
      const void* pr[2];
      float low[1][4], sum[1][4];
      clear<1>(low);
      clear<1>(sum);
#pragma unroll
      for (int h = 0; h < 2; ++h) pr[h] = row + 8 * h < o1 ? g.WP + (size_t)(row + 8 * h) * k + lt * 8 : nullptr;
      dot_steps<1, false, false>(pr[0], pr[1], k, 0, 1, ksteps, op + nb * 8 * stride, stride, 0, NC - nb * 8, low, sum);
      add_low<1>(low, sum);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int t = tb + nb * 8 + 2 * lt + (i & 1), r = row + 8 * (i >> 1);
        if (t < tb + NC && r < o1) io.y[(size_t)t * g.O + r] = sum[0][i];
      }
    }
  }

  // ---- x2: the norms of a token, every CTA's share, by one warp, added in double in a fixed order;
  // the gate.  In small calls every CTA takes every decision (the same sums: the same decision),
  // else token t's is taken by one CTA, which passes it on.
  auto decide = [&](int t) -> bool {
    constexpr int kPer = kFusedMaxGrid / 32;
    Word128 w[kPer];
    bool all = false;
    for (unsigned it = 0; !all && it < g.spin_limit; ++it) {
      all = true;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int c = lane + 32 * i;
        w[i] = Word128{0u, 0u, 0u, tag};
        if (c < G) w[i] = get128(words.norm + (size_t)c * n + t);
      }
#pragma unroll
      for (int i = 0; i < kPer; ++i) all = all && w[i].tag == tag;
      all = __all_sync(0xffffffffu, all);
    }
    ok = ok && all;
    fence_gpu();
    double sr = 0.0, sx = 0.0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      sr += (double)__uint_as_float(w[i].a);
      sx += (double)__uint_as_float(w[i].b);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sr += __shfl_xor_sync(0xffffffffu, sr, o);
      sx += __shfl_xor_sync(0xffffffffu, sx, o);
    }
    const double nr = sqrt(sr), nx = sqrt(sx);
    if (lane == 0) s_rho[t] = (float)(nr / nx);
    return nr < (double)g.eps * nx;   // false for NaN and for x = 0
  };
  if (kDirect || n <= kDecideTokens) {
    if (warp < n) {
      const bool fast = decide(warp);
      if (lane == 0) s_fast[warp] = fast;
    }
  } else {
    for (int t = cta + warp * G; t < n; t += kW * G) {
      const bool fast = decide(t);
      __syncwarp();   // what the lanes have seen (every CTA's r), before the word that announces it
      if (lane == 0) fence_gpu();
      if (lane == 0 && ok) put128(words.gate + t, __float_as_uint(s_rho[t]), fast ? 1u : 0u, 0u, tag);
    }
    __syncwarp();
    if (warp < 2 && warp * 32 + lane < n) {
      // (a first look ahead of the words would hold up their writers: 21 tokens 26.6 -> 26.4 us)
      for (const long long t0 = clock64(); clock64() - t0 < kGateHoldOff;) {}
      Word128 w = get128(words.gate + warp * 32 + lane);
      for (unsigned it = 1; w.tag != tag && it < g.spin_limit; ++it) w = get128(words.gate + warp * 32 + lane);
      ok = ok && w.tag == tag;
      s_fast[warp * 32 + lane] = w.b != 0u;
      s_rho[warp * 32 + lane] = __uint_as_float(w.a);
      fence_gpu();
    }
  }
  if (timed_out(ok)) return false;
  if (tid == 0 && cta > 0) leave_launch(g.tickets);   // (that was the last wait)
  if (warp == 0) {
    int f = 0;
    for (int t0 = 0; t0 < n; t0 += 32) {
      const int t = t0 + lane;
      bool fired = false;
      if (t < n) {
        const bool fast = s_fast[t];
        fired = !fast && !(g.flags & GSI_FLAG_STATIC_PROJECTION);
        if (cta == 0) {
          io.gate[(long long)slot * io.log_step_stride + t] = fast ? 0 : 1;
          float* rho = io.rho ? io.rho + (long long)slot * io.log_step_stride : g.rho_scratch;
          rho[t] = s_rho[t];
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, fired);
      const int at = f + __popc(m & ((1u << lane) - 1u));
      if (fired) {
        s_fired[1 + at] = t;
        if (leave_from && cta == 0) g.fired[at] = t;
      }
      f += __popc(m);
    }
    if (lane == 0) {
      s_fired[0] = f;
      if (leave_from && cta == 0) *g.n_fired = f;
    }
  }
  __syncthreads();
  if (tid == 0 && cta == 0) leave_launch(g.tickets);   // (behind the gates and rho)
  if (s_fired[0] == 0 || (leave_from && s_fired[0] >= leave_from)) return true;

  // ---- C
  if (s_fired[0] <= 8) stream_w<1>(g, io, words.rb, s_fired, smem, o0, o1);
  else if (s_fired[0] <= 16) stream_w<2>(g, io, words.rb, s_fired, smem, o0, o1);
  else stream_w<4>(g, io, words.rb, s_fired, smem, o0, o1);
  return true;
}

template <int NB, bool PF32, bool kDirect>
__global__ void __launch_bounds__(kT, 1) k_forward_fused(const __grid_constant__ GroupParams g, const __grid_constant__ IoRef io,
                                                         int n_tokens, int n_slabs,
                                                         int leave_from) {
  if (forward_fused<NB, PF32, kDirect>(g, io, n_tokens, n_slabs, leave_from)) return;
  // The call's results must not pass for results (the allocation-free entry point has no status word
  // to ask for): NaN in this CTA's rows of y, whose W r may be missing, and in every token's rho.
  const float nan = __int_as_float(0x7fc00000);
  const int cta = blockIdx.x, G = gridDim.x;
  const int o0 = (int)((long long)g.O * cta / G), o1 = (int)((long long)g.O * (cta + 1) / G);
  for (int t = 0; t < n_tokens; ++t)
    for (int row = o0 + (int)threadIdx.x; row < o1; row += kT) io.y[(size_t)t * g.O + row] = nan;
  if (leave_from && cta == 0 && threadIdx.x == 0) *g.n_fired = 0;   // no list of another call for the contraction
  if (cta > 0 && threadIdx.x == 0)
    for (int i = 0; i < kReportPolls && !block0_left(g.tickets); ++i) {}
  __syncthreads();
  let_land();
  report_give_up(g, io, n_tokens);
}

template <int NB, bool PF32, bool kDirect>
cudaError_t launch_fused_t(GroupParams g, IoRef io, int n_tokens, int n_slabs, int leave, int grid, cudaStream_t st) {
  auto kernel = k_forward_fused<NB, PF32, kDirect>;
  static bool configured[64] = {};   // per device: the attribute belongs to the device's function
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  if (dev >= 64 || !configured[dev]) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemFused);
    if (e != cudaSuccess) return e;
    if (dev < 64) configured[dev] = true;
  }
  void* args[] = {&g, &io, &n_tokens, &n_slabs, &leave};
  return cudaLaunchCooperativeKernel((void*)kernel, dim3(grid), dim3(kT), args, kSmemFused, st);
}
template <int NB, bool kDirect>
cudaError_t launch_fused_p(const GroupParams& g, const IoRef& io, int n, int slabs, int leave, int grid, cudaStream_t st) {
  return g.p_f32 ? launch_fused_t<NB, true, kDirect>(g, io, n, slabs, leave, grid, st)
                 : launch_fused_t<NB, false, kDirect>(g, io, n, slabs, leave, grid, st);
}

}  // namespace

size_t fused_words_bytes(int d, int k, int max_tokens) {
  return 8 * ((size_t)kFusedMaxGrid * (max_tokens * (kCols + 2) + 4) + (size_t)max_tokens * (k + 2) + d) +
         (size_t)max_tokens * term_bytes(d);
}

namespace {
template <typename F>
F driver_function(const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
    return nullptr;
  return reinterpret_cast<F>(p);
}
}  // namespace

unsigned long long context_id() {
  static const auto id_of = driver_function<CUresult (*)(CUcontext, unsigned long long*)>("cuCtxGetId");
  static const auto current = driver_function<CUresult (*)(CUcontext*)>("cuCtxGetCurrent");
  int dev = 0;
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;   // (makes a context current)
  return id_of && current && current(&ctx) == CUDA_SUCCESS && ctx && id_of(ctx, &id) == CUDA_SUCCESS ? id : 0;
}

// (The number of SMs is asked of a context once per thread: 0.3 us.)
int fused_grid() {
  static const auto resource_of =
      driver_function<CUresult (*)(CUcontext, CUdevResource*, CUdevResourceType)>("cuCtxGetDevResource");
  static const auto current = driver_function<CUresult (*)(CUcontext*)>("cuCtxGetCurrent");
  static thread_local unsigned long long last_id = 0;
  static thread_local int last_grid = 0;
  const unsigned long long id = context_id();
  int dev = 0, grid = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  CUcontext ctx = nullptr;
  const bool known = id && resource_of && current && current(&ctx) == CUDA_SUCCESS && ctx;
  if (known && last_grid && id == last_id) return last_grid;
  CUdevResource sm{};
  if (known && resource_of(ctx, &sm, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS && sm.sm.smCount > 0)
    grid = (int)sm.sm.smCount;
  else if (cudaDeviceGetAttribute(&grid, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  if (grid > kFusedMaxGrid) grid = kFusedMaxGrid;
  if (known) {
    last_id = id;
    last_grid = grid;
  }
  return grid;
}

int fused_slabs(int d, int k, int grid) {
  int slabs = grid / ((k + kCols - 1) / kCols);
  if (slabs > (d + 31) / 32) slabs = (d + 31) / 32;
  return slabs < 1 ? 1 : slabs;
}

cudaError_t launch_forward_fused(const GroupParams& g, const IoRef& io, int n_tokens, int leave_from,
                                 cudaStream_t st) {
  return launch_resident([&](int grid) -> cudaError_t {
    const int slabs = fused_slabs(g.d, g.k, grid);
    const bool direct = n_tokens <= kDirectTokens && grid * kCols >= g.k;
    return direct            ? launch_fused_p<1, true>(g, io, n_tokens, slabs, leave_from, grid, st)
           : n_tokens <= 8           ? launch_fused_p<1, false>(g, io, n_tokens, slabs, leave_from, grid, st)
           : n_tokens <= 16          ? launch_fused_p<2, false>(g, io, n_tokens, slabs, leave_from, grid, st)
                                     : launch_fused_p<4, false>(g, io, n_tokens, slabs, leave_from, grid, st);
  });
}

}  // namespace gsi
