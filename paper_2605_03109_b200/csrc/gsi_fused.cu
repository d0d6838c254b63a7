// One call of any supported shape as ONE launch: Algorithm 1 with two grid-wide exchanges inside a
// cooperative kernel (every CTA resident).
//
//   A   partial c of a slab of basis rows x 32 columns per CTA              (line 1)
//   x1  the partials are added in slab order: by every CTA for itself in calls of a few tokens,
//       else each coefficient by one CTA, which passes the sum on to all
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
// the five launches of the per-stage kernels before: one token at 768 x 64 -> 3072 27.3 -> 15.8 us,
// at 4096 x 256 -> 28672 41.7 -> 16.0 us; 21 tokens at 3000 x 200 -> 1576 84 -> 46 us (on CUDA-core
// FMAs this kernel took 112 us there); 16 tokens, fp32 basis, 768 x 128 -> 2304 48.5 -> 23.7 us.
//
// The exchanges are words that carry the call's number (gsi_exchange.cuh): a release / acquire
// barrier would cost two L2 round trips and a fence where these cost one.  Every token's sums run
// in an order that depends on the shape alone: results are reproducible, and a token's are the
// same in a call of any size.
// Every wait is bounded; a wait that gives up sets GSI_ERR_TIMEOUT and the CTA returns.
#include "gsi_exchange.cuh"

namespace gsi {

namespace {

using namespace exchange;

constexpr int kT = 512, kW = kT / 32;
constexpr int kTileRows = 16 * kW;     // rows of a basis slab (and of W) per pass: 16 per warp
constexpr int kPitch = 80;             // bytes between the staged 64-byte pieces: conflict-free ldmatrix
constexpr int kDirectTokens = 4;       // calls of so few tokens gather the slabs' partials themselves
// dynamic shared memory: operand terms (phase A: the slab), then partial sums
constexpr int kOpBytes = 131072, kAuxBytes = 32768;
constexpr int kSmemFused = kOpBytes + kAuxBytes;

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

// Operand of eight-token blocks: 16 bytes (eight neighbours of the contraction) of term q of
// column (token) c at step s (32 of the contraction), lane quarter t.  Only the NC columns that
// exist are stored.
__device__ __forceinline__ int op_at(int s, int q, int c, int t, int NC) { return ((s * 3 + q) * NC + c) * 4 + t; }

template <int NB>
__device__ __forceinline__ void clear(float (&v)[NB][4]) {
#pragma unroll
  for (int nb = 0; nb < NB; ++nb)
#pragma unroll
    for (int i = 0; i < 4; ++i) v[nb][i] = 0.f;
}

// sum[nb] += rows g and g + 8 (p0, p1: this lane's pointers to element 8 t of each row, null when
// the row does not exist) x columns 8 nb .. 8 nb + 7 over steps s0, s0 + ds, .. < s1.  `op` holds
// the operand from step op0 on; K: length of the contraction.  The tensor core's own accumulation
// truncates (a chain of 48 instructions is 2e-6 off, ten times an FMA chain), so the products of
// the leading terms start from zero in every step and are added in fp32; those of the lower
// terms, 2^-8 of the value, go through one accumulator of their own (low).
template <int NB, bool AF32, bool kStream>
__device__ __forceinline__ void dot_steps(const void* p0, const void* p1, int K, int s0, int ds, int s1,
                                          const uint4* op, int op0, int NC, float (&low)[NB][4], float (&sum)[NB][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  constexpr int U = AF32 ? 2 : 4;   // steps in flight
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
          if (nb * 8 + g < NC) b = op[op_at(s - op0, q, nb * 8 + g, t, NC)];
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

// y += W r for the fired tokens, 8 NB at a time.  A warp owns 16 of this CTA's rows of W and every
// ks-th step of the contraction (narrow maps: several warps share 16 rows and their sums meet in
// shared memory); r comes from the exchange words into operand form as much of the width at a
// time as fits.
template <int NB>
__device__ __forceinline__ void stream_w(const GroupParams& g, const IoRef& io, const unsigned long long* rw,
                                         unsigned tag, const int* s_fired, unsigned char* smem, int o0, int o1) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lg = lane >> 2, lt = lane & 3;
  const int d = g.d, n_fired = s_fired[0], steps = (d + 31) / 32;
  uint4* op = reinterpret_cast<uint4*>(smem);
  float* part = reinterpret_cast<float*>(smem + kOpBytes);   // [warp][16 rows][8 NB]
  static_assert(kW * 16 * 8 * NB * 4 <= kAuxBytes, "partial sums of the warps");
  for (int f0 = 0; f0 < n_fired; f0 += 8 * NB) {
    const int NC = min(8 * NB, n_fired - f0);
    const int span = min(steps, kOpBytes / (192 * NC));   // steps whose operand fits (192 bytes per column)
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
          bool ok = true;
          const int octets = (s1 - s0) * 4;   // eight elements each
          for (int i = tid; i < octets * NC; i += kT) {
            const int c = i / octets, o8 = i % octets, e = s0 * 32 + o8 * 8;
            uint4 tm[3];
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = 0.f;
            if (e < d) ok = gather(rw + (size_t)s_fired[1 + f0 + c] * d + e, 1, 8, tag, [&](int q, float x) { v[q] = x; }) && ok;
            split3_x8(v, tm);
#pragma unroll
            for (int q = 0; q < 3; ++q) op[op_at(o8 >> 2, q, c, o8 & 3, NC)] = tm[q];
          }
          if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
            return;
          }
        }
        // step s belongs to warp s % ks (ks a power of two)
        if (active) dot_steps<NB, false, true>(p[0], p[1], d, s0 + ((kq - s0) & (ks - 1)), ks, s1, op, s0, NC, low, sum);
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

// 8 NB tokens at a time.  leave_from > 0: with that many gated tokens or more W r is left to the
// tensor-core contraction that follows (r goes to g.r, the gated tokens to g.fired).
template <int NB, bool PF32>
__global__ void __launch_bounds__(kT, 1) k_forward_fused(GroupParams g, IoRef io, int n_tokens, int n_slabs,
                                                         int leave_from) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float s_x2[kW][8 * NB];                  // the warps' partial norms
  __shared__ double s_norm[GSI_MAX_TOKENS][2];
  __shared__ int s_fired[GSI_MAX_TOKENS + 1];
  constexpr int kTerms = PF32 ? 3 : 1, kTok = 8 * NB;
  float* s_aux = reinterpret_cast<float*>(smem + kOpBytes);
  uint4* op = reinterpret_cast<uint4*>(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lg = lane >> 2, lt = lane & 3;
  const int G = gridDim.x, cta = blockIdx.x;
  const int d = g.d, k = g.k, n = n_tokens;
  const unsigned tag = *g.fused_call + 1u;
  const Words words = words_of(g);
  unsigned long long *cw = words.c, *xw = words.x2, *nw = words.r2, *cf = words.cf, *rw = words.r;
  const int slot = io_slot(io);
  const float* x = io.x + (long long)slot * io.x_step_stride;
  const int o0 = (int)((long long)g.O * cta / G), o1 = (int)((long long)g.O * (cta + 1) / G);
  const int p0 = (int)((long long)d * cta / G), p1 = (int)((long long)d * (cta + 1) / G);

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
  if (cta < n_slabs * n_cb) {
    const int slab = cta / n_cb, cb = cta % n_cb;
    const int r0 = (int)((long long)d * slab / n_slabs), r1 = (int)((long long)d * (slab + 1) / n_slabs);
    for (int tb = 0; tb < n; tb += kTok) {
      float acc[2][NB][4], sx[NB];
#pragma unroll
      for (int nb = 0; nb < NB; ++nb) sx[nb] = 0.f;
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
            for (int h = 0; h < 2; ++h) {
              split3_pair(xv[nb][2 * h], xv[nb][2 * h + 1], xt[nb][h]);
              sx[nb] = fmaf(xv[nb][2 * h], xv[nb][2 * h], sx[nb]);
              sx[nb] = fmaf(xv[nb][2 * h + 1], xv[nb][2 * h + 1], sx[nb]);
            }
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
      if (cb == 0) {
#pragma unroll
        for (int nb = 0; nb < NB; ++nb) {
          float s = sx[nb];
          s += __shfl_xor_sync(0xffffffffu, s, 1);
          s += __shfl_xor_sync(0xffffffffu, s, 2);
          if (lt == 0) s_x2[warp][nb * 8 + lg] = s;
        }
      }
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
      if (cb == 0 && tid < kTok && tb + tid < n) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kW; ++w) s += s_x2[w][tid];
        put(xw + (size_t)slab * n + tb + tid, s, tag);
      }
      __syncthreads();
    }
  }

  // ---- x1.  Sum of a coefficient over the slabs: Q threads, each its slabs in order
  bool ok = true;
  int Q = 1;
  while (2 * Q * k <= kT && Q < 8) Q *= 2;
  auto slab_sum = [&](int i, bool live) -> float {   // i = token * k + j; all lanes of a group of Q
    const int q = tid % Q;
    float s = 0.f;
    if (live) {
      const int a = n_slabs * q / Q, b = n_slabs * (q + 1) / Q;
      ok = gather(cw + (size_t)a * n * k + i, (size_t)n * k, b - a, tag, [&](int, float v) { s += v; }) && ok;
    }
    for (int o = 1; o < Q; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  };
  const bool direct = n <= kDirectTokens;
  if (!direct) {
    const int i0 = (int)((long long)n * k * cta / G), i1 = (int)((long long)n * k * (cta + 1) / G);
    for (int ib = i0; ib < i1; ib += kT / Q) {
      const int i = ib + tid / Q;
      const float s = slab_sum(i, i < i1);
      if (i < i1 && tid % Q == 0) put(cf + i, s, tag);
    }
  }

  // ---- x1 (end) and B
  const int ksteps = (k + 31) / 32;
  for (int tb = 0; tb < n; tb += kTok) {
    const int NC = min(kTok, n - tb), items = NC * k;
    unsigned short* op16 = reinterpret_cast<unsigned short*>(op);
    auto store_c = [&](int i, float v) {   // i = column * k + j: the three terms of a coefficient
      const int c = i / k, j = i - c * k;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        op16[op_at(j >> 5, q, c, (j >> 3) & 3, NC) * 8 + (j & 7)] = __bfloat16_as_ushort(h);
        v -= __bfloat162float(h);
      }
    };
    if (tb > 0) __syncthreads();
    for (int i = tid; i < (ksteps * 32 - k) * NC; i += kT) {   // the operand beyond k
      const int c = i % NC, j = k + i / NC;
#pragma unroll
      for (int q = 0; q < 3; ++q) op16[op_at(j >> 5, q, c, (j >> 3) & 3, NC) * 8 + (j & 7)] = 0;
    }
    if (direct) {
      for (int ib = 0; ib < items; ib += kT / Q) {
        const int i = ib + tid / Q;
        const float s = slab_sum(tb * k + i, i < items);
        if (i < items && tid % Q == 0) store_c(i, s);
      }
    } else {
      for (int ib = 0; ib < items; ib += 8 * kT) {
        const int cnt = items > ib + tid ? min(8, (items - ib - tid + kT - 1) / kT) : 0;
        ok = gather(cf + (size_t)tb * k + ib + tid, kT, cnt, tag, [&](int u, float v) { store_c(ib + tid + u * kT, v); }) && ok;
      }
    }
    if (__syncthreads_or(!ok)) {
      if (tid == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
      if (tid == 0 && cta == 0) *g.fused_call = tag;
      return;
    }
    // units of 16 rows: first the basis rows, then (their norms travel meanwhile) the image rows
    const int pt = (p1 - p0 + 15) / 16, ot = (o1 - o0 + 15) / 16;
    float sr[NB][2];
#pragma unroll
    for (int nb = 0; nb < NB; ++nb) sr[nb][0] = sr[nb][1] = 0.f;
    for (int u = warp; u < pt; u += kW) {
      const int row = p0 + 16 * u + lg;
      const void* pr[2];
      float low[NB][4], sum[NB][4];
      clear<NB>(low);
      clear<NB>(sum);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        pr[h] = row + 8 * h < p1 ? static_cast<const char*>(g.P) + ((size_t)(row + 8 * h) * k + lt * 8) * (PF32 ? 4 : 2)
                                 : nullptr;
      dot_steps<NB, PF32, false>(pr[0], pr[1], k, 0, 1, ksteps, op, 0, NC, low, sum);
      add_low<NB>(low, sum);
#pragma unroll
      for (int nb = 0; nb < NB; ++nb)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int t = tb + nb * 8 + 2 * lt + (i & 1), r = row + 8 * (i >> 1);
          if (t < n && r < p1) {
            const float rv = __ldg(x + (size_t)t * d + r) - sum[nb][i];
            put(rw + (size_t)t * d + r, rv, tag);
            if (leave_from) g.r[(size_t)t * d + r] = rv;
            sr[nb][i & 1] = fmaf(rv, rv, sr[nb][i & 1]);
          }
        }
    }
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        float s = sr[nb][i];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lg == 0) s_x2[warp][nb * 8 + 2 * lt + i] = s;
      }
    __syncthreads();
    if (tid < NC) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < kW; ++w) s += s_x2[w][tid];
      put(nw + (size_t)cta * n + tb + tid, s, tag);
    }
    // (warps without basis rows go first: units are dealt from the last warp down)
    for (int u = kW - 1 - warp; u < ot; u += kW) {
      const int row = o0 + 16 * u + lg;
      const void* pr[2];
      float low[NB][4], sum[NB][4];
      clear<NB>(low);
      clear<NB>(sum);
#pragma unroll
      for (int h = 0; h < 2; ++h) pr[h] = row + 8 * h < o1 ? g.WP + (size_t)(row + 8 * h) * k + lt * 8 : nullptr;
      dot_steps<NB, false, false>(pr[0], pr[1], k, 0, 1, ksteps, op, 0, NC, low, sum);
      add_low<NB>(low, sum);
#pragma unroll
      for (int nb = 0; nb < NB; ++nb)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int t = tb + nb * 8 + 2 * lt + (i & 1), r = row + 8 * (i >> 1);
          if (t < n && r < o1) io.y[(size_t)t * g.O + r] = sum[nb][i];
        }
    }
  }

  // ---- x2: norms, gate (the same sums in the same order on every CTA)
  for (int i = warp; i < 2 * n; i += kW) {
    const int t = i >> 1;
    double s = 0.0;
    ok = ((i & 1) ? warp_gather_sum(xw + t, n, n_slabs, tag, s) : warp_gather_sum(nw + t, n, G, tag, s)) && ok;
    if (lane == 0) s_norm[t][i & 1] = s;
  }
  if (__syncthreads_or(!ok)) {
    if (tid == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
    if (tid == 0 && cta == 0) *g.fused_call = tag;
    return;
  }
  if (warp == 0) {
    int f = 0;
    for (int t0 = 0; t0 < n; t0 += 32) {
      const int t = t0 + lane;
      bool fired = false;
      if (t < n) {
        const double nr = sqrt(s_norm[t][0]), nx = sqrt(s_norm[t][1]);
        const bool fast = nr < (double)g.eps * nx;   // false for NaN and for x = 0
        fired = !fast && !(g.flags & GSI_FLAG_STATIC_PROJECTION);
        if (cta == 0) {
          io.gate[(long long)slot * io.log_step_stride + t] = fast ? 0 : 1;
          float* rho = io.rho ? io.rho + (long long)slot * io.log_step_stride : g.rho_scratch;
          rho[t] = (float)(nr / nx);
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
      if (cta == 0) *g.fused_call = tag;   // every CTA has read the counter: its norms are here
    }
  }
  __syncthreads();
  if (s_fired[0] == 0 || (leave_from && s_fired[0] >= leave_from)) return;

  // ---- C
  stream_w<NB>(g, io, rw, tag, s_fired, smem, o0, o1);
}

template <int NB, bool PF32>
cudaError_t launch_fused_t(GroupParams g, IoRef io, int n_tokens, int n_slabs, int leave, int grid, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_forward_fused<NB, PF32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSmemFused);
  if (e != cudaSuccess) return e;
  void* args[] = {&g, &io, &n_tokens, &n_slabs, &leave};
  return cudaLaunchCooperativeKernel((void*)k_forward_fused<NB, PF32>, dim3(grid), dim3(kT), args, kSmemFused, st);
}
template <int NB>
cudaError_t launch_fused_p(const GroupParams& g, const IoRef& io, int n, int slabs, int leave, int grid, cudaStream_t st) {
  return g.p_f32 ? launch_fused_t<NB, true>(g, io, n, slabs, leave, grid, st)
                 : launch_fused_t<NB, false>(g, io, n, slabs, leave, grid, st);
}

}  // namespace

size_t fused_words_bytes(int d, int k, int max_tokens) {
  return 8 * ((size_t)kFusedMaxGrid * max_tokens * (kCols + 2) + (size_t)max_tokens * (k + d));
}

int fused_grid() {
  static int sms_of[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  int grid = dev < 64 ? sms_of[dev] : 0;
  if (!grid) {
    if (cudaDeviceGetAttribute(&grid, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (dev < 64) sms_of[dev] = grid;
  }
  return grid > kFusedMaxGrid ? kFusedMaxGrid : grid;
}

int fused_slabs(int d, int k, int grid) {
  int slabs = grid / ((k + kCols - 1) / kCols);
  if (slabs > (d + 31) / 32) slabs = (d + 31) / 32;
  return slabs < 1 ? 1 : slabs;
}

cudaError_t launch_forward_fused(const GroupParams& g, const IoRef& io, int n_tokens, int leave_from,
                                 cudaStream_t st) {
  const int grid = fused_grid();
  if (!grid) return cudaErrorInvalidDevice;
  const int slabs = fused_slabs(g.d, g.k, grid);
  // eight-token blocks at a time: those of the call, as far as their c fits (6 bytes per
  // coefficient, padded to 32) and the sums fit the registers (four)
  int nb = 1;
  while (8 * nb < n_tokens && nb < 4 && 2 * nb * 48 * ((g.k + 31) / 32 * 32) <= kOpBytes) nb *= 2;
  switch (nb) {
    case 1: return launch_fused_p<1>(g, io, n_tokens, slabs, leave_from, grid, st);
    case 2: return launch_fused_p<2>(g, io, n_tokens, slabs, leave_from, grid, st);
    default: return launch_fused_p<4>(g, io, n_tokens, slabs, leave_from, grid, st);
  }
}

}  // namespace gsi
