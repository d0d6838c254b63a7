// Batched front end of the gated subspace layer on the 5th-gen tensor cores:
// Algorithm 1 lines 1-5 for a batch of tokens as three skinny contractions,
//
//   c  = P^T x      A = P^T tile [128 of k][d],   B = terms of x [3n][d],  split over d
//   Pc (-> r, gate) A = P tile   [128 of d][k],   B = terms of c [3n][k]
//   y  = W_P c      A = W_P tile [128 of O][k],   B = terms of c [3n][k]
//
// The basis and the images are bf16 already; the fp32 activations and coefficients
// enter as THREE bf16 terms each (v = hi + mid + lo, 24 significant bits), stored as
// rows 3t, 3t+1, 3t+2 of the B operand, so every product is exact and the sums are
// fp32 in tensor memory: the same arithmetic as the CUDA-core kernels up to the order
// of the additions.  The epilogues add the three columns of a token and apply the rest
// of the line: the split-K partial of c; r = x - Pc with the partial sums of ||r||^2
// and ||x||^2 followed by the gate decision (Eq. (3.3)) in the last block; y.
#include "gsi_umma.cuh"

namespace gsi {

namespace {

using namespace umma;

// stages of the projection: in a stack, blocks of 82 KB, which find a slot beside the W streams sooner
// (four stages left a step 2-7 % slower); in a call by itself there is nothing beside them
constexpr int kStages3 = 2, kStages3Alone = 4;
constexpr int kMaxN3 = 192;          // 3 terms x 64 tokens
constexpr int kTmemCols3 = 256;      // power of two >= kMaxN3
// residual / image: K = k is short (four 64-wide blocks at k = 256).  Up to 32 tokens the B
// operand is small enough for four stages with two blocks per SM, so every weight box of a
// tile is requested before the wait on the previous kernel; beyond, two stages.
constexpr int kStagesRI = 2, kStagesRIs = 4;
constexpr int kMaxN3s = 96, kTmemCols3s = 128;   // 3 terms x 32 tokens
constexpr int kSmemRI = Cfg<kStagesRI, kMaxN3>::kSmem;
constexpr int kSmemRIs = Cfg<kStagesRIs, kMaxN3s>::kSmem;

__device__ __forceinline__ uint16_t bf16_bits(float v) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  return *reinterpret_cast<const uint16_t*>(&h);
}
__device__ __forceinline__ float bf16_val(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

// v = hi + mid + lo exactly for every finite fp32 v whose low term is not subnormal.
__device__ __forceinline__ void split3(float v, uint16_t& hi, uint16_t& mid, uint16_t& lo) {
  hi = bf16_bits(v);
  const float r1 = v - bf16_val(hi);
  mid = bf16_bits(r1);
  const float r2 = r1 - bf16_val(mid);
  lo = bf16_bits(r2);
}

__device__ __forceinline__ int rows3(int n_tokens) { return term_rows(n_tokens); }

// src [n_tokens][len] fp32 -> dst [rows3][len] bf16 terms; rows past 3 n_tokens are zero.
// One block row (blockIdx.y) per token slot, 8 elements per thread.
__device__ __forceinline__ void store_terms(const float (&v)[8], bool live, uint16_t* dst, int slot,
                                            int n_rows, size_t len, size_t at) {
  uint32_t w[3][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    uint16_t a[3], b[3];
    if (live) {
      split3(v[2 * e], a[0], a[1], a[2]);
      split3(v[2 * e + 1], b[0], b[1], b[2]);
    } else {
      a[0] = a[1] = a[2] = b[0] = b[1] = b[2] = 0;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) w[c][e] = (uint32_t)a[c] | ((uint32_t)b[c] << 16);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int row = 3 * slot + c;
    if (row < n_rows)
      *reinterpret_cast<uint4*>(dst + (size_t)row * len + at) = make_uint4(w[c][0], w[c][1], w[c][2], w[c][3]);
  }
}

// Elements 8 i8 .. of token slot `slot`, i8 from `first` on in strides of `stride`.
__device__ __forceinline__ void split3_body(const GroupParams& g, const IoRef& io, int n_tokens, int slot, int first,
                                            int stride) {
  const int n_rows = rows3(n_tokens);
  const bool live = slot < n_tokens;
  const float* x = io.x + (long long)io_slot(io) * io.x_step_stride + (size_t)slot * g.d;
  for (int i8 = first; i8 < g.d / 8; i8 += stride) {
    float v[8] = {};
    if (live) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(x) + 2 * i8);
      const float4 b = __ldg(reinterpret_cast<const float4*>(x) + 2 * i8 + 1);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
    store_terms(v, live, g.xb, slot, n_rows, (size_t)g.d, (size_t)i8 * 8);
  }
}

__global__ void __launch_bounds__(256) k_split3_x(GroupParams g, IoRef io, int n_tokens) {
  // first kernel of the chain: wait first, so that nothing of the chain (its successors
  // request weight tiles before their own waits) runs beside an earlier call's kernels
  pdl_wait();   // xb may still be read by the previous call's projection
  pdl_launch_dependents();
  split3_body(g, io, n_tokens, blockIdx.y, blockIdx.x * 256 + threadIdx.x, gridDim.x * 256);
}

// c partials: cpart3[split][t][128*tile + lane row] over this split's share of d.
template <bool kInStack>
__device__ __forceinline__ void proj_body(unsigned char* smem_raw, const GroupParams& g, const TmaMaps& tm,
                                          int n_tokens, int block) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int splits = g.proj_splits;
  const int tile = block / splits, split = block % splits;
  const int nkb = g.d / kTK;
  const int kb0 = (int)((long long)nkb * split / splits), kb1 = (int)((long long)nkb * (split + 1) / splits);
  uint32_t tmem;
  const bool ok = tile_mma<kInStack ? kStages3 : kStages3Alone, kMaxN3, kTmemCols3, kInStack>(
      smem_raw, &tm.pt, tile * kTM, &tm.xb, 0, rows3(n_tokens), kb0, kb1 - kb0, &tmem);
  if (!ok) {
    if (threadIdx.x == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
  } else {
    const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16);
    float* out = g.cpart3 + (size_t)split * g.B * g.k + tile * kTM + warp * 32 + lane;
    for (int q = 0; 16 * q < n_tokens; ++q) {
      float s[16];
      sum3_tokens16(tl, q, s);
#pragma unroll
      for (int tt = 0; tt < 16; ++tt)
        if (16 * q + tt < n_tokens) out[(size_t)(16 * q + tt) * g.k] = s[tt];
    }
  }
  tile_release<kTmemCols3>(tmem);
}

template <bool kInStack>
__global__ void __launch_bounds__(kThreads, 1)
k_proj_tc(GroupParams g, const __grid_constant__ TmaMaps tm, int n_tokens) {
  extern __shared__ unsigned char smem_raw[];
  pdl_launch_dependents();
  proj_body<kInStack>(smem_raw, g, tm, n_tokens, blockIdx.x);
}

// c = sum of the split-K partials in split order; also its three bf16 terms.
// One block per token slot, one coefficient per thread and pass.
__device__ __forceinline__ void reduce_body(const GroupParams& g, int n_tokens, int slot) {
  const int n_rows = rows3(n_tokens);
  const bool live = slot < n_tokens;
  for (int j = threadIdx.x; j < g.k; j += 256) {
    float v = 0.f;
    if (live) {
      const float* p = g.cpart3 + (size_t)slot * g.k + j;
      const size_t stride = (size_t)g.B * g.k;
      int s = 0;
      for (; s + 32 <= g.proj_splits; s += 32) {   // thirty-two partials in flight, summed in order
        float u[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) u[i] = p[(size_t)(s + i) * stride];
#pragma unroll
        for (int i = 0; i < 32; ++i) v += u[i];
      }
      for (; s + 8 <= g.proj_splits; s += 8) {
        float u[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) u[i] = p[(size_t)(s + i) * stride];
#pragma unroll
        for (int i = 0; i < 8; ++i) v += u[i];
      }
      for (; s < g.proj_splits; ++s) v += p[(size_t)s * stride];
      g.c[(size_t)slot * g.k + j] = v;
    }
    uint16_t term[3] = {0, 0, 0};
    if (live) split3(v, term[0], term[1], term[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (3 * slot + c < n_rows) g.cb[(size_t)(3 * slot + c) * g.k + j] = term[c];
  }
}

__global__ void __launch_bounds__(256) k_reduce_split3_c(GroupParams g, int n_tokens) {
  pdl_launch_dependents();
  pdl_wait();
  reduce_body(g, n_tokens, blockIdx.x);
}

// Lane l's result: the sum of v[l] over the lanes.  Every step halves the values and pairs the lanes:
// 31 shuffles for all 32 sums, where one after the other they take 160.
__device__ __forceinline__ float sum32_over_lanes(float (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float give = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  return v[0];
}

// One launch for Algorithm 1 lines 2-5.  Every block contracts one 128-row tile against
// the c terms of a range of 16-token groups (operand rows 48 q_lo .. 48 q_hi - 1):
//   blocks [0, n_resid)   tile of P, one of rs token ranges (rs > 1 spreads the narrow
//                         inputs, d = 4096: 32 tiles, over the machine):
//                         r = x - P c -> bf16 rows of rb, the partial norms of the tile,
//                         and in the block that finishes last the gate
//   blocks [n_resid, ..)  tile of W_P, all tokens: y = W_P c
template <int kStagesT, int kMaxRows, int kTmemColsT, bool kInStack>
__device__ __forceinline__ void resid_image_body(unsigned char* smem_raw, const GroupParams& g, const TmaMaps& tm,
                                                 const IoRef& io, int n_tokens, int rs, int block) {
  __shared__ float s_norm[kThreads / 32][GSI_MAX_TOKENS][2];
  __shared__ int s_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nq = (n_tokens + 15) / 16;
  const int n_resid = (g.d / kTM) * rs;
  const bool image = block >= n_resid;
  const int tile = image ? block - n_resid : block / rs;
  const int part = image ? 0 : block % rs;
  const int per = image ? nq : (nq + rs - 1) / rs;
  const int q_lo = min(part * per, nq), q_hi = min(q_lo + per, nq);
  const int row = tile * kTM + warp * 32 + lane;
  const int slot = io_slot(io);
  const float* x = io.x + (long long)slot * io.x_step_stride + row;

  float xv[16];
  if (!image && q_lo < q_hi) {
#pragma unroll
    for (int tt = 0; tt < 16; ++tt)
      xv[tt] = (16 * q_lo + tt < n_tokens) ? __ldg(x + (size_t)(16 * q_lo + tt) * g.d) : 0.f;
  }
  uint32_t tmem = 0;
  bool ok = true;
  if (q_lo < q_hi) {   // block-uniform
    const int n_rows = min(48 * (q_hi - q_lo), rows3(n_tokens) - 48 * q_lo);
    ok = tile_mma<kStagesT, kMaxRows, kTmemColsT, kInStack>(smem_raw, image ? &tm.wp : &tm.p, tile * kTM, &tm.cb,
                                                48 * q_lo, n_rows, 0, g.k / kTK, &tmem);
    if (!ok && threadIdx.x == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
    const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16);
    for (int q = q_lo; q < q_hi && ok; ++q) {
      float s[16];
      sum3_tokens16(tl, q - q_lo, s);
      if (image) {
#pragma unroll
        for (int tt = 0; tt < 16; ++tt)
          if (16 * q + tt < n_tokens) io.y[(size_t)(16 * q + tt) * g.O + row] = s[tt];
        continue;
      }
      float xn[16];   // the next group's x, in flight while this group is reduced
#pragma unroll
      for (int tt = 0; tt < 16; ++tt)
        xn[tt] = (q + 1 < q_hi && 16 * (q + 1) + tt < n_tokens) ? __ldg(x + (size_t)(16 * (q + 1) + tt) * g.d)
                                                                 : 0.f;
      float sq[32];   // ||r||^2 of the sixteen tokens, then ||x||^2
#pragma unroll
      for (int tt = 0; tt < 16; ++tt) {
        const int t = 16 * q + tt;
        const float rv = xv[tt] - s[tt];
        if (t < n_tokens) g.rb[(size_t)t * g.d + row] = bf16_bits(rv);
        sq[tt] = rv * rv;
        sq[16 + tt] = xv[tt] * xv[tt];
        xv[tt] = xn[tt];
      }
      const float sum = sum32_over_lanes(sq);
      const int t = 16 * q + (lane & 15);
      if (t < n_tokens) s_norm[warp][t][lane >> 4] = sum;
    }
    tile_release<kTmemColsT>(tmem);
  }
  if (image) return;
  __syncthreads();
  for (int i = threadIdx.x; i < 32 * (q_hi - q_lo); i += kThreads) {
    const int t = 16 * q_lo + (i >> 1), w = i & 1;
    if (t < n_tokens) {
      float sum = 0.f;
#pragma unroll
      for (int wp = 0; wp < kThreads / 32; ++wp) sum += ok ? s_norm[wp][t][w] : 0.f;
      g.normpart3[((size_t)tile * g.B + t) * 2 + w] = sum;
    }
  }
  decide_gate_last_block(g, io, slot, n_tokens, g.normpart3, g.d / kTM, (unsigned)n_resid, &s_last);
}

template <int kStagesT, int kMaxRows, int kTmemColsT, bool kInStack>
__global__ void __launch_bounds__(kThreads, 2)
k_resid_image_tc(GroupParams g, const __grid_constant__ TmaMaps tm, IoRef io, int n_tokens, int rs) {
  extern __shared__ unsigned char smem_raw[];
  pdl_launch_dependents();
  resid_image_body<kStagesT, kMaxRows, kTmemColsT, kInStack>(smem_raw, g, tm, io, n_tokens, rs, blockIdx.x);
}

// ---- the same for all groups of a range of a stack in one launch each -------------------
// (a block finds its group in the table; WideGroup)
// A step in a chain of five launches per group is the latency of its chains and the tails of small
// grids: 28 GPT-J layers, 64 tokens, a tenth gated, 477 launches 3.34 ms; the same kernels over all
// groups, whose inputs are staged before the step, 2.58 ms, with the persistent one below 2.49 (W r at the copy
// bandwidth); 12 GPT-2 layers, k = 256, 636 -> 153 -> 137 us.
__global__ void __launch_bounds__(256) k_split3_x_wide(WideParams p, int n_tokens, int slots) {
  pdl_wait();   // (first of the chain, as above)
  pdl_launch_dependents();
  int block;
  const WideGroup& w = p.find(kWideSplit, &block);
  const IoRef io = p.io_of(w);
  split3_body(w.g, io, n_tokens, block % slots, block / slots * 256 + threadIdx.x, (w.g.d / 8 + 255) / 256 * 256);
}

__global__ void __launch_bounds__(kThreads, 1) k_proj_wide(WideParams p, int n_tokens) {
  extern __shared__ unsigned char smem_raw[];
  pdl_launch_dependents();
  int block;
  const WideGroup& w = p.find(kWideProj, &block);
  if (threadIdx.x < 32) {
    acquire_map(&w.tm.pt);
    acquire_map(&w.tm.xb);
  }
  proj_body<true>(smem_raw, w.g, w.tm, n_tokens, block);
}

__global__ void __launch_bounds__(256) k_reduce_wide(WideParams p, int n_tokens, int slots) {
  pdl_launch_dependents();
  pdl_wait();
  reduce_body(p.table[blockIdx.x / slots].g, n_tokens, blockIdx.x % slots);
}

// Residual and image tiles of all groups, persistent: a CTA takes an even share of the tiles, in
// order, and with it the terms of c of few groups, which it keeps in shared memory while weight tiles
// stream through the ring (112 KB and more in flight).  Two accumulators: while four warps take one to
// r, norms and y, the next tile is contracted into the other.
//   warp 0 asks for the weight tiles (ahead of the wait on the kernel before), warp 1 for the terms, and
//   issues the contractions; warps 2-5 and 6-9 take the accumulators in turn.
// As a block per tile each lived 12 us (search, tensor maps, tensor memory, one round trip of the copies,
// epilogue) for 64 KB of weights: eight GPT-J layers at 8 tokens 175 -> 77 us (the step 463 -> 370), at 64 193 -> 167
// (760 -> 741; there the epilogue is what bounds it: 64 columns per row to store, and to add up for the residual).
constexpr int kThreadsW = 320, kSmemW = 220 * 1024, kBarBytesW = 512, kMostStagesW = 13;
constexpr int kTermBytesW = 100 * 1024;   // shared memory for the terms of c at most
constexpr int kTmemColsW = 512;

__global__ void __launch_bounds__(kThreadsW, 1) k_resid_image_wide(WideParams p, int n_tiles, int n_tokens) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ float s_norm[2][4][GSI_MAX_TOKENS][2];
  __shared__ unsigned char s_gate[2][GSI_MAX_TOKENS];
  __shared__ int s_last[2], s_fail, s_issued, s_terms;
  pdl_launch_dependents();
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kSmemW - 1024 - kBarBytesW);
  uint64_t *full = bars, *empty = bars + kMostStagesW, *tfull = empty + kMostStagesW, *tempty = tfull + 2,
           *terms = tempty + 2, *read = terms + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(read + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nq = (n_tokens + 15) / 16, rows_all = rows3(n_tokens);
  unsigned char* s_terms_at = smem;
  unsigned char* s_ring = smem + p.term_bytes;
  const int stages = min(kMostStagesW, (kSmemW - 1024 - kBarBytesW - p.term_bytes) / kABytes);
  if (tid == 0) {
    for (int s = 0; s < kMostStagesW; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int e = 0; e < 2; ++e) {
      mbar_init(&tfull[e], 1);
      mbar_init(&tempty[e], 128);
    }
    mbar_init(terms, 1);
    mbar_init(read, 1);
    s_fail = s_issued = s_terms = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(tmem_slot)), "r"(kTmemColsW) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  // This CTA's tiles, group by group, in passes over the tokens whose terms fit; every role goes through
  // the same list.  `tile` is called with (group, tile of the group, first 16-token block, last), `open`
  // and `close` around each pass; they return false to give up.
  const int t0 = (int)((long long)n_tiles * blockIdx.x / gridDim.x), t1 = (int)((long long)n_tiles * (blockIdx.x + 1) / gridDim.x);
  auto walk = [&](auto&& open, auto&& tile, auto&& close) {
    const int* first = p.first + kWideResid * (p.n + 1);
    int gi = 0;
    for (int b = p.n; b - gi > 1;) {   // the last group that begins at or before tile t0
      const int m = (gi + b) / 2;
      if (first[m] <= t0) gi = m;
      else b = m;
    }
    for (; gi < p.n && first[gi] < t1; ++gi) {
      const int a = max(0, t0 - first[gi]), b = min(t1, first[gi + 1]) - first[gi];
      if (a >= b) continue;
      const WideGroup& w = p.table[gi];
      const int per = max(1, p.term_bytes / (48 * w.g.k * 2));   // 16-token blocks of a pass
      for (int q0 = 0; q0 < nq; q0 += per) {
        const int q1 = min(nq, q0 + per);
        if (!open(w, q0, q1)) return;
        for (int t = a; t < b; ++t)
          if (!tile(w, t, q0, q1)) return;
        if (!close()) return;
      }
    }
  };
  auto nothing = [] { return true; };

  if (warp == 0) {
    if (lane == 0) {   // weight tiles
      int n = 0;
      const WideGroup* last = nullptr;
      walk([](const WideGroup&, int, int) { return true; },
           [&](const WideGroup& w, int t, int, int) {
             if (&w != last) {
               acquire_map(&w.tm.p);
               acquire_map(&w.tm.wp);
               last = &w;
             }
             const int dt = w.g.d / kTM;
             const CUtensorMap* map = t < dt ? &w.tm.p : &w.tm.wp;
             const int row = (t < dt ? t : t - dt) * kTM;
             for (int kb = 0; kb < w.g.k / kTK; ++kb, ++n) {
               const int s = n % stages;
               if (n >= stages && !mbar_wait(&empty[s], ((n / stages) - 1) & 1)) {
                 s_fail = 1;
                 return false;
               }
               mbar_expect_tx(&full[s], (uint32_t)kABytes);
               tma_load_2d(s32(s_ring + s * kABytes), map, kb * kTK, row, &full[s]);
               s_issued = n + 1;
             }
             return true;
           },
           nothing);
    }
    __syncwarp();
    pdl_wait();
  } else if (warp == 1) {
    pdl_wait();
    int n = 0, n_tile = 0, n_pass = 0;
    bool ok = true;   // (the same for the whole warp)
    walk(
        [&](const WideGroup& w, int q0, int q1) {   // the terms of c of the pass, a lane per box
          const int N = min(48 * (q1 - q0), rows_all - 48 * q0), boxes = N / kBBox, all = w.g.k / kTK * boxes;
          acquire_map(&w.tm.cb);
          if (n_pass > 0) ok = __all_sync(0xffffffffu, mbar_wait(read, (n_pass - 1) & 1));   // those before are read
          if (!ok) return false;
          if (lane == 0) mbar_expect_tx(terms, (uint32_t)(all * kBBox * kTK * 2));
          if (lane == 0) s_terms = n_pass + 1;
          __syncwarp();
          for (int i = lane; i < all; i += 32) {
            const int kb = i / boxes, r = i - kb * boxes;
            tma_load_2d(s32(s_terms_at) + (kb * N + r * kBBox) * (kTK * 2), &w.tm.cb, kb * kTK, 48 * q0 + r * kBBox, terms);
          }
          ok = __all_sync(0xffffffffu, mbar_wait(terms, n_pass & 1));
          ++n_pass;
          return ok;
        },
        [&](const WideGroup& w, int, int q0, int q1) {
          const int N = min(48 * (q1 - q0), rows_all - 48 * q0), e = n_tile & 1;
          if (lane == 0) {
            const uint32_t idesc = instr_desc(kTM, N);
            if (n_tile >= 2) ok = mbar_wait(&tempty[e], ((n_tile >> 1) - 1) & 1, kSpin * 8);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int kb = 0; ok && kb < w.g.k / kTK; ++kb) {
              const int s = (n + kb) % stages;
              ok = mbar_wait(&full[s], ((n + kb) / stages) & 1);
              if (!ok) break;
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              const uint32_t a0 = s32(s_ring + s * kABytes), b0 = s32(s_terms_at) + kb * N * (kTK * 2);
#pragma unroll
              for (int k = 0; k < kTK / 16; ++k)
                umma_bf16(tmem + e * 256, smem_desc_sw128(a0 + k * 32), smem_desc_sw128(b0 + k * 32), idesc, (kb > 0 || k > 0) ? 1u : 0u);
              umma_commit(&empty[s]);
            }
            if (ok) umma_commit(&tfull[e]);
          }
          ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
          n += w.g.k / kTK;
          ++n_tile;
          return ok;
        },
        [&] {
          if (lane == 0) umma_commit(read);
          __syncwarp();
          return true;
        });
    // (no arrival is on its way to the barrier when the block leaves)
    if (ok && n_pass > 0) ok = __all_sync(0xffffffffu, mbar_wait(read, (n_pass - 1) & 1));
    if (!ok && lane == 0) s_fail = 1;
  } else {
    pdl_wait();
    const int e = (warp - 2) >> 2, quarter = warp & 3, tid4 = quarter * 32 + lane;
    const uint32_t tl = tmem + e * 256 + ((uint32_t)(quarter * 32) << 16);
    auto sync = [&] { asm volatile("bar.sync %0, 128;" ::"r"(1 + e) : "memory"); };
    int n_tile = 0;
    bool ok = true;   // after a wait that ran out: NaN, and every arrival that others count on
    walk([](const WideGroup&, int, int) { return true; },
         [&](const WideGroup& w, int tile, int q0, int q1) {
           if ((n_tile & 1) != e) {
             ++n_tile;
             return true;
           }
           const GroupParams& g = w.g;
           // (in registers: the table lies in memory that the stores below could reach, for all the compiler knows)
           const int d = g.d, O = g.O, dt = d / kTM;
           uint16_t* rb = g.rb;
           const bool image = tile >= dt;
           const int row = (image ? tile - dt : tile) * kTM + quarter * 32 + lane;
           const IoRef io = p.io_of(w);
           const int slot = io_slot(io);
           float* y = io.y;
           const float* x = io.x + (long long)slot * io.x_step_stride + row;
           float xv[16];
           if (!image)
#pragma unroll
             for (int tt = 0; tt < 16; ++tt)
               xv[tt] = 16 * q0 + tt < n_tokens ? __ldg(x + (size_t)(16 * q0 + tt) * d) : 0.f;
           if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&tfull[e], (n_tile >> 1) & 1, kSpin * 8));
           if (!ok && lane == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
           asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
           for (int q = q0; q < q1; ++q) {
             float s[16];
             if (ok) {
               sum3_tokens16(tl, q - q0, s);
             } else {
#pragma unroll
               for (int tt = 0; tt < 16; ++tt) s[tt] = __int_as_float(0x7fc00000);
             }
             if (q + 1 == q1) {   // the accumulator is read
               asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
               mbar_arrive(&tempty[e]);
             }
             if (image) {
#pragma unroll
               for (int tt = 0; tt < 16; ++tt)
                 if (16 * q + tt < n_tokens) y[(size_t)(16 * q + tt) * O + row] = s[tt];
               continue;
             }
             float xn[16], sq[32];
#pragma unroll
             for (int tt = 0; tt < 16; ++tt)
               xn[tt] = (q + 1 < q1 && 16 * (q + 1) + tt < n_tokens) ? __ldg(x + (size_t)(16 * (q + 1) + tt) * d) : 0.f;
#pragma unroll
             for (int tt = 0; tt < 16; ++tt) {
               const int t = 16 * q + tt;
               const float rv = xv[tt] - s[tt];
               if (t < n_tokens) rb[(size_t)t * d + row] = bf16_bits(rv);
               sq[tt] = rv * rv;
               sq[16 + tt] = xv[tt] * xv[tt];
               xv[tt] = xn[tt];
             }
             const float sum = sum32_over_lanes(sq);
             const int t = 16 * q + (lane & 15);
             if (t < n_tokens) s_norm[e][quarter][t][lane >> 4] = sum;
           }
           ++n_tile;
           if (image) return true;
           sync();
           for (int i = tid4; i < 32 * (q1 - q0); i += 128) {
             const int t = 16 * q0 + (i >> 1), h = i & 1;
             if (t < n_tokens) {
               float sum = 0.f;
#pragma unroll
               for (int c = 0; c < 4; ++c) sum += s_norm[e][c][t][h];
               g.normpart3[((size_t)tile * g.B + t) * 2 + h] = sum;
             }
           }
           const int per = max(1, p.term_bytes / (48 * g.k * 2)), passes = (nq + per - 1) / per;
           decide_gate_last(g, io, slot, n_tokens, g.normpart3, dt, (unsigned)(dt * passes), &s_last[e], s_gate[e], tid4, 128, sync);
           sync();   // (s_last and s_norm are read)
           return true;
         },
         nothing);
    if (!ok) s_fail = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (s_fail && tid == 0) {   // copies that were asked for: a bounded time to land before the block exits
    for (int i = max(0, s_issued - stages); i < s_issued; ++i) (void)mbar_wait(&full[i % stages], (i / stages) & 1, 1u << 16);
    if (s_terms > 0) (void)mbar_wait(terms, (s_terms - 1) & 1, 1u << 16);
  }
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemColsW) : "memory");
}

// PT[j][i] = P[i][j], 32 x 32 tiles through shared memory.
__global__ void __launch_bounds__(256) k_transpose_bf16(const uint16_t* __restrict__ P, int d, int k,
                                                        uint16_t* __restrict__ PT) {
  __shared__ uint16_t tile[32][33];
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int r = ty; r < 32; r += 8)
    if (i0 + r < d && j0 + tx < k) tile[r][tx] = P[(size_t)(i0 + r) * k + j0 + tx];
  __syncthreads();
  for (int r = ty; r < 32; r += 8)
    if (j0 + r < k && i0 + tx < d) PT[(size_t)(j0 + r) * d + i0 + tx] = tile[tx][r];
}

}  // namespace

int front_rows(int max_tokens) { return (3 * max_tokens + 15) & ~15; }

int front_proj_splits(int d, int k) {
  const int tiles = k / kTM, nkb = d / kTK;
  int s = 148 / tiles;
  if (s > nkb / 2) s = nkb / 2;
  if (s > 32) s = 32;   // more partials cost the reduction more than they save the projection (measured)
  if (s < 1) s = 1;
  return s;
}

cudaError_t launch_transpose_bf16(const void* P, int d, int k, void* PT, cudaStream_t st) {
  k_transpose_bf16<<<dim3((k + 31) / 32, (d + 31) / 32), 256, 0, st>>>(
      static_cast<const uint16_t*>(P), d, k, static_cast<uint16_t*>(PT));
  return cudaGetLastError();
}

cudaError_t launch_split3_x(const GroupParams& g, const IoRef& io, int n_tokens, cudaStream_t st) {
  const int slots = (front_rows(n_tokens) + 2) / 3;
  k_split3_x<<<dim3((g.d / 8 + 255) / 256, slots), 256, 0, st>>>(g, io, n_tokens);
  return cudaGetLastError();
}

template <bool kInStack>
static cudaError_t launch_front(const GroupParams& g, const TmaMaps& tm, const IoRef& io, int n_tokens,
                                cudaStream_t st) {
  constexpr int kSmem3 = Cfg<kInStack ? kStages3 : kStages3Alone, kMaxN3>::kSmem;
  auto proj = k_proj_tc<kInStack>;
  auto wide = k_resid_image_tc<kStagesRI, kMaxN3, kTmemCols3, kInStack>;
  auto narrow = k_resid_image_tc<kStagesRIs, kMaxN3s, kTmemCols3s, kInStack>;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(proj, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem3)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(wide, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemRI)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(narrow, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemRIs)) != cudaSuccess)
    return e;
  const bool small = term_rows(n_tokens) <= kMaxN3s;
  const int slots = (front_rows(n_tokens) + 2) / 3;   // token slots covering every operand row
  const int nq = (n_tokens + 15) / 16, tiles = g.d / kTM;
  int rs = tiles <= 37 ? 4 : tiles <= 148 ? 2 : 1;   // token ranges per residual tile (measured: 4 for all is slower)
  if (rs > nq) rs = nq;
  // the x the residual blocks read before their wait is an input of the call, complete before
  // k_split3_x was launched
  if ((e = launch_pdl(k_split3_x, dim3((g.d / 8 + 255) / 256, slots), dim3(256), 0, st, g, io, n_tokens)) !=
          cudaSuccess ||
      (e = launch_pdl(proj, dim3((g.k / kTM) * g.proj_splits), dim3(kThreads), kSmem3, st, g, tm, n_tokens)) !=
          cudaSuccess ||
      (e = launch_pdl(k_reduce_split3_c, dim3(slots), dim3(256), 0, st, g, n_tokens)) != cudaSuccess ||
      (e = launch_pdl(small ? narrow : wide, dim3((g.d / kTM) * rs + g.O / kTM), dim3(kThreads),
                      small ? kSmemRIs : kSmemRI, st, g, tm, io, n_tokens, rs)) != cudaSuccess)
    return e;
  return cudaGetLastError();
}

cudaError_t launch_front_tc(const GroupParams& g, const TmaMaps& tm, const IoRef& io, int n_tokens, bool in_stack,
                            cudaStream_t st, int* n_launches) {
  if (n_launches) *n_launches += 4;
  return in_stack ? launch_front<true>(g, tm, io, n_tokens, st) : launch_front<false>(g, tm, io, n_tokens, st);
}

int wide_split_blocks(int d, int n_tokens) { return (d / 8 + 255) / 256 * ((front_rows(n_tokens) + 2) / 3); }

int wide_term_bytes(int most_k, int n_tokens) {
  const int nq = (n_tokens + 15) / 16, one = 48 * most_k * 2;
  int q = kTermBytesW / one;
  q = q < 1 ? 1 : q > nq ? nq : q;
  return (q * one + 1023) / 1024 * 1024;
}

cudaError_t launch_front_wide(const WideParams& p, const int* blocks, int n_tokens, int grid, cudaStream_t st) {
  constexpr int kSmem3 = Cfg<kStages3, kMaxN3>::kSmem;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_proj_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem3)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(k_resid_image_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemW)) != cudaSuccess)
    return e;
  const int slots = (front_rows(n_tokens) + 2) / 3, tiles = blocks[kWideResid];
  if ((e = launch_pdl(k_split3_x_wide, dim3(blocks[kWideSplit]), dim3(256), 0, st, p, n_tokens, slots)) != cudaSuccess ||
      (e = launch_pdl(k_proj_wide, dim3(blocks[kWideProj]), dim3(kThreads), kSmem3, st, p, n_tokens)) != cudaSuccess ||
      (e = launch_pdl(k_reduce_wide, dim3(p.n * slots), dim3(256), 0, st, p, n_tokens, slots)) != cudaSuccess ||
      (e = launch_pdl(k_resid_image_wide, dim3(tiles < grid ? tiles : grid), dim3(kThreadsW), kSmemW, st, p, tiles, n_tokens)) !=
          cudaSuccess)
    return e;
  return cudaGetLastError();
}

}  // namespace gsi
