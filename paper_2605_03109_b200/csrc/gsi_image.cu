// Cached image W_P = bf16(W P) of Eq. (3.2) / Section 4.2 on the 5th-gen tensor cores, any
// o, d, k that are multiples of 8.
//
//   D[128 rows of W][kN columns of P] = W tile . P tile, fp32 in tensor memory
//
//   A   W  [o][d], K-major: boxes of 128 rows x 64 elements, 128-byte swizzle (TMA)
//   B   P  [d][k]: the contraction runs over its ROWS, so the tile is an MN-major operand: boxes
//       of 64 rows x 64 columns, 128-byte swizzle, one per 64 columns (TMA) - no transposed
//       copy of the basis and no workspace.  An fp32 basis enters as three bf16 terms
//       (hi + mid + lo = the fp32 value), split by four warps into the same layout; all products
//       are exact then, and the three terms share one accumulator.
//
// What bounds it: a CTA of a 128 x 256 tile takes 48 KB per 64 of the depth through the L2 (at
// GPT-J's fc, 16384 x 4096 and k = 256, 393 MB in all at 10 TB/s; W alone from HBM is 134 MB,
// 21 us, the tensor cores need 17 us).  Measured there: 43 us, 0.8 PFLOP/s; the CUDA-core kernel
// before took 1935 us (18 TFLOP/s).
//
// The tensor core's own accumulation truncates: over the 1024 instructions of d = 16384 that
// costs five times the error of an fp32 FMA chain (bf16 entries that fall on the other side of a
// rounding boundary: 4e-3 of all against 5e-4).  So a chunk of 512 of the depth is accumulated
// in tensor memory, two accumulators in turn, and eight warps add the chunks up in fp32
// registers: as exact as the FMA chain, beside the next chunk's instructions.
//
// One CTA per tile and share of the depth.  Narrow maps leave SMs idle, so a cluster of S CTAs may
// split the depth: the partial tiles meet in distributed shared memory and are added in rank
// order (reproducible).  Ragged edges are the tensor maps' zero fill plus guarded stores.
// Every wait is bounded; a tile whose wait ran out is written as NaN, never as a wrong number, and the
// status word, where the caller has one, says so.
#include "gsi_umma.cuh"

namespace gsi {

namespace {

using namespace umma;

constexpr int kAccFirst = 4, kAccWarps = 8;   // warp 0: TMA, warp 1: MMA, warps 4..11: sums and stores
constexpr int kConvFirst = kAccFirst + kAccWarps;   // fp32 basis: warps 12..15 split it
constexpr int kConv = 128;
constexpr int kChunkBlocks = 8;   // blocks of the depth one accumulator takes

struct ImageMaps {
  CUtensorMap w, p;
};

template <int kN, bool kF32>
struct ICfg {
  static constexpr int kBBytes = kN * kTK * 2;
  static constexpr int kTerms = kF32 ? 3 : 1;
  static constexpr int kStageBytes = kABytes + kTerms * kBBytes;
  static constexpr int kStages = 196608 / kStageBytes > 8 ? 8 : 196608 / kStageBytes;
  static constexpr int kRing = kStages * kStageBytes;
  static constexpr int kSmem = 1024 + kRing + 256;
  static constexpr int kTmem = 2 * kN;   // two accumulators
  static constexpr int kThreads = 32 * kConvFirst + (kF32 ? kConv : 0);
  static_assert(kN * kTM * 4 <= kRing, "the partial tile of a split lies in the ring");
};

// MN-major operand in the 128-byte swizzle: 64 elements (128 bytes) per row of the depth, eight
// depth rows 1024 bytes apart, the next 64 elements one box (64 depth rows) on.
__device__ __forceinline__ uint64_t smem_desc_mn_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((kTK * 128) >> 4) << 16;   // leading offset: from 64 elements to the next 64
  d |= (uint64_t)(1024 >> 4) << 32;          // stride offset: from eight depth rows to the next
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// Two fp32 values -> their hi, mid and lo bf16 terms, packed in pairs.
__device__ __forceinline__ void split3_pair(float a, float b, uint32_t (&t)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    t[i] = pack_bf16(a, b);
    a -= __uint_as_float(t[i] << 16);
    b -= __uint_as_float(t[i] & 0xFFFF0000u);
  }
}

template <int kN, bool kF32>
__global__ void __launch_bounds__(ICfg<kN, kF32>::kThreads, 1)
k_image_tc(const __grid_constant__ ImageMaps tm, const float* __restrict__ Pf, int o, int d, int k, int splits,
           uint16_t* __restrict__ WP, int* status) {
  using C = ICfg<kN, kF32>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bar_full = reinterpret_cast<uint64_t*>(smem + C::kRing);
  uint64_t* bar_empty = bar_full + C::kStages;
  uint64_t* acc_full = bar_empty + C::kStages;   // [2]
  uint64_t* acc_empty = acc_full + 2;            // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  int* s_fail = reinterpret_cast<int*>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int split = blockIdx.x % splits;                 // rank in the cluster
  const int row0 = (int)(blockIdx.x / splits) * kTM, col0 = blockIdx.y * kN;
  const int nkb = (d + kTK - 1) / kTK;
  const int kb0 = (int)((long long)nkb * split / splits), kb1 = (int)((long long)nkb * (split + 1) / splits);
  const int nloc = kb1 - kb0;

  if (tid == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&bar_full[s], kF32 ? 1 + kConv : 1);
      mbar_init(&bar_empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kAccWarps);
    }
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(tmem_slot)),
                 "r"(C::kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {   // producer
      for (int i = 0; i < nloc; ++i) {
        const int stage = i % C::kStages;
        if (i >= C::kStages && !mbar_wait(&bar_empty[stage], ((i / C::kStages) - 1) & 1)) {
          *s_fail = 1;
          break;
        }
        const uint32_t sa = s32(smem + stage * C::kStageBytes);
        const int x = (kb0 + i) * kTK;
        mbar_expect_tx(&bar_full[stage], (uint32_t)(kF32 ? kABytes : C::kStageBytes));
        tma_load_2d(sa, &tm.w, x, row0, &bar_full[stage]);
        if constexpr (!kF32) {
          // (boxes that lie past column k arrive as zeros and count in full)
#pragma unroll
          for (int j = 0; j < kN / 64; ++j)
            tma_load_2d(sa + kABytes + j * (kTK * 128), &tm.p, col0 + 64 * j, x, &bar_full[stage]);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {   // MMA issuer
      const uint32_t idesc = instr_desc(kTM, kN) | (1u << 16);   // B is MN-major
      bool ok = true;
      for (int i = 0; i < nloc && ok; ++i) {
        const int stage = i % C::kStages, chunk = i / kChunkBlocks, buf = chunk & 1;
        const bool first = i % kChunkBlocks == 0;
        ok = (!first || chunk < 2 || mbar_wait(&acc_empty[buf], ((chunk >> 1) - 1) & 1)) &&
             mbar_wait(&bar_full[stage], (i / C::kStages) & 1);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a0 = s32(smem + stage * C::kStageBytes), b0 = a0 + kABytes;
#pragma unroll
        for (int t = 0; t < C::kTerms; ++t)
#pragma unroll
          for (int q = 0; q < kTK / 16; ++q)   // sixteen depth rows of B are 2048 bytes
            umma_bf16(tmem + buf * kN, smem_desc_sw128(a0 + q * 32),
                      smem_desc_mn_sw128(b0 + t * C::kBBytes + q * 2048), idesc,
                      (!first || q > 0 || t > 0) ? 1u : 0u);
        umma_commit(&bar_empty[stage]);
        if (i + 1 == nloc || (i + 1) % kChunkBlocks == 0) umma_commit(&acc_full[buf]);
      }
      if (!ok) *s_fail = 1;
    }
    __syncwarp();
  } else if (kF32 && warp >= kConvFirst) {
    // fp32 basis: chunk c of a block = eight columns of one depth row; the next block's values are
    // requested before this block's are split
    constexpr int kPer = kTK * kN / 8 / kConv;
    const int ct = tid - 32 * kConvFirst;
    float4 v[2][kPer][2];
    auto request = [&](int i, float4 (&r)[kPer][2]) {
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int c = ct + u * kConv, row = (kb0 + i) * kTK + c / (kN / 8), col = col0 + (c % (kN / 8)) * 8;
        r[u][0] = r[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < d && col < k) {   // (k is a multiple of 8)
          const float4* src = reinterpret_cast<const float4*>(Pf + (size_t)row * k + col);
          r[u][0] = __ldg(src);
          r[u][1] = __ldg(src + 1);
        }
      }
    };
    auto store = [&](int i, const float4 (&r)[kPer][2]) -> bool {
      const int stage = i % C::kStages;
      if (i >= C::kStages && !mbar_wait(&bar_empty[stage], ((i / C::kStages) - 1) & 1)) return false;
      unsigned char* sb = smem + stage * C::kStageBytes + kABytes;
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int c = ct + u * kConv, row = c / (kN / 8), c8 = c % (kN / 8);
        uint32_t t[4][3];
        split3_pair(r[u][0].x, r[u][0].y, t[0]);
        split3_pair(r[u][0].z, r[u][0].w, t[1]);
        split3_pair(r[u][1].x, r[u][1].y, t[2]);
        split3_pair(r[u][1].z, r[u][1].w, t[3]);
        const int at = (c8 >> 3) * (kTK * 128) + row * 128 + (((c8 & 7) ^ (row & 7)) << 4);
#pragma unroll
        for (int q = 0; q < 3; ++q)
          *reinterpret_cast<uint4*>(sb + q * C::kBBytes + at) = make_uint4(t[0][q], t[1][q], t[2][q], t[3][q]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(&bar_full[stage]);
      return true;
    };
    bool ok = true;
    if (nloc > 0) request(0, v[0]);
#pragma unroll 2
    for (int i = 0; i < nloc && ok; ++i) {
      if (i + 1 < nloc) request(i + 1, v[(i + 1) & 1]);
      ok = store(i, v[i & 1]);
    }
    if (!ok) *s_fail = 1;
  }

  // lane of tensor memory = row of the tile; warps 4..7 own the first half of the columns, 8..11 the second
  const bool acc_warp = warp >= kAccFirst && warp < kConvFirst;
  const int r = 32 * (warp & 3) + lane, row = row0 + r;
  constexpr int kHalf = kN / 2;
  const int ch = ((warp - kAccFirst) >> 2) * kHalf;
  float sum[kHalf];
  bool mine = true;
  if (acc_warp) {
#pragma unroll
    for (int e = 0; e < kHalf; ++e) sum[e] = 0.f;
    const int chunks = (nloc + kChunkBlocks - 1) / kChunkBlocks;
    for (int c = 0; c < chunks && mine; ++c) {
      const int buf = c & 1;
      mine = __all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (c >> 1) & 1, kSpin * 8));
      if (!mine) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + buf * kN + ch;
#pragma unroll
      for (int c0 = 0; c0 < kHalf; c0 += 16) {
        uint32_t u[16];
        tmem_ld16(tl + c0, u);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) sum[c0 + e] += __uint_as_float(u[e]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
  }
  if (*reinterpret_cast<volatile int*>(s_fail)) mine = false;
  const bool done = __syncthreads_and(mine ? 1 : 0) != 0;
  if (!done && tid == 0) {   // copies issued but not consumed: a bounded time to land
    if (status) atomicExch(status, (int)GSI_ERR_TIMEOUT);
    for (int s = 0; s < C::kStages && s < nloc; ++s) {
      const int last = ((nloc - 1 - s) / C::kStages) * C::kStages + s;
      (void)mbar_wait(&bar_full[s], (last / C::kStages) & 1, 1u << 16);
    }
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  if (!done) {
#pragma unroll
    for (int e = 0; e < kHalf; ++e) sum[e] = __int_as_float(0x7fc00000);
  }
  if (splits == 1) {
    if (acc_warp && row < o) {
#pragma unroll
      for (int c0 = 0; c0 < kHalf; c0 += 8)
        if (col0 + ch + c0 < k)
          *reinterpret_cast<uint4*>(WP + (size_t)row * k + col0 + ch + c0) =
              make_uint4(pack_bf16(sum[c0], sum[c0 + 1]), pack_bf16(sum[c0 + 2], sum[c0 + 3]),
                         pack_bf16(sum[c0 + 4], sum[c0 + 5]), pack_bf16(sum[c0 + 6], sum[c0 + 7]));
    }
  } else {
    // the partial tile, column by column of 128 rows, into the ring (its last stage is consumed);
    // then every rank adds its share of the columns over the ranks, in rank order
    float* part = reinterpret_cast<float*>(smem);
    if (acc_warp) {
#pragma unroll
      for (int e = 0; e < kHalf; ++e) part[(ch + e) * kTM + r] = sum[e];
    }
    cluster_sync();
    const int per = kN / 8 / splits * 8;   // columns of a rank: kN >= 64, splits <= 8
    const int rr = tid & 127, rowr = row0 + rr;
    for (int c0 = split * per + 8 * (warp >> 2); c0 < (split + 1) * per && col0 + c0 < k; c0 += C::kThreads / 16) {
      float s[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) s[e] = 0.f;
      for (int q = 0; q < splits; ++q)
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] += ld_cluster(s32(part + (c0 + e) * kTM + rr), q);
      if (rowr < o)
        *reinterpret_cast<uint4*>(WP + (size_t)rowr * k + col0 + c0) =
            make_uint4(pack_bf16(s[0], s[1]), pack_bf16(s[2], s[3]), pack_bf16(s[4], s[5]), pack_bf16(s[6], s[7]));
    }
    cluster_sync();   // nobody leaves while its partial tile is being read
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmem) : "memory");
}

template <int kN, bool kF32>
cudaError_t launch_n(const ImageMaps& tm, const void* P, int o, int d, int k, int splits, void* WP, int* status,
                     cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_image_tc<kN, kF32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       ICfg<kN, kF32>::kSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(((o + kTM - 1) / kTM) * splits, (k + kN - 1) / kN);
  cfg.blockDim = dim3(ICfg<kN, kF32>::kThreads);
  cfg.dynamicSmemBytes = ICfg<kN, kF32>::kSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = splits;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_image_tc<kN, kF32>, tm, static_cast<const float*>(kF32 ? P : nullptr), o, d, k,
                            splits, static_cast<uint16_t*>(WP), status);
}

}  // namespace

cudaError_t launch_build_image(const void* W, const void* P, int o, int d, int k, bool p_f32, void* WP,
                               int* status, cudaStream_t st) {
  ImageMaps tm;
  if (!encode_bf16_map(&tm.w, W, o, d, kTM)) return cudaErrorNotSupported;
  if (!p_f32 && !encode_bf16_map(&tm.p, P, d, k, kTK)) return cudaErrorNotSupported;
  // Tile width and depth split with the shortest critical path: waves of CTAs x (blocks of a
  // share of the depth x the bytes a block brings through an SM's L2 port, about 110 bytes per
  // nanosecond, plus 3 us of start and end; a split adds its exchange).
  const int mt = (o + kTM - 1) / kTM, nkb = (d + kTK - 1) / kTK;
  int best_n = 64, best_s = 1;
  double best = 1e30;
  for (int n = 64; n <= (p_f32 ? 64 : 256); n *= 2) {
    if (n > 64 && n / 2 >= k) break;   // a narrower tile covers every column
    for (int s = 1; s <= 8 && (s == 1 || 4 * s <= nkb); s *= 2) {
      const long long ctas = (long long)mt * ((k + n - 1) / n) * s;
      const double waves = (double)((ctas + 147) / 148), blocks = (nkb + s - 1) / s;
      const double per = (kABytes + (p_f32 ? 4.0 : 2.0) * n * kTK) / 110.0;
      const double t = waves * (blocks * per + 3000.0 + (s > 1 ? 1500.0 + 4.0 * n : 0.0));
      if (t < best) {
        best = t;
        best_n = n;
        best_s = s;
      }
    }
  }
  if (p_f32) return launch_n<64, true>(tm, P, o, d, k, best_s, WP, status, st);
  switch (best_n) {
    case 64: return launch_n<64, false>(tm, P, o, d, k, best_s, WP, status, st);
    case 128: return launch_n<128, false>(tm, P, o, d, k, best_s, WP, status, st);
    default: return launch_n<256, false>(tm, P, o, d, k, best_s, WP, status, st);
  }
}

}  // namespace gsi
