// One call whose basis fits the shared memory of sixteen SMs as ONE launch of independent clusters.
//
// A cluster of sixteen CTAs keeps the whole basis in shared memory (a slab of rows per CTA) and runs
// Algorithm 1 lines 1-4 for itself: the partial c, ||r||^2 and ||x||^2 meet by st.async in
// distributed shared memory.  Every cluster does the same sums in the same order, so all take the
// same decision without a word between them; the rows of the images and of W are dealt over the
// clusters, and within one in units of 16 rows over its CTAs.
//
//   A   partial c of this CTA's rows of P, from shared memory                (line 1)
//   x1  the sixteen partials of a coefficient are added in rank order: by every CTA for itself
//       where they are few, else each by one CTA, which passes the sum on
//   B   r of the same rows, then y = W_P c of its image rows                 (lines 2, 5)
//   x2  the norms of all ranks, the gate                                     (lines 3-4, Eq. (3.3))
//   C   gated tokens: every CTA contracts its own rows of r, which never leave it, with its columns of
//       all W rows of the cluster; the owner of a row adds the sixteen partials to y (Eq. (3.2))
//
// What bounds it: a chain of latencies.  An exchange through the L2 between the CTAs of a
// cooperative grid costs 2 us (gsi_fused.cu), one between the CTAs of a cluster 0.4, and nothing is
// kept between calls but the count of the launches (for the report of a CTA that gave up).  The price is that every
// cluster reads the basis (from the L2, but for one), and seven clusters of sixteen leave 36 of 148
// SMs idle; W r makes up for that with 128 KB in flight per SM (5.5 TB/s where the cooperative launch,
// by loads into registers, reaches 4.7).  Kernel times in a captured graph, cooperative launch -> this: one
// token at 768 x 64 -> 3072 10.3 -> 5.3 us, 4096 x 256 -> 28672 13.5 -> 13.1 (gated 64 -> 57); 16 tokens, fp32
// basis, 768 x 128 -> 2304 19 -> 10.3.
//
// Every wait is bounded; a CTA whose wait ran out goes no further, sets GSI_ERR_TIMEOUT, leaves NaN, and
// stays until its peers are gone.
#include <cuda.h>

#include "gsi_mma.cuh"
#include "gsi_exchange.cuh"

namespace gsi {

namespace {

using namespace mma16;

constexpr int kC = 16;                  // CTAs of a cluster
constexpr int kT = 512, kW = kT / 32;
constexpr int kSmemCluster = 225 * 1024;
// Coefficients up to which every CTA adds all partials itself: one exchange, but sixteen times the words
// (one token, in a graph: k = 64 5.2 us either way, k = 256 13.8 us, as two exchanges 13.1).
constexpr int kDirectValues = 128;
constexpr int kMostColumns = 512;
constexpr int kMostPlane = 24576;       // bytes of a term of an fp32 basis per CTA
constexpr int kMaxBatches = 4096;       // of W r: more than any call makes (bounds the stay of a CTA that gave up)

// The ring of W: slots of 16 rows x 64 elements per warp.  A lane copies what it reads itself (16 bytes
// of rows g and g + 8 per step), so a slot needs no barrier, only the lane's own cp.async groups.
constexpr int kSlotBytes = 2048, kDeepSlots = 5, kShallowSlots = 3;
__host__ __device__ constexpr int ring_bytes(int slots) { return kW * slots * kSlotBytes; }

// Sizes and places in dynamic shared memory, worked out on the host.
struct ClusterPlan {
  int pitch, plane, xp;           // bytes of a basis row and of a term of the slab; floats between tokens of x
  int nbs;                        // eight-token blocks of a pass
  int steps;                      // 32-row steps of the fullest CTA
  int mt, ks_log2;                // 16-column tiles of c; log2 of the warps that share the rows of a tile
  int direct;
  unsigned kq_magic;              // ceil(2^32 / (k / 4)): token of a float4 of coefficients
  int lpr_log2;                   // lanes that load a basis row
  int unit_base, unit_rem;        // 16-row units of the images per cluster, and clusters with one more
  int xt, wsum, recv, recv2, front_bytes, op, xs, norm, unit, total;
};

template <int NB, bool PF32>
bool make_plan(int d, int k, int n, ClusterPlan* p) {
  const int kTok = 8 * NB, tok = n < kTok ? n : kTok, nbs = (tok + 7) / 8;
  const int U = (d + 15) / 16, units = (U + kC - 1) / kC, R = 16 * units;
  p->pitch = ((k / 8) | 1) * 16;        // an odd number of 16-byte pieces: ldmatrix without conflicts
  p->plane = R * p->pitch;
  p->xp = R % 32 ? R + 24 : R + 8;      // 8 modulo 32 floats: eight tokens x four row pairs without conflicts
  p->steps = (R + 31) / 32;
  p->mt = (k + 15) / 16;
  p->ks_log2 = 0;
  while ((2 << p->ks_log2) * p->mt <= kW) ++p->ks_log2;
  p->direct = n <= kTok && n * k <= kDirectValues;
  p->kq_magic = (unsigned)(((1ull << 32) + k / 4 - 1) / (k / 4));
  p->lpr_log2 = 0;
  while ((1 << p->lpr_log2) < k / 8 && p->lpr_log2 < 5) ++p->lpr_log2;
  long long at = 0;
  auto take = [&](long long bytes) {
    const int o = (int)at;
    at = (at + bytes + 127) / 128 * 128;
    return o;
  };
  if (n * (long long)p->xp * 4 > kSmemCluster) return false;
  if (PF32 && p->plane > kMostPlane) return false;
  take((long long)p->plane * (PF32 ? 3 : 1) + 64);
  p->nbs = nbs;
  p->xt = take((long long)units * nbs * 3 * 256);
  p->wsum = take((long long)(1 << p->ks_log2) * nbs * 8 * p->mt * 64);
  const int V = tok * k / 4, per = (V + kC - 1) / kC;
  p->recv = take((long long)kC * (p->direct ? V : per) * 16);
  p->recv2 = take(p->direct ? 0 : (long long)V * 16);
  // W r takes this first part over: r as operand, the ring, two buffers of partials
  const int least = 8 * op_stride(p->steps) + ring_bytes(kShallowSlots) + 2 * 8 * 1024;
  if (at < least) at = (least + 127) / 128 * 128;
  p->front_bytes = (int)at;
  p->op = take((long long)tok * op_stride((k + 31) / 32));
  p->xs = take((long long)n * p->xp * 4);
  p->norm = take((long long)kC * n * 8);
  p->unit = take((long long)units * nbs * 64);
  if (at > kSmemCluster) return false;
  const int spare = (int)((kSmemCluster - at) / 128 * 128);   // goes to the first part
  p->front_bytes += spare;
  p->op += spare;
  p->xs += spare;
  p->norm += spare;
  p->unit += spare;
  p->total = (int)at + spare;
  return true;
}

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t peer(uint32_t local, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  return a;
}
// Into a peer's shared memory; the bytes count towards the peer's barrier.
__device__ __forceinline__ void send16(uint32_t to, uint32_t bar, const float4& v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(to),
               "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
               "r"(__float_as_uint(v.w)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void send8(uint32_t to, uint32_t bar, float a, float b) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(to),
               "r"(__float_as_uint(a)), "r"(__float_as_uint(b)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s32(bar)), "r"(bytes) : "memory");
}
// The first look does not wait at all, the others up to a microsecond each.
__device__ __forceinline__ bool arrived(uint64_t* bar, uint32_t parity, unsigned limit) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(s32(bar)), "r"(parity)
      : "memory");
#pragma unroll 1
  for (unsigned it = 1; !ok && it < limit; ++it)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(s32(bar)), "r"(parity), "r"(1000u)
        : "memory");
  return ok != 0;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint4 ld_shared16(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void add4(float4& s, const float4& v) {
  s.x += v.x;
  s.y += v.y;
  s.z += v.z;
  s.w += v.w;
}
// Sixteen partials, `pitch` apart, in rank order.
__device__ __forceinline__ float4 sum_ranks(const float4* p, int pitch) {
  float4 s = p[0];
#pragma unroll
  for (int q = 1; q < kC; ++q) add4(s, p[q * pitch]);
  return s;
}

// What every part of the kernel knows of its CTA.
struct Cta {
  int rank;
  int r0, units, rows;   // its rows of the basis: first, 16-row units, rows
  int u0, n_units;       // the cluster's 16-row units of the images and of W; unit u (of n_units) is CTA u % kC's
};

template <int kSlots>
__device__ __forceinline__ void wait_slot() {   // all but the last kSlots - 1 groups
  asm volatile("cp.async.wait_group %0;" ::"n"(kSlots - 1) : "memory");
}
// y += W r for the fired tokens, 8 NB at a time.  False when a wait ran out (for every thread of the CTA):
// the batches from there on are left out, what the peers wait for among them, which stop in turn.
template <int NB>
__device__ __forceinline__ bool stream_w(const GroupParams& g, const IoRef& io, const ClusterPlan& pl, const Cta& me,
                                         const int* s_fired, unsigned char* smem, uint64_t* s_bar) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lg = lane >> 2, lt = lane & 3;
  const int n_fired = s_fired[0], stride = op_stride(pl.steps);   // (places alike on all CTAs)
  const float* xs = reinterpret_cast<const float*>(smem + pl.xs);
  const int most = min(8 * NB, n_fired);                      // tokens of a pass
  const int all_slots = (me.n_units + kC - 1) / kC, passes = (n_fired + 8 * NB - 1) / (8 * NB);
  // r as operand, the ring, one buffer of partials [slot][rank][token][16 rows] or two
  const int ring = most * stride, left = pl.front_bytes - ring, one = most * 1024;
  const bool deep = left - ring_bytes(kDeepSlots) >= (passes > 1 ? 2 : 1) * all_slots * one;
  const int n_ring = deep ? kDeepSlots : kShallowSlots;
  const int part = ring + ring_bytes(n_ring);
  const int slots = deep ? all_slots : max(1, min(all_slots, (pl.front_bytes - part) / 2 / one));
  const int batch_units = slots * kC, per_pass = (me.n_units + batch_units - 1) / batch_units;
  const int batches = per_pass * passes;
  auto tokens_of = [&](int b) { return min(8 * NB, n_fired - b / per_pass * 8 * NB); };
  auto own_slots = [&](int b) {   // units of batch b that are this CTA's
    const int n = min(batch_units, me.n_units - b % per_pass * batch_units) - me.rank;
    return n > 0 ? (n + kC - 1) / kC : 0;
  };
  // This warp's slots, in order: units warp, warp + kW, ... of every pass, `sp` slots each.
  const int steps = (me.rows + 31) / 32, sp = (steps + 1) / 2;
  const int per_warp = me.n_units > warp ? (me.n_units - warp + kW - 1) / kW * sp : 0;
  const uint32_t mine = s32(smem + ring) + warp * n_ring * kSlotBytes + lane * 16;
  const uint16_t* w[2] = {nullptr, nullptr};
  int at_unit = warp, at_part = 0, issued = 0, slot_in = 0;
  auto issue = [&]() {
    if (issued < per_warp * passes) {
      if (at_part == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int row = (me.u0 + at_unit) * 16 + lg + 8 * h;
          w[h] = nullptr;
          if (row < g.O) {
            int j = 0;
            while (j + 1 < g.n_maps && row >= g.off[j + 1]) ++j;
            w[h] = g.W[j] + (size_t)(row - g.off[j]) * g.d + me.r0 + lt * 8;
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int e = (at_part * 2 + q) * 32;
          const bool in = w[h] && e + lt * 8 < me.rows;
          const uint16_t* p = in ? w[h] + e : g.W[0];
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(mine + slot_in * kSlotBytes + (q * 2 + h) * 512),
                       "l"(p), "r"(in ? 16 : 0)
                       : "memory");
        }
      ++issued;
      if (++at_part == sp) {
        at_part = 0;
        at_unit += kW;
        if (at_unit >= me.n_units) at_unit = warp;   // the next tokens
      }
      if (++slot_in == n_ring) slot_in = 0;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll 1
  for (int i = 0; i < n_ring - 1; ++i) issue();
  int slot_out = 0;
#pragma unroll 1
  for (int b = 0; b <= batches; ++b) {
    if (b < batches) {
      const int f0 = b / per_pass * 8 * NB, NC = tokens_of(b), first = b % per_pass * batch_units;
      if (tid == 0) expect(&s_bar[b & 1], (uint32_t)(own_slots(b) * NC * 1024));
      if (b % per_pass == 0) {   // r of these tokens as operand
        if (b > 0) __syncthreads();
        for (int c = warp; c < NC; c += kW) {
          const float* r = xs + s_fired[1 + f0 + c] * pl.xp;
          for (int e = lane; e < steps * 4; e += 32) {
            float v[8] = {};
            if (e * 8 < me.rows) {
              const float4 lo = *reinterpret_cast<const float4*>(r + e * 8), hi = *reinterpret_cast<const float4*>(r + e * 8 + 4);
              v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w;
              v[4] = hi.x; v[5] = hi.y; v[6] = hi.z; v[7] = hi.w;
            }
            uint4 t[3];
            split3_x8(v, t);
            unsigned char* to = smem + c * stride + (e >> 2) * 192 + (e & 3) * 16;
#pragma unroll
            for (int q = 0; q < 3; ++q) *reinterpret_cast<uint4*>(to + q * 64) = t[q];
          }
        }
        __syncthreads();
      }
      if (b >= 2) cluster_wait();   // every CTA has added batch b - 2: its buffer is free
#pragma unroll 1
      for (int u = warp; u < batch_units && first + u < me.n_units; u += kW) {
        float low[NB][4], sum[NB][4];
        clear<NB>(low);
        clear<NB>(sum);
        uint32_t slot = mine;
#pragma unroll 1
        for (int s0 = 0; s0 < steps; s0 += 2) {
          issue();
          if (deep) wait_slot<kDeepSlots>();
          else wait_slot<kShallowSlots>();
          slot = mine + slot_out * kSlotBytes;
          if (++slot_out == n_ring) slot_out = 0;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (s0 + q >= steps) break;
            const uint4 a0 = ld_shared16(slot + q * 1024), a1 = ld_shared16(slot + q * 1024 + 512);
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) {
              float hi[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
              for (int r = 0; r < 3; ++r) {
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (nb * 8 + lg < NC) v = ld_shared16(s32(smem) + (nb * 8 + lg) * stride + ((s0 + q) * 3 + r) * 64 + lt * 16);
                float(&to)[4] = r == 0 ? hi : low[nb];
                mma(to, a0.x, a1.x, a0.y, a1.y, v.x, v.y);
                mma(to, a0.z, a1.z, a0.w, a1.w, v.z, v.w);
              }
#pragma unroll
              for (int i = 0; i < 4; ++i) sum[nb][i] += hi[i];
            }
          }
        }
        add_low<NB>(low, sum);
        // the unit's sums as [token][16 rows], in the slot that was read last, and to the unit's owner
        float* sums = reinterpret_cast<float*>(smem + (slot - lane * 16 - s32(smem)));
        __syncwarp();
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = nb * 8 + 2 * lt + (i & 1);
            if (c < NC) sums[c * 16 + lg + 8 * (i >> 1)] = sum[nb][i];
          }
        __syncwarp();
        const int to = u % kC;
        const uint32_t at = peer(s32(smem + part + ((b & 1) * slots + u / kC) * one + me.rank * NC * 64), to);
        const uint32_t bar = peer(s32(&s_bar[b & 1]), to);
        for (int i = lane; i < NC * 4; i += 32) send16(at + i * 16, bar, *reinterpret_cast<const float4*>(sums + i * 4));
        __syncwarp();
      }
    }
    if (b > 0) {   // the batch before: this CTA's units
      const int a = b - 1, f0 = a / per_pass * 8 * NB, NC = tokens_of(a), first = a % per_pass * batch_units;
      // (a barrier whose words have not come may not be armed again: they would count towards another batch)
      if (__syncthreads_or(!arrived(&s_bar[a & 1], (a >> 1) & 1, g.spin_limit))) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        return false;
      }
      for (int i = tid; i < own_slots(a) * NC * 4; i += kT) {
        const int q = i & 3, sc = i >> 2, slot = sc / NC, c = sc - slot * NC;
        const float4 v = sum_ranks(reinterpret_cast<const float4*>(smem + part + ((a & 1) * slots + slot) * one) + c * 4 + q, NC * 4);
        const int row = (me.u0 + first + slot * kC + me.rank) * 16 + q * 4;
        if (row < g.O) {
          float4* y = reinterpret_cast<float4*>(io.y + (size_t)s_fired[1 + f0 + c] * g.O + row);
          float4 t = *y;
          add4(t, v);
          *y = t;
        }
      }
      if (a + 2 < batches) cluster_arrive();
    }
  }
  return true;
}

// Everything up to the gate.  False when a wait ran out (for every thread of the CTA); s_fired: the
// number of gated tokens whose W r this launch adds, and which.
template <int NB, bool PF32>
__device__ __forceinline__ bool front(const GroupParams& g, const IoRef& io, const ClusterPlan& pl, const Cta& me, int n,
                                      int leave_from, unsigned char* smem, int* s_fired, uint64_t* s_bar) {
  constexpr int kTok = 8 * NB, kTerms = PF32 ? 3 : 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lg = lane >> 2, lt = lane & 3;
  const int d = g.d, k = g.k, kq = k / 4, units = me.units, rows = me.rows, cid = blockIdx.x / kC;
  float* xs = reinterpret_cast<float*>(smem + pl.xs);
  uint2* xt = reinterpret_cast<uint2*>(smem + pl.xt);   // x as operand: [unit][eight tokens][term][lane]
  unsigned char* op = smem + pl.op;
  const int own = me.n_units > me.rank ? (me.n_units - me.rank + kC - 1) / kC : 0;   // its units of the images
  const int ksteps = (k + 31) / 32, stride = op_stride(ksteps), nbs = NB == 1 ? 1 : pl.nbs, kTokB = 8 * nbs;

  pdl_wait();
  const int slot = io_slot(io);
  const float* x = io.x + (long long)slot * io.x_step_stride + me.r0;
  // ---- the slab of P (the clusters begin at different rows), x of later passes
  {
    const int KV = k / 8, rpp = 32 >> pl.lpr_log2, all = 16 * units, rot = (all * (cid & 7)) >> 3;
    for (int b = warp * rpp + (lane >> pl.lpr_log2); b < all; b += kW * rpp) {
      const int row = b + rot < all ? b + rot : b + rot - all;
      for (int c = lane & ((1 << pl.lpr_log2) - 1); c < KV; c += 1 << pl.lpr_log2) {
        unsigned char* to = smem + row * pl.pitch + c * 16;
        if constexpr (PF32) {
          float v[8] = {};
          uint4 t[3];
          if (row < rows) load8<true>(g.P, (size_t)(me.r0 + row) * KV + c, v);
          split3_x8(v, t);
#pragma unroll
          for (int q = 0; q < 3; ++q) *reinterpret_cast<uint4*>(to + q * pl.plane) = t[q];
        } else if (row < rows) {
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s32(to)),
                       "l"(static_cast<const uint4*>(g.P) + (size_t)(me.r0 + row) * KV + c)
                       : "memory");
        } else {
          *reinterpret_cast<uint4*>(to) = make_uint4(0u, 0u, 0u, 0u);
        }
      }
    }
  }
  for (int t = kTok + warp; t < n; t += kW)
    for (int c = lane; c < rows / 4; c += 32)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s32(xs + t * pl.xp + 4 * c)),
                   "l"(x + (size_t)t * d + 4 * c)
                   : "memory");
  auto x_terms = [&](int u, int nb, const float2& a, const float2& b) {
    uint32_t ta[3], tc[3];
    split3_pair(a.x, a.y, ta);
    split3_pair(b.x, b.y, tc);
#pragma unroll
    for (int q = 0; q < 3; ++q) xt[((u * nbs + nb) * 3 + q) * 32 + lane] = make_uint2(ta[q], tc[q]);
  };
  // x of the first pass: as operand, and as it is
  for (int it = warp; it < units * NB; it += kW) {
    const int u = it / NB, nb = it % NB, t = nb * 8 + lg, row = 16 * u + 2 * lt;
    if (nb >= nbs) continue;
    float2 a = make_float2(0.f, 0.f), b = a;
    if (t < n && row < rows) a = __ldg(reinterpret_cast<const float2*>(x + (size_t)t * d + row));
    if (t < n && row + 8 < rows) b = __ldg(reinterpret_cast<const float2*>(x + (size_t)t * d + row + 8));
    if (t < n) {
      *reinterpret_cast<float2*>(xs + t * pl.xp + row) = a;
      *reinterpret_cast<float2*>(xs + t * pl.xp + row + 8) = b;
    }
    x_terms(u, nb, a, b);
  }
  // the image rows are asked into the L2 while c is on its way
  for (int i = tid; i < own; i += kT) {
    const int row = (me.u0 + me.rank + i * kC) * 16;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(g.WP + (size_t)row * k),
                 "r"((unsigned)(min(16, g.O - row) * k * 2))
                 : "memory");
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  bool ok = true;
  int phase = 0;
#pragma unroll 1
  for (int tb = 0; tb < n; tb += kTok, phase ^= 1) {
    const int NC = min(kTok, n - tb), ncb = NB == 1 ? 1 : (NC + 7) / 8;
    const int V = NC * kq, per = (V + kC - 1) / kC, mine = (V - me.rank + kC - 1) / kC;   // float4 v is CTA v % kC's
    if (tid == 0) {
      expect(&s_bar[0], (uint32_t)(kC * 16 * (pl.direct ? V : mine)));
      if (!pl.direct) expect(&s_bar[1], (uint32_t)(V * 16));
    }
    if (tb > 0) {
      __syncthreads();   // the operands before are read
      for (int it = warp; it < units * NB; it += kW) {
        const int u = it / NB, nb = it % NB, t = tb + nb * 8 + lg, row = 16 * u + 2 * lt;
        if (nb >= nbs) continue;
        float2 a = make_float2(0.f, 0.f), b = a;
        if (t < n && row < rows) a = *reinterpret_cast<const float2*>(xs + t * pl.xp + row);
        if (t < n && row + 8 < rows) b = *reinterpret_cast<const float2*>(xs + t * pl.xp + row + 8);
        x_terms(u, nb, a, b);
      }
      __syncthreads();
    }
    // ---- A
    float* wsum = reinterpret_cast<float*>(smem + pl.wsum);   // [share of the rows][token][16 mt columns]
    const int wpitch = pl.mt * 16;
    {
      // (a tile x eight tokens at a time: with the tokens inside, 3000 x 200 and 21 tokens took 12 us here)
      const int ks = 1 << pl.ks_log2, share = warp & (ks - 1);
      for (int it = warp >> pl.ks_log2; it < pl.mt * ncb; it += kW >> pl.ks_log2) {
        int m = it, nb = 0;
        if constexpr (NB > 1)
          for (; m >= pl.mt; m -= pl.mt) ++nb;
        float sum[4] = {}, low[4] = {}, low2[4] = {};
        const uint32_t at = s32(smem) + ((lane & 7) + ((lane >> 4) << 3)) * pl.pitch + m * 32 + ((lane >> 3) & 1) * 16;
#pragma unroll 4
        for (int u = share; u < units; u += ks) {
          uint32_t a[kTerms][4];
#pragma unroll
          for (int r = 0; r < kTerms; ++r)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                         : "=r"(a[r][0]), "=r"(a[r][1]), "=r"(a[r][2]), "=r"(a[r][3])
                         : "r"(at + u * 16 * pl.pitch + r * pl.plane));
          float hi[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const uint2 b = xt[((u * nbs + nb) * 3 + q) * 32 + lane];
#pragma unroll
            for (int r = 0; r < kTerms; ++r) mma((q == 0 && r == 0) ? hi : q == 1 ? low : low2, a[r][0], a[r][1], a[r][2], a[r][3], b.x, b.y);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) sum[i] += hi[i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = nb * 8 + 2 * lt + (i & 1);
          if (c < NC) wsum[(share * kTokB + c) * wpitch + m * 16 + lg + 8 * (i >> 1)] = sum[i] + (low[i] + low2[i]);
        }
      }
    }
    __syncthreads();

    // ---- x1
    if (tb == 0) cluster_wait();   // every CTA of the cluster has its barriers
    auto partial = [&](int v) {    // over the warps that shared the rows
      const int c = (int)__umulhi((unsigned)v, pl.kq_magic);
      const float* p = wsum + c * wpitch + 4 * (v - c * kq);
      float4 s = *reinterpret_cast<const float4*>(p);
      for (int q = 1; q < 1 << pl.ks_log2; ++q) add4(s, *reinterpret_cast<const float4*>(p + q * kTokB * wpitch));
      return s;
    };
    auto terms = [&](int v, const float4& s) {
      const int c = (int)__umulhi((unsigned)v, pl.kq_magic), j = 4 * (v - c * kq);
      uint32_t t[2][3];
      split3_pair(s.x, s.y, t[0]);
      split3_pair(s.z, s.w, t[1]);
      unsigned char* to = op + c * stride;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        *reinterpret_cast<uint2*>(to + op_pair(j, q)) = make_uint2(t[0][q], t[1][q]);
        if (j + 4 == k)   // zeros past the end
          for (int e = k; e & 31; e += 4) *reinterpret_cast<uint2*>(to + op_pair(e, q)) = make_uint2(0u, 0u);
      }
    };
    const float4* recv = reinterpret_cast<const float4*>(smem + pl.recv);
    if (pl.direct) {
      const int to = tid % kC;
      const uint32_t base = peer(s32(recv + me.rank * V), to), bar = peer(s32(&s_bar[0]), to);
      for (int v = tid / kC; v < V; v += kT / kC) send16(base + v * 16, bar, partial(v));
      ok = arrived(&s_bar[0], phase, g.spin_limit);
      if (ok && tid < V) terms(tid, sum_ranks(recv + tid, V));   // (V <= kDirectValues / 4)
    } else {
      for (int v = tid; v < V; v += kT) {
        const int to = v % kC;
        send16(peer(s32(recv + me.rank * per + v / kC), to), peer(s32(&s_bar[0]), to), partial(v));
      }
      ok = arrived(&s_bar[0], phase, g.spin_limit);
      const float4* recv2 = reinterpret_cast<const float4*>(smem + pl.recv2);
      if (ok) {
        const int to = tid % kC;
        const uint32_t base = peer(s32(recv2 + me.rank), to), bar = peer(s32(&s_bar[1]), to);
        for (int i = tid / kC; i < mine; i += kT / kC) send16(base + i * kC * 16, bar, sum_ranks(recv + i, per));
        ok = arrived(&s_bar[1], phase, g.spin_limit);
      }
      if (ok)
        for (int v = tid; v < V; v += kT) terms(v, recv2[v]);
    }
    if (__syncthreads_or(!ok)) return false;

    // ---- B: a unit x eight tokens per warp; r takes the place of x
    float2* s_unit = reinterpret_cast<float2*>(smem + pl.unit);   // [unit][token]: ||r||^2, ||x||^2
    for (int it = warp; it < units * NB; it += kW) {
      const int u = it / NB, nb = it % NB;
      if (nb >= ncb) continue;
      float low[4] = {}, low2[4] = {}, sum[4] = {};
      // (the lower terms in two chains: a dependent instruction waits for some 35 cycles)
      const uint32_t a0 = s32(smem) + (16 * u + lg) * pl.pitch + lt * 16;
      const uint32_t b0 = s32(op) + (nb * 8 + lg) * stride + lt * 16;
#pragma unroll 2
      for (int s = 0; s < ksteps; ++s) {
        uint4 a[2][kTerms];
        const bool in = s * 32 + lt * 8 < k;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int r = 0; r < kTerms; ++r)
            a[h][r] = in ? ld_shared16(a0 + h * 8 * pl.pitch + r * pl.plane + s * 64) : make_uint4(0u, 0u, 0u, 0u);
        float hi[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const uint4 b = nb * 8 + lg < NC ? ld_shared16(b0 + (s * 3 + q) * 64) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
          for (int r = 0; r < kTerms; ++r) {
            float(&to)[4] = (q == 0 && r == 0) ? hi : q == 1 ? low : low2;
            mma(to, a[0][r].x, a[1][r].x, a[0][r].y, a[1][r].y, b.x, b.y);
            mma(to, a[0][r].z, a[1][r].z, a[0][r].w, a[1][r].w, b.z, b.w);
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) sum[i] += hi[i];
      }
      float sr[2] = {0.f, 0.f}, sx[2] = {0.f, 0.f};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int t = tb + nb * 8 + 2 * lt + (i & 1), row = 16 * u + lg + 8 * (i >> 1);
        if (t < n && row < rows) {
          const float xv = xs[t * pl.xp + row], rv = xv - (sum[i] + (low[i] + low2[i]));
          xs[t * pl.xp + row] = rv;
          if (leave_from && cid == 0) g.r[(size_t)t * d + me.r0 + row] = rv;
          sr[i & 1] = fmaf(rv, rv, sr[i & 1]);
          sx[i & 1] = fmaf(xv, xv, sx[i & 1]);
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          sr[i] += __shfl_xor_sync(0xffffffffu, sr[i], o);
          sx[i] += __shfl_xor_sync(0xffffffffu, sx[i], o);
        }
        if (lg == 0) s_unit[u * kTokB + nb * 8 + 2 * lt + i] = make_float2(sr[i], sx[i]);
      }
    }
    // The first warp adds the units' norms in order and sends them off; the others go on to the image.
    if (warp > 0) {
      asm volatile("bar.arrive 1, %0;" ::"n"(kT) : "memory");
    } else {
      asm volatile("bar.sync 1, %0;" ::"n"(kT) : "memory");
      double sr[4] = {}, sx[4] = {};
      if (lane < NC)
        for (int u0 = 0; u0 < units; u0 += 4)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (u0 + e < units) {
              const float2 v = s_unit[(u0 + e) * kTokB + lane];
              sr[e] += (double)v.x;
              sx[e] += (double)v.y;
            }
      const float fr = (float)((sr[0] + sr[1]) + (sr[2] + sr[3])), fx = (float)((sx[0] + sx[1]) + (sx[2] + sx[3]));
      const int to = lane % kC;
      const uint32_t base = peer(s32(smem + pl.norm) + (me.rank * n + tb) * 8, to), bar = peer(s32(&s_bar[2]), to);
      for (int t2 = 0; t2 < NC; t2 += 2) {
        const int t = t2 + lane / kC;
        const float a = __shfl_sync(0xffffffffu, fr, t & 31), b = __shfl_sync(0xffffffffu, fx, t & 31);
        if (t < NC) send8(base + t * 8, bar, a, b);
      }
    }
    // image rows (the last warps, which have no basis rows in narrow calls, go first)
    for (int it = kW - 1 - warp; it < own * NB; it += kW) {
      const int i = it / NB, nb = it % NB, row = (me.u0 + me.rank + i * kC) * 16 + lg;
      if (nb >= ncb) continue;
      const void* pr[2];
      float low[1][4], sum[1][4];
      clear<1>(low);
      clear<1>(sum);
#pragma unroll
      for (int h = 0; h < 2; ++h) pr[h] = row + 8 * h < g.O ? g.WP + (size_t)(row + 8 * h) * k + lt * 8 : nullptr;
      dot_steps<1, false, false>(pr[0], pr[1], k, 0, 1, ksteps, op + nb * 8 * stride, stride, 0, NC - nb * 8, low, sum);
      add_low<1>(low, sum);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int t = tb + nb * 8 + 2 * lt + (e & 1), r = row + 8 * (e >> 1);
        if (t < n && t < tb + NC && r < g.O) io.y[(size_t)t * g.O + r] = sum[0][e];
      }
    }
  }

  // ---- x2 and the gate: the same sums in the same order on every CTA
  if (warp == 0) {
    ok = arrived(&s_bar[2], 0, g.spin_limit);
    int f = 0;
    for (int t0 = 0; t0 < n; t0 += 32) {
      const int t = t0 + lane;
      bool fired = false;
      if (t < n) {
        const float2* norm = reinterpret_cast<const float2*>(smem + pl.norm) + t;
        double a[kC], b[kC];   // by a tree: sixteen additions one after the other take half a microsecond
#pragma unroll
        for (int q = 0; q < kC; ++q) {
          const float2 v = norm[q * n];
          a[q] = (double)v.x;
          b[q] = (double)v.y;
        }
#pragma unroll
        for (int h = 1; h < kC; h *= 2)
#pragma unroll
          for (int q = 0; q < kC; q += 2 * h) {
            a[q] += a[q + h];
            b[q] += b[q + h];
          }
        const double sr = a[0], sx = b[0];
        // ||r|| < eps ||x||, false for NaN and for x = 0; away from equality the squares decide (roots and
        // quotients in double take a microsecond)
        const double bound = (double)g.eps * g.eps * sx;
        bool fast = sr < bound * (1.0 - 1e-9);
        if (!fast && !(sr > bound * (1.0 + 1e-9))) fast = sqrt(sr) < (double)g.eps * sqrt(sx);
        fired = !fast && !(g.flags & GSI_FLAG_STATIC_PROJECTION);
        if (blockIdx.x == 0) {
          io.gate[(long long)slot * io.log_step_stride + t] = fast ? 0 : 1;
          float* rho = io.rho ? io.rho + (long long)slot * io.log_step_stride : g.rho_scratch;
          if (ok) rho[t] = sr == 0.0 && sx > 0.0 ? 0.f : (float)(sr * rsqrt(sr * sx));   // sqrt(sr / sx)
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, fired);
      const int at = f + __popc(m & ((1u << lane) - 1u));
      if (fired) {
        s_fired[1 + at] = t;
        if (leave_from && blockIdx.x == 0) g.fired[at] = t;
      }
      f += __popc(m);
    }
    if (lane == 0) {
      s_fired[0] = leave_from && f >= leave_from ? 0 : f;
      if (leave_from && blockIdx.x == 0) *g.n_fired = f;
    }
  }
  return !__syncthreads_or(!ok);
}

template <int NB, bool PF32>
__global__ void __launch_bounds__(kT, 1)
k_forward_cluster(const __grid_constant__ GroupParams g, const __grid_constant__ IoRef io, const __grid_constant__ ClusterPlan pl,
                  int n_tokens, int leave_from) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[5];   // partials of c, sums of c, norms, partials of W r (two buffers)
  __shared__ int s_fired[GSI_MAX_TOKENS + 1];
  if (threadIdx.x == 0) {
    for (uint64_t& b : s_bar) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s32(&b)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    expect(&s_bar[2], (uint32_t)(kC * n_tokens * 8));
  }
  cluster_arrive();   // (waited for ahead of the first word to a peer)
  pdl_launch_dependents();
  const int cid = blockIdx.x / kC, U = (g.d + 15) / 16;
  Cta me;
  me.rank = blockIdx.x % kC;
  me.r0 = U * me.rank / kC;
  me.units = U * (me.rank + 1) / kC - me.r0;
  me.r0 *= 16;
  me.rows = max(0, min(g.d - me.r0, 16 * me.units));
  me.u0 = cid * pl.unit_base + min(cid, pl.unit_rem);
  me.n_units = pl.unit_base + (cid < pl.unit_rem ? 1 : 0);
  bool ok = front<NB, PF32>(g, io, pl, me, n_tokens, leave_from, smem, s_fired, s_bar);
  if (ok) {
    const int f = s_fired[0];
    if (f == 0) {   // (all that its peers sent to this CTA has arrived)
      if (threadIdx.x == 0) exchange::leave_launch(g.tickets);
      return;
    }
    // as many tokens at a time as there are and as the first part of shared memory holds
    const int op = op_stride(pl.steps);
    auto fits = [&](int NC) { return NC * op + ring_bytes(kShallowSlots) + 2 * NC * 1024 <= pl.front_bytes; };
    if (f > 16 && fits(min(f, 32))) ok = stream_w<4>(g, io, pl, me, s_fired, smem, s_bar + 3);
    else if (f > 8 && fits(min(f, 16))) ok = stream_w<2>(g, io, pl, me, s_fired, smem, s_bar + 3);
    else ok = stream_w<1>(g, io, pl, me, s_fired, smem, s_bar + 3);
    if (ok) {   // (likewise)
      if (threadIdx.x == 0) exchange::leave_launch(g.tickets);
      return;
    }
  }
  if (threadIdx.x == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
  // The call's results must not pass for results: NaN in this CTA's rows of y and in every token's rho.
  const float nan = __int_as_float(0x7fc00000);
  for (int t = 0; t < n_tokens; ++t)
    for (int i = threadIdx.x; i < 16 * me.n_units; i += kT) {
      const int row = me.u0 * 16 + i;
      if ((i >> 4) % kC == me.rank && row < g.O) io.y[(size_t)t * g.O + row] = nan;
    }
  if (leave_from && blockIdx.x == 0 && threadIdx.x == 0) *g.n_fired = 0;
  __syncthreads();
  // Peers may still send to this CTA: it stays until they have left (an exited thread counts as
  // arrived, one that goes on with W r arrives once per batch), and for the words then in flight.
  // Meanwhile block 0, of this cluster or another, leaves.
  bool told = blockIdx.x == 0;
#pragma unroll 1
  for (int i = 0; i < kMaxBatches || (!told && i < exchange::kReportPolls); ++i) {
    cluster_arrive();
    cluster_wait();
    if (!told) told = __syncthreads_or(threadIdx.x == 0 && exchange::block0_left(g.tickets));
  }
  exchange::let_land();
  exchange::report_give_up(g, io, n_tokens);
}

// Clusters that the current context (for this stream) holds at a time; 0: none, or it cannot be told.
template <typename K>
int resident_clusters(K kernel, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kC);
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = kSmemCluster;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kC;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

template <int NB, bool PF32>
bool launch_t(const GroupParams& g, const IoRef& io, int n, int leave, cudaStream_t st, cudaError_t* e) {
  ClusterPlan pl;
  if (!make_plan<NB, PF32>(g.d, g.k, n, &pl)) return false;
  auto kernel = k_forward_cluster<NB, PF32>;
  // per thread and context (whose id is never used again): the kernel's attributes, the clusters that fit
  static thread_local unsigned long long known = 0;
  static thread_local int clusters = 0;
  const unsigned long long id = context_id();
  if (!id || id != known) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCluster) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
    clusters = resident_clusters(kernel, st);
    known = id;
  }
  if (clusters < 1) return false;
  const int units = (g.O + 15) / 16, most = (units + kC - 1) / kC;   // a unit of rows per CTA at least
  const int grid = clusters < most ? clusters : most;
  pl.unit_base = units / grid;
  pl.unit_rem = units % grid;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kC * grid);
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = kSmemCluster;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kC;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  *e = cudaLaunchKernelEx(&cfg, kernel, g, io, pl, n, leave);
  if (*e == cudaErrorInvalidClusterSize || *e == cudaErrorLaunchOutOfResources) {   // a stream with fewer SMs than its context
    (void)cudaGetLastError();
    return false;
  }
  return true;
}

// Which calls run here.  The shape has to fit with any number of tokens of the handle's (handles for one
// or two tokens: with those).  Every cluster does all of the contractions with P, which the cooperative launch
// shares out: up to 16 tokens that pays as far as (tokens rounded up to 8) d k <= 1.2e7, beyond up to 4.5e6.  A tenth gated, us per call,
// cooperative launch / this: 3000 x 200 -> 1576 at 8 tokens 15.1 / 10.7, 16 17.3 / 15.7, 24 24.3 / 25.3, 32 24.7 / 32.2;
// 4000 x 200 -> 1000 at 8 15.9 / 12.0, 16 16.9 / 17.4; 8000 x 104 -> 1000 at 8 17.0 / 12.4, 16 18.6 / 20.4; 1000 x 400 ->
// 2000 at 16 22.3 / 19.0, 24 24.1 / 26.5; 304 x 296 -> 600 at 32 22.8 / 19.9; 760 x 128 -> 2304, fp32 basis, at 32 24.4 / 17.9; 1000 x 72 -> 4000 at 48
// 25.7 / 21.8, 64 28.0 / 28.0.  Nine to 16 tokens have to fit in one pass (1800 x 400 -> 3000 at 16 19.5 / 22.0, 1408 x 504 -> 3000
// at 12 23.3 / 26.0, -> 64 18.7 / 20.1; but 1288 x 440 -> 64 at 16 20.6 / 19.6).  Where the rows outnumber the width by far,
// twenty to forty times, a quarter gated, the 112 SMs of seven clusters are behind: 520 x 512 -> 16000 at 8 24.3 / 24.2, 16 27.0 /
// 32.6, but 20.7 / 20.6 with 1 % gated, at 4 16.7 / 11.4; 768 x 64 -> 20480 at 32 33.1 / 38.0.
template <bool PF32>
bool launch_p(const GroupParams& g, const IoRef& io, int n, int leave, cudaStream_t st, cudaError_t* e) {
  ClusterPlan pl;
  if (g.k > kMostColumns) return false;
  if ((double)((n + 7) / 8 * 8) * g.d * g.k > (n <= 16 ? 1.2e7 : 4.5e6)) return false;
  if (g.B > 2 && !make_plan<1, PF32>(g.d, g.k, GSI_MAX_TOKENS, &pl)) return false;
  if (n > 16 && launch_t<4, PF32>(g, io, n, leave, st, e)) return true;
  return n > 8 ? launch_t<2, PF32>(g, io, n, leave, st, e) : launch_t<1, PF32>(g, io, n, leave, st, e);
}

}  // namespace

bool launch_forward_cluster(const GroupParams& g, const IoRef& io, int n_tokens, int leave_from, cudaStream_t st,
                            cudaError_t* e) {
  return g.p_f32 ? launch_p<true>(g, io, n_tokens, leave_from, st, e) : launch_p<false>(g, io, n_tokens, leave_from, st, e);
}

}  // namespace gsi
