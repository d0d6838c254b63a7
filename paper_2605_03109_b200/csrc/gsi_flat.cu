// Decode step of a stack of many small groups, one token: three launches over all groups, none of
// which waits for another CTA.
//
//   k_flat_project   partial c of every CTA's rows of the bases             (line 1)
//   k_flat_residual  c from the partials; r and the partial norms of the same rows   (line 2)
//   k_flat_rows      every CTA takes all gates (Eq. (3.3)) and an even share, in bytes, of the rows that
//                    are to be read: y = W_P c, and + W r where the group is gated    (lines 3-5, Eq. (3.2))
//
// The inputs of a step are staged before it, so no group waits for another.  The persistent kernel
// (gsi_persistent_impl.cuh) goes through a stack phase by phase, 3.5 us each whatever a phase carries; with
// small groups that is most of the step.  Here a step is three passes at the speed of the memory
// system; the price is that the bases are read twice, so they have to fit the L2.  12 GPT-2 layers,
// k = 128, 70 % gated: 120 -> 51 us; by themselves the launches take 8, 10 and 37 (140 MB of images and W; held
// up by the decisions at its start and by rows of 1.5 to 6 KB, W flows at 4.5 TB/s).  What a CTA needs of the
// tables, and the first rows of the basis in the second launch, are read ahead of the wait on the launch before:
// 4 us a step in small stacks (two GPT-2 layers, 1 % gated, 26.8 -> 22.7; the persistent kernel takes 23.0).
//
// All sums run in an order that depends on the shapes and the grid alone.
#include "gsi_flat.cuh"

namespace gsi {

namespace {

constexpr int kT = 512, kW = kT / 32;
constexpr int kMaxVec = 4;   // 16-byte vectors of a basis row per lane (k <= 1024)

__device__ __forceinline__ IoRef io_of(const WideGroup& w, int use_counter) {
  IoRef io = w.io;
  if (!use_counter) io.step = nullptr;
  return io;
}
__device__ __forceinline__ float dot8(const uint4& v, const float4& lo, const float4& hi, float s) {
  float f[8];
  unpack_bf16x8(v, f);
  s = fmaf(f[0], lo.x, s); s = fmaf(f[1], lo.y, s); s = fmaf(f[2], lo.z, s); s = fmaf(f[3], lo.w, s);
  s = fmaf(f[4], hi.x, s); s = fmaf(f[5], hi.y, s); s = fmaf(f[6], hi.z, s); s = fmaf(f[7], hi.w, s);
  return s;
}

// Lanes of a warp over a basis row of KV vectors: `lpr` lanes per row, VPL vectors per lane.
struct Lanes {
  int lpr, rpp, sub, cl;
  __device__ __forceinline__ explicit Lanes(int KV) {
    const int lane = threadIdx.x & 31;
    lpr = 1;
    while (lpr < KV && lpr < 32) lpr <<= 1;
    rpp = 32 / lpr;
    sub = lane / lpr;
    cl = lane % lpr;
  }
};

// What the first two kernels need of a group, in registers: read ahead of the wait on the kernel before.
struct Rows {
  const uint4* P;
  float *cpart, *c, *r;
  IoRef io;
  int k, d, r0, r1, slot, slots;
  __device__ __forceinline__ Rows(const FlatParams& p, int i) {
    const FlatShare sh = p.shares[i];
    const WideGroup& w = p.table[sh.group];
    P = static_cast<const uint4*>(w.g.P);
    cpart = w.g.cpart;
    c = w.g.c;
    r = w.g.r;
    k = w.g.k;
    d = w.g.d;
    io = io_of(w, p.use_counter);
    slots = p.groups[sh.group].slots;
    slot = sh.slot;
    r0 = sh.r0;
    r1 = min(d, sh.r1);
  }
  __device__ __forceinline__ const float* x() const {
    return io.x + (io.step ? (long long)(__ldcg(io.step) % io.n_steps) * io.x_step_stride : 0);
  }
};
template <int VPL>
__device__ constexpr int in_flight() { return VPL == 1 ? 8 : VPL == 2 ? 4 : 2; }   // rows per lane
// Rows base, base + stride, ... of the basis, and their x.
template <int VPL, int U>
__device__ __forceinline__ void load_rows(const Rows& g, const float* x, const Lanes& L, int base, uint4 (&q)[U][VPL],
                                          float (&xv)[U]) {
  const int KV = g.k / 8, stride = kW * L.rpp;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int row = base + u * stride;
    xv[u] = row < g.r1 ? __ldcg(x + row) : 0.f;
#pragma unroll
    for (int v = 0; v < VPL; ++v)
      q[u][v] = row < g.r1 && L.cl + v * 32 < KV ? __ldg(g.P + (size_t)row * KV + L.cl + v * 32) : make_uint4(0u, 0u, 0u, 0u);
  }
}

template <int VPL>
__device__ __forceinline__ void project(const Rows& g, float* s_sum) {
  constexpr int U = in_flight<VPL>();
  const int KV = g.k / 8, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Lanes L(KV);
  const float* x = g.x();
  float acc[VPL][8];
#pragma unroll
  for (int v = 0; v < VPL; ++v)
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[v][e] = 0.f;
  for (int base = g.r0 + warp * L.rpp + L.sub; base < g.r1; base += U * kW * L.rpp) {
    uint4 p[U][VPL];
    float xv[U];
    load_rows<VPL, U>(g, x, L, base, p, xv);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        float f[8];
        unpack_bf16x8(p[u][v], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[v][e] = fmaf(f[e], xv[u], acc[v][e]);
      }
  }
  for (int o = L.lpr; o < 32; o <<= 1)
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[v][e] += __shfl_xor_sync(0xffffffffu, acc[v][e], o);
  __syncthreads();
#pragma unroll
  for (int v = 0; v < VPL; ++v)
    if (lane < L.lpr && lane + v * 32 < KV) {
      float4* to = reinterpret_cast<float4*>(s_sum + warp * g.k + (lane + v * 32) * 8);
      to[0] = make_float4(acc[v][0], acc[v][1], acc[v][2], acc[v][3]);
      to[1] = make_float4(acc[v][4], acc[v][5], acc[v][6], acc[v][7]);
    }
  __syncthreads();
  for (int j = threadIdx.x; j < g.k; j += kT) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kW; ++w) s += s_sum[w * g.k + j];
    g.cpart[(size_t)g.slot * g.k + j] = s;
  }
}

__global__ void __launch_bounds__(kT, 1) k_flat_project(FlatParams p) {
  extern __shared__ __align__(16) float s_sum[];   // [warp][k]
  const int i0 = p.first[blockIdx.x], i1 = p.first[blockIdx.x + 1];   // (written when the stack is bound)
  Rows g(p, min(i0, p.n_shares - 1));
  // First of the chain: nothing of it runs beside an earlier step, whose outputs and step the other two
  // may so take for granted ahead of their own waits.
  pdl_wait();
  pdl_launch_dependents();
  for (int i = i0; i < i1; ++i) {
    if (i > i0) g = Rows(p, i);
    if (g.k <= 256) project<1>(g, s_sum);
    else if (g.k <= 512) project<2>(g, s_sum);
    else project<kMaxVec>(g, s_sum);
  }
}

// r and the norms of a share's rows; the first rows are on their way while c comes together.
template <int VPL>
__device__ __forceinline__ void residual(const Rows& g, bool wait, float* s_c, float& sr, float& sx) {
  constexpr int U = in_flight<VPL>();
  const int KV = g.k / 8, tid = threadIdx.x, warp = tid >> 5;
  const Lanes L(KV);
  const float* x = g.x();
  const int stride = kW * L.rpp;
  int base = g.r0 + warp * L.rpp;
  uint4 q[U][VPL];
  float xv[U], dot[U];
  load_rows<VPL, U>(g, x, L, base + L.sub, q, xv);
  if (wait) pdl_wait();
  __syncthreads();   // c of the share before is read
  for (int j = tid; j < g.k; j += kT) {   // the partials in slot order, eight in flight
    float s = 0.f;
    for (int q0 = 0; q0 < g.slots; q0 += 8) {
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = q0 + e < g.slots ? __ldcg(g.cpart + (size_t)(q0 + e) * g.k + j) : 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) s += v[e];
    }
    s_c[j] = s;
    if (g.slot == 0) g.c[j] = s;
  }
  __syncthreads();
  float4 c[VPL][2];
#pragma unroll
  for (int v = 0; v < VPL; ++v)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      c[v][h] = L.cl + v * 32 < KV ? reinterpret_cast<const float4*>(s_c)[(L.cl + v * 32) * 2 + h] : make_float4(0.f, 0.f, 0.f, 0.f);
  while (base < g.r1) {   // (warp-uniform)
#pragma unroll
    for (int u = 0; u < U; ++u) {
      dot[u] = 0.f;
#pragma unroll
      for (int v = 0; v < VPL; ++v) dot[u] = dot8(q[u][v], c[v][0], c[v][1], dot[u]);
    }
    for (int o = 1; o < L.lpr; o <<= 1)
#pragma unroll
      for (int u = 0; u < U; ++u) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], o);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = base + L.sub + u * stride;
      if (row < g.r1 && L.cl == 0) {
        const float rv = xv[u] - dot[u];
        g.r[row] = rv;
        sr = fmaf(rv, rv, sr);
        sx = fmaf(xv[u], xv[u], sx);
      }
    }
    base += U * stride;
    if (base < g.r1) load_rows<VPL, U>(g, x, L, base + L.sub, q, xv);
  }
}

__global__ void __launch_bounds__(kT, 1) k_flat_residual(FlatParams p) {
  __shared__ __align__(16) float s_c[1024];
  __shared__ float2 s_norm[kW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  const int i0 = p.first[blockIdx.x], i1 = p.first[blockIdx.x + 1];
  for (int i = i0; i < i1; ++i) {   // (a CTA without a share: its index may lie past the list)
    const Rows g(p, i);
    float sr = 0.f, sx = 0.f;
    if (g.k <= 256) residual<1>(g, i == i0, s_c, sr, sx);
    else if (g.k <= 512) residual<2>(g, i == i0, s_c, sr, sx);
    else residual<kMaxVec>(g, i == i0, s_c, sr, sx);
    sr = warp_sum(sr);
    sx = warp_sum(sx);
    if (lane == 0) s_norm[warp] = make_float2(sr, sx);
    __syncthreads();
    if (tid == 0) {
      double a = 0.0, b = 0.0;
#pragma unroll
      for (int q = 0; q < kW; ++q) {
        a += (double)s_norm[q].x;
        b += (double)s_norm[q].y;
      }
      p.norms[i] = make_float2((float)a, (float)b);
    }
  }
}

// ---- rows of the images and of W ---------------------------------------------------------------
constexpr int kChunk = 512;       // rows at a time (their partial sums meet in shared memory)
constexpr int kTeamCols = 1024;   // columns of a row of W per warp: four 16-byte loads per lane
constexpr int kAhead = 3;         // rows of W in flight per warp: 6 KB, 96 KB per SM

// Image rows [r0, r1): to y, or to s_y (from row r0 on) where W r is still to come.
template <int VPL>
__device__ __forceinline__ void image_rows(const GroupParams& g, int r0, int r1, const float* s_c, float* s_y, float* y) {
  constexpr int U = VPL == 1 ? 8 : VPL == 2 ? 4 : 2;   // rows in flight per lane
  const int KV = g.k / 8, warp = threadIdx.x >> 5;
  const Lanes L(KV);
  const uint4* WP = reinterpret_cast<const uint4*>(g.WP);
  float4 c[VPL][2];
#pragma unroll
  for (int v = 0; v < VPL; ++v)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      c[v][h] = L.cl + v * 32 < KV ? reinterpret_cast<const float4*>(s_c)[(L.cl + v * 32) * 2 + h] : make_float4(0.f, 0.f, 0.f, 0.f);
  const int stride = kW * L.rpp;
  for (int base = r0 + warp * L.rpp; base < r1; base += U * stride) {   // (warp-uniform)
    uint4 q[U][VPL];
    float dot[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = base + L.sub + u * stride;
#pragma unroll
      for (int v = 0; v < VPL; ++v)
        q[u][v] = row < r1 && L.cl + v * 32 < KV ? ld_stream(WP + (size_t)row * KV + L.cl + v * 32) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      dot[u] = 0.f;
#pragma unroll
      for (int v = 0; v < VPL; ++v) dot[u] = dot8(q[u][v], c[v][0], c[v][1], dot[u]);
    }
    for (int o = 1; o < L.lpr; o <<= 1)
#pragma unroll
      for (int u = 0; u < U; ++u) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], o);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = base + L.sub + u * stride;
      if (row < r1 && L.cl == 0) {
        if (s_y) s_y[row - r0] = dot[u];
        else y[row] = dot[u];
      }
    }
  }
}

__global__ void __launch_bounds__(kT, 1) k_flat_rows(FlatParams p) {
  __shared__ __align__(16) float s_c[1024];
  __shared__ float s_y[kChunk], s_part[kChunk * kW];
  __shared__ unsigned long long s_start[kFlatMaxGroups + 1];   // bytes to read before every group
  __shared__ unsigned char s_gate[kFlatMaxGroups];
  __shared__ unsigned long long s_scan[kW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  pdl_wait();

  // ---- all gates, by every CTA: the same sums in the same order
  for (int i = tid; i < p.n; i += kT) {
    const FlatGroup g = p.groups[i];
    const float2* np = p.norms + g.first;
    const int n = g.slots;
    double sr = 0.0, sx = 0.0;
    for (int q0 = 0; q0 < n; q0 += 8) {
      float2 v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = q0 + e < n ? __ldcg(np + q0 + e) : make_float2(0.f, 0.f);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        sr += (double)v[e].x;
        sx += (double)v[e].y;
      }
    }
    // ||r|| < eps ||x||, false for NaN and for x = 0; away from equality the squares decide
    const double bound = (double)g.eps * g.eps * sx;
    bool fast = sr < bound * (1.0 - 1e-9);
    if (!fast && !(sr > bound * (1.0 + 1e-9))) fast = sqrt(sr) < (double)g.eps * sqrt(sx);
    s_gate[i] = !fast && !(g.flags & GSI_FLAG_STATIC_PROJECTION);
    if (blockIdx.x == 0) {
      const IoRef io = io_of(p.table[i], p.use_counter);
      const long long at = (long long)io_slot(io) * io.log_step_stride;
      io.gate[at] = fast ? 0 : 1;
      if (io.rho) io.rho[at] = sr == 0.0 && sx > 0.0 ? 0.f : (float)(sr * rsqrt(sr * sx));   // sqrt(sr / sx)
    }
  }
  __syncthreads();
  {   // bytes of the rows that are to be read, added up over the groups
    unsigned long long before = 0;
    for (int i0 = 0; i0 < p.n; i0 += kT) {
      const int i = i0 + tid;
      unsigned long long v = 0;
      if (i < p.n) {
        const FlatGroup g = p.groups[i];
        v = (unsigned long long)g.O * (2u * (unsigned)(g.k + (s_gate[i] ? g.d : 0)));
      }
      unsigned long long sum = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += u;
      }
      if (lane == 31) s_scan[warp] = sum;
      __syncthreads();
      unsigned long long w = before;
      for (int q = 0; q < warp; ++q) w += s_scan[q];
      if (i < p.n) s_start[i] = w + sum - v;
      if (i == p.n - 1) s_start[p.n] = w + sum;
      for (int q = 0; q < kW; ++q) before += s_scan[q];
      __syncthreads();
    }
  }
  if (tid == 0 && p.use_counter) {   // every CTA has read the step: the last one to come here moves it on
    const int prev = atomicAdd(p.arrived, 1);
    if (prev == (int)gridDim.x - 1) {
      *p.arrived = 0;
      *p.step = *p.step + 1;
    }
  }
  const unsigned long long all = s_start[p.n];
  const unsigned long long lo = all / gridDim.x * blockIdx.x + min((unsigned long long)blockIdx.x, all % gridDim.x);
  const unsigned long long hi = lo + all / gridDim.x + (blockIdx.x < all % gridDim.x ? 1 : 0);
  // first row of group i that begins at byte `at` or later, in pairs of rows
  auto row_at = [&](int i, unsigned long long at) -> int {
    if (at <= s_start[i]) return 0;
    const FlatGroup g = p.groups[i];
    const unsigned pair = 4u * (unsigned)(g.k + (s_gate[i] ? g.d : 0));
    const unsigned long long r = (at - s_start[i] + pair - 1) / pair * 2;
    return r < (unsigned long long)g.O ? (int)r : g.O;
  };
  int g0 = 0;
  {   // the last group that begins at or before byte lo
    int a = 0, b = p.n;
    while (b - a > 1) {
      const int m = (a + b) / 2;
      if (s_start[m] <= lo) a = m;
      else b = m;
    }
    g0 = a;
  }
#pragma unroll 1
  for (int gi = g0; gi < p.n && s_start[gi] < hi; ++gi) {
    const int a = row_at(gi, lo), b = row_at(gi, hi);
    if (a >= b) continue;   // (the same for the whole CTA)
    const WideGroup& w = p.table[gi];
    const GroupParams& g = w.g;
    const int d = g.d, k = g.k;
    const bool gated = s_gate[gi];
    float* y = w.io.y;
    __syncthreads();   // c of the group before is read
    for (int j = tid; j < k / 4; j += kT) reinterpret_cast<float4*>(s_c)[j] = __ldcg(reinterpret_cast<const float4*>(g.c) + j);
    __syncthreads();
    auto image = [&](int r0, int r1, float* to) {
      if (k <= 256) image_rows<1>(g, r0, r1, s_c, to, y);
      else if (k <= 512) image_rows<2>(g, r0, r1, s_c, to, y);
      else image_rows<kMaxVec>(g, r0, r1, s_c, to, y);
    };
    if (!gated) {
      image(a, b, nullptr);
      continue;
    }
    // W: teams of `ts` warps take a row at a time, each warp its share of the columns, whose r it keeps
    const int ts = (d + kTeamCols - 1) / kTeamCols, teams = kW / ts, team = warp / ts, part = warp % ts;
    const int c0 = part * kTeamCols + lane * 8;
    float4 r[4][2];
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        r[v][h] = team < teams && c0 + v * 256 < d ? __ldcg(reinterpret_cast<const float4*>(g.r + c0 + v * 256) + h)
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
    int j = 0;
#pragma unroll 1
    for (int r0 = a, r1; r0 < b; r0 = r1) {
      while (r0 >= g.off[j + 1]) ++j;
      r1 = min(min(b, r0 + kChunk), g.off[j + 1]);   // (rows of one map)
      const uint16_t* W = g.W[j] + (size_t)(r0 - g.off[j]) * d + c0;
      const int n = team < teams ? (r1 - r0 - team + teams - 1) / teams : 0;   // this team's rows (n <= 0: none)
      uint4 q[kAhead][4];
      auto load = [&](int i, uint4 (&to)[4]) {
#pragma unroll
        for (int v = 0; v < 4; ++v)
          to[v] = i < n && c0 + v * 256 < d
                      ? ld_stream(reinterpret_cast<const uint4*>(W + (size_t)(team + i * teams) * d + v * 256))
                      : make_uint4(0u, 0u, 0u, 0u);
      };
      if (lane < kAhead && lane < n) {   // the first rows are asked into the L2 beside the image
        const uint16_t* at = W - lane * 8 + (size_t)(team + lane * teams) * d;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(at), "r"((unsigned)min(kTeamCols, d - part * kTeamCols) * 2)
                     : "memory");
      }
      image(r0, r1, s_y);
#pragma unroll
      for (int e = 0; e < kAhead; ++e) load(e, q[e]);
#pragma unroll 1
      for (int i = 0; i < n; i += kAhead)
#pragma unroll
        for (int e = 0; e < kAhead; ++e) {
          float s = 0.f, t = 0.f;
          s = dot8(q[e][0], r[0][0], r[0][1], s);
          t = dot8(q[e][1], r[1][0], r[1][1], t);
          s = dot8(q[e][2], r[2][0], r[2][1], s);
          t = dot8(q[e][3], r[3][0], r[3][1], t);
          load(i + e + kAhead, q[e]);
          s = warp_sum(s + t);
          if (lane == 0 && i + e < n) s_part[(team + (i + e) * teams) * ts + part] = s;
        }
      __syncthreads();
      for (int row = r0 + tid; row < r1; row += kT) {
        float v = s_y[row - r0];
        for (int e = 0; e < ts; ++e) v += s_part[(row - r0) * ts + e];
        y[row] = v;
      }
      __syncthreads();
    }
  }
}

}  // namespace

cudaError_t launch_flat_step(const FlatParams& p, int grid, int most_k, cudaStream_t st) {
  const int smem1 = kW * most_k * 4;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_flat_project, cudaFuncAttributeMaxDynamicSharedMemorySize, smem1)) != cudaSuccess ||
      (e = launch_pdl(k_flat_project, dim3(grid), dim3(kT), smem1, st, p)) != cudaSuccess ||
      (e = launch_pdl(k_flat_residual, dim3(grid), dim3(kT), 0, st, p)) != cudaSuccess ||
      (e = launch_pdl(k_flat_rows, dim3(grid), dim3(kT), 0, st, p)) != cudaSuccess)
    return e;
  return cudaGetLastError();
}

}  // namespace gsi
