// Online extension of the basis by one vector (the paper's "time-dimension tracking",
// Section 5.4, and "online basis adaptation", Section 7.2): a token is tested against
// the basis in use; if rho = ||x - P P^T x|| / ||x|| exceeds a threshold, the residual,
// orthogonalised against P twice (Gram-Schmidt with one re-orthogonalisation, "DGKS") and
// normalised, becomes column k_active of P, and W times that column (Section 4.2) becomes
// column k_active of every cached image.  Columns [k_active, k) of P are zero before, so
// every other kernel of the library keeps working on the full width k.
//
// ONE cooperative launch (every CTA resident), CUDA-core FMAs in fp32, no host
// synchronisation; nearly every token ends after the first pass.
//
//   pass 1   c = P^T x, r1 = x - P c, rho
//   (rho <= tau, no free column or a non-finite token: done)
//   pass 2   c = P^T r1, r2 = r1 - P c, ||r2||
//   store    v = r2 / ||r2|| rounded to the basis type: column of P, of its transposed copy and
//            of the tiled copy; max|P|
//   image    W v for this CTA's rows: column of the image and of its tiled copy (FP8: the
//            sixteen-row blocks are quantised again, their scales may change)
//
// What bounds it: the chain of two exchanges per pass (words that carry their validity,
// gsi_exchange.cuh) and 2 MB of basis.  Before, fourteen launches whether a column was appended
// or not: 107 us for a token inside the subspace at 4096 x 256 and 28672 image rows, now 12.1 us a
// call (the kernel 9.5); with a column appended (235 MB of W) 168 us, now 78 us.
#include "gsi_exchange.cuh"
#include "gsi_pack.cuh"

namespace gsi {

namespace {

using namespace exchange;

constexpr int kT = 512, kW = kT / 32;
constexpr int kHoldOff = 400;  // cycles between a CTA's norm word and its first look at the others'
constexpr int kStage = 4096;   // floats of x, r1 or v in shared memory at a time

__device__ __forceinline__ uint16_t to_bf16_bits(float v) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  return *reinterpret_cast<const uint16_t*>(&h);
}

// Elements [i0, i0 + n) of a vector into shared memory, from plain floats or from tagged words.
__device__ __forceinline__ bool stage(float* s, const float* x, const unsigned long long* words, unsigned tag,
                                      unsigned limit, int i0, int n) {
  bool ok = true;
  for (int ib = 0; ib < n; ib += 8 * kT) {
    if (x) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = ib + (int)threadIdx.x + u * kT;
        if (i < n) s[i] = __ldg(x + i0 + i);
      }
    } else {
      const int first = ib + (int)threadIdx.x;
      const int cnt = n > first ? min(8, (n - first + kT - 1) / kT) : 0;
      ok = gather(words + i0 + first, kT, cnt, tag, limit, [&](int u, float v) { s[first + u * kT] = v; }) && ok;
    }
  }
  return ok;
}

template <int VPL, bool PF32>
__global__ void __launch_bounds__(kT, 1) k_extend(GroupParams g, ExtendArgs a, int n_slabs) {
  __shared__ float s_v[kStage];
  __shared__ __align__(8) float s_part[kW * kCols];
  __shared__ float s_c[1024];
  __shared__ float s_scale[16];
  __shared__ double s_norm[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, cta = blockIdx.x, d = g.d, k = g.k, KV = k / 8;
  const unsigned tag1 = first_tag(g.tickets);
  const int col = *a.k_active;
  const Area words = area_of(g);
  const int p0 = (int)((long long)d * cta / G), p1 = (int)((long long)d * (cta + 1) / G);
  const int n_cb = (k + kCols - 1) / kCols;
  int lpr = 1;
  while (lpr < KV && lpr < 32) lpr <<= 1;
  const int rpp = 32 / lpr, rsub = lane / lpr, cl = lane % lpr;
  auto give_up = [&](bool ok) -> bool {   // the same answer for every thread
    if (!__syncthreads_or(!ok)) return false;
    if (tid == 0) atomicExch(g.status, (int)GSI_ERR_TIMEOUT);
    if (tid == 0) leave_launch(g.tickets);
    return true;
  };

  if (cta == 0 && tid == 0) {   // what a call that gives up leaves
    if (a.appended_out) *a.appended_out = 0;
    if (a.rho_out) *a.rho_out = __int_as_float(0x7fc00000);
  }

  float inv = 0.f;
#pragma unroll 1
  for (int pass = 1; pass <= 2; ++pass) {
    const unsigned tag = tag1 + (unsigned)(pass - 1);
    bool ok = true;
    // partial c of a slab of rows x 32 columns
    for (int part = cta; part < n_slabs * n_cb; part += G) {   // (a small grid may have fewer CTAs than column blocks)
      const int slab = part / n_cb, cb = part % n_cb;
      const int r0 = (int)((long long)d * slab / n_slabs), r1 = (int)((long long)d * (slab + 1) / n_slabs);
      const int sub = lane >> 2, c = cb * kCols + (lane & 3) * 8;
      float acc[8], sx = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] = 0.f;
      for (int rb = r0; rb < r1; rb += kStage) {
        const int n = min(kStage, r1 - rb);
        __syncthreads();
        ok = stage(s_v, pass == 1 ? a.x : nullptr, words.ext_r, tag1, g.spin_limit, rb, n) && ok;
        __syncthreads();
        for (int base = warp * 8 + sub; base < n; base += kW * 8 * 4) {
          float p[4][8];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = base + u * kW * 8;
#pragma unroll
            for (int e = 0; e < 8; ++e) p[u][e] = 0.f;
            if (i < n && c < k) load8<PF32>(g.P, (size_t)(rb + i) * KV + c / 8, p[u]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = base + u * kW * 8;
            const float v = i < n ? s_v[i] : 0.f;
            sx = fmaf(v, v, sx);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] = fmaf(p[u][e], v, acc[e]);
          }
        }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e)
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) sx += __shfl_xor_sync(0xffffffffu, sx, o);
      if (lane < 4)
#pragma unroll
        for (int e = 0; e < 8; ++e) s_part[warp * kCols + lane * 8 + e] = acc[e];
      if (lane == 0) s_c[warp] = sx;
      __syncthreads();
      if (tid < kCols) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kW; ++w) s += s_part[w * kCols + tid];
        if (cb * kCols + tid < k) put(words.c + (size_t)slab * k + cb * kCols + tid, s, tag);
      } else if (pass == 1 && tid == kCols && cb == 0) {   // (pass 2 needs no ||x||^2)
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kW; ++w) s += s_c[w];
        put(words.ext_x2 + slab, s, tag);
      }
      __syncthreads();
    }
    // c: every CTA adds all partials in slab order
    for (int j = tid; j < k; j += kT) {
      float s = 0.f;
      ok = gather(words.c + j, k, n_slabs, tag, g.spin_limit, [&](int, float v) { s += v; }) && ok;
      s_c[j] = s;
    }
    if (give_up(ok)) return;
    // this CTA's rows of the residual
    float c8[VPL][8], sr = 0.f;
    double sr2 = 0.0;   // pass 2: the column is divided by this norm, whatever the scale of x (squares of 1e-21 are not fp32 numbers)
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
      for (int e = 0; e < 8; ++e) c8[v][e] = cl + v * lpr < KV ? s_c[(cl + v * lpr) * 8 + e] : 0.f;
    for (int base = p0 + warp * rpp; base < p1; base += kW * rpp) {
      const int row = base + rsub;
      float dot = 0.f;
      if (row < p1) {
#pragma unroll
        for (int v = 0; v < VPL; ++v)
          if (cl + v * lpr < KV) {
            float p8[8];
            load8<PF32>(g.P, (size_t)row * KV + cl + v * lpr, p8);
#pragma unroll
            for (int e = 0; e < 8; ++e) dot = fmaf(p8[e], c8[v][e], dot);
          }
      }
      for (int o = lpr >> 1; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
      if (row < p1 && cl == 0) {
        const float rv = (pass == 1 ? __ldg(a.x + row) : g.r[row]) - dot;   // (g.r: written here in pass 1)
        g.r[row] = rv;
        if (pass == 1) put(words.ext_r + row, rv, tag);
        if (pass == 1) sr = fmaf(rv, rv, sr);
        else sr2 = fma((double)rv, (double)rv, sr2);
      }
    }
    // (each pass has norm words of its own: the first CTAs are done with pass 1, and at those of pass 2,
    // while a late one may still read)
    if (pass == 1) {
      sr = warp_sum(sr);
      if (lane == 0) s_part[warp] = sr;
      __syncthreads();
      if (tid == 0) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kW; ++w) s += s_part[w];
        put(words.ext_r2 + cta, s, tag);
      }
    } else {
      double* s_part2 = reinterpret_cast<double*>(s_part);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sr2 += __shfl_xor_sync(0xffffffffu, sr2, o);
      if (lane == 0) s_part2[warp] = sr2;
      __syncthreads();
      if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < kW; ++w) s += s_part2[w];
        put128(words.ext_r2d + cta, (uint32_t)__double2loint(s), (uint32_t)__double2hiint(s), 0u, tag);
      }
    }
    if (pass == 2) {
      if (warp == 0) {
        double s = 0.0;
        const int mine = G > lane ? (G - lane + 31) / 32 : 0;
        ok = gather128([&](int u) { return words.ext_r2d + lane + 32 * u; }, mine, tag, g.spin_limit,
                       [&](int, const Word128& w) { s += __hiloint2double((int)w.b, (int)w.a); });
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) s_norm[0] = s;
      }
    } else if (warp < 2) {
      // (First polls that arrive ahead of the words hold them up: all CTAs read the same few lines.  Asking
      // at once, this exchange took 1.7 or 2.7 to 4 us, by where the words lie in memory.)
      for (const long long t0 = clock64(); clock64() - t0 < kHoldOff;) {}
      double s = 0.0;
      ok = warp ? warp_gather_sum(words.ext_x2, 1, n_slabs, tag, g.spin_limit, s) : warp_gather_sum(words.ext_r2, 1, G, tag, g.spin_limit, s);
      if (lane == 0) s_norm[warp] = s;
    }
    if (give_up(ok)) return;
    // the same sums in the same order on every CTA: the same decision
    bool go;
    if (pass == 1) {
      const float rho = (float)(sqrt(s_norm[0]) / sqrt(s_norm[1]));
      // rho > tau is false for NaN: a non-finite token never extends the basis
      go = rho > a.tau && col >= 0 && col < k;
      if (cta == 0 && tid == 0 && a.rho_out) *a.rho_out = rho;
    } else {
      go = s_norm[0] > 0.0 && s_norm[0] < 1e300;
      inv = go ? (float)(1.0 / sqrt(s_norm[0])) : 0.f;
    }
    if (!go || pass == 2) {
      if (cta == 0 && tid == 0) {
        if (a.appended_out) *a.appended_out = go ? 1 : 0;
        if (go) *a.k_active = col + 1;   // (every CTA has read it: its norms are here)
      }
      if (!go) {
        if (tid == 0) leave_launch(g.tickets);
        return;
      }
    }
    __syncthreads();
  }

  // ---- store: the image column is W times what the basis really holds
  const unsigned tag = tag1 + 2u;
  float m = 0.f;
  for (int i = p0 + tid; i < p1; i += kT) {
    const float v = g.r[i] * inv;
    float stored = v;
    if constexpr (PF32) {
      const_cast<float*>(static_cast<const float*>(g.P))[(size_t)i * k + col] = v;
    } else {
      const uint16_t b = to_bf16_bits(v);
      const_cast<uint16_t*>(static_cast<const uint16_t*>(g.P))[(size_t)i * k + col] = b;
      if (a.PT) a.PT[(size_t)col * d + i] = b;
      if (a.P16) a.P16[pack::t16_slot(i, col, k)] = b;
      stored = __uint_as_float((uint32_t)b << 16);
    }
    put(words.ext_r + i, stored, tag);
    m = fmaxf(m, fabsf(stored));
  }
  if (a.pmax) {   // non-negative floats order like their bit patterns
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0 && m > 0.f) atomicMax(reinterpret_cast<int*>(a.pmax), __float_as_int(m));
  }

  // ---- image: blocks of sixteen rows, a row per warp, four 16-byte loads of W in flight per lane
  const int blocks = (g.O + 15) / 16;
  const int o0 = (int)((long long)blocks * cta / G) * 16;
  const int o1 = min(g.O, (int)((long long)blocks * (cta + 1) / G) * 16);
  uint16_t* WP = const_cast<uint16_t*>(g.WP);
  for (int c0 = 0; c0 < d; c0 += kStage) {
    const int n = min(kStage, d - c0);
    const bool last = c0 + n == d;
    __syncthreads();
    if (give_up(stage(s_v, nullptr, words.ext_r, tag, g.spin_limit, c0, n))) return;
    for (int row = o0 + warp; row < o1; row += kW) {
      int j = 0;
      while (j + 1 < g.n_maps && row >= g.off[j + 1]) ++j;
      const uint4* w = reinterpret_cast<const uint4*>(g.W[j] + (size_t)(row - g.off[j]) * d + c0);
      float s = 0.f;
      for (int v0 = lane; v0 < n / 8; v0 += 4 * 32) {
        uint4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          q[u] = v0 + 32 * u < n / 8 ? ld_stream(w + v0 + 32 * u) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (v0 + 32 * u < n / 8) {
            float f[8];
            unpack_bf16x8(q[u], f);
            const float4* x4 = reinterpret_cast<const float4*>(s_v + (v0 + 32 * u) * 8);
            const float4 lo = x4[0], hi = x4[1];
            s = fmaf(f[0], lo.x, s); s = fmaf(f[1], lo.y, s); s = fmaf(f[2], lo.z, s); s = fmaf(f[3], lo.w, s);
            s = fmaf(f[4], hi.x, s); s = fmaf(f[5], hi.y, s); s = fmaf(f[6], hi.z, s); s = fmaf(f[7], hi.w, s);
          }
      }
      s = warp_sum(s);
      if (lane == 0) {
        if (c0 > 0) s += a.y_scratch[row];
        if (!last) {
          a.y_scratch[row] = s;
        } else {
          const uint16_t b = to_bf16_bits(s);
          WP[(size_t)row * k + col] = b;
          if (a.WP16) a.WP16[pack::t16_slot(row, col, k)] = b;
        }
      }
    }
  }
  if (tid == 0) leave_launch(g.tickets);
  if (a.WP8) {
    __syncthreads();   // the column is in this CTA's rows
    for (int R = o0 / 16; R * 16 < o1; ++R) {
      pack::fp8_rows16(WP, g.O, k, a.WP8, R, s_scale);
      __syncthreads();
    }
  }
}

template <int VPL>
cudaError_t launch_t(GroupParams g, ExtendArgs a, int slabs, int grid, cudaStream_t st) {
  void* args[] = {&g, &a, &slabs};
  return g.p_f32 ? cudaLaunchCooperativeKernel((void*)k_extend<VPL, true>, dim3(grid), dim3(kT), args, 0, st)
                 : cudaLaunchCooperativeKernel((void*)k_extend<VPL, false>, dim3(grid), dim3(kT), args, 0, st);
}

}  // namespace

cudaError_t launch_extend_basis(const GroupParams& g, const ExtendArgs& a, cudaStream_t st) {
  return launch_resident([&](int grid) -> cudaError_t {
    const int slabs = fused_slabs(g.d, g.k, grid);
    return g.k <= 256   ? launch_t<1>(g, a, slabs, grid, st)
           : g.k <= 512 ? launch_t<2>(g, a, slabs, grid, st)
                        : launch_t<4>(g, a, slabs, grid, st);
  });
}

}  // namespace gsi
