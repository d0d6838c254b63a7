// C ABI of the gated subspace layer: argument checking, workspace layout,
// handle and stack bookkeeping, kernel sequencing.  No arithmetic lives here.
#include <chrono>
#include <cmath>
#include <algorithm>
#include <new>
#include <vector>
#include <cstring>

#include "gsi_common.cuh"
#include "gsi_umma.cuh"
#include "gsi_persistent.cuh"
#include "gsi_flat.cuh"

using namespace gsi;

namespace {

constexpr size_t kAlign = 256;
constexpr int kSlabTarget = 148;  // one basis slab per SM of a B200

inline size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

struct Layout {
  size_t wp, c, cpart, r, normpart, ctrl, fired, rho, x_stage, y_stage, gate_stage, rho_stage,
      pk_acc, pk_slot, tc_rb, tc_ypart, f_pt, f_xb, f_cb, f_cpart, f_normpart, pk_pp, pk_wpp, fused, total;
  int O, n_slabs, slab_rows;
  bool tc, front, dense_tc, packed;
};

constexpr int kTcMinFired = 5;  // fewer fired tokens: one pass of the CUDA-core GEMV
constexpr double kOwnStreamBytes = 262144.0;   // W rows of a CTA up to which a gated residual stays on its group's share
constexpr int kChains = 2;   // chains of a batched step side by side
constexpr int kMaxSegments = 12;   // of a step with host buffers
// Batched stacks of fewer groups keep a chain of launches per group (one GPT-J layer, three groups, 64 tokens, a
// tenth gated: 134 us against 152 in five launches; four groups, one GPT-2 layer 60 against 45, one OPT layer at 8
// tokens 123 against 117, at 33 139 against 143, but 117 against 104 with 1 % gated).
constexpr int kWideMinGroups = 4;
// Single-token stacks that step in three launches (gsi_flat.cu) instead of the persistent kernel: groups enough
// for their phases to add up, images that are small per group, bases that stay in the L2 (us a step,
// persistent / three launches: 12 GPT-2 layers, k = 128, 70 % gated 120 / 51, k = 512 126 / 70; two layers, eight
// groups, 39.5 / 29.8, 1 % gated 23.0 / 22.7; OPT layers, k = 128, images of 2.4 MB, a tenth gated, two 42.6 / 38.0, 12
// 160 / 147; k = 256, 4.7 MB, six layers 99 / 102, 1 % gated 71 / 73.  Between the two lines lie GPT-J layers at k = 128,
// 3.1 MB, three 57.9 / 52.6, 14 165 / 154).
constexpr int kFlatMinGroups = 8;
constexpr double kFlatBasisBytes = 96.0e6, kFlatImageBytes = 3.0e6;
constexpr int kWideGemmSlots = 296;   // blocks of the contraction that are resident at a time
constexpr int kWideBlocks = 592;   // projection blocks of a wide step: two waves of two per SM
constexpr int kFrontMinTokens = 2;  // single-token calls never take the tcgen05 front end (nor small ones: takes_fused)

bool tc_shapes_ok(const gsi_desc_t* d) {
  for (int j = 0; j < d->n_maps; ++j)
    if (d->d_out[j] % 128) return false;
  return true;
}

gsi_status_t check_desc(const gsi_desc_t* d) {
  if (!d || !d->d_out) return GSI_ERR_INVALID_ARG;
  if (d->d <= 0 || d->n_maps <= 0 || d->max_tokens <= 0) return GSI_ERR_INVALID_ARG;
  if (d->n_maps > GSI_MAX_MAPS || d->max_tokens > GSI_MAX_TOKENS) return GSI_ERR_UNSUPPORTED;
  if (d->p_dtype != GSI_BF16 && d->p_dtype != GSI_F32) return GSI_ERR_INVALID_ARG;
  if (d->d % 8) return GSI_ERR_UNSUPPORTED;
  for (int j = 0; j < d->n_maps; ++j) {
    if (d->d_out[j] <= 0) return GSI_ERR_INVALID_ARG;
    if (d->d_out[j] % 8) return GSI_ERR_UNSUPPORTED;
  }
  if ((d->flags & GSI_FLAG_FP8_IMAGE) && (d->flags & GSI_FLAG_DENSE)) return GSI_ERR_INVALID_ARG;
  if (!(d->flags & GSI_FLAG_DENSE)) {
    if (d->k <= 0) return GSI_ERR_INVALID_ARG;
    if (d->k % 8 || d->k > 1024 || d->k > d->d) return GSI_ERR_UNSUPPORTED;
    if (!(d->eps >= 0.f)) return GSI_ERR_INVALID_ARG;  // also rejects NaN
  }
  return GSI_OK;
}

Layout make_layout_ws(const gsi_desc_t* d) {
  Layout L{};
  const bool dense = d->flags & GSI_FLAG_DENSE;
  const size_t B = d->max_tokens, k = dense ? 0 : d->k;
  int O = 0;
  for (int j = 0; j < d->n_maps; ++j) O += d->d_out[j];
  L.O = O;
  int slab = (d->d + kSlabTarget - 1) / kSlabTarget;
  if (slab < 8) slab = 8;
  L.slab_rows = slab;
  L.n_slabs = (d->d + slab - 1) / slab;
  size_t at = 0;
  auto take = [&](size_t bytes) { size_t o = at; at += align_up(bytes); return o; };
  L.wp = take((size_t)O * k * 2);
  L.c = take(B * k * 4);
  L.cpart = take((size_t)L.n_slabs * B * k * 4);
  L.r = take(dense ? 0 : B * d->d * 4);
  L.normpart = take((size_t)L.n_slabs * B * 2 * 4);
  L.ctrl = take(256);
  L.fired = take(B * 4);
  L.rho = take(B * 4);
  L.x_stage = take(B * d->d * 4);
  L.y_stage = take(B * (size_t)O * 4);
  L.gate_stage = take(B);
  L.rho_stage = take(B * 4);
  L.pk_acc = take(2 * (k + 4) * 8);                 // persistent kernel: accumulators of c, ||x||^2, ||r||^2
  L.pk_slot = take((size_t)kPersistMaxGrid * 8);    // persistent kernel: tagged max|x| words, published ||x||^2
  // tensor-core kernels: batched handles only
  const bool tc_any = d->max_tokens >= kFrontMinTokens && d->d % 64 == 0 && tc_shapes_ok(d);
  const bool tc = !dense && tc_any;
  const bool dense_tc = dense && tc_any;   // the dense baseline of batched calls, same tile routine
  L.tc_rb = take(tc_any ? (size_t)65 * d->d * 2 : 0);   // row 64 stays zero
  L.tc_ypart = take(tc_any && tc_partials(O, d->d, dense) ? (size_t)tc_splits(O, d->d) * 64 * O * 4 : 0);
  L.tc = tc;
  L.dense_tc = dense_tc;
  // tensor-core projection / residual / image for batched calls
  const bool front = tc && d->max_tokens >= kFrontMinTokens && d->p_dtype == GSI_BF16 && d->k % 128 == 0 &&
                     d->d % 128 == 0 && O % 128 == 0;
  const size_t rows = front ? front_rows(d->max_tokens) : 0;
  L.f_pt = take(front ? (size_t)d->k * d->d * 2 : 0);
  L.f_xb = take(rows * d->d * 2);
  L.f_cb = take(rows * k * 2);
  L.f_cpart = take(front ? (size_t)front_proj_splits(d->d, d->k) * B * k * 4 : 0);
  L.f_normpart = take(front ? (size_t)(d->d / 128) * B * 2 * 4 : 0);
  L.front = front;
  // persistent kernel: the basis and the images once more, as 16 x 16 tiles in the operand
  // order of the tensor-core instruction (rows padded to a multiple of 16)
  const bool packed = !dense && d->p_dtype == GSI_BF16 && d->k >= 64 && d->k <= 512 &&
                      (d->k & (d->k - 1)) == 0 && d->max_tokens <= kPersistMaxTokens;
  L.pk_pp = take(packed ? (size_t)((d->d + 15) / 16 * 16) * k * 2 : 0);
  L.pk_wpp = take(packed ? (size_t)((O + 15) / 16) * persist_image_row_bytes(d->k, d->flags & GSI_FLAG_FP8_IMAGE) : 0);
  L.packed = packed;
  L.fused = take(dense ? 0 : fused_words_bytes(d->d, d->k, d->max_tokens));
  L.total = at;
  return L;
}

}  // namespace

struct gsi_layer {
  gsi_desc_t desc;
  int d_out[GSI_MAX_MAPS];
  Layout lay;
  GroupParams gp;
  TmaMaps tm;          // tensor maps of the tensor-core kernels' operands
  bool has_tm = false;
  char* ws;
  float* pmax;     // device: max |P| (bf16 basis only)
  unsigned* bar;   // device: [2] barrier counters of the persistent kernel
  cudaStream_t last_stream;
};

struct gsi_stack {
  int mode;                 // 0 auto, 1 generic kernels, 2 persistent kernel required
  bool persistent;          // the persistent kernel is in use
  int grid;                 // CTAs of the persistent kernel (= SMs)
  bool has_pairs;           // some phase of the persistent schedule holds several groups
  int common_k;             // rank shared by every gated group of the persistent schedule, or 0
  PersistGroup* dev_groups; // device table
  int* dev_phase_first;     // device: first group of every phase of the persistent schedule
  int n_phases;
  std::vector<int> host_phase_first;
  unsigned spin_limit;      // polls a cross-CTA wait of the persistent kernel may take
  std::vector<PersistGroup> host_groups;
  std::vector<const float*> host_pmax_ptrs;
  int* epoch;               // device
  int* status;              // device
  unsigned long long* trace; // device, optional
  std::vector<gsi_layer*> groups;
  std::vector<char> pair_first;   // group i and i+1 declared independent of each other
  std::vector<gsi_stack_io_t> io;
  int B;
  int n_steps;
  unsigned char* gate_log;
  float* rho_log;
  int* step;  // device
  bool bound;
  int seek_value;
  cudaStream_t last_stream;
  // per-stage / batched path: the second group of a concurrent pair runs on a stream of
  // the stack's own, forked from and joined to the caller's stream by events
  cudaStream_t aux = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  // batched steps: the chains of small kernels (projection, residual, gate, image) run on two
  // streams of the stack's own with the highest priority; the gated-residual contractions stay
  // on the caller's stream: a contraction is ordered behind its group's gate by an event and
  // runs beside the chains of the groups that follow (inputs are staged before the step).
  // alternate: small maps, where a step is the latency of its chains: those of consecutive groups
  // on alternating streams (GPT-2 at 8 tokens, a quarter gated: 0.76 -> 0.55 ms).  With large
  // maps the W stream sets the time, and a second chain only takes its SM slots (OPT at 64
  // tokens 0.93 -> 1.02 ms for six layers): there it is for the second group of a declared pair.
  cudaStream_t front[kChains] = {};
  bool alternate = false;
  // steps with host buffers: the groups in up to kMaxSegments segments, whose inputs, work and
  // outputs overlap (a copy stream per direction); segment i begins with group (persistent
  // schedule: phase) segment[i]
  std::vector<int> segment;
  cudaStream_t copy_in = nullptr, copy_out = nullptr;
  cudaEvent_t ev_begin = nullptr, ev_in[kMaxSegments] = {}, ev_run[kMaxSegments] = {};
  cudaEvent_t ev_resid = nullptr, ev_front_fork = nullptr, ev_front_join = nullptr;
  // batched steps in five launches over all groups (WideParams): the table, and for the whole step
  // and for every segment the blocks before each group
  struct WideRange {
    int g0, g1;
    const int *first, *order;   // device
    int blocks[kWideStages];
    int splits;                 // of the depth, in the contraction
  };
  char* wide_area;           // device, null when the workspace has no room for it
  bool wide = false;
  int wide_k = 0;            // the largest rank
  std::vector<WideRange> wide_ranges;
  std::vector<WideGroup> wide_table;
  std::vector<int> wide_ints;
  // single-token steps of small groups in three launches (gsi_flat.cu): table and shares in the same area
  bool flat = false;
  int flat_grid = 0, flat_k = 0;
  FlatParams flat_params;
  ~gsi_stack() {
    if (ev_fork) cudaEventDestroy(ev_fork);
    if (ev_join) cudaEventDestroy(ev_join);
    if (aux) cudaStreamDestroy(aux);
    if (ev_resid) cudaEventDestroy(ev_resid);
    if (ev_front_fork) cudaEventDestroy(ev_front_fork);
    if (ev_front_join) cudaEventDestroy(ev_front_join);
    for (cudaStream_t f : front)
      if (f) cudaStreamDestroy(f);
    if (copy_in) cudaStreamDestroy(copy_in);
    if (copy_out) cudaStreamDestroy(copy_out);
    if (ev_begin) cudaEventDestroy(ev_begin);
    for (cudaEvent_t e : ev_in)
      if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : ev_run)
      if (e) cudaEventDestroy(e);
  }
};

// The tiled copies of the basis and of the images that the persistent kernel streams.
static bool repack(gsi_layer* h, cudaStream_t stream) {
  const Layout& L = h->lay;
  if (launch_pack_t16(h->gp.P, h->desc.d, h->desc.k, h->ws + L.pk_pp, stream) != cudaSuccess) return false;
  return ((h->desc.flags & GSI_FLAG_FP8_IMAGE)
              ? launch_pack_t16_fp8(h->ws + L.wp, L.O, h->desc.k, h->ws + L.pk_wpp, stream)
              : launch_pack_t16(h->ws + L.wp, L.O, h->desc.k, h->ws + L.pk_wpp, stream)) == cudaSuccess;
}

extern "C" {

const char* gsi_status_string(gsi_status_t s) {
  switch (s) {
    case GSI_OK: return "ok";
    case GSI_ERR_INVALID_ARG: return "invalid argument";
    case GSI_ERR_UNSUPPORTED: return "unsupported shape";
    case GSI_ERR_ALLOC: return "host allocation failed";
    case GSI_ERR_CUDA: return "CUDA runtime error";
    case GSI_ERR_TIMEOUT: return "device-side wait timed out";
    case GSI_ERR_WORKSPACE: return "workspace too small";
  }
  return "unknown status";
}

gsi_status_t gsi_build_image(const void* W, const void* P, int o, int d, int k,
                             gsi_dtype_t p_dtype, void* W_P_out, gsi_stream_t stream) {
  if (!W || !P || !W_P_out || o <= 0 || d <= 0 || k <= 0) return GSI_ERR_INVALID_ARG;
  if (p_dtype != GSI_BF16 && p_dtype != GSI_F32) return GSI_ERR_INVALID_ARG;
  if (!aligned16(W) || !aligned16(P) || !aligned16(W_P_out)) return GSI_ERR_INVALID_ARG;
  if (o % 8 || d % 8 || k % 8) return GSI_ERR_UNSUPPORTED;
  return launch_build_image(W, P, o, d, k, p_dtype == GSI_F32, W_P_out, nullptr, stream) == cudaSuccess
             ? GSI_OK
             : GSI_ERR_CUDA;
}

size_t gsi_workspace_bytes(const gsi_desc_t* desc) {
  if (check_desc(desc) != GSI_OK) return 0;
  return make_layout_ws(desc).total;
}

gsi_status_t gsi_create(const gsi_desc_t* desc, const void* const* W, const void* P,
                        void* workspace, size_t workspace_bytes, gsi_stream_t stream,
                        gsi_handle_t* out) {
  if (!out) return GSI_ERR_INVALID_ARG;
  *out = nullptr;
  gsi_status_t st = check_desc(desc);
  if (st != GSI_OK) return st;
  const bool dense = desc->flags & GSI_FLAG_DENSE;
  if (!W || !workspace || (!dense && !P)) return GSI_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(workspace) % kAlign) || (P && !aligned16(P)))
    return GSI_ERR_INVALID_ARG;
  for (int j = 0; j < desc->n_maps; ++j)
    if (!W[j] || !aligned16(W[j])) return GSI_ERR_INVALID_ARG;
  Layout L = make_layout_ws(desc);
  if ((desc->flags & GSI_FLAG_FP8_IMAGE) && !L.packed) return GSI_ERR_UNSUPPORTED;   // the persistent kernel alone reads FP8 images
  if (workspace_bytes < L.total) return GSI_ERR_WORKSPACE;

  gsi_layer* h = new (std::nothrow) gsi_layer();
  if (!h) return GSI_ERR_ALLOC;
  h->desc = *desc;
  std::memcpy(h->d_out, desc->d_out, sizeof(int) * desc->n_maps);
  h->desc.d_out = h->d_out;
  h->lay = L;
  h->ws = static_cast<char*>(workspace);
  h->last_stream = stream;

  GroupParams& g = h->gp;
  std::memset(&g, 0, sizeof g);
  g.d = desc->d;
  g.k = dense ? 8 : desc->k;
  g.O = L.O;
  g.B = desc->max_tokens;
  g.p_f32 = desc->p_dtype == GSI_F32;
  g.eps = desc->eps;
  g.flags = desc->flags;
  g.P = P;
  g.WP = reinterpret_cast<const uint16_t*>(h->ws + L.wp);
  g.n_maps = desc->n_maps;
  int off = 0;
  for (int j = 0; j < desc->n_maps; ++j) {
    g.W[j] = static_cast<const uint16_t*>(W[j]);
    g.d_out[j] = desc->d_out[j];
    g.off[j] = off;
    off += desc->d_out[j];
  }
  g.off[desc->n_maps] = off;
  g.c = reinterpret_cast<float*>(h->ws + L.c);
  g.cpart = reinterpret_cast<float*>(h->ws + L.cpart);
  g.r = reinterpret_cast<float*>(h->ws + L.r);
  g.normpart = reinterpret_cast<float*>(h->ws + L.normpart);
  int* ctrl = reinterpret_cast<int*>(h->ws + L.ctrl);
  g.n_fired = ctrl + 0;
  g.counter = reinterpret_cast<unsigned*>(ctrl + 1);
  g.status = ctrl + 2;
  g.fired = reinterpret_cast<int*>(h->ws + L.fired);
  g.rho_scratch = reinterpret_cast<float*>(h->ws + L.rho);
  g.n_slabs = L.n_slabs;
  g.slab_rows = L.slab_rows;
  g.tc_min_fired = L.tc ? kTcMinFired : 0;
  g.rb = reinterpret_cast<uint16_t*>(h->ws + L.tc_rb);
  g.ypart = reinterpret_cast<float*>(h->ws + L.tc_ypart);
  g.front_min_tokens = (L.front || L.dense_tc) ? kFrontMinTokens : 0;
  g.proj_splits = L.front ? front_proj_splits(desc->d, desc->k) : 0;
  g.PT = reinterpret_cast<const uint16_t*>(h->ws + L.f_pt);
  g.xb = reinterpret_cast<uint16_t*>(h->ws + L.f_xb);
  g.cb = reinterpret_cast<uint16_t*>(h->ws + L.f_cb);
  g.cpart3 = reinterpret_cast<float*>(h->ws + L.f_cpart);
  g.normpart3 = reinterpret_cast<float*>(h->ws + L.f_normpart);
  g.fused_words = reinterpret_cast<unsigned long long*>(h->ws + L.fused);
  g.tickets = reinterpret_cast<unsigned long long*>(ctrl + 32);
  g.spin_limit = kFusedSpinLimit;
  g.area_B = g.B;
  g.area_k = g.k;
  g.area_d = g.d;

  if (L.tc || L.dense_tc) {
    if (!build_tma_maps(g, L.front, desc->max_tokens, &h->tm)) {
      delete h;
      return GSI_ERR_CUDA;
    }
    h->has_tm = true;
  }

  const auto begin = std::chrono::steady_clock::now();
  if (cudaMemsetAsync(ctrl, 0, 256, stream) != cudaSuccess ||
      cudaMemsetAsync(h->ws + L.pk_acc, 0, L.total - L.pk_acc, stream) != cudaSuccess) {
    delete h;
    return GSI_ERR_CUDA;
  }
  h->pmax = reinterpret_cast<float*>(ctrl + 8);
  h->bar = reinterpret_cast<unsigned*>(ctrl + 16);
  if (!dense && !g.p_f32 &&
      launch_abs_max_bf16(P, (size_t)desc->d * desc->k, h->pmax, stream) != cudaSuccess) {
    delete h;
    return GSI_ERR_CUDA;
  }
  if (L.front &&
      launch_transpose_bf16(P, desc->d, desc->k, h->ws + L.f_pt, stream) != cudaSuccess) {
    delete h;
    return GSI_ERR_CUDA;
  }
  if (!dense) {
    for (int j = 0; j < desc->n_maps; ++j) {
      void* dst = h->ws + L.wp + (size_t)g.off[j] * desc->k * 2;
      if (launch_build_image(W[j], P, desc->d_out[j], desc->d, desc->k, g.p_f32, dst, g.status, stream) !=
          cudaSuccess) {
        delete h;
        return GSI_ERR_CUDA;
      }
    }
  }
  if (L.packed && !repack(h, stream)) {
    delete h;
    return GSI_ERR_CUDA;
  }
  // A set-up call: return only when the images, max|P| and the cleared state are in
  // place, so the handle may be used from any stream afterwards.
  // A wait of the image kernel that runs out takes 2^22 polls of twenty cycles at least, 43 ms: the
  // status word (10 us to read) is looked at when the work took long enough to hold one.
  int status = 0;
  if (cudaStreamSynchronize(stream) != cudaSuccess ||
      (std::chrono::steady_clock::now() - begin > std::chrono::milliseconds(20) &&
       cudaMemcpy(&status, g.status, sizeof status, cudaMemcpyDeviceToHost) != cudaSuccess) ||
      status != 0) {
    delete h;
    return status ? (gsi_status_t)status : GSI_ERR_CUDA;   // (an image with a tile that was given up)
  }
  *out = h;
  return GSI_OK;
}

gsi_status_t gsi_forward_n(gsi_handle_t h, const float* x, int n_tokens, float* y,
                           unsigned char* gate_mask_out, float* rho_out, gsi_stream_t stream) {
  if (!h || n_tokens < 0 || n_tokens > h->desc.max_tokens) return GSI_ERR_INVALID_ARG;
  if (h->desc.flags & GSI_FLAG_FP8_IMAGE) return GSI_ERR_UNSUPPORTED;   // stacks on the persistent kernel only
  if (n_tokens == 0) return GSI_OK;
  if (!x || !y || !gate_mask_out) return GSI_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(y)) return GSI_ERR_INVALID_ARG;
  IoRef io{};
  io.x = x;
  io.y = y;
  io.gate = gate_mask_out;
  io.rho = rho_out;
  io.step = nullptr;
  io.n_steps = 1;
  h->last_stream = stream;
  return launch_generic_forward(h->gp, h->has_tm ? &h->tm : nullptr, io, n_tokens, stream, nullptr) == cudaSuccess ? GSI_OK
                                                                                      : GSI_ERR_CUDA;
}

gsi_status_t gsi_forward(gsi_handle_t h, const float* x, float* y, unsigned char* gate_mask_out,
                         gsi_stream_t stream) {
  if (!h) return GSI_ERR_INVALID_ARG;
  return gsi_forward_n(h, x, h->desc.max_tokens, y, gate_mask_out, nullptr, stream);
}

gsi_status_t gsi_forward_host(gsi_handle_t h, const float* x_host, int n_tokens, float* y_host,
                              unsigned char* gate_mask_host, float* rho_host,
                              gsi_stream_t stream) {
  if (!h || n_tokens < 0 || n_tokens > h->desc.max_tokens) return GSI_ERR_INVALID_ARG;
  if (n_tokens == 0) return GSI_OK;
  if (!x_host || !y_host || !gate_mask_host) return GSI_ERR_INVALID_ARG;
  const Layout& L = h->lay;
  float* xs = reinterpret_cast<float*>(h->ws + L.x_stage);
  float* ys = reinterpret_cast<float*>(h->ws + L.y_stage);
  unsigned char* gs = reinterpret_cast<unsigned char*>(h->ws + L.gate_stage);
  float* rs = reinterpret_cast<float*>(h->ws + L.rho_stage);
  const size_t n = n_tokens;
  if (cudaMemcpyAsync(xs, x_host, n * h->desc.d * 4, cudaMemcpyHostToDevice, stream) != cudaSuccess)
    return GSI_ERR_CUDA;
  gsi_status_t st = gsi_forward_n(h, xs, n_tokens, ys, gs, rs, stream);
  if (st != GSI_OK) return st;
  // rows of y are contiguous because the device buffer is [n][O] for any n
  if (cudaMemcpyAsync(y_host, ys, n * L.O * 4, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaMemcpyAsync(gate_mask_host, gs, n, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
    return GSI_ERR_CUDA;
  if (rho_host &&
      cudaMemcpyAsync(rho_host, rs, n * 4, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
    return GSI_ERR_CUDA;
  return cudaStreamSynchronize(stream) == cudaSuccess ? GSI_OK : GSI_ERR_CUDA;
}

gsi_status_t gsi_extend_basis(gsi_handle_t h, const float* x, float tau, int* k_active,
                              int* appended_out, float* rho_out, gsi_stream_t stream) {
  if (!h || !x || !k_active || !aligned16(x) || !(tau >= 0.f)) return GSI_ERR_INVALID_ARG;
  if (h->desc.flags & GSI_FLAG_DENSE) return GSI_ERR_UNSUPPORTED;
  const Layout& L = h->lay;
  const bool fp8 = h->desc.flags & GSI_FLAG_FP8_IMAGE;
  ExtendArgs a{};
  a.x = x;
  a.tau = tau;
  a.k_active = k_active;
  a.appended_out = appended_out;
  a.rho_out = rho_out;
  a.y_scratch = reinterpret_cast<float*>(h->ws + L.y_stage);
  a.pmax = h->gp.p_f32 ? nullptr : h->pmax;
  a.PT = L.front ? const_cast<uint16_t*>(h->gp.PT) : nullptr;
  if (L.packed) {
    a.P16 = reinterpret_cast<uint16_t*>(h->ws + L.pk_pp);
    if (fp8) a.WP8 = reinterpret_cast<unsigned char*>(h->ws + L.pk_wpp);
    else a.WP16 = reinterpret_cast<uint16_t*>(h->ws + L.pk_wpp);
  }
  h->last_stream = stream;
  return launch_extend_basis(h->gp, a, stream) == cudaSuccess ? GSI_OK : GSI_ERR_CUDA;
}

gsi_status_t gsi_get_image(gsi_handle_t h, int map, const void** out) {
  if (!h || !out || map < 0 || map >= h->desc.n_maps) return GSI_ERR_INVALID_ARG;
  if (h->desc.flags & GSI_FLAG_DENSE) return GSI_ERR_UNSUPPORTED;
  *out = h->ws + h->lay.wp + (size_t)h->gp.off[map] * h->desc.k * 2;
  return GSI_OK;
}

gsi_status_t gsi_get_image_fp8(gsi_handle_t h, const void** out, size_t* bytes_out) {
  if (!h || !out || !bytes_out) return GSI_ERR_INVALID_ARG;
  if (!(h->desc.flags & GSI_FLAG_FP8_IMAGE)) return GSI_ERR_UNSUPPORTED;
  *out = h->ws + h->lay.pk_wpp;
  *bytes_out = (size_t)((h->lay.O + 15) / 16) * persist_image_row_bytes(h->desc.k, true);
  return GSI_OK;
}

gsi_status_t gsi_get_status(gsi_handle_t h, int* device_status) {
  if (!h || !device_status) return GSI_ERR_INVALID_ARG;
  if (cudaStreamSynchronize(h->last_stream) != cudaSuccess) return GSI_ERR_CUDA;
  if (cudaMemcpy(device_status, h->gp.status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return GSI_ERR_CUDA;
  return GSI_OK;
}

gsi_status_t gsi_set_spin_limit(gsi_handle_t h, unsigned polls) {
  if (!h) return GSI_ERR_INVALID_ARG;
  h->gp.spin_limit = polls ? polls : kFusedSpinLimit;
  return GSI_OK;
}

gsi_status_t gsi_destroy(gsi_handle_t h) {
  if (!h) return GSI_ERR_INVALID_ARG;
  delete h;
  return GSI_OK;
}

// ------------------------------------------------------------------ stack
static size_t stack_tables_bytes(int n_groups) {
  static_assert(sizeof(PersistGroup) <= 512, "group descriptor outgrew its slot");
  return align_up(256) + align_up((size_t)n_groups * 512) + align_up((size_t)n_groups * 8) +
         align_up((size_t)n_groups * 4);
}
static size_t wide_ints(int n_groups) {   // of the whole step and of the segments, or of a flat step
  const size_t wide = 2 * (kWideStages + 1) * (size_t)n_groups + kWideStages * (kMaxSegments + 1);
  const size_t flat = 14 * (size_t)n_groups + 7 * kFlatMaxGrid + 8;   // shares and their norms, groups, first shares
  return wide > flat ? wide : flat;
}

size_t gsi_stack_workspace_bytes(int n_groups) {
  if (n_groups <= 0) return 0;
  return stack_tables_bytes(n_groups) + align_up(n_groups * sizeof(WideGroup)) + align_up(4 * wide_ints(n_groups));
}

gsi_status_t gsi_stack_create(int n_groups, const gsi_handle_t* groups, void* workspace,
                              size_t workspace_bytes, gsi_stream_t stream, gsi_stack_t* out) {
  if (!out) return GSI_ERR_INVALID_ARG;
  *out = nullptr;
  if (n_groups <= 0 || !groups || !workspace) return GSI_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) % kAlign) return GSI_ERR_INVALID_ARG;
  if (workspace_bytes < stack_tables_bytes(n_groups)) return GSI_ERR_WORKSPACE;
  for (int i = 0; i < n_groups; ++i) {
    if (!groups[i]) return GSI_ERR_INVALID_ARG;
    if (groups[i]->desc.max_tokens != groups[0]->desc.max_tokens) return GSI_ERR_INVALID_ARG;
    // a handle's exchange state and scratch serve one use per step
    for (int j = 0; j < i; ++j)
      if (groups[j] == groups[i]) return GSI_ERR_INVALID_ARG;
  }
  gsi_stack* s = new (std::nothrow) gsi_stack();
  if (!s) return GSI_ERR_ALLOC;
  s->groups.assign(groups, groups + n_groups);
  s->pair_first.assign(n_groups, 0);
  s->io.resize(n_groups);
  s->B = groups[0]->desc.max_tokens;
  s->n_steps = 0;
  s->gate_log = nullptr;
  s->rho_log = nullptr;
  s->step = static_cast<int*>(workspace);
  s->epoch = s->step + 1;
  s->status = s->step + 2;
  s->dev_groups = reinterpret_cast<PersistGroup*>(static_cast<char*>(workspace) + 256);
  s->dev_phase_first = reinterpret_cast<int*>(static_cast<char*>(workspace) + align_up(256) +
                                              align_up((size_t)n_groups * 512) + align_up((size_t)n_groups * 8));
  s->wide_area = workspace_bytes >= gsi_stack_workspace_bytes(n_groups)
                     ? static_cast<char*>(workspace) + stack_tables_bytes(n_groups) : nullptr;
  s->spin_limit = kPersistSpinLimitDefault;
  s->mode = 0;
  s->trace = nullptr;
  s->persistent = false;
  s->grid = 0;
  s->bound = false;
  s->last_stream = stream;
  if (cudaMemsetAsync(workspace, 0, 256, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    delete s;
    return GSI_ERR_CUDA;
  }
  *out = s;
  return GSI_OK;
}

// Basis rows and image rows are dealt to the CTAs of a group's shares in units of 16 rows: the
// least shares whose rows fit a CTA's buffers.
static int p_tiles(const gsi_layer* h) { return (h->desc.d + 15) / 16; }
static int o_tiles(const gsi_layer* h) { return (h->lay.O + 15) / 16; }
static int least_p_share(const gsi_layer* h) { return (p_tiles(h) + kPersistMaxPRows / 16 - 1) / (kPersistMaxPRows / 16); }
static int least_o_share(const gsi_layer* h) { return (o_tiles(h) + kPersistMaxORows / 16 - 1) / (kPersistMaxORows / 16); }
static bool rows_fit(const gsi_layer* h, int ctas) {
  if ((h->desc.flags & GSI_FLAG_DENSE) || h->desc.k <= 0) return true;
  return std::max(least_p_share(h), least_o_share(h)) <= ctas;
}

// W stream geometry of a CTA's `rows` rows: whole rows per contiguous piece of at most 32 KB, fewer
// where that leaves teams of consumer warps idle (see w_geometry in the kernel; two rows at least, the
// step of a team).  d = 768, 62 rows: five rows on 15 teams, against 21 on three (12 GPT-2 layers with
// 67 % gated 127 -> 117 us); cutting smaller where all teams have work costs (28 GPT-J
// layers, all gated, 16 KB pieces: 2.23 -> 2.57 ms).
static int w_piece_rows(int d, int rows) {
  const int most = std::max(1, kPersistPieceBytes / (d * 2));
  const int teams = std::max(1, kPersistConsumerWarps / ((d / 8 + 127) / 128));
  return std::min(most, std::max(2, (rows + teams - 1) / teams));
}

// A row of W fits a piece, and the per-warp partial results of the W stream hold every row a
// CTA owns of every map of a group.
static bool w_rows_fit(const gsi_layer* h, int grid) {
  if (h->desc.d > kPersistMaxD) return false;
  int total = 0;
  for (int j = 0; j < h->desc.n_maps; ++j) total += (h->d_out[j] + grid - 1) / grid;
  return total <= kPersistMaxWRows;
}

// Can this stack run on the persistent kernel?  (one or two tokens per step, bf16 basis
// with a power-of-two rank up to 512, rows that fit the per-CTA buffers and the ring.)
static bool persistent_eligible(const gsi_stack* s, int grid) {
  if (s->B > kPersistMaxTokens || grid <= 0 || grid > kPersistMaxGrid) return false;
  if ((int)s->groups.size() + 2 > kPersistMaxTicks) return false;   // the launch's plan lives in shared memory
  for (const gsi_layer* h : s->groups) {
    const gsi_desc_t& d = h->desc;
    const bool dense = d.flags & GSI_FLAG_DENSE;
    if (dense && s->B > 1) return false;   // a dense group streams W: once for all tokens (batched GEMM)
    if (d.d % 16) return false;
    if (!rows_fit(h, grid) || !w_rows_fit(h, grid)) return false;
    if (!dense && !h->lay.packed) return false;
  }
  return true;
}

// Deals `grid` CTAs to `len` groups, at least least[j] to each, the next one always to the group
// with the most load per CTA.  False when they do not suffice.
static bool deal_ctas(int grid, int len, const double* load, const int* least, int* ncta) {
  int left = grid;
  for (int j = 0; j < len; ++j) left -= ncta[j] = least[j];
  if (left < 0) return false;
  for (; left > 0; --left) {
    int at = 0;
    for (int j = 1; j < len; ++j)
      if (load[j] / ncta[j] > load[at] / ncta[at]) at = j;
    ++ncta[at];
  }
  return true;
}

struct Shares {
  int p = 0, o = 0, w = 0;   // CTAs for the basis rows, for the image rows, for W r beside the others of the phase
};

// Time of a phase of groups [i, i + len) in microseconds as the shares (filled in) leave it, or a
// negative number when the rows do not fit.  Basis and image rows are dealt on their own, so that
// every CTA carries about the same bytes of either: with one share per group, the CTAs of a wide
// basis turn its slab over twice (pass 1, residual) in their ring, 147 KB each time at GPT-J's
// 16384 -> 4096, while those beside them wait (28 GPT-J layers, nothing gated: 254 -> 219 us; 26
// OPT layers at k = 512: 532 -> 518).  A tick costs about 4 us whatever it carries (the
// barriers, the scalar code and the latency of its sections); on top of that either the memory
// system (6 bytes per picosecond), or the CTA with the most rows: rounds of fifteen 16-row units,
// 0.85 us each at k = 256, and pass 1, 0.1 us per unit.
static double phase_cost(const gsi_stack* s, int i, int len, Shares* share) {
  double bytes = 0.0, load[3][kPersistMaxLen];
  int least[2][kPersistMaxLen], one[kPersistMaxLen], n[3][kPersistMaxLen];
  for (int j = 0; j < len; ++j) {
    const gsi_layer* h = s->groups[i + j];
    load[0][j] = (double)h->desc.d * h->desc.k;
    load[1][j] = (double)h->lay.O * h->desc.k;
    load[2][j] = (double)h->lay.O * h->desc.d;
    least[0][j] = least_p_share(h);
    least[1][j] = least_o_share(h);
    one[j] = 1;
    bytes += 2.0 * ((double)h->desc.d + h->lay.O) * h->desc.k;
  }
  if (!deal_ctas(s->grid, len, load[0], least[0], n[0]) || !deal_ctas(s->grid, len, load[1], least[1], n[1]) ||
      !deal_ctas(s->grid, len, load[2], one, n[2]))
    return -1.0;
  double pt = 0.0, ot = 0.0;   // most units of one CTA, in units of k = 256
  for (int j = 0; j < len; ++j) {
    const gsi_layer* h = s->groups[i + j];
    pt = std::max(pt, (p_tiles(h) + n[0][j] - 1) / n[0][j] * h->desc.k / 256.0);
    ot = std::max(ot, (o_tiles(h) + n[1][j] - 1) / n[1][j] * h->desc.k / 256.0);
    share[j].p = n[0][j];
    share[j].o = n[1][j];
    share[j].w = n[2][j];
  }
  const double rows = 0.85 * std::ceil((pt + ot) / kPersistConsumerWarps) + 0.1 * pt;
  return 4.0 + std::max(bytes / 6.0e6, rows);
}

// The phases of the persistent schedule: consecutive groups in one phase as far as that shortens
// the step (inputs are staged before it), chosen over all partitions of the order.
static void plan_phases(gsi_stack* s, std::vector<int>* first, std::vector<Shares>* share) {
  const int G = (int)s->groups.size();
  std::vector<double> best(G + 1, 0.0);   // cost of groups [i, G)
  std::vector<int> len(G, 1);
  Shares parts[kPersistMaxLen];
  auto dense = [&](int i) { return (s->groups[i]->desc.flags & GSI_FLAG_DENSE) != 0; };
  for (int i = G - 1; i >= 0; --i) {
    best[i] = -1.0;
    for (int l = 1; l <= kPersistMaxLen && i + l <= G; ++l) {
      if (l > 1 && (dense(i) || dense(i + l - 1))) break;   // a dense group is a phase of its own
      const double c = dense(i) ? 4.0 : phase_cost(s, i, l, parts);
      if (c < 0.0) break;
      if (best[i] < 0.0 || c + best[i + l] < best[i]) {
        best[i] = c + best[i + l];
        len[i] = l;
      }
    }
  }
  first->clear();
  share->assign(G, Shares{s->grid, s->grid, s->grid});
  for (int i = 0; i < G; i += len[i]) {
    first->push_back(i);
    if (!dense(i)) (void)phase_cost(s, i, len[i], share->data() + i);
  }
}

gsi_status_t gsi_stack_set_concurrent(gsi_stack_t s, int first_group, int enable) {
  if (!s || first_group < 0 || first_group + 1 >= (int)s->groups.size()) return GSI_ERR_INVALID_ARG;
  // a group belongs to at most one pair
  if (enable && ((first_group > 0 && s->pair_first[first_group - 1]) || s->pair_first[first_group + 1]))
    return GSI_ERR_INVALID_ARG;
  s->pair_first[first_group] = enable ? 1 : 0;
  s->bound = false;  // applied at bind time
  return GSI_OK;
}

gsi_status_t gsi_stack_set_mode(gsi_stack_t s, int mode) {
  if (!s || mode < 0 || mode > 2) return GSI_ERR_INVALID_ARG;
  s->mode = mode;
  s->bound = false;  // the choice is taken at bind time
  return GSI_OK;
}

static bool plan_segments(gsi_stack* s);

// A step of one token in three launches over all groups?  The persistent kernel takes 3.5 us and more
// per phase; the three launches read the bases twice, the second time from the L2.
static bool flat_eligible(const gsi_stack* s, int grid) {
  const int G = (int)s->groups.size();
  if (s->mode != 0 || s->B != 1 || !s->wide_area || grid <= 0 || grid > kFlatMaxGrid || G < kFlatMinGroups ||
      G > kFlatMaxGroups)
    return false;
  double basis = 0.0, image = 0.0;
  for (const gsi_layer* h : s->groups) {
    const gsi_desc_t& d = h->desc;
    if ((d.flags & (GSI_FLAG_DENSE | GSI_FLAG_FP8_IMAGE)) || h->gp.p_f32 || d.d > kFlatMaxD) return false;
    basis += 2.0 * d.d * d.k;
    image += 2.0 * h->lay.O * d.k;
  }
  return basis <= kFlatBasisBytes && image / G <= kFlatImageBytes;
}

// The rows of all bases in even shares: CTA c has rows of cost [c, c + 1) / grid of the total, in units of
// 16 rows.  False when a basis would have too many shares.
static bool plan_flat(gsi_stack* s, int grid, cudaStream_t stream) {
  const int G = (int)s->groups.size();
  std::vector<int> first(1, 0), slots(G, 0);
  std::vector<FlatShare> shares;
  double total = 0.0, at = 0.0;
  for (const gsi_layer* h : s->groups) total += (double)((h->desc.d + 15) / 16) * h->desc.k;
  const double each = total / grid;
  int gi = 0, unit = 0;
  for (int c = 0; c < grid; ++c) {
    const double end = c + 1 == grid ? total : each * (c + 1);
    while (gi < G) {
      const int units = (s->groups[gi]->desc.d + 15) / 16, k = s->groups[gi]->desc.k;
      int n = c + 1 == grid ? units - unit : (int)((end - at) / k + 0.5);
      n = std::min(n, units - unit);
      if (n <= 0) break;
      shares.push_back({gi, unit * 16, (unit + n) * 16, slots[gi]++});
      at += (double)n * k;
      unit += n;
      if (unit < units) break;
      ++gi;
      unit = 0;
    }
    first.push_back((int)shares.size());
  }
  for (int n : slots)
    if (n > kFlatMaxSlots) return false;
  s->wide_table.assign(G, WideGroup{});
  s->flat_k = 0;
  for (int i = 0; i < G; ++i) {
    WideGroup& w = s->wide_table[i];
    w.g = s->groups[i]->gp;
    w.io = IoRef{s->io[i].x, s->io[i].y, s->gate_log + i, s->rho_log ? s->rho_log + i : nullptr, s->step, s->n_steps,
                 (long long)w.g.d, (long long)G};
    s->flat_k = std::max(s->flat_k, w.g.k);
  }
  // (groups first: their records are read as 16-byte words)
  s->wide_ints.clear();
  for (int i = 0, at_share = 0; i < G; at_share += slots[i++]) {
    const GroupParams& g = s->wide_table[i].g;
    const FlatGroup f{at_share, slots[i], g.O, g.k, g.d, g.eps, g.flags, 0};
    const int* words = reinterpret_cast<const int*>(&f);
    s->wide_ints.insert(s->wide_ints.end(), words, words + sizeof f / 4);
  }
  const size_t at_shares = s->wide_ints.size();
  for (const FlatShare& f : shares) s->wide_ints.insert(s->wide_ints.end(), {f.group, f.r0, f.r1, f.slot});
  const size_t at_norms = s->wide_ints.size(), at_first = at_norms + 2 * shares.size();
  s->wide_ints.resize(at_first, 0);
  s->wide_ints.insert(s->wide_ints.end(), first.begin(), first.end());
  int* ints = reinterpret_cast<int*>(s->wide_area + align_up(G * sizeof(WideGroup)));
  s->flat_grid = grid;
  s->flat_params = FlatParams{reinterpret_cast<const WideGroup*>(s->wide_area), ints + at_first,
                              reinterpret_cast<const FlatShare*>(ints + at_shares), reinterpret_cast<const FlatGroup*>(ints),
                              reinterpret_cast<float2*>(ints + at_norms), G, (int)shares.size(), 0, s->step, s->step + 4};
  return cudaMemsetAsync(s->step + 4, 0, sizeof(int), stream) == cudaSuccess &&
         cudaMemcpyAsync(s->wide_area, s->wide_table.data(), G * sizeof(WideGroup), cudaMemcpyHostToDevice, stream) ==
             cudaSuccess &&
         cudaMemcpyAsync(ints, s->wide_ints.data(), s->wide_ints.size() * 4, cudaMemcpyHostToDevice, stream) == cudaSuccess;
}

// Does every group of a batched stack take the tensor-core front end, and are there enough of them
// to fill the launches of a wide step?
static bool wide_eligible(const gsi_stack* s) {
  const int G = (int)s->groups.size();
  if (s->persistent || s->flat || s->mode != 0 || !s->wide_area || G < kWideMinGroups || G > kWideMaxGroups) return false;
  for (const gsi_layer* h : s->groups)
    if (!h->has_tm || !h->lay.front || s->B < h->gp.front_min_tokens || (h->desc.flags & GSI_FLAG_DENSE)) return false;
  return true;
}

// The table of a wide step and the blocks of its launches, for the whole step and for every segment.
static bool plan_wide(gsi_stack* s, cudaStream_t stream) {
  const int G = (int)s->groups.size();
  long long kblocks = 0;
  s->wide_k = 0;
  for (const gsi_layer* h : s->groups) {
    kblocks += (long long)(h->desc.d / umma::kTK) * (h->desc.k / umma::kTM);
    s->wide_k = std::max(s->wide_k, h->desc.k);
  }
  const int per_split = (int)std::max(4ll, (kblocks + kWideBlocks - 1) / kWideBlocks);
  s->wide_table.assign(G, WideGroup{});
  for (int i = 0; i < G; ++i) {
    gsi_layer* h = s->groups[i];
    WideGroup& w = s->wide_table[i];
    w.tm = h->tm;
    w.g = h->gp;
    const int nkb = h->desc.d / umma::kTK;
    w.g.proj_splits = std::max(1, std::min(h->gp.proj_splits, (nkb + per_split - 1) / per_split));
    w.io = IoRef{s->io[i].x, s->io[i].y, s->gate_log + (size_t)i * s->B,
                 s->rho_log ? s->rho_log + (size_t)i * s->B : nullptr, s->step, s->n_steps,
                 (long long)s->B * h->desc.d, (long long)G * s->B};
  }
  char* ints_dev = s->wide_area + align_up(G * sizeof(WideGroup));
  s->wide_ints.clear();
  s->wide_ranges.clear();
  auto add_range = [&](int g0, int g1) {
    const int n = g1 - g0;
    gsi_stack::WideRange r{g0, g1, nullptr, nullptr, {}, 1};
    std::vector<int> order(n);
    for (int i = 0; i < n; ++i) order[i] = i;
    // the contraction: deep tiles, which take longest, first
    std::stable_sort(order.begin(), order.end(),
                     [&](int a, int b) { return s->groups[g0 + a]->desc.d > s->groups[g0 + b]->desc.d; });
    r.first = reinterpret_cast<const int*>(ints_dev) + s->wide_ints.size();
    for (int stage = 0; stage < kWideStages; ++stage) {
      int at = 0;
      for (int i = 0; i < n; ++i) {
        s->wide_ints.push_back(at);
        const int gi = g0 + (stage == kWideGemm ? order[i] : i);
        const WideGroup& w = s->wide_table[gi];
        const int d = w.g.d, O = w.g.O;
        at += stage == kWideSplit   ? wide_split_blocks(d, s->B)
              : stage == kWideProj  ? w.g.k / umma::kTM * w.g.proj_splits
              : stage == kWideResid ? (d + O) / umma::kTM
              : (w.g.flags & GSI_FLAG_STATIC_PROJECTION) ? 0 : O / umma::kTM;
      }
      s->wide_ints.push_back(at);
      r.blocks[stage] = at;
    }
    // So many splits that the deepest tile takes no longer than an even share of all, none below a
    // depth of 2048 (64 tokens, a tenth gated: two GPT-J layers 237 us without, 227 with eight; 12 GPT-2
    // layers, depth 3072, 151 without, 172 with two).
    double work = 0.0, deepest = 0.0;
    for (int i = 0; i < n; ++i) {
      const GroupParams& g = s->wide_table[g0 + i].g;
      work += (double)g.O / umma::kTM * g.d;
      deepest = std::max(deepest, (double)g.d);
    }
    while (r.splits < 8 && deepest / r.splits > work / kWideGemmSlots && deepest / (2 * r.splits) >= 2048) r.splits *= 2;
    r.order = reinterpret_cast<const int*>(ints_dev) + s->wide_ints.size();
    s->wide_ints.insert(s->wide_ints.end(), order.begin(), order.end());
    s->wide_ranges.push_back(r);
  };
  add_range(0, G);
  for (size_t i = 0; s->segment.size() > 2 && i + 1 < s->segment.size(); ++i) add_range(s->segment[i], s->segment[i + 1]);
  return cudaMemcpyAsync(s->wide_area, s->wide_table.data(), G * sizeof(WideGroup), cudaMemcpyHostToDevice, stream) ==
             cudaSuccess &&
         cudaMemcpyAsync(ints_dev, s->wide_ints.data(), s->wide_ints.size() * 4, cudaMemcpyHostToDevice, stream) ==
             cudaSuccess;
}

static gsi_status_t wide_enqueue(gsi_stack* s, int g0, int g1, bool use_counter, cudaStream_t stream) {
  for (const gsi_stack::WideRange& r : s->wide_ranges) {
    if (r.g0 != g0 || r.g1 != g1) continue;
    const WideParams p{reinterpret_cast<const WideGroup*>(s->wide_area) + g0, r.first, r.order, g1 - g0, use_counter ? 1 : 0,
                       wide_term_bytes(s->wide_k, s->B)};
    for (int i = g0; i < g1; ++i) s->groups[i]->last_stream = stream;
    if (launch_front_wide(p, r.blocks, s->B, s->grid, stream) != cudaSuccess) return GSI_ERR_CUDA;
    if (r.blocks[kWideGemm] && launch_gemm_wide(p, r.blocks[kWideGemm], r.splits, s->B, stream) != cudaSuccess) return GSI_ERR_CUDA;
    return GSI_OK;
  }
  return GSI_ERR_CUDA;
}

gsi_status_t gsi_stack_bind(gsi_stack_t s, const gsi_stack_io_t* io, int n_steps,
                            unsigned char* gate_log, float* rho_log, gsi_stream_t stream) {
  if (!s || !io || n_steps <= 0 || !gate_log) return GSI_ERR_INVALID_ARG;
  const int G = (int)s->groups.size();
  for (int i = 0; i < G; ++i)
    if (!io[i].x || !io[i].y || !aligned16(io[i].x) || !aligned16(io[i].y))
      return GSI_ERR_INVALID_ARG;
  std::copy(io, io + G, s->io.begin());
  s->n_steps = n_steps;
  s->gate_log = gate_log;
  s->rho_log = rho_log;
  s->last_stream = stream;

  s->persistent = s->flat = false;
  if (s->mode != 1) {
    int dev = 0, sms = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess)
      return GSI_ERR_CUDA;
    s->grid = sms;
    s->flat = flat_eligible(s, sms) && plan_flat(s, sms, stream);
    s->persistent = !s->flat && coop && persistent_eligible(s, sms);
    if (s->mode == 2 && !s->persistent) return GSI_ERR_UNSUPPORTED;
  }
  if (!s->persistent)
    for (const gsi_layer* h : s->groups)
      if (h->desc.flags & GSI_FLAG_FP8_IMAGE) return GSI_ERR_UNSUPPORTED;
  s->wide = wide_eligible(s);
  if (!s->persistent && !s->flat && !s->wide && !s->aux) {
    bool any = false;
    for (char c : s->pair_first) any = any || c;
    int least = 0, greatest = 0;
    if (any && (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess ||
                cudaStreamCreateWithPriority(&s->aux, cudaStreamNonBlocking, greatest) != cudaSuccess ||
                cudaEventCreateWithFlags(&s->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
                cudaEventCreateWithFlags(&s->ev_join, cudaEventDisableTiming) != cudaSuccess))
      return GSI_ERR_CUDA;
  }
  if (!s->persistent && !s->flat && !s->wide && !s->ev_front_join) {
    bool any = false;   // some group takes the tensor-core front end at this batch
    for (const gsi_layer* h : s->groups)
      any = any || (h->has_tm && h->gp.front_min_tokens > 0 && s->B >= h->gp.front_min_tokens &&
                    !(h->desc.flags & (GSI_FLAG_DENSE | GSI_FLAG_STATIC_PROJECTION)));
    int least = 0, greatest = 0;
    if (any && (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess ||
                cudaEventCreateWithFlags(&s->ev_resid, cudaEventDisableTiming) != cudaSuccess ||
                cudaEventCreateWithFlags(&s->ev_front_fork, cudaEventDisableTiming) != cudaSuccess ||
                cudaEventCreateWithFlags(&s->ev_front_join, cudaEventDisableTiming) != cudaSuccess))
      return GSI_ERR_CUDA;
    s->alternate = true;
    for (const gsi_layer* h : s->groups) s->alternate = s->alternate && (double)h->lay.O * h->desc.d <= 8388608.0;
    for (cudaStream_t& f : s->front)
      if (any && cudaStreamCreateWithPriority(&f, cudaStreamNonBlocking, greatest) != cudaSuccess) return GSI_ERR_CUDA;
  }
  if (s->persistent) {
    // The cross-CTA exchange state of every group (accumulators, exchange words, arrival
    // counters) is tied to THIS stack's launch counter: start both from zero.  A handle
    // can therefore serve only one bound stack at a time.
    if (cudaMemsetAsync(s->epoch, 0, sizeof(int), stream) != cudaSuccess ||
        cudaMemsetAsync(s->status, 0, 2 * sizeof(int), stream) != cudaSuccess)   // a fresh start also after a time-out (status word, site of the wait that gave up)
      return GSI_ERR_CUDA;
    for (int i = 0; i < G; ++i) {
      const gsi_layer* h = s->groups[i];
      if (cudaMemsetAsync(h->ws + h->lay.pk_acc, 0, h->lay.tc_rb - h->lay.pk_acc, stream) !=
              cudaSuccess ||
          cudaMemsetAsync(h->bar, 0, 6 * sizeof(unsigned), stream) != cudaSuccess)
        return GSI_ERR_CUDA;
    }
    s->host_groups.assign(G, PersistGroup{});
    s->host_pmax_ptrs.assign(G, nullptr);
    for (int i = 0; i < G; ++i) {
      const gsi_layer* h = s->groups[i];
      PersistGroup& pg = s->host_groups[i];
      const GroupParams& gp = h->gp;
      pg.P = reinterpret_cast<const uint16_t*>(h->ws + h->lay.pk_pp);
      pg.WP = reinterpret_cast<const uint16_t*>(h->ws + h->lay.pk_wpp);
      for (int j = 0; j < gp.n_maps; ++j) pg.W[j] = gp.W[j];
      for (int j = 0; j <= gp.n_maps; ++j) pg.off[j] = gp.off[j];
      pg.n_maps = gp.n_maps;
      pg.d = gp.d;
      const bool dense_g = gp.flags & GSI_FLAG_DENSE;
      pg.k = dense_g ? 256 : gp.k;
      pg.O = gp.O;
      pg.eps = gp.eps;
      pg.flags = gp.flags;
      pg.pmax = 0.f;
      s->host_pmax_ptrs[i] = (gp.flags & GSI_FLAG_DENSE) ? nullptr : h->pmax;
      pg.x = io[i].x;
      pg.y = io[i].y;
      pg.r = gp.r;
      pg.acc = reinterpret_cast<unsigned long long*>(h->ws + h->lay.pk_acc);
      pg.xmax = reinterpret_cast<unsigned*>(h->ws + h->lay.pk_slot);
      pg.pub = reinterpret_cast<unsigned long long*>(h->ws + h->lay.pk_slot + (size_t)kPersistMaxGrid * 4);
      pg.bar = h->bar;
      pg.x_step_stride = (long long)s->B * gp.d;
    }
    std::vector<Shares> share;
    plan_phases(s, &s->host_phase_first, &share);
    s->has_pairs = false;
    s->common_k = -1;
    for (size_t ph = 0; ph < s->host_phase_first.size(); ++ph) {
      const int i0 = s->host_phase_first[ph];
      const int i1 = ph + 1 < s->host_phase_first.size() ? s->host_phase_first[ph + 1] : G;
      if (i1 - i0 > 1) s->has_pairs = true;
      Shares at;
      for (int i = i0; i < i1; ++i) {
        PersistGroup& pg = s->host_groups[i];
        const gsi_layer* h = s->groups[i];
        pg.cta0 = at.p;
        pg.ncta = share[i].p;
        pg.o_cta0 = at.o;
        pg.o_ncta = share[i].o;
        pg.phase_len = i1 - i0;
        // rows are dealt in groups of 16: CTA c of the share owns groups [c n / ncta, (c + 1) n / ncta)
        // (the first n CTAs one group each when there are fewer groups than CTAs)
        pg.p_rows = 16 * ((p_tiles(h) + pg.ncta - 1) / pg.ncta);
        pg.n_contrib = std::min(pg.ncta, p_tiles(h));
        // W r on a share of the group's own where a CTA's rows are few pieces: such a stream is a chain
        // of latencies (2.5 us whatever its size), and those of a phase then run side by side
        const bool own = !(pg.flags & GSI_FLAG_DENSE) && w_rows_fit(h, share[i].w) &&
                         (double)((pg.O + share[i].w - 1) / share[i].w) * pg.d * 2 <= kOwnStreamBytes;
        pg.w_cta0 = (short)(own ? at.w : 0);
        pg.w_ncta = (short)(own ? share[i].w : s->grid);
        at.p += share[i].p;
        at.o += share[i].o;
        at.w += share[i].w;
        int w_rows = 0;
        for (int j = 0; j < h->gp.n_maps; ++j)
          w_rows += pg.w_rows[j] = (short)((h->gp.d_out[j] + pg.w_ncta - 1) / pg.w_ncta);
        pg.w_pr = w_piece_rows(pg.d, w_rows);
        if (!(pg.flags & GSI_FLAG_DENSE)) s->common_k = s->common_k < 0 || s->common_k == pg.k ? pg.k : 0;
      }
    }
    if (s->common_k < 0) s->common_k = 0;
    s->n_phases = (int)s->host_phase_first.size();
    const float** dev_ptrs = reinterpret_cast<const float**>(
        reinterpret_cast<char*>(s->dev_groups) + (size_t)G * 512);
    if (cudaMemcpyAsync(s->dev_groups, s->host_groups.data(), sizeof(PersistGroup) * G,
                        cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        cudaMemcpyAsync(dev_ptrs, s->host_pmax_ptrs.data(), sizeof(float*) * G,
                        cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        cudaMemcpyAsync(s->dev_phase_first, s->host_phase_first.data(),
                        s->host_phase_first.size() * sizeof(int), cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        launch_patch_pmax(s->dev_groups, dev_ptrs, G, stream) != cudaSuccess)
      return GSI_ERR_CUDA;
  }
  if (!plan_segments(s)) return GSI_ERR_CUDA;
  if (s->wide && !plan_wide(s, stream)) return GSI_ERR_CUDA;
  // A set-up call: the descriptor table and the cleared exchange state must be in
  // device memory before a step may be enqueued on ANY stream.
  if (cudaStreamSynchronize(stream) != cudaSuccess) return GSI_ERR_CUDA;
  s->bound = true;
  return GSI_OK;
}

gsi_status_t gsi_stack_seek(gsi_stack_t s, int step, gsi_stream_t stream) {
  if (!s || step < 0) return GSI_ERR_INVALID_ARG;
  s->last_stream = stream;
  s->seek_value = step;  // pageable source: staged by the runtime before the call returns
  return cudaMemcpyAsync(s->step, &s->seek_value, sizeof(int), cudaMemcpyHostToDevice, stream) ==
                 cudaSuccess
             ? GSI_OK
             : GSI_ERR_CUDA;
}

// The groups [g0, g1) of a step (persistent schedule: the phases [g0, g1)) whose inputs are there
// once `ready` (null: everything enqueued on `stream` so far) has happened.  `first` / `last`: the
// range opens / closes the step.
static gsi_status_t stack_enqueue_range(gsi_stack_t s, int g0, int g1, bool first, bool last, bool use_counter,
                                        cudaEvent_t ready, gsi_stream_t stream) {
  const int G = (int)s->groups.size();
  if (ready && cudaStreamWaitEvent(stream, ready, 0) != cudaSuccess) return GSI_ERR_CUDA;
  if (s->persistent) {
    PersistParams p{};
    p.groups = s->dev_groups;
    p.n_groups = G;
    p.phase_first = s->dev_phase_first + g0;
    p.n_phases = g1 - g0;
    p.step = s->step;
    p.epoch = s->epoch;
    p.n_steps = s->n_steps;
    p.use_counter = use_counter ? 1 : 0;
    p.gate_log = s->gate_log;
    p.rho_log = s->rho_log;
    p.log_step_stride = G;
    p.status = s->status;
    p.trace = s->trace;
    p.spin_limit = s->spin_limit - 1;   // the kernels give up when a wait has polled more than this many times without success
    p.n_tokens = s->B;
    p.last = last ? 1 : 0;
    // one launch per token of the step (up to kPersistMaxTokens; larger batches take the
    // batched kernels): each is a complete decode step of that token, the last one advances
    for (int t = 0; t < s->B; ++t) {
      p.token = t;
      p.advance = t == s->B - 1;
      if (launch_decode_step(p, s->grid, s->has_pairs, s->common_k, stream) != cudaSuccess) return GSI_ERR_CUDA;
    }
    return GSI_OK;
  }
  if (s->flat) {   // (one segment)
    FlatParams p = s->flat_params;
    p.use_counter = use_counter ? 1 : 0;
    for (gsi_layer* h : s->groups) h->last_stream = stream;
    return launch_flat_step(p, s->flat_grid, s->flat_k, stream) == cudaSuccess ? GSI_OK : GSI_ERR_CUDA;
  }
  if (s->wide) {
    const gsi_status_t st = wide_enqueue(s, g0, g1, use_counter, stream);
    if (st != GSI_OK) return st;
    if (last && use_counter && launch_advance_step(s->step, stream) != cudaSuccess) return GSI_ERR_CUDA;
    return GSI_OK;
  }
  ResidualLane lane{stream, s->ev_resid, false};
  const bool chains = s->front[0] != nullptr;
  if (chains) {
    if (first && cudaEventRecord(s->ev_front_fork, stream) != cudaSuccess) return GSI_ERR_CUDA;
    for (cudaStream_t f : s->front)
      if ((first && cudaStreamWaitEvent(f, s->ev_front_fork, 0) != cudaSuccess) ||
          (ready && cudaStreamWaitEvent(f, ready, 0) != cudaSuccess))
        return GSI_ERR_CUDA;
  }
  auto enqueue_group = [&](int i, cudaStream_t st) -> bool {
    gsi_layer* h = s->groups[i];
    IoRef io{};
    io.x = s->io[i].x;
    io.y = s->io[i].y;
    io.gate = s->gate_log + (size_t)i * s->B;
    io.rho = s->rho_log ? s->rho_log + (size_t)i * s->B : nullptr;
    io.step = use_counter ? s->step : nullptr;
    io.n_steps = s->n_steps;
    io.x_step_stride = (long long)s->B * h->desc.d;
    io.log_step_stride = (long long)G * s->B;
    h->last_stream = stream;   // the joins below put all of the step's work in the caller's stream order
    return launch_generic_forward(h->gp, h->has_tm ? &h->tm : nullptr, io, s->B, st, nullptr,
                                  chains ? &lane : nullptr, true, s->mode == 1) == cudaSuccess;
  };
  for (int i = g0; i < g1; ++i) {
    if (chains && s->alternate) {
      if (!enqueue_group(i, s->front[i % kChains])) return GSI_ERR_CUDA;
      continue;
    }
    const cudaStream_t main = chains ? s->front[0] : stream, side = chains ? s->front[1] : s->aux;
    if (side && i + 1 < g1 && s->pair_first[i]) {
      // groups i and i+1 do not read each other's outputs: two chains of dependent launches
      // side by side (under stream capture this becomes a fork and a join in the graph)
      if (cudaEventRecord(s->ev_fork, main) != cudaSuccess || cudaStreamWaitEvent(side, s->ev_fork, 0) != cudaSuccess)
        return GSI_ERR_CUDA;
      if (!enqueue_group(i, main) || !enqueue_group(i + 1, side)) return GSI_ERR_CUDA;
      if (cudaEventRecord(s->ev_join, side) != cudaSuccess || cudaStreamWaitEvent(main, s->ev_join, 0) != cudaSuccess)
        return GSI_ERR_CUDA;
      ++i;
      continue;
    }
    if (!enqueue_group(i, main)) return GSI_ERR_CUDA;
  }
  if (chains)   // the chains join the caller's stream, which holds the contractions
    for (cudaStream_t f : s->front)
      if (cudaEventRecord(s->ev_front_join, f) != cudaSuccess ||
          cudaStreamWaitEvent(stream, s->ev_front_join, 0) != cudaSuccess)
        return GSI_ERR_CUDA;
  if (last && use_counter && launch_advance_step(s->step, stream) != cudaSuccess) return GSI_ERR_CUDA;
  return GSI_OK;
}

static gsi_status_t stack_enqueue(gsi_stack_t s, bool use_counter, gsi_stream_t stream) {
  return stack_enqueue_range(s, 0, s->persistent ? s->n_phases : (int)s->groups.size(), true, true, use_counter,
                             nullptr, stream);
}

// First group of unit u (a phase of the persistent schedule, else a group).
static int unit_group(const gsi_stack* s, int u) {
  if (!s->persistent) return u;
  return u < s->n_phases ? s->host_phase_first[u] : (int)s->groups.size();
}

// Segments of a batched step in launches over all groups.  A further segment costs the tails of five
// launches, some 40 us, and spares a part of the first copy in and the last one out; where the copies of
// one direction take longer than the step it costs nothing until it outgrows what they hide.  (us a step, a tenth
// gated, by segments: 12 GPT-2 layers at 24 tokens 2 311, 4 324, 12 621; at 64 3 634, 5 582, 12 780; eight GPT-J
// layers at 8 1 693, 3 582, 12 865; at 24 1 1437, 3 941, 5 965, 12 1179; at 64 3 2022, 8 1832, 12 1847.)
static int wide_segments(const gsi_stack* s) {
  double in = 0.0, out = 0.0, run = 0.0;   // us: copies at 20 per MB, the step as measured at 33 to 64 tokens
  for (const gsi_layer* h : s->groups) {
    in += 80e-6 * s->B * h->desc.d;
    out += 80e-6 * s->B * h->lay.O;
    run += 2.0 + 2.0 * h->lay.O * h->desc.d / 4.2e6;
  }
  if (in + out < 100.0) return 1;   // (two GPT-J layers at 8 tokens, 79 us of copies: 217, in two 227; 24 layers at 3, 350: 1047, 930)
  return (int)std::max(0.6 + std::sqrt((in + out) / 40.0), (std::max(in, out) - run) / 45.0);
}

// Cuts a step with host buffers into segments of about equal bytes, and makes the streams and
// events that overlap them.
static bool plan_segments(gsi_stack* s) {
  const int units = s->persistent ? s->n_phases : (int)s->groups.size();
  auto bytes = [&](int u) {
    double b = 0.0;
    for (int i = unit_group(s, u); i < unit_group(s, u + 1); ++i)
      b += 4.0 * s->B * ((double)s->groups[i]->desc.d + s->groups[i]->lay.O);
    return b;
  };
  double total = 0.0;
  for (int u = 0; u < units; ++u) total += bytes(u);
  // A copy of 1 MB takes 20 us.  A further launch of the persistent kernel costs about that (its
  // opening and closing ticks), so two halves from 3 MB on (28 GPT-J groups: 776 us in one piece,
  // 729 in two); the chains of batched steps go on from segment to segment without a gap: 3 MB each.
  int n = s->flat ? 1 : s->persistent ? (s->B == 1 && total >= 3.0e6 ? 2 : 1) : (int)(total / 3.0e6);
  if (s->wide) n = wide_segments(s);
  n = std::max(1, std::min(n, std::min(units, kMaxSegments)));
  s->segment.assign(1, 0);
  double at = 0.0;
  for (int u = 0; u < units && (int)s->segment.size() < n; ++u) {
    at += bytes(u);
    const bool inside_pair = !s->persistent && !s->wide && s->pair_first[u];   // (a pair shares streams)
    if (at >= total * s->segment.size() / n && !inside_pair && u + 1 < units) s->segment.push_back(u + 1);
  }
  s->segment.push_back(units);
  if (s->segment.size() == 2 || s->copy_in) return true;
  bool ok = cudaStreamCreateWithFlags(&s->copy_in, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamCreateWithFlags(&s->copy_out, cudaStreamNonBlocking) == cudaSuccess &&
            cudaEventCreateWithFlags(&s->ev_begin, cudaEventDisableTiming) == cudaSuccess;
  for (cudaEvent_t& e : s->ev_in) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
  for (cudaEvent_t& e : s->ev_run) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
  return ok;
}

gsi_status_t gsi_stack_step(gsi_stack_t s, gsi_stream_t stream) {
  if (!s || !s->bound) return GSI_ERR_INVALID_ARG;
  s->last_stream = stream;
  return stack_enqueue(s, true, stream);
}

gsi_status_t gsi_stack_launches_per_step(gsi_stack_t s, int* n_out) {
  if (!s || !n_out || !s->bound) return GSI_ERR_INVALID_ARG;
  if (s->persistent) {
    *n_out = s->B;
    return GSI_OK;
  }
  if (s->flat) {
    *n_out = 3;
    return GSI_OK;
  }
  if (s->wide) {
    *n_out = 4 + (s->wide_ranges[0].blocks[kWideGemm] ? 1 : 0) + 1;
    return GSI_OK;
  }
  int n = 0;
  for (gsi_layer* h : s->groups) {
    n += generic_launch_count(h->gp, s->B, s->mode == 1);
  }
  *n_out = n + 1;
  return GSI_OK;
}

gsi_status_t gsi_stack_step_host(gsi_stack_t s, const float* const* x_host, float* const* y_host,
                                 unsigned char* gate_host, gsi_stream_t stream) {
  if (!s || !s->bound || !x_host || !y_host || !gate_host) return GSI_ERR_INVALID_ARG;
  const int G = (int)s->groups.size();
  for (int i = 0; i < G; ++i)
    if (!x_host[i] || !y_host[i]) return GSI_ERR_INVALID_ARG;
  // Runs of groups whose buffers are adjacent both on the host and on the device
  // (a caller that carves them out of one arena) travel as ONE copy.
  auto copy_runs = [&](bool to_device, int g0, int g1, cudaStream_t st) -> bool {
    bool merge = true;
    for (int i = g0; i < g1;) {
      const char* h0 = to_device ? reinterpret_cast<const char*>(x_host[i])
                                 : reinterpret_cast<const char*>(y_host[i]);
      const char* d0 = to_device ? reinterpret_cast<const char*>(s->io[i].x)
                                 : reinterpret_cast<const char*>(s->io[i].y);
      size_t bytes = 0;
      int j = i;
      for (; j < g1 && (merge || j == i); ++j) {
        const size_t b = to_device ? (size_t)s->B * s->groups[j]->desc.d * 4
                                   : (size_t)s->B * s->groups[j]->lay.O * 4;
        const char* hj = to_device ? reinterpret_cast<const char*>(x_host[j])
                                   : reinterpret_cast<const char*>(y_host[j]);
        const char* dj = to_device ? reinterpret_cast<const char*>(s->io[j].x)
                                   : reinterpret_cast<const char*>(s->io[j].y);
        if (hj != h0 + bytes || dj != d0 + bytes) break;
        bytes += b;
      }
      const cudaError_t e =
          to_device ? cudaMemcpyAsync(const_cast<char*>(d0), h0, bytes, cudaMemcpyHostToDevice, st)
                    : cudaMemcpyAsync(const_cast<char*>(h0), d0, bytes, cudaMemcpyDeviceToHost, st);
      if (e != cudaSuccess) {
        if (j == i + 1) return false;
        (void)cudaGetLastError();   // neighbours by chance, in allocations of their own: one copy each
        merge = false;
        continue;
      }
      i = j;
    }
    return true;
  };
  s->last_stream = stream;
  const int n = (int)s->segment.size() - 1;
  if (n == 1) {
    if (!copy_runs(true, 0, G, stream)) return GSI_ERR_CUDA;
    gsi_status_t st = stack_enqueue(s, false, stream);
    if (st != GSI_OK) return st;
    if (!copy_runs(false, 0, G, stream)) return GSI_ERR_CUDA;
    if (cudaMemcpyAsync(gate_host, s->gate_log, (size_t)G * s->B, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
      return GSI_ERR_CUDA;
    return cudaStreamSynchronize(stream) == cudaSuccess ? GSI_OK : GSI_ERR_CUDA;
  }
  // Segment i + 1 is copied in and segment i - 1 copied out while segment i runs.
  auto ok = [](cudaError_t e) { return e == cudaSuccess; };
  if (!ok(cudaEventRecord(s->ev_begin, stream)) || !ok(cudaStreamWaitEvent(s->copy_in, s->ev_begin, 0)))
    return GSI_ERR_CUDA;
  for (int i = 0; i < n; ++i)
    if (!copy_runs(true, unit_group(s, s->segment[i]), unit_group(s, s->segment[i + 1]), s->copy_in) ||
        !ok(cudaEventRecord(s->ev_in[i], s->copy_in)))
      return GSI_ERR_CUDA;
  for (int i = 0; i < n; ++i) {
    gsi_status_t st = stack_enqueue_range(s, s->segment[i], s->segment[i + 1], i == 0, i + 1 == n, false, s->ev_in[i], stream);
    if (st != GSI_OK) return st;
    if (!ok(cudaEventRecord(s->ev_run[i], stream))) return GSI_ERR_CUDA;
  }
  // A host buffer that is y of one segment and x of a later one must be read before it is written: no
  // copy out starts before the last copy in then.  (Looked at here: the segments are on their way.)
  auto overlap = [&]() -> bool {
    for (int i = 0; i + 1 < n; ++i)
      for (int a = unit_group(s, s->segment[i]); a < unit_group(s, s->segment[i + 1]); ++a) {
        const uintptr_t y0 = (uintptr_t)y_host[a], y1 = y0 + (size_t)s->B * s->groups[a]->lay.O * 4;
        for (int b = unit_group(s, s->segment[i + 1]); b < G; ++b) {
          const uintptr_t x0 = (uintptr_t)x_host[b], x1 = x0 + (size_t)s->B * s->groups[b]->desc.d * 4;
          if (x0 < y1 && y0 < x1) return true;
        }
      }
    return false;
  };
  if (overlap() && !ok(cudaStreamWaitEvent(s->copy_out, s->ev_in[n - 1], 0))) return GSI_ERR_CUDA;
  for (int i = 0; i < n; ++i)   // (after all work is enqueued: a copy to pageable memory holds the host)
    if (!ok(cudaStreamWaitEvent(s->copy_out, s->ev_run[i], 0)) ||
        !copy_runs(false, unit_group(s, s->segment[i]), unit_group(s, s->segment[i + 1]), s->copy_out))
      return GSI_ERR_CUDA;
  if (!ok(cudaMemcpyAsync(gate_host, s->gate_log, (size_t)G * s->B, cudaMemcpyDeviceToHost, stream)) ||
      !ok(cudaEventRecord(s->ev_begin, s->copy_out)) || !ok(cudaStreamWaitEvent(stream, s->ev_begin, 0)))
    return GSI_ERR_CUDA;
  return ok(cudaStreamSynchronize(stream)) ? GSI_OK : GSI_ERR_CUDA;
}

gsi_status_t gsi_stack_set_trace(gsi_stack_t s, unsigned long long* cycles) {
  if (!s) return GSI_ERR_INVALID_ARG;
  s->trace = cycles;
  return GSI_OK;
}

gsi_status_t gsi_stack_set_spin_limit(gsi_stack_t s, unsigned polls) {
  if (!s) return GSI_ERR_INVALID_ARG;
  s->spin_limit = polls ? polls : kPersistSpinLimitDefault;
  return GSI_OK;
}

gsi_status_t gsi_stack_is_persistent(gsi_stack_t s, int* out) {
  if (!s || !out || !s->bound) return GSI_ERR_INVALID_ARG;
  *out = s->persistent ? 1 : 0;
  return GSI_OK;
}

gsi_status_t gsi_stack_get_status(gsi_stack_t s, int* device_status) {
  if (!s || !device_status) return GSI_ERR_INVALID_ARG;
  if (cudaStreamSynchronize(s->last_stream) != cudaSuccess) return GSI_ERR_CUDA;
  *device_status = 0;
  if (cudaMemcpy(device_status, s->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return GSI_ERR_CUDA;
  if (*device_status) return GSI_OK;
  for (gsi_layer* h : s->groups) {
    int v = 0;
    if (cudaMemcpy(&v, h->gp.status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
      return GSI_ERR_CUDA;
    if (v) {
      *device_status = v;
      break;
    }
  }
  return GSI_OK;
}

gsi_status_t gsi_stack_destroy(gsi_stack_t s) {
  if (!s) return GSI_ERR_INVALID_ARG;
  delete s;
  return GSI_OK;
}

}  // extern "C"
