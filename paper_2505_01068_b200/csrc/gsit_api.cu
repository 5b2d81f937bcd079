// C ABI of the IM attention library: argument validation, workspace carving, kernel sequencing.
#include <math.h>

#include "common.cuh"
#include "ptx.cuh"

namespace gsit {

extern int g_attn_variant;  // attn_bf16.cu
__device__ unsigned int g_device_status_word = 0;

namespace {

constexpr int MAX_DEVICES = 64;
unsigned int* g_status_ptr[MAX_DEVICES] = {};

// Address of this device's status word (looked up once per device).
cudaError_t status_ptr(unsigned int** p) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  if (g_status_ptr[dev] == nullptr) {
    void* sym = nullptr;
    e = cudaGetSymbolAddress(&sym, g_device_status_word);
    if (e != cudaSuccess) return e;
    g_status_ptr[dev] = static_cast<unsigned int*>(sym);
  }
  *p = g_status_ptr[dev];
  return cudaSuccess;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

gsit_status allowed_bits(const gsit_shape* s, uint32_t* bits) {
  switch (s->phase) {
    case GSIT_PHASE_INTER_FWD: *bits = (1u << 1) | (1u << 5) | (1u << 6); return GSIT_OK;  // 0->1, 1->2, 2->0
    case GSIT_PHASE_INTER_BWD: *bits = (1u << 2) | (1u << 3) | (1u << 7); return GSIT_OK;  // 0->2, 1->0, 2->1
    case GSIT_PHASE_INTRA:     *bits = (1u << 0) | (1u << 4) | (1u << 8); return GSIT_OK;  // s->s
    case GSIT_PHASE_CUSTOM:
      if (s->custom_mask > 0x1FFu) return GSIT_ERR_INVALID_ARG;
      *bits = s->custom_mask;
      return GSIT_OK;
    default: return GSIT_ERR_INVALID_ARG;
  }
}

// Validates the shape and fills the kernel-side geometry (without the status pointer).
gsit_status make_geometry(const gsit_shape* s, Geometry* g) {
  if (s == nullptr) return GSIT_ERR_INVALID_ARG;
  if (s->batch < 1 || s->heads < 1 || s->d_model < 1 || s->d_model % s->heads != 0) return GSIT_ERR_INVALID_ARG;
  if (s->dtype != GSIT_F32 && s->dtype != GSIT_BF16) return GSIT_ERR_INVALID_ARG;
  int64_t L = 0;
  for (int i = 0; i < 3; ++i) {
    if (s->seg_len[i] < 0) return GSIT_ERR_INVALID_ARG;
    L += s->seg_len[i];
  }
  if (L < 1) return GSIT_ERR_INVALID_ARG;
  if (L * (int64_t)s->batch > 0x7fffffffLL / 4) return GSIT_ERR_UNSUPPORTED;
  uint32_t bits = 0;
  gsit_status st = allowed_bits(s, &bits);
  if (st != GSIT_OK) return st;
  g->batch = s->batch;
  g->L = (int)L;
  g->d = s->d_model;
  g->heads = s->heads;
  g->hd = s->d_model / s->heads;
  for (int i = 0; i < 3; ++i) g->seg_len[i] = s->seg_len[i];
  g->seg_off[0] = 0;
  g->seg_off[1] = s->seg_len[0];
  g->seg_off[2] = s->seg_len[0] + s->seg_len[1];
  g->allowed = bits;
  g->valid_len = s->valid_len;
  g->status = nullptr;
  g->row_start = s->row_start;
  g->out_rows = nullptr;
  g->capacity = 0;
  if (s->row_start != nullptr) {  // packed row layout
    if (s->valid_len == nullptr || s->packed_capacity < 1) return GSIT_ERR_INVALID_ARG;
    if ((int64_t)s->packed_capacity > 0x7fffffffLL / 4) return GSIT_ERR_UNSUPPORTED;
    g->capacity = s->packed_capacity;
  }
  if (s->dtype == GSIT_BF16) {
    if (g->d % 16 != 0) return GSIT_ERR_UNSUPPORTED;
    if (g->hd != 8 && g->hd != 16 && g->hd != 32 && g->hd != 64) return GSIT_ERR_UNSUPPORTED;
    const int cw = (g->d % 64 == 0) ? 64 : (g->d % 32 == 0) ? 32 : 16;
    if (g->hd > cw || g->batch > 65535) return GSIT_ERR_UNSUPPORTED;
  } else {
    if (g->hd > 256) return GSIT_ERR_UNSUPPORTED;
  }
  return GSIT_OK;
}

gsit_status from_cuda(cudaError_t e) {
  if (e == cudaSuccess) return GSIT_OK;
  return (e == cudaErrorNotSupported) ? GSIT_ERR_UNSUPPORTED : GSIT_ERR_CUDA;
}

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

constexpr size_t ATTENTION_SCRATCH = 256;  // bytes gsit_im_attention_fwd can use (one work counter)

// Scratch layout of one layer call; every region 256-byte aligned.
struct LayerScratch {
  size_t h, qkv, att, y1, f, sched, total;
};
LayerScratch layer_scratch(const Geometry& g, int dtype, int d_ff) {
  // packed layout: every call addresses the packed matrices by absolute row, whatever part of the batch it covers
  const size_t rows = (size_t)matrix_rows(g), es = (dtype == GSIT_BF16) ? 2 : 4;
  LayerScratch s;
  size_t off = 0;
  s.h = off;   off += align_up(rows * g.d * es, 256);       // LN1(x), later LN2(y1)
  s.qkv = off; off += align_up(rows * 3 * g.d * es, 256);
  s.att = off; off += align_up(rows * g.d * es, 256);
  s.y1 = off;  off += align_up(rows * g.d * 4, 256);        // float residual stream after attention
  s.f = off;   off += align_up(rows * (size_t)d_ff * es, 256);
  s.sched = off; off += ATTENTION_SCRATCH;                   // work counter of the attention kernel
  s.total = off;
  return s;
}

// ---- optional event tracing of the library's launches ----
struct TraceRec { cudaEvent_t beg, end; int kind; };
constexpr int TRACE_CAP = 8192;
bool g_trace_on = false;
int g_trace_n = 0;            // records in use
int g_trace_created = 0;      // event pairs created so far (reused after a reset)
TraceRec g_trace[TRACE_CAP];

struct TraceScope {
  cudaStream_t st;
  TraceRec* rec = nullptr;
  TraceScope(int kind, cudaStream_t s) : st(s) {
    if (!g_trace_on || g_trace_n >= TRACE_CAP) return;
    TraceRec* r = &g_trace[g_trace_n];
    if (g_trace_n >= g_trace_created) {
      if (cudaEventCreate(&r->beg) != cudaSuccess || cudaEventCreate(&r->end) != cudaSuccess) return;
      ++g_trace_created;
    }
    r->kind = kind;
    if (cudaEventRecord(r->beg, st) != cudaSuccess) return;
    rec = r;
    ++g_trace_n;
  }
  ~TraceScope() { if (rec) cudaEventRecord(rec->end, st); }
};

gsit_status run_linear(const Geometry& g, int dtype, const LinearArgs& a, cudaStream_t st) {
  TraceScope t(GSIT_KERNEL_LINEAR, st);
  return from_cuda(dtype == GSIT_BF16 ? launch_linear_bf16(g, a, st) : launch_linear_f32(g, a, st));
}

gsit_status run_layernorm(const Geometry& g, const float* x, int64_t ldx, const float* gamma, const float* beta,
                          float eps, void* y, int out_bf16, cudaStream_t st) {
  TraceScope t(GSIT_KERNEL_LAYERNORM, st);
  return from_cuda(launch_layernorm(g, x, ldx, gamma, beta, eps, y, out_bf16, st));
}

gsit_status run_attention(const Geometry& g, int dtype, const void* q, const void* k, const void* v,
                          int64_t row_stride, void* out, float* lse, float scale, void* scratch, cudaStream_t st,
                          bool scratch_cleared = false) {
  TraceScope t(GSIT_KERNEL_ATTENTION, st);
  if (dtype == GSIT_BF16)
    return from_cuda(launch_attn_bf16(g, static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k),
                                      static_cast<const __nv_bfloat16*>(v), row_stride,
                                      static_cast<__nv_bfloat16*>(out), lse, scale, static_cast<int*>(scratch), st,
                                      scratch_cleared));
  return from_cuda(launch_attn_f32(g, static_cast<const float*>(q), static_cast<const float*>(k),
                                   static_cast<const float*>(v), row_stride, static_cast<float*>(out), lse, scale, st));
}

// Bounded waits whose barrier expects one arrival that nobody makes, by the loop that the kernels wait with: warp 0 must run out after 4096
// polls; warp 1, whose own limit is sixteen times that, must then see that the CTA has given up.  Both also wait for a phase that is over.
// `status` and `drained` take the flags of warps 0 and 1; answers (may be null): 2 warps x (phase over, phase never over) x 32 lanes.
__global__ void expire_wait_kernel(unsigned int* status, unsigned int* drained, uint32_t* answers, int cluster_form) {
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ uint32_t gave_up;
  const uint32_t never = smem_u32(&bar[0]), over = smem_u32(&bar[1]);
  if (threadIdx.x == 0) {
    gave_up = 0;
    ptx::mbar_init(never, 1);
    ptx::mbar_init(over, 1);
    ptx::mbar_init_fence();
    ptx::mbar_arrive(over);
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const ptx::WaitCtx wc{warp == 0 ? status : drained, smem_u32(&gave_up)};
  auto wait = [&](uint32_t b, int limit) { return cluster_form ? ptx::mbar_wait_cluster(wc, b, 0, limit) : ptx::mbar_wait_warp(wc, b, 0, limit); };
  for (int w = 0; w < 2; ++w) {
    if (warp == w) {
      const bool first = wait(over, 1 << 12), second = wait(never, w == 0 ? 1 << 12 : 1 << 16);
      if (answers != nullptr) {
        answers[64 * w + lane] = first;
        answers[64 * w + 32 + lane] = second;
      }
    }
    __syncthreads();
  }
}

// Lets its successor start at once, then takes its time before it writes (about delay_us, at most twice that).
__global__ void late_write_kernel(uint4* dst, const uint4* src, size_t n, int delay_us) {
  ptx::grid_dep_launch();
  for (int i = 0; i < delay_us; ++i) __nanosleep(1000);
  for (size_t i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// Which kernels run the two halves of a bf16 layer around the attention.
enum Halves { HALVES_NONE = 0, HALVES_ROWS, HALVES_TC, HALVES_TC128, HALVES_LEGACY };
Halves pick_halves(const Geometry& g, int d_ff) {
  const bool packed = g.row_start != nullptr;
  if (!packed && g_attn_variant == GSIT_ATTN_UNFUSED) return HALVES_NONE;
  if (!packed && g_attn_variant == GSIT_ATTN_LEGACY) return fused_layer_supported(g, d_ff) ? HALVES_LEGACY : HALVES_NONE;
  if (fused_rows_supported(g, d_ff) && fused_rows_preferred(g)) return HALVES_ROWS;
  if (fused_layer_tc_supported(g, d_ff)) return HALVES_TC;
  if (fused_layer_tc128_supported(g, d_ff)) return HALVES_TC128;
  if (!packed && fused_layer_supported(g, d_ff)) return HALVES_LEGACY;
  return HALVES_NONE;
}

FusedHalfArgs half_args(const gsit_layer_weights* w, const float* x, int64_t ldx, __nv_bfloat16* qkv, __nv_bfloat16* att, float* y, int64_t ldy) {
  auto b = [](const void* p) { return static_cast<const __nv_bfloat16*>(p); };
  return FusedHalfArgs{x, ldx, w->ln1_gamma, w->ln1_beta, b(w->w_qkv), w->b_qkv, qkv, att, b(w->w_o), w->b_o, w->ln2_gamma, w->ln2_beta,
                       b(w->w_1), w->b_1, b(w->w_2), w->b_2, y, ldy};
}

// Do `n` layers of this geometry, side by side, run as one launch behind their first projection?  (The row-tile kernels on mma.sync, for a problem
// whose attention is the mma.sync kernel as well: the same bits as three launches.)  in_encoder: layers of an encoder call, or on packed rows.
bool one_launch_layers(const Geometry& g, int dtype, const uint32_t* allowed, int n, int d_ff, bool in_encoder) {
  if (dtype != GSIT_BF16 || g_attn_variant != GSIT_ATTN_DEFAULT || pick_halves(g, d_ff) != HALVES_ROWS) return false;
  if (!layer_tail_supported(g, d_ff) || !layer_tail_preferred(g, allowed, n, in_encoder || g.row_start != nullptr)) return false;
  for (int i = 0; i < n; ++i)
    if (attn_uses_tensor_memory(g, allowed[i])) return false;
  return true;
}

float pick_scale(const gsit_shape* s, const Geometry& g) {
  return (s->scale > 0.f) ? s->scale : 1.0f / sqrtf((float)g.hd);
}

// `depth` layers of n (1 or 2) problems of geometry g side by side, each layer behind the first projection in one launch.  The layers of
// problem i read x[i] and write y[i * depth + j]; ws holds one layer_scratch per problem.
struct LayerChain {
  const gsit_layer_weights* const* w[2];
  const float* x[2];
  int64_t ldx[2];
  float* const* y[2];
  const int64_t* ldy[2];
  uint32_t allowed[2];
};
float eps_of(const gsit_layer_weights* w) { return (w->ln_eps > 0.f) ? w->ln_eps : 1e-5f; }

gsit_status run_chain(const Geometry& g, const LayerChain& c, int n, int depth, float scale, uint8_t* ws, size_t ws_stride, const LayerScratch& sc,
                      cudaStream_t cs) {
  // a launch reads one projection and writes the next layer's: they take turns in the scratch of qkv and that of att and y1, which lie
  // side by side (2 d + 4 d bytes a row) and have no other use here
  static_assert(sizeof(float) == 2 * sizeof(__nv_bfloat16), "att and y1 together hold the three projections");
  auto qkv = [&](int i, int j) { return reinterpret_cast<__nv_bfloat16*>(ws + i * ws_stride + ((j & 1) ? sc.att : sc.qkv)); };
  FusedHalfArgs h[2];
  for (int i = 0; i < n; ++i) h[i] = half_args(c.w[i][0], c.x[i], c.ldx[i], qkv(i, 0), nullptr, nullptr, 0);
  {
    TraceScope t(GSIT_KERNEL_LINEAR, cs);
    const gsit_status st = from_cuda(launch_ln_qkv_rows(g, h, n, eps_of(c.w[0][0]), nullptr, cs));
    if (st != GSIT_OK) return st;
  }
  for (int j = 0; j < depth; ++j) {
    LayerTailArgs a[2];
    for (int i = 0; i < n; ++i) {
      const bool next = j + 1 < depth;
      a[i].qkv = qkv(i, j);
      a[i].h = half_args(c.w[i][j], j == 0 ? c.x[i] : c.y[i][j - 1], j == 0 ? c.ldx[i] : c.ldy[i][j - 1], nullptr, nullptr, c.y[i][j], c.ldy[i][j]);
      a[i].allowed = c.allowed[i];
      const FusedHalfArgs nx = half_args(c.w[i][next ? j + 1 : j], nullptr, 0, nullptr, nullptr, nullptr, 0);
      a[i].h.ln1_gamma = nx.ln1_gamma; a[i].h.ln1_beta = nx.ln1_beta;
      a[i].h.w_qkv = nx.w_qkv; a[i].h.b_qkv = nx.b_qkv;
      a[i].h.qkv = next ? qkv(i, j + 1) : nullptr;
    }
    TraceScope t(GSIT_KERNEL_ATTENTION, cs);
    const gsit_status st = from_cuda(launch_layer_tail(g, a, n, scale, eps_of(c.w[0][j]), eps_of(c.w[0][j + 1 < depth ? j + 1 : j]), c.w[0][j]->d_ff, cs));
    if (st != GSIT_OK) return st;
  }
  return GSIT_OK;
}

}  // namespace
}  // namespace gsit

using namespace gsit;

extern "C" {

gsit_status gsit_im_qkv_proj(const gsit_shape* shape, const void* x, int64_t x_row_stride, const void* w_qkv,
                             const float* b_qkv, void* qkv, gsit_stream stream) {
  Geometry g;
  gsit_status st = make_geometry(shape, &g);
  if (st != GSIT_OK) return st;
  if (!x || !w_qkv || !qkv || x_row_stride < g.d) return GSIT_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(w_qkv) || !aligned16(qkv)) return GSIT_ERR_INVALID_ARG;
  if (shape->dtype == GSIT_BF16 && x_row_stride % 8 != 0) return GSIT_ERR_INVALID_ARG;
  if (from_cuda(status_ptr(&g.status)) != GSIT_OK) return GSIT_ERR_CUDA;
  LinearArgs a = {};
  a.A = x; a.lda = x_row_stride; a.W = w_qkv; a.bias = b_qkv;
  a.C = qkv; a.ldc = 3 * (int64_t)g.d;
  a.M = (int)matrix_rows(g); a.N = 3 * g.d; a.K = g.d;
  a.mask_rows = 1;
  if (shape->dtype == GSIT_BF16 && g_attn_variant == GSIT_ATTN_DEFAULT && qkv_rows_preferred(g) && (g.row_start == nullptr || linear_tc_supported(a))) {
    TraceScope t(GSIT_KERNEL_LINEAR, static_cast<cudaStream_t>(stream));
    return from_cuda(launch_qkv_rows(g, a, static_cast<cudaStream_t>(stream)));
  }
  if (g.row_start != nullptr) {
    // packed rows: the tcgen05 kernel computes and writes this call's row range only (widths it covers: multiples of 64)
    if (shape->dtype != GSIT_BF16 || !linear_tc_supported(a)) return GSIT_ERR_UNSUPPORTED;
    TraceScope t(GSIT_KERNEL_LINEAR, static_cast<cudaStream_t>(stream));
    return from_cuda(launch_linear_tc_bf16(g, a, static_cast<cudaStream_t>(stream)));
  }
  return run_linear(g, shape->dtype, a, static_cast<cudaStream_t>(stream));
}

gsit_status gsit_im_attention_fwd(const gsit_shape* shape, const void* q, const void* k, const void* v,
                                  int64_t row_stride, void* out, float* lse, void* workspace,
                                  size_t workspace_bytes, gsit_stream stream) {
  Geometry g;
  gsit_status st = make_geometry(shape, &g);
  if (st != GSIT_OK) return st;
  if (!q || !k || !v || !out || row_stride < g.d) return GSIT_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out)) return GSIT_ERR_INVALID_ARG;
  if (shape->dtype == GSIT_BF16 && row_stride % 8 != 0) return GSIT_ERR_INVALID_ARG;
  if (g.row_start != nullptr && shape->dtype != GSIT_BF16) return GSIT_ERR_UNSUPPORTED;  // every bf16 kernel takes the packed layout
  if (from_cuda(status_ptr(&g.status)) != GSIT_OK) return GSIT_ERR_CUDA;
  // optional scratch: with it the bf16 kernels hand out their work items through a counter instead of a fixed assignment
  void* scratch = (workspace != nullptr && workspace_bytes >= sizeof(int) && (reinterpret_cast<uintptr_t>(workspace) & 3u) == 0)
                      ? workspace : nullptr;
  return run_attention(g, shape->dtype, q, k, v, row_stride, out, lse, pick_scale(shape, g), scratch,
                       static_cast<cudaStream_t>(stream));
}

static gsit_status layer_fwd(const gsit_shape* shape, const gsit_layer_weights* w, const float* x, int64_t x_row_stride, float* y,
                             int64_t y_row_stride, const int32_t* row_map, void* workspace, size_t workspace_bytes, gsit_stream stream) {
  Geometry g;
  gsit_status st = make_geometry(shape, &g);
  if (st != GSIT_OK) return st;
  if (!w || !x || !y || x_row_stride < g.d || y_row_stride < g.d) return GSIT_ERR_INVALID_ARG;
  if (!w->w_qkv || !w->w_o || !w->w_1 || !w->w_2 || w->d_ff < 1) return GSIT_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(y) || !aligned16(w->w_qkv) || !aligned16(w->w_o) || !aligned16(w->w_1) ||
      !aligned16(w->w_2))
    return GSIT_ERR_INVALID_ARG;
  if (x_row_stride % 4 != 0 || y_row_stride % 4 != 0) return GSIT_ERR_INVALID_ARG;
  const int dtype = shape->dtype;
  if (dtype == GSIT_BF16 && w->d_ff % 8 != 0) return GSIT_ERR_UNSUPPORTED;
  const LayerScratch sc = layer_scratch(g, dtype, w->d_ff);
  if (!workspace || workspace_bytes < sc.total || (reinterpret_cast<uintptr_t>(workspace) & 255u))
    return GSIT_ERR_WORKSPACE;
  if (from_cuda(status_ptr(&g.status)) != GSIT_OK) return GSIT_ERR_CUDA;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  void *h = ws + sc.h, *qkv = ws + sc.qkv, *att = ws + sc.att, *f = ws + sc.f;
  float* y1 = reinterpret_cast<float*>(ws + sc.y1);
  const float eps = (w->ln_eps > 0.f) ? w->ln_eps : 1e-5f;
  const int bf = (dtype == GSIT_BF16);
  const int es = bf ? 2 : 4;
  const int M = g.batch * g.L, d = g.d;
  const Halves halves = bf ? pick_halves(g, w->d_ff) : HALVES_NONE;
  if (row_map != nullptr && (g.row_start == nullptr || halves != HALVES_TC128)) return GSIT_ERR_UNSUPPORTED;
  g.out_rows = row_map;
  if (g.row_start != nullptr && (halves == HALVES_NONE || g.hd > 32))
    return GSIT_ERR_UNSUPPORTED;  // the packed layout is implemented by the fused halves and the mma.sync / tensor-memory attention

  if (one_launch_layers(g, dtype, &g.allowed, 1, w->d_ff, false)) {
    const LayerChain c = {{&w, nullptr}, {x, nullptr}, {x_row_stride, 0}, {&y, nullptr}, {&y_row_stride, nullptr}, {g.allowed, 0}};
    return run_chain(g, c, 1, 1, pick_scale(shape, g), ws, 0, sc, cs);
  }
  if (halves != HALVES_NONE) {
    // three launches: LN1 + shared projection, IM attention, out-projection + residual + LN2 + MLP + residual
    const FusedHalfArgs h = half_args(w, x, x_row_stride, static_cast<__nv_bfloat16*>(qkv), static_cast<__nv_bfloat16*>(att), y, y_row_stride);
    int* counter = reinterpret_cast<int*>(ws + sc.sched);
    {
      TraceScope t(GSIT_KERNEL_LINEAR, cs);
      st = from_cuda(halves == HALVES_ROWS    ? launch_ln_qkv_rows(g, &h, 1, eps, counter, cs)
                     : halves == HALVES_TC    ? launch_ln_qkv_tc(g, x, x_row_stride, h.ln1_gamma, h.ln1_beta, eps, h.w_qkv, h.b_qkv, h.qkv, counter, cs)
                     : halves == HALVES_TC128 ? launch_ln_qkv_tc128(g, x, x_row_stride, h.ln1_gamma, h.ln1_beta, eps, h.w_qkv, h.b_qkv, h.qkv, counter, cs)
                                              : launch_ln_qkv_bf16(g, x, x_row_stride, h.ln1_gamma, h.ln1_beta, eps, h.w_qkv, h.b_qkv, h.qkv, cs));
    }
    if (st != GSIT_OK) return st;
    // the first halves clear the attention kernel's work counter (but the legacy one), so no memset separates the three kernels
    if ((st = run_attention(g, dtype, h.qkv, h.qkv + d, h.qkv + 2 * d, 3 * (int64_t)d, att, nullptr, pick_scale(shape, g), counter, cs,
                            halves != HALVES_LEGACY)) != GSIT_OK) return st;
    TraceScope t(GSIT_KERNEL_LINEAR, cs);
    if (halves == HALVES_ROWS) return from_cuda(launch_proj_mlp_rows(g, &h, 1, eps, w->d_ff, cs));
    auto second = halves == HALVES_TC ? launch_proj_mlp_tc : halves == HALVES_TC128 ? launch_proj_mlp_tc128 : launch_proj_mlp_bf16;
    return from_cuda(second(g, h.att, x, x_row_stride, h.w_o, h.b_o, h.ln2_gamma, h.ln2_beta, eps, h.w_1, h.b_1, h.w_2, h.b_2, w->d_ff, y,
                            y_row_stride, cs));
  }
  if (!bf && g_attn_variant != GSIT_ATTN_UNFUSED && fused_layer_f32_supported(g, w->d_ff)) {  // the same three launches for float operands
    auto f32 = [](const void* p) { return static_cast<const float*>(p); };
    float *fq = static_cast<float*>(qkv), *fa = static_cast<float*>(att);
    {
      TraceScope t(GSIT_KERNEL_LINEAR, cs);
      st = from_cuda(launch_ln_qkv_f32(g, x, x_row_stride, w->ln1_gamma, w->ln1_beta, eps, f32(w->w_qkv), w->b_qkv, fq, cs));
      if (st != GSIT_OK) return st;
    }
    if ((st = run_attention(g, dtype, fq, fq + d, fq + 2 * d, 3 * (int64_t)d, fa, nullptr, pick_scale(shape, g), nullptr, cs)) != GSIT_OK)
      return st;
    TraceScope t(GSIT_KERNEL_LINEAR, cs);
    return from_cuda(launch_proj_mlp_f32(g, fa, x, x_row_stride, f32(w->w_o), w->b_o, w->ln2_gamma, w->ln2_beta, eps, f32(w->w_1), w->b_1,
                                         f32(w->w_2), w->b_2, w->d_ff, y, y_row_stride, cs));
  }
  // h = LN1(x)
  if ((st = run_layernorm(g, x, x_row_stride, w->ln1_gamma, w->ln1_beta, eps, h, bf, cs)) != GSIT_OK) return st;
  // qkv = h W_qkv^T + b_qkv   (shared projection of the whole concatenated sequence)
  LinearArgs a = {};
  a.A = h; a.lda = d; a.W = w->w_qkv; a.bias = w->b_qkv; a.C = qkv; a.ldc = 3 * (int64_t)d;
  a.M = M; a.N = 3 * d; a.K = d; a.mask_rows = 1;
  if ((st = run_linear(g, dtype, a, cs)) != GSIT_OK) return st;
  // att = IM attention over the open blocks
  const uint8_t* qb = static_cast<const uint8_t*>(qkv);
  if ((st = run_attention(g, dtype, qb, qb + (size_t)d * es, qb + (size_t)2 * d * es, 3 * (int64_t)d, att, nullptr,
                          pick_scale(shape, g), ws + sc.sched, cs)) != GSIT_OK) return st;
  // y1 = x + att W_o^T + b_o   (float)
  a = LinearArgs{};
  a.A = att; a.lda = d; a.W = w->w_o; a.bias = w->b_o; a.residual = x; a.ldr = x_row_stride;
  a.C = y1; a.ldc = d; a.M = M; a.N = d; a.K = d; a.out_f32 = 1; a.mask_rows = 1;
  if ((st = run_linear(g, dtype, a, cs)) != GSIT_OK) return st;
  // h = LN2(y1)
  if ((st = run_layernorm(g, y1, d, w->ln2_gamma, w->ln2_beta, eps, h, bf, cs)) != GSIT_OK) return st;
  // f = relu(h W_1^T + b_1)
  a = LinearArgs{};
  a.A = h; a.lda = d; a.W = w->w_1; a.bias = w->b_1; a.C = f; a.ldc = w->d_ff;
  a.M = M; a.N = w->d_ff; a.K = d; a.relu = 1; a.mask_rows = 1;
  if ((st = run_linear(g, dtype, a, cs)) != GSIT_OK) return st;
  // y = y1 + f W_2^T + b_2   (float), padded rows zero
  a = LinearArgs{};
  a.A = f; a.lda = w->d_ff; a.W = w->w_2; a.bias = w->b_2; a.residual = y1; a.ldr = d;
  a.C = y; a.ldc = y_row_stride; a.M = M; a.N = d; a.K = w->d_ff; a.out_f32 = 1; a.mask_rows = 1;
  return run_linear(g, dtype, a, cs);
}

gsit_status gsit_im_layer_fwd(const gsit_shape* shape, const gsit_layer_weights* w, const float* x, int64_t x_row_stride, float* y,
                              int64_t y_row_stride, void* workspace, size_t workspace_bytes, gsit_stream stream) {
  return layer_fwd(shape, w, x, x_row_stride, y, y_row_stride, nullptr, workspace, workspace_bytes, stream);
}

int32_t gsit_layer_scatters(const gsit_shape* shape, int32_t d_ff) {
  Geometry g;
  return make_geometry(shape, &g) == GSIT_OK && g.row_start != nullptr && shape->dtype == GSIT_BF16 && d_ff >= 1 && d_ff % 8 == 0 && g.hd <= 32 &&
         pick_halves(g, d_ff) == HALVES_TC128;
}

gsit_status gsit_im_layer_scatter_fwd(const gsit_shape* shape, const gsit_layer_weights* w, const float* x, int64_t x_row_stride,
                                      const int32_t* row_map, float* y, int64_t y_row_stride, void* workspace, size_t workspace_bytes,
                                      gsit_stream stream) {
  if (!row_map) return GSIT_ERR_INVALID_ARG;
  return layer_fwd(shape, w, x, x_row_stride, y, y_row_stride, row_map, workspace, workspace_bytes, stream);
}

gsit_status gsit_im_layer_pair_fwd(const gsit_shape* shape_a, const gsit_shape* shape_b, const gsit_layer_weights* w_a,
                                   const gsit_layer_weights* w_b, const float* x_a, int64_t x_a_row_stride, const float* x_b,
                                   int64_t x_b_row_stride, float* y_a, int64_t y_a_row_stride, float* y_b, int64_t y_b_row_stride,
                                   void* workspace, size_t workspace_bytes, gsit_stream stream) {
  Geometry ga, gb;
  gsit_status st = make_geometry(shape_a, &ga);
  if (st != GSIT_OK) return st;
  if ((st = make_geometry(shape_b, &gb)) != GSIT_OK) return st;
  if (!w_a || !w_b) return GSIT_ERR_INVALID_ARG;
  // the two problems must agree in everything but their tensors and block pattern
  if (ga.batch != gb.batch || ga.d != gb.d || ga.heads != gb.heads || ga.valid_len != gb.valid_len || ga.row_start != gb.row_start ||
      ga.capacity != gb.capacity || shape_a->dtype != shape_b->dtype || shape_a->scale != shape_b->scale || w_a->d_ff != w_b->d_ff)
    return GSIT_ERR_INVALID_ARG;
  for (int i = 0; i < 3; ++i)
    if (ga.seg_len[i] != gb.seg_len[i]) return GSIT_ERR_INVALID_ARG;
  if (w_a->d_ff < 1) return GSIT_ERR_INVALID_ARG;
  const LayerScratch sc = layer_scratch(ga, shape_a->dtype, w_a->d_ff);
  if (!workspace || workspace_bytes < 2 * sc.total || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return GSIT_ERR_WORKSPACE;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  const float eps_a = (w_a->ln_eps > 0.f) ? w_a->ln_eps : 1e-5f, eps_b = (w_b->ln_eps > 0.f) ? w_b->ln_eps : 1e-5f;
  const Halves halves = shape_a->dtype == GSIT_BF16 ? pick_halves(ga, w_a->d_ff) : HALVES_NONE;
  const bool one_launch = (halves == HALVES_ROWS || halves == HALVES_TC) && eps_a == eps_b && ga.hd <= 32;
  if (!one_launch) {  // shapes the paired kernels do not cover: the two layers one after the other, same results
    st = gsit_im_layer_fwd(shape_a, w_a, x_a, x_a_row_stride, y_a, y_a_row_stride, ws, sc.total, stream);
    if (st != GSIT_OK) return st;
    return gsit_im_layer_fwd(shape_b, w_b, x_b, x_b_row_stride, y_b, y_b_row_stride, ws + sc.total, sc.total, stream);
  }
  const gsit_layer_weights* w[2] = {w_a, w_b};
  const float* x[2] = {x_a, x_b};
  float* y[2] = {y_a, y_b};
  const int64_t ldx[2] = {x_a_row_stride, x_b_row_stride}, ldy[2] = {y_a_row_stride, y_b_row_stride};
  for (int i = 0; i < 2; ++i) {
    if (!x[i] || !y[i] || ldx[i] < ga.d || ldy[i] < ga.d || ldx[i] % 4 != 0 || ldy[i] % 4 != 0) return GSIT_ERR_INVALID_ARG;
    if (!w[i]->w_qkv || !w[i]->w_o || !w[i]->w_1 || !w[i]->w_2) return GSIT_ERR_INVALID_ARG;
    if (!aligned16(x[i]) || !aligned16(y[i]) || !aligned16(w[i]->w_qkv) || !aligned16(w[i]->w_o) || !aligned16(w[i]->w_1) ||
        !aligned16(w[i]->w_2))
      return GSIT_ERR_INVALID_ARG;
  }
  if (from_cuda(status_ptr(&ga.status)) != GSIT_OK) return GSIT_ERR_CUDA;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  FusedHalfArgs h[2];
  AttnOperands ops[2];
  const uint32_t allowed[2] = {ga.allowed, gb.allowed};
  if (one_launch_layers(ga, shape_a->dtype, allowed, 2, w_a->d_ff, false)) {
    const LayerChain c = {{&w_a, &w_b}, {x_a, x_b}, {x_a_row_stride, x_b_row_stride}, {&y_a, &y_b}, {&y_a_row_stride, &y_b_row_stride}, {allowed[0], allowed[1]}};
    return run_chain(ga, c, 2, 1, pick_scale(shape_a, ga), ws, sc.total, sc, cs);
  }
  for (int i = 0; i < 2; ++i) {
    uint8_t* wsi = ws + i * sc.total;
    __nv_bfloat16* qkv = reinterpret_cast<__nv_bfloat16*>(wsi + sc.qkv);
    __nv_bfloat16* att = reinterpret_cast<__nv_bfloat16*>(wsi + sc.att);
    h[i] = half_args(w[i], x[i], ldx[i], qkv, att, y[i], ldy[i]);
    ops[i] = AttnOperands{qkv, qkv + ga.d, qkv + 2 * ga.d, att, nullptr, allowed[i]};
  }
  {
    TraceScope t(GSIT_KERNEL_LINEAR, cs);
    int* counter = reinterpret_cast<int*>(ws + sc.sched);
    st = from_cuda(halves == HALVES_ROWS ? launch_ln_qkv_rows(ga, h, 2, eps_a, counter, cs) : launch_ln_qkv_tc_pair(ga, h, eps_a, counter, cs));
    if (st != GSIT_OK) return st;
  }
  {
    TraceScope t(GSIT_KERNEL_ATTENTION, cs);
    if ((st = from_cuda(launch_attn_bf16_n(ga, ops, 2, 3 * (int64_t)ga.d, pick_scale(shape_a, ga),
                                           reinterpret_cast<int*>(ws + sc.sched), cs, true))) != GSIT_OK)
      return st;
  }
  TraceScope t(GSIT_KERNEL_LINEAR, cs);
  return from_cuda(halves == HALVES_ROWS ? launch_proj_mlp_rows(ga, h, 2, eps_a, w_a->d_ff, cs) : launch_proj_mlp_tc_pair(ga, h, eps_a, w_a->d_ff, cs));
}

int32_t gsit_encoder_runs_chained(const gsit_shape* const* shapes, int32_t problems, int32_t d_ff) {
  Geometry g[2];
  if (!shapes || problems < 1 || problems > 2 || d_ff < 1) return 0;
  uint32_t allowed[2];
  for (int i = 0; i < problems; ++i) {
    if (make_geometry(shapes[i], &g[i]) != GSIT_OK) return 0;
    allowed[i] = g[i].allowed;
  }
  return one_launch_layers(g[0], shapes[0]->dtype, allowed, problems, d_ff, true);
}

gsit_status gsit_im_encoder_fwd(const gsit_shape* const* shapes, int32_t problems, const gsit_layer_weights* const* const* weights, int32_t depth,
                                const float* const* x, const int64_t* x_row_stride, float* const* const* y, const int64_t* const* y_row_stride,
                                void* workspace, size_t workspace_bytes, gsit_stream stream) {
  if (!shapes || !weights || !x || !x_row_stride || !y || !y_row_stride || problems < 1 || problems > 2 || depth < 1) return GSIT_ERR_INVALID_ARG;
  for (int i = 0; i < problems; ++i) {
    if (!shapes[i] || !weights[i] || !y[i] || !y_row_stride[i]) return GSIT_ERR_INVALID_ARG;
    for (int j = 0; j < depth; ++j)
      if (!weights[i][j]) return GSIT_ERR_INVALID_ARG;
  }
  // the layers one call each, unless they can follow each other launch by launch; the calls also report what is wrong with an argument
  Geometry g[2] = {};
  LayerChain c = {};
  bool chained = depth > 1;
  int max_ff = 1;
  for (int i = 0; i < problems && chained; ++i) {
    chained = make_geometry(shapes[i], &g[i]) == GSIT_OK;
    c.w[i] = weights[i]; c.x[i] = x[i]; c.ldx[i] = x_row_stride[i]; c.y[i] = y[i]; c.ldy[i] = y_row_stride[i];
    c.allowed[i] = g[i].allowed;
    const Geometry &a = g[0], &b = g[i];
    chained = chained && a.batch == b.batch && a.d == b.d && a.heads == b.heads && a.valid_len == b.valid_len && a.row_start == b.row_start &&
              a.capacity == b.capacity && shapes[0]->dtype == shapes[i]->dtype && shapes[0]->scale == shapes[i]->scale &&
              a.seg_len[0] == b.seg_len[0] && a.seg_len[1] == b.seg_len[1] && a.seg_len[2] == b.seg_len[2];
    chained = chained && x[i] && aligned16(x[i]) && x_row_stride[i] >= a.d && x_row_stride[i] % 4 == 0;
    for (int j = 0; j < depth && chained; ++j) {
      const gsit_layer_weights *w = weights[i][j], *w0 = weights[0][j];
      chained = w->w_qkv && w->w_o && w->w_1 && w->w_2 && aligned16(w->w_qkv) && aligned16(w->w_o) && aligned16(w->w_1) && aligned16(w->w_2) &&
                w->d_ff >= 1 && w->d_ff == w0->d_ff && eps_of(w) == eps_of(w0) && y[i][j] && aligned16(y[i][j]) && y_row_stride[i][j] >= a.d &&
                y_row_stride[i][j] % 4 == 0;
      if (chained && w->d_ff > max_ff) max_ff = w->d_ff;
    }
  }
  for (int j = 0; j < depth && chained; ++j) chained = one_launch_layers(g[0], shapes[0]->dtype, c.allowed, problems, weights[0][j]->d_ff, true);
  if (chained) {
    const LayerScratch sc = layer_scratch(g[0], shapes[0]->dtype, max_ff);
    if (!workspace || workspace_bytes < problems * sc.total || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return GSIT_ERR_WORKSPACE;
    if (from_cuda(status_ptr(&g[0].status)) != GSIT_OK) return GSIT_ERR_CUDA;
    return run_chain(g[0], c, problems, depth, pick_scale(shapes[0], g[0]), static_cast<uint8_t*>(workspace), sc.total, sc,
                     static_cast<cudaStream_t>(stream));
  }
  for (int j = 0; j < depth; ++j) {
    const float* in[2];
    int64_t ld[2];
    for (int i = 0; i < problems; ++i) {
      in[i] = j == 0 ? x[i] : y[i][j - 1];
      ld[i] = j == 0 ? x_row_stride[i] : y_row_stride[i][j - 1];
    }
    const gsit_status st =
        problems == 1 ? gsit_im_layer_fwd(shapes[0], weights[0][j], in[0], ld[0], y[0][j], y_row_stride[0][j], workspace, workspace_bytes, stream)
                      : gsit_im_layer_pair_fwd(shapes[0], shapes[1], weights[0][j], weights[1][j], in[0], ld[0], in[1], ld[1], y[0][j],
                                               y_row_stride[0][j], y[1][j], y_row_stride[1][j], workspace, workspace_bytes, stream);
    if (st != GSIT_OK) return st;
  }
  return GSIT_OK;
}

gsit_status gsit_plan_rows(const gsit_shape* shape, int32_t split_sample, int32_t* row_start, gsit_stream stream) {
  if (shape == nullptr || row_start == nullptr || shape->valid_len == nullptr) return GSIT_ERR_INVALID_ARG;
  gsit_shape sh = *shape;  // only batch, seg_len and valid_len matter here: make the rest valid
  sh.d_model = 16; sh.heads = 1; sh.phase = GSIT_PHASE_INTRA; sh.dtype = GSIT_F32; sh.row_start = nullptr; sh.packed_capacity = 0;
  Geometry g;
  gsit_status st = make_geometry(&sh, &g);
  if (st != GSIT_OK) return st;
  if (split_sample < 0) return GSIT_ERR_INVALID_ARG;
  if (from_cuda(status_ptr(&g.status)) != GSIT_OK) return GSIT_ERR_CUDA;
  return from_cuda(launch_plan_rows(g, split_sample, row_start, static_cast<cudaStream_t>(stream)));
}

static gsit_status move_rows(const gsit_shape* shape, bool pack, const float* src, int64_t src_stride, float* dst,
                             int64_t dst_stride, int32_t cols, gsit_stream stream) {
  if (shape == nullptr || shape->row_start == nullptr || !src || !dst) return GSIT_ERR_INVALID_ARG;
  if (cols < 4 || cols % 4 != 0 || src_stride < cols || dst_stride < cols || src_stride % 4 != 0 || dst_stride % 4 != 0)
    return GSIT_ERR_INVALID_ARG;
  if (!aligned16(src) || !aligned16(dst)) return GSIT_ERR_INVALID_ARG;
  gsit_shape sh = *shape;
  sh.d_model = 16; sh.heads = 1; sh.phase = GSIT_PHASE_INTRA; sh.dtype = GSIT_F32;
  Geometry g;
  gsit_status st = make_geometry(&sh, &g);
  if (st != GSIT_OK) return st;
  if (from_cuda(status_ptr(&g.status)) != GSIT_OK) return GSIT_ERR_CUDA;
  return from_cuda(launch_move_rows(g, pack, src, src_stride, dst, dst_stride, cols, static_cast<cudaStream_t>(stream)));
}

gsit_status gsit_pack_rows(const gsit_shape* shape, const float* x, int64_t x_row_stride, float* x_packed,
                           int64_t packed_row_stride, int32_t cols, gsit_stream stream) {
  return move_rows(shape, true, x, x_row_stride, x_packed, packed_row_stride, cols, stream);
}

static gsit_status plan_pack(const gsit_shape* shape, int32_t* row_start, const float* x, int64_t x_row_stride, float* x_packed,
                             int64_t packed_row_stride, int32_t cols, int32_t* row_map, float* y, int64_t y_row_stride, gsit_stream stream) {
  if (shape == nullptr || row_start == nullptr || shape->valid_len == nullptr || !x || !x_packed) return GSIT_ERR_INVALID_ARG;
  if (cols < 4 || cols % 4 != 0 || x_row_stride < cols || packed_row_stride < cols || x_row_stride % 4 != 0 || packed_row_stride % 4 != 0)
    return GSIT_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(x_packed)) return GSIT_ERR_INVALID_ARG;
  gsit_shape sh = *shape;
  sh.d_model = 16; sh.heads = 1; sh.phase = GSIT_PHASE_INTRA; sh.dtype = GSIT_F32; sh.row_start = nullptr; sh.packed_capacity = 0;
  Geometry g;
  gsit_status st = make_geometry(&sh, &g);
  if (st != GSIT_OK) return st;
  if (from_cuda(status_ptr(&g.status)) != GSIT_OK) return GSIT_ERR_CUDA;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  if (plan_pack_supported(g))
    return from_cuda(launch_plan_pack(g, row_start, x, x_row_stride, x_packed, packed_row_stride, cols, row_map, y, y_row_stride, cs));
  if (row_map != nullptr) return GSIT_ERR_UNSUPPORTED;
  if ((st = from_cuda(launch_plan_rows(g, 0, row_start, cs))) != GSIT_OK) return st;
  g.row_start = row_start;
  return from_cuda(launch_move_rows(g, true, x, x_row_stride, x_packed, packed_row_stride, cols, cs));
}

gsit_status gsit_plan_pack_rows(const gsit_shape* shape, int32_t* row_start, const float* x, int64_t x_row_stride, float* x_packed,
                                int64_t packed_row_stride, int32_t cols, gsit_stream stream) {
  return plan_pack(shape, row_start, x, x_row_stride, x_packed, packed_row_stride, cols, nullptr, nullptr, 0, stream);
}

gsit_status gsit_plan_pack_map_rows(const gsit_shape* shape, int32_t* row_start, int32_t* row_map, const float* x, int64_t x_row_stride,
                                    float* x_packed, int64_t packed_row_stride, int32_t cols, float* y, int64_t y_row_stride, gsit_stream stream) {
  if (!row_map || !y || !aligned16(y) || y_row_stride < 2 * (int64_t)cols || y_row_stride % 4 != 0) return GSIT_ERR_INVALID_ARG;
  return plan_pack(shape, row_start, x, x_row_stride, x_packed, packed_row_stride, cols, row_map, y, y_row_stride, stream);
}

gsit_status gsit_unpack_rows(const gsit_shape* shape, const float* y_packed, int64_t packed_row_stride, float* y,
                             int64_t y_row_stride, int32_t cols, gsit_stream stream) {
  return move_rows(shape, false, y_packed, packed_row_stride, y, y_row_stride, cols, stream);
}

gsit_status gsit_stack_head_fwd(const gsit_shape* shape, const float* c, int64_t c_row_stride, int32_t d_c, const void* w_f,
                                const float* b_f, float* out, int32_t out_features, gsit_stream stream) {
  if (shape == nullptr || !c || !w_f || !out || d_c < 1 || out_features < 1 || c_row_stride < d_c) return GSIT_ERR_INVALID_ARG;
  gsit_shape sh = *shape;  // only batch, seg_len, valid_len and dtype matter here: make the rest valid
  sh.d_model = 16; sh.heads = 1; sh.phase = GSIT_PHASE_INTRA;
  sh.row_start = nullptr; sh.packed_capacity = 0;  // c is in the padded layout
  Geometry g;
  gsit_status st = make_geometry(&sh, &g);
  if (st != GSIT_OK) return st;
  if ((size_t)3 * d_c * sizeof(float) > 48 * 1024) return GSIT_ERR_UNSUPPORTED;
  if (from_cuda(status_ptr(&g.status)) != GSIT_OK) return GSIT_ERR_CUDA;
  return from_cuda(launch_stack_head(g, shape->dtype, c, c_row_stride, d_c, w_f, b_f, out, out_features,
                                     static_cast<cudaStream_t>(stream)));
}

size_t gsit_workspace_bytes(const gsit_shape* shape, int which_call, int32_t d_ff) {
  Geometry g;
  if (make_geometry(shape, &g) != GSIT_OK) return (size_t)-1;
  if (which_call == GSIT_CALL_LAYER) {
    if (d_ff < 1) return (size_t)-1;
    return layer_scratch(g, shape->dtype, d_ff).total;
  }
  if (which_call == GSIT_CALL_ATTENTION) return (shape->dtype == GSIT_BF16) ? ATTENTION_SCRATCH : 0;
  if (which_call == GSIT_CALL_QKV_PROJ) return 0;
  return (size_t)-1;
}

int32_t gsit_attention_uses_workspace(const gsit_shape* shape) {
  Geometry g;
  if (make_geometry(shape, &g) != GSIT_OK) return -1;
  return shape->dtype == GSIT_BF16 && attn_uses_tensor_memory(g, g.allowed) && (g.hd != 64 || attn_tc_hd64_uses_counter(g));
}

gsit_status gsit_last_device_status(gsit_stream stream, uint32_t* flags) {
  unsigned int* p = nullptr;
  if (status_ptr(&p) != cudaSuccess) return GSIT_ERR_CUDA;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  unsigned int host = 0;
  if (cudaMemcpyAsync(&host, p, sizeof(host), cudaMemcpyDeviceToHost, cs) != cudaSuccess) return GSIT_ERR_CUDA;
  if (cudaMemsetAsync(p, 0, sizeof(host), cs) != cudaSuccess) return GSIT_ERR_CUDA;
  if (cudaStreamSynchronize(cs) != cudaSuccess) return GSIT_ERR_CUDA;
  if (flags) *flags = host;
  return (host & GSIT_DEVFLAG_TIMEOUT) ? GSIT_ERR_TIMEOUT : GSIT_OK;
}

gsit_status gsit_trace_enable(int on) {
  g_trace_on = (on != 0);
  return GSIT_OK;
}

gsit_status gsit_trace_reset(void) {
  g_trace_n = 0;
  return GSIT_OK;
}

gsit_status gsit_trace_read(int kernel_kind, float* total_ms, int32_t* launches) {
  if (!total_ms || !launches) return GSIT_ERR_INVALID_ARG;
  float sum = 0.f;
  int n = 0;
  for (int i = 0; i < g_trace_n; ++i) {
    if (g_trace[i].kind != kernel_kind) continue;
    if (cudaEventSynchronize(g_trace[i].end) != cudaSuccess) return GSIT_ERR_CUDA;
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, g_trace[i].beg, g_trace[i].end) != cudaSuccess) return GSIT_ERR_CUDA;
    sum += ms;
    ++n;
  }
  *total_ms = sum;
  *launches = n;
  return GSIT_OK;
}

gsit_status gsit_trace_launches(int kernel_kind, float* out_ms, int32_t capacity, int32_t* launches) {
  if (!out_ms || !launches || capacity < 0) return GSIT_ERR_INVALID_ARG;
  int n = 0;
  for (int i = 0; i < g_trace_n && n < capacity; ++i) {
    if (g_trace[i].kind != kernel_kind) continue;
    if (cudaEventSynchronize(g_trace[i].end) != cudaSuccess) return GSIT_ERR_CUDA;
    if (cudaEventElapsedTime(&out_ms[n], g_trace[i].beg, g_trace[i].end) != cudaSuccess) return GSIT_ERR_CUDA;
    ++n;
  }
  *launches = n;
  return GSIT_OK;
}

const char* gsit_status_string(gsit_status s) {
  switch (s) {
    case GSIT_OK: return "ok";
    case GSIT_ERR_INVALID_ARG: return "invalid argument";
    case GSIT_ERR_UNSUPPORTED: return "unsupported shape or dtype";
    case GSIT_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case GSIT_ERR_CUDA: return "CUDA error";
    case GSIT_ERR_TIMEOUT: return "device-side wait timed out";
    default: return "unknown status";
  }
}

gsit_status gsit_test_expire_wait(gsit_stream stream) {
  unsigned int* p = nullptr;
  if (status_ptr(&p) != cudaSuccess) return GSIT_ERR_CUDA;
  expire_wait_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream)>>>(p, p, nullptr, 0);
  return from_cuda(cudaGetLastError());
}

gsit_status gsit_test_wait_answers(uint32_t* answers, int32_t cluster_form, gsit_stream stream) {
  if (!answers || (cluster_form != 0 && cluster_form != 1)) return GSIT_ERR_INVALID_ARG;
  expire_wait_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream)>>>(answers + 128, answers + 129, answers, cluster_form);
  return from_cuda(cudaGetLastError());
}

gsit_status gsit_test_late_write(void* dst, const void* src, size_t bytes, int32_t delay_us, gsit_stream stream) {
  if (!dst || !src || bytes % 16 != 0 || !aligned16(dst) || !aligned16(src) || delay_us < 0 || delay_us > 1000) return GSIT_ERR_INVALID_ARG;
  late_write_kernel<<<1, 256, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<uint4*>(dst), static_cast<const uint4*>(src), bytes / 16, delay_us);
  return from_cuda(cudaGetLastError());
}

gsit_status gsit_tune_attention(int choice) {
  if (choice != GSIT_ATTN_DEFAULT && choice != GSIT_ATTN_UNFUSED && choice != GSIT_ATTN_LEGACY && choice != GSIT_ATTN_TMEM)
    return GSIT_ERR_INVALID_ARG;
  g_attn_variant = choice;
  return GSIT_OK;
}

int gsit_version(void) { return 100; }

}  // extern "C"
