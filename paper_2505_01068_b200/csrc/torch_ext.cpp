// Native argument marshalling between torch tensors and the C ABI of libgsit.so (CPython extension `_native`).
//
// A small call of this library is one or two kernels of a few microseconds; marshalling it through ctypes in Python (struct
// building, shape checks, attribute look-ups, allocations through the dispatcher) took 20 - 25 us per call and was what
// bounded every call that the GPU finishes in less.  Here the same checks and the same allocations take about 2 us, so the
// launches themselves (about 2 us each) are what is left of the host path.  Nothing here computes.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <deque>
#include <exception>
#include <vector>

#include "gsit.h"

namespace {

PyObject* g_error = nullptr;  // binding.GsitError, set once by init()

struct PyFail {};  // a Python exception is set

[[noreturn]] void fail(PyObject* type, const char* msg) {
  PyErr_SetString(type, msg);
  throw PyFail{};
}
void require(bool ok, const char* what) {
  if (!ok) fail(PyExc_AssertionError, what);
}
void check(gsit_status st, const char* what) {
  if (st == GSIT_OK) return;
  PyObject* e = PyObject_CallFunction(g_error, "is", (int)st, what);
  if (e != nullptr) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  throw PyFail{};
}

const at::Tensor* opt_tensor(PyObject* o) {
  if (o == Py_None || o == nullptr) return nullptr;
  if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a torch tensor");
  return &THPVariable_Unpack(o);
}
const at::Tensor& tensor(PyObject* o) {
  const at::Tensor* t = opt_tensor(o);
  if (t == nullptr) fail(PyExc_TypeError, "expected a torch tensor, got None");
  return *t;
}
void* ptr(const at::Tensor* t) { return t == nullptr ? nullptr : t->data_ptr(); }

int64_t as_int(PyObject* o) {
  if (PyLong_CheckExact(o)) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyFail{};
    return v;
  }
  PyObject* n = PyNumber_Long(o);
  if (n == nullptr) throw PyFail{};
  const long long v = PyLong_AsLongLong(n);
  Py_DECREF(n);
  if (v == -1 && PyErr_Occurred()) throw PyFail{};
  return v;
}
double as_float(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyFail{};
  return v;
}
bool as_bool(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw PyFail{};
  return v != 0;
}

void read_segments(PyObject* seg, int32_t (&out)[3]) {
  PyObject* f = PySequence_Fast(seg, "seg_len must be a sequence of three lengths");
  if (f == nullptr) throw PyFail{};
  if (PySequence_Fast_GET_SIZE(f) != 3) {
    Py_DECREF(f);
    fail(PyExc_ValueError, "seg_len must hold three lengths");
  }
  try {
    for (int i = 0; i < 3; ++i) out[i] = (int32_t)as_int(PySequence_Fast_GET_ITEM(f, i));
  } catch (...) {
    Py_DECREF(f);
    throw;
  }
  Py_DECREF(f);
}

void require_vector(const at::Tensor* bias) {
  require(bias == nullptr || (bias->scalar_type() == at::kFloat && bias->is_contiguous()), "bias: contiguous float32");
}
int32_t dtype_code(const at::Tensor& t) {
  if (t.scalar_type() == at::kFloat) return GSIT_F32;
  if (t.scalar_type() == at::kBFloat16) return GSIT_BF16;
  fail(PyExc_TypeError, "unsupported dtype (float32 and bfloat16 are)");
}

gsit_shape make_shape(int64_t batch, PyObject* seg, int64_t d, int64_t heads, const at::Tensor* valid, int32_t dtype, int64_t phase,
                      int64_t mask, double scale, const at::Tensor* row_start = nullptr, int64_t capacity = 0) {
  gsit_shape s = {};
  s.batch = (int32_t)batch;
  read_segments(seg, s.seg_len);
  s.d_model = (int32_t)d;
  s.heads = (int32_t)heads;
  if (valid != nullptr) {
    require(valid->is_cuda() && valid->scalar_type() == at::kInt && valid->is_contiguous(), "valid_len: contiguous int32 device tensor");
    require(valid->dim() == 2 && valid->size(0) == batch && valid->size(1) == 3, "valid_len: shape [batch, 3]");
    s.valid_len = static_cast<const int32_t*>(valid->data_ptr());
  }
  if (row_start != nullptr) {
    require(row_start->is_cuda() && row_start->scalar_type() == at::kInt && row_start->is_contiguous(),
            "row_start: contiguous int32 device tensor");
    require(row_start->numel() >= 3 * batch + 1 && valid != nullptr && capacity >= 1, "row_start: 3 * batch + 1 entries, with valid_len");
    s.row_start = static_cast<const int32_t*>(row_start->data_ptr());
    s.packed_capacity = (int32_t)capacity;
  }
  s.dtype = dtype;
  s.phase = (int32_t)phase;
  s.custom_mask = (uint32_t)mask;
  s.scale = (float)scale;
  return s;
}

at::Tensor empty(at::IntArrayRef sizes, at::ScalarType t, const at::Device& dev) {
  return at::detail::empty_cuda(sizes, t, dev, std::nullopt);
}
size_t scratch_bytes(const gsit_shape& s, gsit_call call, int32_t d_ff) {
  const size_t n = gsit_workspace_bytes(&s, call, d_ff);
  if (n == (size_t)-1) check(GSIT_ERR_INVALID_ARG, "gsit_workspace_bytes");
  return n;
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

struct NoGil {  // a launch may block when the stream's queue is full: other Python threads go on meanwhile
  PyThreadState* s;
  NoGil() : s(PyEval_SaveThread()) {}
  ~NoGil() { PyEval_RestoreThread(s); }
};

// ---- layer weights ----
enum WKey { LN1_G, LN1_B, W_QKV, B_QKV, W_O, B_O, LN2_G, LN2_B, W_1, B_1, W_2, B_2, N_WKEYS };
const char* const W_NAMES[N_WKEYS] = {"ln1_g", "ln1_b", "w_qkv", "b_qkv", "w_o", "b_o", "ln2_g", "ln2_b", "w_1", "b_1", "w_2", "b_2"};
PyObject* g_wkeys[N_WKEYS];
PyObject* g_get;

// Owned references to the tensors of a layer's weights, kept until the call has been issued.  A plain dict is read directly; any
// other mapping (nn.ParameterDict, a subclass with its own look-up) as w[key] for the matrices and w.get(key) for the rest.
struct WeightRefs {
  PyObject* o[N_WKEYS] = {};
  WeightRefs() = default;
  WeightRefs(const WeightRefs&) = delete;
  ~WeightRefs() {
    for (PyObject* p : o) Py_XDECREF(p);
  }
};
bool is_matrix(int key) { return key == W_QKV || key == W_O || key == W_1 || key == W_2; }
void read_weights(PyObject* map, WeightRefs& r) {
  const bool dict = PyDict_CheckExact(map);
  for (const bool matrices : {true, false})
    for (int i = 0; i < N_WKEYS; ++i) {
      if (is_matrix(i) != matrices) continue;
      if (dict) r.o[i] = Py_XNewRef(PyDict_GetItemWithError(map, g_wkeys[i]));
      else r.o[i] = matrices ? PyObject_GetItem(map, g_wkeys[i]) : PyObject_CallMethodOneArg(map, g_get, g_wkeys[i]);
      if (r.o[i] == nullptr && matrices && !PyErr_Occurred()) PyErr_SetObject(PyExc_KeyError, g_wkeys[i]);
      if (r.o[i] == nullptr && PyErr_Occurred()) throw PyFail{};
    }
}

gsit_layer_weights layer_weights(PyObject* map, double eps, int32_t* dtype, WeightRefs& refs) {
  read_weights(map, refs);
  const void* p[N_WKEYS];
  gsit_layer_weights w = {};
  for (int i = 0; i < N_WKEYS; ++i) {
    const at::Tensor* t = opt_tensor(refs.o[i]);
    if (is_matrix(i)) {
      require(t != nullptr && t->is_cuda() && t->is_contiguous(), "layer weights: contiguous device matrices");
      if (i == W_QKV) *dtype = dtype_code(*t);
      require(dtype_code(*t) == *dtype, "layer weights: matrices of one type");
      if (i == W_1) w.d_ff = (int32_t)t->size(0);
    } else if (t != nullptr) {
      require(t->scalar_type() == at::kFloat && t->is_contiguous(), "layer weights: contiguous float32 vectors");
    }
    p[i] = ptr(t);
  }
  auto f = [&](int i) { return static_cast<const float*>(p[i]); };
  w.ln1_gamma = f(LN1_G); w.ln1_beta = f(LN1_B);
  w.w_qkv = p[W_QKV]; w.b_qkv = f(B_QKV);
  w.w_o = p[W_O]; w.b_o = f(B_O);
  w.ln2_gamma = f(LN2_G); w.ln2_beta = f(LN2_B);
  w.w_1 = p[W_1]; w.b_1 = f(B_1);
  w.w_2 = p[W_2]; w.b_2 = f(B_2);
  w.ln_eps = (float)eps;
  return w;
}

// ---- the calls; arguments in the order of the Python functions in binding.py ----

// x, w_qkv, b_qkv, seg_len, heads, valid_len, out, row_start
PyObject* im_qkv_proj(PyObject* const* a) {
  const at::Tensor &x = tensor(a[0]), &w = tensor(a[1]);
  const at::Tensor *bias = opt_tensor(a[2]), *valid = opt_tensor(a[5]), *out = opt_tensor(a[6]), *row_start = opt_tensor(a[7]);
  const int64_t heads = as_int(a[4]);
  require(x.is_cuda() && w.is_contiguous(), "x on the device, contiguous w_qkv");
  require(w.scalar_type() == x.scalar_type(), "x and w_qkv of one type");  // the call reads both in the type of x
  require_vector(bias);
  at::Tensor made;
  gsit_shape s;
  int64_t ldx;
  if (row_start != nullptr) {
    require(x.dim() == 2 && x.stride(1) == 1 && valid != nullptr, "packed x [capacity, d] with valid_len");
    s = make_shape(valid->size(0), a[3], x.size(1), heads, valid, dtype_code(x), GSIT_PHASE_INTRA, 0, 0.0, row_start, x.size(0));
    ldx = x.stride(0);
    if (out == nullptr) made = empty({x.size(0), 3, heads, x.size(1) / heads}, x.scalar_type(), x.device()).zero_();
  } else {
    require(x.dim() == 3 && x.stride(2) == 1 && x.stride(0) == x.size(1) * x.stride(1), "x [B, L, d] with a uniform row stride");
    s = make_shape(x.size(0), a[3], x.size(2), heads, valid, dtype_code(x), GSIT_PHASE_INTRA, 0, 0.0);
    ldx = x.stride(1);
    if (out == nullptr) made = empty({x.size(0), x.size(1), 3, heads, x.size(2) / heads}, x.scalar_type(), x.device());
  }
  void* dst = out != nullptr ? out->data_ptr() : made.data_ptr();
  gsit_status st;
  {
    NoGil n;
    st = gsit_im_qkv_proj(&s, x.data_ptr(), ldx, w.data_ptr(), static_cast<const float*>(ptr(bias)), dst, stream());
  }
  check(st, "gsit_im_qkv_proj");
  if (out != nullptr) return Py_NewRef(a[6]);
  return THPVariable_Wrap(std::move(made));
}

// q, k, v, seg_len, valid_len, phase, custom_mask, scale, want_lse, out, workspace
PyObject* im_attention_fwd(PyObject* const* a) {
  const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]);
  const at::Tensor *valid = opt_tensor(a[4]), *out = opt_tensor(a[9]), *ws = opt_tensor(a[10]);
  require(q.is_cuda() && k.is_cuda() && v.is_cuda() && q.dim() == 4, "q, k, v: [B, L, H, hd] on the device");
  for (const at::Tensor* t : {&k, &v})
    require(t->sizes() == q.sizes() && t->strides() == q.strides() && t->scalar_type() == q.scalar_type(), "q, k, v share shape, strides and dtype");
  const int64_t B = q.size(0), L = q.size(1), H = q.size(2), hd = q.size(3);
  require(q.stride(3) == 1 && q.stride(2) == hd && q.stride(0) == L * q.stride(1), "q, k, v: heads contiguous, uniform row stride");
  const gsit_shape s = make_shape(B, a[3], H * hd, H, valid, dtype_code(q), as_int(a[5]), as_int(a[6]), as_float(a[7]));
  const bool want_lse = as_bool(a[8]);
  at::Tensor made, lse, made_ws;
  if (out == nullptr) made = empty({B, L, H * hd}, q.scalar_type(), q.device());
  if (want_lse) lse = empty({B, H, L}, at::kFloat, q.device());
  // (an allocation is a quarter of what a small call takes on the host: only for the kernels that read their scratch)
  if (const int uses = ws == nullptr ? gsit_attention_uses_workspace(&s) : 0; uses != 0) {
    if (const size_t need = scratch_bytes(s, GSIT_CALL_ATTENTION, 0); need > 0) {  // an invalid shape raises here
      made_ws = empty({(int64_t)need}, at::kByte, q.device());
      ws = &made_ws;
    }
  }
  void* dst = out != nullptr ? out->data_ptr() : made.data_ptr();
  float* lse_p = want_lse ? static_cast<float*>(lse.data_ptr()) : nullptr;
  void* ws_p = ptr(ws);
  const size_t ws_n = ws == nullptr ? 0 : (size_t)ws->numel();
  gsit_status st;
  {
    NoGil n;
    st = gsit_im_attention_fwd(&s, q.data_ptr(), k.data_ptr(), v.data_ptr(), q.stride(1), dst, lse_p, ws_p, ws_n, stream());
  }
  check(st, "gsit_im_attention_fwd");
  PyObject* o = out != nullptr ? Py_NewRef(a[9]) : THPVariable_Wrap(std::move(made));
  if (!want_lse || o == nullptr) return o;
  PyObject* l = THPVariable_Wrap(std::move(lse));
  PyObject* pair = l == nullptr ? nullptr : PyTuple_Pack(2, o, l);
  Py_DECREF(o);
  Py_XDECREF(l);
  return pair;
}

// x, weights, seg_len, heads, valid_len, phase, custom_mask, scale, ln_eps, out, workspace, row_start, static scratch?
PyObject* im_layer_fwd(PyObject* const* a) {
  const at::Tensor& x = tensor(a[0]);
  const at::Tensor *valid = opt_tensor(a[4]), *out = opt_tensor(a[9]), *ws = opt_tensor(a[10]), *row_start = opt_tensor(a[11]);
  const bool use_static = as_bool(a[12]);
  int32_t dtype = GSIT_F32;
  WeightRefs refs;
  const gsit_layer_weights w = layer_weights(a[1], as_float(a[8]), &dtype, refs);
  require(x.is_cuda() && x.scalar_type() == at::kFloat && x.stride(-1) == 1, "x: float32 on the device, features contiguous");
  const int64_t heads = as_int(a[3]);
  at::Tensor made, made_ws;
  gsit_shape s;
  int64_t ldx, ldy;
  if (row_start != nullptr) {
    require(x.dim() == 2 && valid != nullptr && out != nullptr && out->size(0) == x.size(0) && out->stride(1) == 1,
            "packed rows: x and out [capacity, d], with valid_len");
    s = make_shape(valid->size(0), a[2], x.size(1), heads, valid, dtype, as_int(a[5]), as_int(a[6]), as_float(a[7]), row_start, x.size(0));
    ldx = x.stride(0);
    ldy = out->stride(0);
  } else {
    require(x.dim() == 3 && x.stride(0) == x.size(1) * x.stride(1), "x [B, L, d] with a uniform row stride");
    s = make_shape(x.size(0), a[2], x.size(2), heads, valid, dtype, as_int(a[5]), as_int(a[6]), as_float(a[7]));
    ldx = x.stride(1);
    if (out == nullptr) {
      made = empty(x.sizes(), at::kFloat, x.device());
      ldy = x.size(2);
    } else {
      require(out->dim() == 3 && out->stride(2) == 1 && out->stride(0) == x.size(1) * out->stride(1), "out [B, L, d] with a uniform row stride");
      ldy = out->stride(1);
    }
  }
  float* dst = static_cast<float*>(out != nullptr ? out->data_ptr() : made.data_ptr());
  if (!use_static && ws == nullptr) {
    made_ws = empty({(int64_t)scratch_bytes(s, GSIT_CALL_LAYER, w.d_ff)}, at::kByte, x.device());
    ws = &made_ws;
  }
  const float* src = static_cast<const float*>(x.data_ptr());
  void* ws_p = ptr(ws);
  const size_t ws_n = ws == nullptr ? 0 : (size_t)ws->numel();
  gsit_status st;
  {
    NoGil n;
    st = use_static ? gsit_im_layer_fwd_static(&s, &w, src, ldx, dst, ldy, stream())
                    : gsit_im_layer_fwd(&s, &w, src, ldx, dst, ldy, ws_p, ws_n, stream());
  }
  check(st, use_static ? "gsit_im_layer_fwd_static" : "gsit_im_layer_fwd");
  if (out != nullptr) return Py_NewRef(a[9]);
  return THPVariable_Wrap(std::move(made));
}

// c, w_f, b_f, seg_len, valid_len, out
PyObject* stack_head_fwd(PyObject* const* a) {
  const at::Tensor &c = tensor(a[0]), &w = tensor(a[1]);
  const at::Tensor *bias = opt_tensor(a[2]), *valid = opt_tensor(a[4]), *out = opt_tensor(a[5]);
  require(c.is_cuda() && c.scalar_type() == at::kFloat && c.dim() == 3 && c.stride(2) == 1 && c.stride(0) == c.size(1) * c.stride(1),
          "c: float32 [B, L, dc] on the device with a uniform row stride");
  require(w.is_contiguous() && w.dim() == 2 && w.size(1) == 3 * c.size(2), "w_f: contiguous [out_features, 3 * dc]");
  require_vector(bias);
  const gsit_shape s = make_shape(c.size(0), a[3], 16, 1, valid, dtype_code(w), GSIT_PHASE_INTRA, 0, 0.0);
  at::Tensor made;
  if (out == nullptr) made = empty({c.size(0), w.size(0)}, at::kFloat, c.device());
  float* dst = static_cast<float*>(out != nullptr ? out->data_ptr() : made.data_ptr());
  gsit_status st;
  {
    NoGil n;
    st = gsit_stack_head_fwd(&s, static_cast<const float*>(c.data_ptr()), c.stride(1), (int32_t)c.size(2), w.data_ptr(),
                             static_cast<const float*>(ptr(bias)), dst, (int32_t)w.size(0), stream());
  }
  check(st, "gsit_stack_head_fwd");
  if (out != nullptr) return Py_NewRef(a[5]);
  return THPVariable_Wrap(std::move(made));
}

// x_a, x_b, weights_a, weights_b, seg_len, heads, valid_len, phase_a, phase_b, ln_eps, out_a, out_b, workspace, row_start
PyObject* im_layer_pair_fwd(PyObject* const* a) {
  const at::Tensor &xa = tensor(a[0]), &xb = tensor(a[1]);
  const at::Tensor *valid = opt_tensor(a[6]), *oa = opt_tensor(a[10]), *ob = opt_tensor(a[11]), *ws = opt_tensor(a[12]), *row_start = opt_tensor(a[13]);
  int32_t dtype = GSIT_F32, other = GSIT_F32;
  WeightRefs refs_a, refs_b;
  const gsit_layer_weights wa = layer_weights(a[2], as_float(a[9]), &dtype, refs_a), wb = layer_weights(a[3], as_float(a[9]), &other, refs_b);
  require(dtype == other, "both layers' weights of one type");
  at::Tensor made[2], made_ws;
  const bool packed = row_start != nullptr;
  if (packed) require(xa.dim() == 2 && valid != nullptr && oa != nullptr && ob != nullptr, "packed rows: x and out [capacity, d], with valid_len");
  else require(xa.dim() == 3, "x [B, L, d]");
  if (oa == nullptr) { made[0] = empty(xa.sizes(), at::kFloat, xa.device()); oa = &made[0]; }
  if (ob == nullptr) { made[1] = empty(xa.sizes(), at::kFloat, xa.device()); ob = &made[1]; }
  for (const at::Tensor* t : {&xa, &xb, oa, ob})
    require(t->is_cuda() && t->scalar_type() == at::kFloat && t->sizes() == xa.sizes() && t->stride(-1) == 1,
            "x and out: float32 device tensors of one shape, features contiguous");
  const int64_t heads = as_int(a[5]), d = xa.size(-1), rows = packed ? valid->size(0) : xa.size(0);
  const gsit_shape sa = make_shape(rows, a[4], d, heads, valid, dtype, as_int(a[7]), 0, 0.0, row_start, packed ? xa.size(0) : 0);
  const gsit_shape sb = make_shape(rows, a[4], d, heads, valid, dtype, as_int(a[8]), 0, 0.0, row_start, packed ? xa.size(0) : 0);
  if (ws == nullptr) {
    made_ws = empty({(int64_t)(2 * scratch_bytes(sa, GSIT_CALL_LAYER, wa.d_ff))}, at::kByte, xa.device());
    ws = &made_ws;
  }
  const int sd = packed ? 0 : 1;
  gsit_status st;
  {
    NoGil n;
    st = gsit_im_layer_pair_fwd(&sa, &sb, &wa, &wb, static_cast<const float*>(xa.data_ptr()), xa.stride(sd),
                                static_cast<const float*>(xb.data_ptr()), xb.stride(sd), static_cast<float*>(oa->data_ptr()), oa->stride(sd),
                                static_cast<float*>(ob->data_ptr()), ob->stride(sd), ws->data_ptr(), (size_t)ws->numel(), stream());
  }
  check(st, "gsit_im_layer_pair_fwd");
  PyObject* ya = made[0].defined() ? THPVariable_Wrap(std::move(made[0])) : Py_NewRef(a[10]);
  PyObject* yb = made[1].defined() ? THPVariable_Wrap(std::move(made[1])) : Py_NewRef(a[11]);
  PyObject* pair = (ya == nullptr || yb == nullptr) ? nullptr : PyTuple_Pack(2, ya, yb);
  Py_XDECREF(ya);
  Py_XDECREF(yb);
  return pair;
}

// ---- the fusion stack: every launch of one forward issued from here ----

struct Layer {
  WeightRefs refs;
  int32_t dtype = GSIT_F32;
  gsit_layer_weights w;
};
std::deque<Layer> all_layers(PyObject* list, double eps) {
  require(PyList_Check(list), "layers: a list of weight mappings");
  std::deque<Layer> layers;
  for (Py_ssize_t i = 0; i < PyList_GET_SIZE(list); ++i) {
    Layer& l = layers.emplace_back();
    l.w = layer_weights(PyList_GET_ITEM(list, i), eps, &l.dtype, l.refs);
  }
  return layers;
}

// Are all layers of one type, of equal MLP width in a pair?  Then an encoder (pair) goes through one call.
bool uniform(const std::deque<Layer>& a, const std::deque<Layer>& b) {
  for (size_t i = 0; i < a.size(); ++i)
    if (a[i].dtype != a[0].dtype || b[i].dtype != a[0].dtype || a[i].w.d_ff != b[i].w.d_ff) return false;
  return true;
}
bool chained(const at::Tensor& x, PyObject* seg, int64_t heads, int64_t intra_heads, const at::Tensor* valid, const std::deque<Layer>& fwd,
             const std::deque<Layer>& bwd, const std::deque<Layer>& intra) {
  if (!uniform(fwd, bwd) || !uniform(intra, intra)) return false;
  auto all = [&](const std::deque<Layer>& layers, int64_t width, int64_t h, int problems) {
    for (const Layer& l : layers) {
      gsit_shape s[2];
      for (int i = 0; i < 2; ++i)
        s[i] = make_shape(x.size(0), seg, width, h, valid, l.dtype, problems == 1 ? GSIT_PHASE_INTRA : i ? GSIT_PHASE_INTER_BWD : GSIT_PHASE_INTER_FWD, 0, 0.0);
      const gsit_shape* shapes[2] = {&s[0], &s[1]};
      if (!gsit_encoder_runs_chained(shapes, problems, l.w.d_ff)) return false;
    }
    return true;
  };
  return all(fwd, x.size(2), heads, 2) && all(intra, 2 * x.size(2), intra_heads, 1);
}

// Do two float matrices of uniform row stride touch the same bytes anywhere between their first and last element?
bool overlap(const at::Tensor& a, const at::Tensor& b) {
  auto range = [](const at::Tensor& t, const char*& lo, const char*& hi) {
    lo = hi = static_cast<const char*>(t.data_ptr());
    if (t.numel() == 0) return;
    int64_t last = 0;
    for (int64_t i = 0; i < t.dim(); ++i) last += (t.size(i) - 1) * t.stride(i);
    hi += (last + 1) * t.element_size();
  };
  const char *a0, *a1, *b0, *b1;
  range(a, a0, a1);
  range(b, b0, b1);
  return a0 < b1 && b0 < a1;
}

// x, valid_len, y, fwd, bwd, intra, seg_len, heads, intra_heads, ln_eps, buffers
//   buffers = (plan or None, workspace, ring_a0, ring_a1, ring_b0, ring_b1, x_packed or None, wide_0, wide_1, row_map or None): with a
//   plan the packed row layout is used (x gathered into x_packed; the result scattered into y, by the last layer itself where it
//   can), without one the padded layout.
// Everything runs on the caller's stream, the whole batch per launch: every kernel then starts under the tail of the one
// before it.  (Halves of the batch on two streams in the intra encoder, 820 us against 784 at 64 x 1050 rows, 234 against
// 225 at 2 x 1050: the fork and the join each cost one such overlap.)
// Returns the status of the first call that did not succeed (0: all is issued).
PyObject* stack_forward(PyObject* const* a) {
  const at::Tensor &x = tensor(a[0]), &y = tensor(a[2]);
  const at::Tensor* valid = opt_tensor(a[1]);
  require(x.is_cuda() && x.scalar_type() == at::kFloat && x.dim() == 3 && x.stride(2) == 1 && x.stride(0) == x.size(1) * x.stride(1),
          "x: float32 [B, L, d] on the device with a uniform row stride");
  const double eps = as_float(a[9]);
  const std::deque<Layer> intra = all_layers(a[5], eps), fwd = all_layers(a[3], eps), bwd = all_layers(a[4], eps);
  require(fwd.size() == bwd.size() && !fwd.empty(), "rings of equal depth");
  require(PyTuple_Check(a[10]) && PyTuple_GET_SIZE(a[10]) == 10, "buffers: ten tensors");
  const at::Tensor* b[10];
  for (int i = 0; i < 10; ++i) b[i] = opt_tensor(PyTuple_GET_ITEM(a[10], i));
  // x may lie in y (a view of an earlier result): then it is gathered, or copied, before anything of y is written.  The gather must not
  // clear y's padding in the same launch, and no layer may read x while another kernel of the call writes y.
  const bool x_in_y = overlap(x, y);
  // layers that run as one launch each do no work for padding in the padded layout either: no plan, no copies between layouts then
  const at::Tensor* plan = b[0];
  if (plan != nullptr && !x_in_y && chained(x, a[6], as_int(a[7]), as_int(a[8]), valid, fwd, bwd, intra)) plan = nullptr;
  const int64_t B = x.size(0), d = x.size(2), cap = plan != nullptr ? b[6]->size(0) : 0;
  const gsit_shape ring_shape = make_shape(B, a[6], d, as_int(a[7]), valid, fwd[0].dtype, GSIT_PHASE_INTER_FWD, 0, 0.0, plan, cap);
  const gsit_shape intra_shape = make_shape(B, a[6], 2 * d, as_int(a[8]), valid, fwd[0].dtype, GSIT_PHASE_INTRA, 0, 0.0, plan, cap);
  uint8_t* ws = static_cast<uint8_t*>(b[1]->data_ptr());
  const size_t ws_n = (size_t)b[1]->numel(), ws_half = ws_n / 2;
  auto f = [](const at::Tensor* t) { return static_cast<float*>(t->data_ptr()); };
  float *ping_a[2] = {f(b[2]), f(b[3])}, *ping_b[2] = {f(b[4]), f(b[5])}, *wide[2] = {f(b[7]), f(b[8])};
  float* out = f(&y);
  at::Tensor copy;
  if (x_in_y && plan == nullptr && fwd.size() == 1 && intra.empty()) copy = x.clone(at::MemoryFormat::Contiguous);  // a first layer that is also the last
  const float* x_in = static_cast<const float*>(copy.defined() ? copy.data_ptr() : x.data_ptr());
  int64_t ldx = copy.defined() ? d : x.stride(1);
  gsit_stream cs = stream();

  auto issue = [&]() -> gsit_status {
    gsit_status st = GSIT_OK;
    int32_t* row_map = nullptr;  // the last layer writes the padded result itself
    if (plan != nullptr) {
      float* xp = f(b[6]);
      int32_t* starts = static_cast<int32_t*>(plan->data_ptr());
      if (!x_in_y && !intra.empty() && B <= 1024) {
        gsit_shape last = intra_shape;
        last.dtype = intra.back().dtype;
        if (gsit_layer_scatters(&last, intra.back().w.d_ff)) row_map = static_cast<int32_t*>(b[9]->data_ptr());
      }
      st = row_map != nullptr ? gsit_plan_pack_map_rows(&ring_shape, starts, row_map, x_in, ldx, xp, d, (int32_t)d, out, 2 * d, cs)
                              : gsit_plan_pack_rows(&ring_shape, starts, x_in, ldx, xp, d, (int32_t)d, cs);
      if (st != GSIT_OK) return st;
      x_in = xp;
      ldx = d;
    }
    // both rings side by side; the last layers write the halves of the concatenated rows
    float* c = (plan == nullptr && intra.empty()) ? out : wide[0];
    gsit_shape sa = ring_shape, sb = ring_shape;
    sb.phase = GSIT_PHASE_INTER_BWD;
    std::vector<float*> ya, yb, yi;
    std::vector<int64_t> ldr, ldi;
    std::vector<const gsit_layer_weights*> wf, wb, wi;
    for (size_t i = 0; i < fwd.size(); ++i) {
      const bool last = i + 1 == fwd.size();
      ya.push_back(last ? c : ping_a[i & 1]);
      yb.push_back(last ? c + d : ping_b[i & 1]);
      ldr.push_back(last ? 2 * d : d);
      wf.push_back(&fwd[i].w);
      wb.push_back(&bwd[i].w);
    }
    if (uniform(fwd, bwd)) {
      const gsit_shape* shapes[2] = {&sa, &sb};
      const gsit_layer_weights* const* w[2] = {wf.data(), wb.data()};
      const float* xs[2] = {x_in, x_in};
      const int64_t ldxs[2] = {ldx, ldx};
      float* const* ys[2] = {ya.data(), yb.data()};
      const int64_t* ldys[2] = {ldr.data(), ldr.data()};
      st = gsit_im_encoder_fwd(shapes, 2, w, (int32_t)fwd.size(), xs, ldxs, ys, ldys, ws, ws_n, cs);
      if (st != GSIT_OK) return st;
    } else {
      for (size_t i = 0; i < fwd.size(); ++i) {  // every layer in the type of its own weights; a pair of one type goes through one call
        const float *cur_a = i == 0 ? x_in : ya[i - 1], *cur_b = i == 0 ? x_in : yb[i - 1];
        const int64_t ld = i == 0 ? ldx : ldr[i - 1];
        sa.dtype = fwd[i].dtype;
        sb.dtype = bwd[i].dtype;
        if (sa.dtype == sb.dtype && fwd[i].w.d_ff == bwd[i].w.d_ff) {
          st = gsit_im_layer_pair_fwd(&sa, &sb, wf[i], wb[i], cur_a, ld, cur_b, ld, ya[i], ldr[i], yb[i], ldr[i], ws, ws_n, cs);
        } else {
          st = gsit_im_layer_fwd(&sa, wf[i], cur_a, ld, ya[i], ldr[i], ws, ws_half, cs);
          if (st == GSIT_OK) st = gsit_im_layer_fwd(&sb, wb[i], cur_b, ld, yb[i], ldr[i], ws + ws_half, ws_half, cs);
        }
        if (st != GSIT_OK) return st;
      }
    }
    int in_wide = 0;
    for (size_t i = 0; i < intra.size(); ++i) {
      yi.push_back((i + 1 == intra.size() && plan == nullptr) ? out : wide[in_wide ^ 1]);
      ldi.push_back(2 * d);
      wi.push_back(&intra[i].w);
      in_wide ^= 1;
    }
    gsit_shape si = intra_shape;
    const size_t plain = intra.size() - (row_map != nullptr ? 1 : 0);  // layers before the one that scatters
    if (plain > 0 && uniform(intra, intra)) {
      si.dtype = intra[0].dtype;
      const gsit_shape* shape = &si;
      const gsit_layer_weights* const* w = wi.data();
      const float* xs = wide[0];
      const int64_t ldxs = 2 * d;
      float* const* ys = yi.data();
      const int64_t* ldys = ldi.data();
      st = gsit_im_encoder_fwd(&shape, 1, &w, (int32_t)plain, &xs, &ldxs, &ys, &ldys, ws, ws_n, cs);
      if (st != GSIT_OK) return st;
    } else {
      for (size_t i = 0; i < plain; ++i) {
        si.dtype = intra[i].dtype;
        st = gsit_im_layer_fwd(&si, wi[i], i == 0 ? wide[0] : yi[i - 1], 2 * d, yi[i], 2 * d, ws, ws_n, cs);
        if (st != GSIT_OK) return st;
      }
    }
    if (row_map != nullptr) {
      si.dtype = intra[plain].dtype;
      return gsit_im_layer_scatter_fwd(&si, wi[plain], plain == 0 ? wide[0] : yi[plain - 1], 2 * d, row_map, out, 2 * d, ws, ws_n, cs);
    }
    if (plan != nullptr) st = gsit_unpack_rows(&ring_shape, wide[in_wide], 2 * d, out, 2 * d, (int32_t)(2 * d), cs);
    return st;
  };
  gsit_status st;
  {
    NoGil n;
    st = issue();
  }
  return PyLong_FromLong(st);
}

// ---- module ----
template <PyObject* (*F)(PyObject* const*), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
    return nullptr;
  }
  try {
    return F(args);
  } catch (const PyFail&) {
  } catch (...) {
    // as torch itself raises it: a failed allocation is torch.OutOfMemoryError, which callers catch to go on with a smaller batch
    try {
      torch::translate_exception_to_python(std::current_exception());
    } catch (...) {
    }
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, "unknown C++ exception");
  }
  return nullptr;
}

PyObject* init(PyObject* const* a) {
  Py_INCREF(a[0]);
  g_error = a[0];
  Py_RETURN_NONE;
}

template <PyObject* (*F)(PyObject* const*), int N>
PyMethodDef def(const char* name) {
  return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<F, N>)), METH_FASTCALL, nullptr};
}
PyMethodDef methods[] = {def<init, 1>("init"),
                         def<im_qkv_proj, 8>("im_qkv_proj"),
                         def<im_attention_fwd, 11>("im_attention_fwd"),
                         def<im_layer_fwd, 13>("im_layer_fwd"),
                         def<im_layer_pair_fwd, 14>("im_layer_pair_fwd"),
                         def<stack_head_fwd, 6>("stack_head_fwd"),
                         def<stack_forward, 11>("stack_forward"),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  for (int i = 0; i < N_WKEYS; ++i) g_wkeys[i] = PyUnicode_InternFromString(W_NAMES[i]);
  g_get = PyUnicode_InternFromString("get");
  return PyModule_Create(&module);
}
