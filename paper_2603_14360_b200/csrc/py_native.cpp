// Native half of the Python binding: argument checks, output allocation and the call into
// libm2rnn.so for the entry points a model runs on every layer and token.
//
// A small call (one decoded token: a few microseconds on the GPU) is bound by its host path.  The same
// marshalling in Python -- shape tuples, one ctypes argument object per pointer, torch.empty through
// the dispatcher -- took 18-24 us a call (B200 host, 60 us for the three calls of a decoded token's
// layer); here a check is a few compares on the tensor's own size and stride arrays and an output is
// one call of the caching allocator.  binding.py keeps the signatures and documentation and passes
// its arguments on by position.  Errors are the binding's: ValueError (shape, layout, device),
// TypeError (element type), M2RNNError (a status of the library).
#include <Python.h>

#include <ATen/core/TensorBody.h>
#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/zeros.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdarg>
#include <mutex>
#include <vector>

#include "m2rnn.h"

namespace {

using at::Tensor;
using at::ScalarType;

PyObject *g_error_class = nullptr;   // binding.M2RNNError

[[noreturn]] void fail(PyObject *type, const char *fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  PyErr_FormatV(type, fmt, ap);
  va_end(ap);
  throw python_error();
}

void check_rc(int rc, const char *where) {
  if (rc == M2RNN_OK) return;
  PyObject *e = PyObject_CallFunction(g_error_class, "is", rc, where);
  if (e) {
    PyErr_SetObject(g_error_class, e);
    Py_DECREF(e);
  }
  throw python_error();
}

// ---- arguments by position
const Tensor *opt_tensor(PyObject *o, const char *name) {
  if (o == Py_None) return nullptr;
  if (!THPVariable_Check(o)) fail(PyExc_TypeError, "%s must be a tensor, got %s", name, Py_TYPE(o)->tp_name);
  return &THPVariable_Unpack(o);
}
const Tensor &tensor(PyObject *o, const char *name) {
  const Tensor *t = opt_tensor(o, name);
  if (!t) fail(PyExc_TypeError, "%s must be a tensor, got None", name);
  return *t;
}
long integer(PyObject *o) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) throw python_error();
  return v;
}
double real(PyObject *o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw python_error();
  return v;
}
bool truth(PyObject *o) {
  if (o == Py_True) return true;
  if (o == Py_False || o == Py_None) return false;
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw python_error();
  return v != 0;
}
void want_args(Py_ssize_t got, Py_ssize_t want) {
  if (got != want) fail(PyExc_TypeError, "%zd arguments expected, got %zd", want, got);
}

void *stream_of(PyObject *o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw python_error();
  void *s = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (!s && PyErr_Occurred()) throw python_error();
  return s;
}

int32_t io_code(const Tensor &t) {
  if (t.scalar_type() == ScalarType::Float) return M2RNN_F32;
  if (t.scalar_type() == ScalarType::BFloat16) return M2RNN_BF16;
  fail(PyExc_TypeError, "unsupported I/O dtype %s", c10::toString(t.scalar_type()));
}

std::string shape_text(at::IntArrayRef s) {
  std::string r = "(";
  for (size_t i = 0; i < s.size(); ++i) r += (i ? ", " : "") + std::to_string(s[i]);
  return r + (s.size() == 1 ? ",)" : ")");
}

// shape, type and place of a tensor (absent ones pass); strided: the token layout is checked elsewhere
void check(const Tensor *t, const char *name, at::IntArrayRef shape, ScalarType dtype, bool strided = false) {
  if (!t) return;
  if (!t->is_cuda()) fail(PyExc_ValueError, "%s must be a CUDA tensor", name);
  if (t->sizes() != shape)
    fail(PyExc_ValueError, "%s: expected shape %s, got %s", name, shape_text(shape).c_str(), shape_text(t->sizes()).c_str());
  if (t->scalar_type() != dtype)
    fail(PyExc_TypeError, "%s: expected %s, got %s", name, c10::toString(dtype), c10::toString(t->scalar_type()));
  if (!strided && !t->is_contiguous()) fail(PyExc_ValueError, "%s must be contiguous", name);
}
void check(const Tensor &t, const char *name, at::IntArrayRef shape, ScalarType dtype, bool strided = false) {
  check(&t, name, shape, dtype, strided);
}
void need_dims(const Tensor &t, const char *name, int64_t d) {
  if (t.dim() != d) fail(PyExc_ValueError, "%s: expected %lld axes, got %lld", name, (long long)d, (long long)t.dim());
}

Tensor empty(at::IntArrayRef shape, ScalarType dtype, const at::Device &dev) {
  return Tensor(at::detail::empty_cuda(shape, dtype, dev, std::nullopt));
}
// the caller's tensor, or a new one
Tensor given_or_empty(const Tensor *t, at::IntArrayRef shape, ScalarType dtype, const at::Device &dev) {
  return t ? *t : empty(shape, dtype, dev);
}

void *ptr(const Tensor &t) { return t.defined() ? t.data_ptr() : nullptr; }
void *ptr(const Tensor *t) { return t ? t->data_ptr() : nullptr; }
template <typename P> float *fptr(const P &t) { return static_cast<float *>(ptr(t)); }

PyObject *wrap(const Tensor &t) {
  if (!t.defined()) Py_RETURN_NONE;
  return THPVariable_Wrap(t);
}
// an output as a Python object: the caller's own object where one was given
PyObject *back(PyObject *given, const Tensor &t) {
  if (given != Py_None) { Py_INCREF(given); return given; }
  return wrap(t);
}

// The int32 words that kernels raise when a bounded wait runs out: one per device, kept for the life
// of the process (never destroyed: the CUDA context may be gone by then).
std::mutex g_status_mutex;
std::vector<Tensor> &status_words() {
  static auto *v = new std::vector<Tensor>();
  return *v;
}
int32_t *status_ptr(int idx);
Tensor status_word_of(int idx) {
  std::lock_guard<std::mutex> lock(g_status_mutex);
  auto &v = status_words();
  if ((int)v.size() <= idx) v.resize(idx + 1);
  if (!v[idx].defined()) v[idx] = at::zeros({1}, at::TensorOptions().dtype(at::kInt).device(at::kCUDA, idx));
  return v[idx];
}
int32_t *status_ptr(int idx) {
  constexpr int kMax = 64;
  static int32_t *cached[kMax] = {};   // written once per device, under the GIL
  if (idx >= 0 && idx < kMax && cached[idx]) return cached[idx];
  int32_t *p = static_cast<int32_t *>(status_word_of(idx).data_ptr());
  if (idx >= 0 && idx < kMax) cached[idx] = p;
  return p;
}
int32_t *status_of(const Tensor &t) { return status_ptr(t.device().index()); }

// Elements between consecutive tokens of q, k or v ([B,T,heads,dim] or packed [tokens,heads,dim]);
// 0 stands for the dense layout
int64_t token_stride(const Tensor &t, const char *name) {
  if (t.numel() == 0) return 0;
  const auto sz = t.sizes(), st = t.strides();
  const size_t d = sz.size();
  if (st[d - 1] != 1 || st[d - 2] != sz[d - 1]) fail(PyExc_ValueError, "%s: the heads of a token must be contiguous", name);
  const int64_t tok = st[d - 3];
  if (d == 4 && sz[0] > 1 && st[0] != sz[1] * tok)
    fail(PyExc_ValueError, "%s: batch entries must follow one another along the token axis", name);
  return tok == sz[d - 2] * sz[d - 1] ? 0 : tok;
}

struct Scan {
  m2rnn_params p{};
  int64_t lead[2];
  int nlead;
  ScalarType io;
  c10::SmallVector<int64_t, 4> tok(int64_t heads, int64_t dim) const {   // a per-token tensor's shape
    c10::SmallVector<int64_t, 4> s(lead, lead + nlead);
    s.push_back(heads); s.push_back(dim);
    return s;
  }
  c10::SmallVector<int64_t, 4> gate() const {
    c10::SmallVector<int64_t, 4> s(lead, lead + nlead);
    s.push_back(p.N);
    return s;
  }
};

Scan scan_params(const Tensor &q, const Tensor &k, const Tensor &v, long gate_kind, long ckpt_interval, double dh_clip,
                 const Tensor *cu, PyObject *max_seqlen) {
  Scan s;
  m2rnn_params &p = s.p;
  s.io = q.scalar_type();
  if (cu) {
    if (cu->scalar_type() != ScalarType::Int || !cu->is_cuda() || !cu->is_contiguous())
      fail(PyExc_TypeError, "cu_seqlens must be a contiguous int32 CUDA tensor of B + 1 offsets");
    if (max_seqlen == Py_None) fail(PyExc_ValueError, "max_seqlen (the longest sequence) is required with cu_seqlens");
    need_dims(q, "q", 3); need_dims(k, "k", 3); need_dims(v, "v", 3);
    p.total_tokens = q.size(0);
    p.B = (int32_t)(cu->numel() - 1);
    PyObject *n = PyNumber_Long(max_seqlen);
    if (!n) throw python_error();
    p.T = (int32_t)PyLong_AsLong(n);
    Py_DECREF(n);
    if (PyErr_Occurred()) throw python_error();
    p.cu_seqlens = static_cast<const int32_t *>(cu->data_ptr());
    s.lead[0] = q.size(0); s.nlead = 1;
  } else {
    need_dims(q, "q", 4); need_dims(k, "k", 4); need_dims(v, "v", 4);
    p.B = (int32_t)q.size(0); p.T = (int32_t)q.size(1);
    s.lead[0] = p.B; s.lead[1] = p.T; s.nlead = 2;
  }
  p.Nq = (int32_t)q.size(-2); p.K = (int32_t)q.size(-1);
  p.Nk = (int32_t)k.size(-2);
  p.N = (int32_t)v.size(-2); p.V = (int32_t)v.size(-1);
  p.io_dtype = io_code(q);
  p.gate_kind = (int32_t)gate_kind;
  p.ckpt_interval = (int32_t)ckpt_interval;
  p.dh_clip = (float)dh_clip;
  p.q_stride = token_stride(q, "q"); p.k_stride = token_stride(k, "k"); p.v_stride = token_stride(v, "v");
  return s;
}

void check_scan(const Scan &s, const Tensor &q, const Tensor &k, const Tensor &v, const Tensor &gate, const Tensor &W,
                const Tensor *h0, const Tensor *alpha, const Tensor *beta, const Tensor *w_r) {
  const m2rnn_params &p = s.p;
  check(q, "q", s.tok(p.Nq, p.K), s.io, true);
  check(k, "k", s.tok(p.Nk, p.K), s.io, true);
  check(v, "v", s.tok(p.N, p.V), s.io, true);
  check(gate, "gate", s.gate(), ScalarType::Float);
  check(W, "W", {p.N, p.V, p.V}, s.io);
  check(h0, "h0", {p.B, p.N, p.K, p.V}, ScalarType::Float);
  check(w_r, "w_r", {p.N, p.V}, s.io);
  check(alpha, "alpha", {p.N}, ScalarType::Float);
  check(beta, "beta", {p.N}, ScalarType::Float);
}

int interval(const m2rnn_params &p) {
  const int c = m2rnn_ckpt_interval(&p);
  if (c <= 0) check_rc(c, "m2rnn_ckpt_interval");
  return c;
}

size_t bytes_of(const Tensor &t) { return t.defined() ? (size_t)t.numel() : 0; }

// fwd(q, k, v, gate, W, h0, gate_kind, alpha, beta, w_r, save_ckpt, ckpt_interval, want_hT, y, hT, ckpt, workspace, stream,
//     cu_seqlens, max_seqlen) -> (y, hT, ckpt)
PyObject *py_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  want_args(n, 20);
  const Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v"), &gate = tensor(a[3], "gate"), &W = tensor(a[4], "W");
  const Tensor *h0 = opt_tensor(a[5], "h0"), *alpha = opt_tensor(a[7], "alpha"), *beta = opt_tensor(a[8], "beta"), *w_r = opt_tensor(a[9], "w_r");
  const Tensor *cu = opt_tensor(a[18], "cu_seqlens");
  const Scan s = scan_params(q, k, v, integer(a[6]), integer(a[11]), 0.0, cu, a[19]);
  const m2rnn_params &p = s.p;
  check_scan(s, q, k, v, gate, W, h0, alpha, beta, w_r);
  const at::Device dev = q.device();
  const Tensor y = given_or_empty(opt_tensor(a[13], "y"), s.tok(p.N, p.V), s.io, dev);
  Tensor hT, ckpt, ws;
  if (const Tensor *t = opt_tensor(a[14], "hT")) hT = *t;
  else if (truth(a[12])) hT = empty({p.B, p.N, p.K, p.V}, ScalarType::Float, dev);
  if (const Tensor *t = opt_tensor(a[15], "ckpt")) {
    ckpt = *t;
    if (!ckpt.is_cuda()) fail(PyExc_ValueError, "ckpt must be a CUDA tensor");
    if (ckpt.nbytes() < m2rnn_ckpt_bytes(&p)) fail(PyExc_ValueError, "ckpt: smaller than m2rnn_ckpt_bytes");   // (the call itself cannot tell)
  }
  else if (truth(a[10])) {
    const int C = interval(p);
    ckpt = empty({p.B, p.N, (p.T + C - 1) / C, p.K, p.V}, ScalarType::Float, dev);
  }
  check(y, "y", s.tok(p.N, p.V), s.io);
  check(hT.defined() ? &hT : nullptr, "hT", {p.B, p.N, p.K, p.V}, ScalarType::Float);
  if (const Tensor *t = opt_tensor(a[16], "workspace")) ws = *t;
  else if (const size_t need = m2rnn_fwd_workspace_bytes(&p)) ws = empty({(int64_t)need}, ScalarType::Byte, dev);
  void *st = stream_of(a[17]);
  int32_t *status = status_of(q);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = m2rnn_fwd(&p, ptr(q), ptr(k), ptr(v), fptr(gate), ptr(W), fptr(h0), fptr(alpha), fptr(beta), ptr(w_r), ptr(y), fptr(hT),
                 fptr(ckpt), ptr(ws), bytes_of(ws), status, st);
  Py_END_ALLOW_THREADS
  check_rc(rc, "m2rnn_fwd");
  PyObject *r = PyTuple_New(3);
  if (!r) throw python_error();
  PyTuple_SET_ITEM(r, 0, back(a[13], y));
  PyTuple_SET_ITEM(r, 1, back(a[14], hT));
  PyTuple_SET_ITEM(r, 2, back(a[15], ckpt));
  return r;
  END_HANDLE_TH_ERRORS
}

struct Out { const char *name; PyObject *given; const Tensor *t; };
PyObject *dict_of(std::initializer_list<Out> items) {
  PyObject *d = PyDict_New();
  if (!d) throw python_error();
  for (const Out &o : items) {
    PyObject *v = o.given ? back(o.given, *o.t) : wrap(*o.t);
    if (!v || PyDict_SetItemString(d, o.name, v)) throw python_error();
    Py_DECREF(v);
  }
  return d;
}

// bwd(q, k, v, gate, W, h0, dy, d_hT, ckpt, gate_kind, alpha, beta, w_r, ckpt_interval, dh_clip, want_dh0, workspace, dq, dk, dv,
//     dgate, dW, dh0, stream, cu_seqlens, max_seqlen) -> dict
PyObject *py_bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  want_args(n, 26);
  const Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v"), &gate = tensor(a[3], "gate"), &W = tensor(a[4], "W");
  const Tensor *h0 = opt_tensor(a[5], "h0"), &dy = tensor(a[6], "dy"), *d_hT = opt_tensor(a[7], "d_hT"), *ckpt = opt_tensor(a[8], "ckpt");
  const Tensor *alpha = opt_tensor(a[10], "alpha"), *beta = opt_tensor(a[11], "beta"), *w_r = opt_tensor(a[12], "w_r");
  const Tensor *cu = opt_tensor(a[24], "cu_seqlens");
  const Scan s = scan_params(q, k, v, integer(a[9]), integer(a[13]), real(a[14]), cu, a[25]);
  const m2rnn_params &p = s.p;
  check_scan(s, q, k, v, gate, W, h0, alpha, beta, w_r);
  check(dy, "dy", s.tok(p.N, p.V), s.io);
  check(d_hT, "d_hT", {p.B, p.N, p.K, p.V}, ScalarType::Float);
  if (ckpt && p.T > 0) {
    const int C = interval(p);
    check(ckpt, "ckpt", {p.B, p.N, (p.T + C - 1) / C, p.K, p.V}, ScalarType::Float);
  }
  const at::Device dev = q.device();
  const Tensor dq = given_or_empty(opt_tensor(a[17], "dq"), q.sizes(), s.io, dev);
  const Tensor dk = given_or_empty(opt_tensor(a[18], "dk"), k.sizes(), s.io, dev);
  const Tensor dv = given_or_empty(opt_tensor(a[19], "dv"), v.sizes(), s.io, dev);
  const Tensor dgate = given_or_empty(opt_tensor(a[20], "dgate"), gate.sizes(), ScalarType::Float, dev);
  const Tensor dW = given_or_empty(opt_tensor(a[21], "dW"), {p.N, p.V, p.V}, ScalarType::Float, dev);
  Tensor dh0, ws;
  if (const Tensor *t = opt_tensor(a[22], "dh0")) dh0 = *t;
  else if (truth(a[15])) dh0 = empty({p.B, p.N, p.K, p.V}, ScalarType::Float, dev);
  check(dq, "dq", q.sizes(), s.io);
  check(dk, "dk", k.sizes(), s.io);
  check(dv, "dv", v.sizes(), s.io);
  if (const Tensor *t = opt_tensor(a[16], "workspace")) ws = *t;
  else {
    const size_t need = m2rnn_bwd_workspace_bytes(&p, ckpt != nullptr);
    ws = empty({(int64_t)(need ? need : 1)}, ScalarType::Byte, dev);
  }
  void *st = stream_of(a[23]);
  int32_t *status = status_of(q);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = m2rnn_bwd(&p, ptr(q), ptr(k), ptr(v), fptr(gate), ptr(W), fptr(h0), fptr(alpha), fptr(beta), ptr(w_r), fptr(ckpt), ptr(dy),
                 fptr(d_hT), ptr(dq), ptr(dk), ptr(dv), fptr(dgate), fptr(dW), fptr(dh0), ptr(ws), bytes_of(ws), status, st);
  Py_END_ALLOW_THREADS
  check_rc(rc, "m2rnn_bwd");
  return dict_of({{"dq", a[17], &dq}, {"dk", a[18], &dk}, {"dv", a[19], &dv}, {"dgate", a[20], &dgate}, {"dW", a[21], &dW}, {"dh0", a[22], &dh0}});
  END_HANDLE_TH_ERRORS
}

// decode_step(q, k, v, gate, W, state, gate_kind, alpha, beta, w_r, y, stream) -> y
PyObject *py_decode_step(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  want_args(n, 12);
  const Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v"), &gate = tensor(a[3], "gate"), &W = tensor(a[4], "W");
  const Tensor &state = tensor(a[5], "state"), *alpha = opt_tensor(a[7], "alpha"), *beta = opt_tensor(a[8], "beta"), *w_r = opt_tensor(a[9], "w_r");
  need_dims(q, "q", 3); need_dims(k, "k", 3); need_dims(v, "v", 3);
  m2rnn_params p{};
  p.B = (int32_t)q.size(0); p.T = 1; p.Nq = (int32_t)q.size(1); p.K = (int32_t)q.size(2);
  p.Nk = (int32_t)k.size(1); p.N = (int32_t)v.size(1); p.V = (int32_t)v.size(2);
  p.io_dtype = io_code(q);
  p.gate_kind = (int32_t)integer(a[6]);
  const ScalarType io = q.scalar_type();
  check(q, "q", {p.B, p.Nq, p.K}, io);
  check(k, "k", {p.B, p.Nk, p.K}, io);
  check(v, "v", {p.B, p.N, p.V}, io);
  check(gate, "gate", {p.B, p.N}, ScalarType::Float);
  check(W, "W", {p.N, p.V, p.V}, io);
  check(state, "state", {p.B, p.N, p.K, p.V}, ScalarType::Float);
  check(w_r, "w_r", {p.N, p.V}, io);
  check(alpha, "alpha", {p.N}, ScalarType::Float);
  check(beta, "beta", {p.N}, ScalarType::Float);
  const Tensor y = given_or_empty(opt_tensor(a[10], "y"), {p.B, p.N, p.V}, io, q.device());
  check(y, "y", {p.B, p.N, p.V}, io);
  void *st = stream_of(a[11]);
  int32_t *status = status_of(q);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = m2rnn_decode_step(&p, ptr(q), ptr(k), ptr(v), fptr(gate), ptr(W), fptr(alpha), fptr(beta), ptr(w_r), fptr(state), ptr(y), status, st);
  Py_END_ALLOW_THREADS
  check_rc(rc, "m2rnn_decode_step");
  return back(a[10], y);
  END_HANDLE_TH_ERRORS
}

// tokens and features of y [..., N, V]
void norm_dims(const Tensor &y, int64_t &tokens, int64_t &d) {
  if (y.dim() < 2) fail(PyExc_ValueError, "y needs at least the two trailing axes [N, V]");
  d = y.size(-2) * y.size(-1);
  tokens = d ? y.numel() / d : 0;
}

// gated_norm_fwd(y, g_in, w, eps, silu, out, rstd, stream) -> (out, rstd)
PyObject *py_gated_norm_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  want_args(n, 8);
  const Tensor &y = tensor(a[0], "y"), &g = tensor(a[1], "g_in"), &w = tensor(a[2], "w");
  int64_t tokens, d;
  norm_dims(y, tokens, d);
  const ScalarType io = y.scalar_type();
  check(y, "y", y.sizes(), io);
  check(g, "g_in", y.sizes(), io);
  check(w, "w", w.sizes(), io);
  if (w.numel() != d) fail(PyExc_ValueError, "w has %lld entries, the rows have %lld", (long long)w.numel(), (long long)d);
  const at::IntArrayRef rows = y.sizes().slice(0, y.dim() - 2);
  const Tensor out = given_or_empty(opt_tensor(a[5], "out"), y.sizes(), io, y.device());
  const Tensor rstd = given_or_empty(opt_tensor(a[6], "rstd"), rows, ScalarType::Float, y.device());
  check(out, "out", y.sizes(), io);
  check(rstd, "rstd", rows, ScalarType::Float);
  const double eps = real(a[3]);
  const int silu = truth(a[4]);
  const int32_t code = io_code(y);
  void *st = stream_of(a[7]);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = m2rnn_gated_norm_fwd(tokens, (int32_t)d, code, ptr(y), ptr(g), ptr(w), (float)eps, silu, ptr(out), fptr(rstd), st);
  Py_END_ALLOW_THREADS
  check_rc(rc, "m2rnn_gated_norm_fwd");
  PyObject *r = PyTuple_New(2);
  if (!r) throw python_error();
  PyTuple_SET_ITEM(r, 0, back(a[5], out));
  PyTuple_SET_ITEM(r, 1, back(a[6], rstd));
  return r;
  END_HANDLE_TH_ERRORS
}

// gated_norm_bwd(y, g_in, w, rstd, dout, silu, workspace, dy, dg, dw, stream) -> dict
PyObject *py_gated_norm_bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  want_args(n, 11);
  const Tensor &y = tensor(a[0], "y"), &g = tensor(a[1], "g_in"), &w = tensor(a[2], "w"), &rstd = tensor(a[3], "rstd"), &dout = tensor(a[4], "dout");
  int64_t tokens, d;
  norm_dims(y, tokens, d);
  const ScalarType io = y.scalar_type();
  check(y, "y", y.sizes(), io);
  check(g, "g_in", y.sizes(), io);
  check(dout, "dout", y.sizes(), io);
  check(w, "w", w.sizes(), io);
  if (w.numel() != d) fail(PyExc_ValueError, "w has %lld entries, the rows have %lld", (long long)w.numel(), (long long)d);
  check(rstd, "rstd", y.sizes().slice(0, y.dim() - 2), ScalarType::Float);
  const at::Device dev = g.device();
  const Tensor dy = given_or_empty(opt_tensor(a[7], "dy"), y.sizes(), io, dev);
  const Tensor dg = given_or_empty(opt_tensor(a[8], "dg"), y.sizes(), io, dev);
  const Tensor dw = given_or_empty(opt_tensor(a[9], "dw"), {d}, ScalarType::Float, dev);
  check(dy, "dy", y.sizes(), io);
  check(dg, "dg", y.sizes(), io);
  check(dw, "dw", {d}, ScalarType::Float);
  Tensor ws;
  if (const Tensor *t = opt_tensor(a[6], "workspace")) ws = *t;
  else {
    const size_t need = m2rnn_gated_norm_bwd_workspace_bytes(tokens, (int32_t)d);
    ws = empty({(int64_t)(need ? need : 1)}, ScalarType::Byte, dev);
  }
  const int silu = truth(a[5]);
  const int32_t code = io_code(y);
  void *st = stream_of(a[10]);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = m2rnn_gated_norm_bwd(tokens, (int32_t)d, code, ptr(y), ptr(g), ptr(w), fptr(rstd), silu, ptr(dout), ptr(dy), ptr(dg), fptr(dw), ptr(ws),
                            bytes_of(ws), st);
  Py_END_ALLOW_THREADS
  check_rc(rc, "m2rnn_gated_norm_bwd");
  return dict_of({{"dy", a[7], &dy}, {"dg", a[8], &dg}, {"dw", a[9], &dw}});
  END_HANDLE_TH_ERRORS
}

// [B,T,C] with contiguous channels and a regular token axis -> token stride in elements
int64_t row_stride(const Tensor &t, const char *name) {
  if (t.dim() == 3 && t.numel() == 0) return t.size(2);
  if (t.dim() != 3 || t.stride(2) != 1 || (t.size(0) > 1 && t.stride(0) != t.size(1) * t.stride(1)))
    fail(PyExc_ValueError, "%s: expected [B,T,C] with contiguous channels and batch entries one after the other", name);
  return t.stride(1);
}

// conv_silu_fwd(x, w, bias, prev, out, stream) -> out
PyObject *py_conv_silu_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  want_args(n, 6);
  const Tensor &x = tensor(a[0], "x"), &w = tensor(a[1], "w"), *bias = opt_tensor(a[2], "bias"), *prev = opt_tensor(a[3], "prev");
  need_dims(x, "x", 3);
  const int64_t B = x.size(0), T = x.size(1), C = x.size(2);
  const ScalarType io = x.scalar_type();
  check(x, "x", {B, T, C}, io, true);
  check(w, "w", {C, 4}, io);
  check(bias, "bias", {C}, io);
  check(prev, "prev", {B, 3, C}, io);
  const Tensor out = given_or_empty(opt_tensor(a[4], "out"), {B, T, C}, io, x.device());
  check(out, "out", {B, T, C}, io, true);
  const int32_t code = io_code(x);
  const int64_t xs = row_stride(x, "x"), os = row_stride(out, "out");
  void *st = stream_of(a[5]);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = m2rnn_conv_silu_fwd((int32_t)B, (int32_t)T, (int32_t)C, code, ptr(x), xs, ptr(w), ptr(bias), ptr(prev), ptr(out), os, st);
  Py_END_ALLOW_THREADS
  check_rc(rc, "m2rnn_conv_silu_fwd");
  return back(a[4], out);
  END_HANDLE_TH_ERRORS
}

// conv_silu_bwd(x, w, dout, bias, prev, workspace, dx, dw, dbias, dprev, stream) -> (dx, dw, dbias, dprev)
PyObject *py_conv_silu_bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  want_args(n, 11);
  const Tensor &x = tensor(a[0], "x"), &w = tensor(a[1], "w"), &dout = tensor(a[2], "dout"), *bias = opt_tensor(a[3], "bias"), *prev = opt_tensor(a[4], "prev");
  need_dims(x, "x", 3);
  const int64_t B = x.size(0), T = x.size(1), C = x.size(2);
  const ScalarType io = x.scalar_type();
  check(x, "x", {B, T, C}, io, true);
  check(w, "w", {C, 4}, io);
  check(bias, "bias", {C}, io);
  check(prev, "prev", {B, 3, C}, io);
  check(dout, "dout", {B, T, C}, io, true);
  const at::Device dev = dout.device();
  const Tensor dx = given_or_empty(opt_tensor(a[6], "dx"), {B, T, C}, io, dev);
  const Tensor dw = given_or_empty(opt_tensor(a[7], "dw"), {C, 4}, ScalarType::Float, dev);
  const Tensor dbias = given_or_empty(opt_tensor(a[8], "dbias"), {C}, ScalarType::Float, dev);
  Tensor dprev, ws;
  if (const Tensor *t = opt_tensor(a[9], "dprev")) dprev = *t;
  else if (prev) dprev = empty({B, 3, C}, io, dev);
  check(dx, "dx", {B, T, C}, io, true);
  check(dw, "dw", {C, 4}, ScalarType::Float);
  if (const Tensor *t = opt_tensor(a[5], "workspace")) ws = *t;
  else {
    const size_t need = m2rnn_conv_silu_bwd_workspace_bytes((int32_t)B, (int32_t)T, (int32_t)C);
    ws = empty({(int64_t)(need ? need : 1)}, ScalarType::Byte, dev);
  }
  const int32_t code = io_code(x);
  const int64_t xs = row_stride(x, "x"), ds = row_stride(dout, "dout"), dxs = row_stride(dx, "dx");
  void *st = stream_of(a[10]);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = m2rnn_conv_silu_bwd((int32_t)B, (int32_t)T, (int32_t)C, code, ptr(x), xs, ptr(w), ptr(bias), ptr(prev), ptr(dout), ds, ptr(dx), dxs,
                           fptr(dw), fptr(dbias), ptr(dprev), ptr(ws), bytes_of(ws), st);
  Py_END_ALLOW_THREADS
  check_rc(rc, "m2rnn_conv_silu_bwd");
  PyObject *r = PyTuple_New(4);
  if (!r) throw python_error();
  PyTuple_SET_ITEM(r, 0, back(a[6], dx));
  PyTuple_SET_ITEM(r, 1, back(a[7], dw));
  PyTuple_SET_ITEM(r, 2, back(a[8], dbias));
  PyTuple_SET_ITEM(r, 3, back(a[9], dprev));
  return r;
  END_HANDLE_TH_ERRORS
}

// status_word(device index) -> the device's int32 status tensor
PyObject *py_status_word(PyObject *, PyObject *idx) {
  HANDLE_TH_ERRORS
  return wrap(status_word_of((int)integer(idx)));
  END_HANDLE_TH_ERRORS
}

PyObject *py_set_error_class(PyObject *, PyObject *cls) {
  Py_INCREF(cls);
  Py_XDECREF(g_error_class);
  g_error_class = cls;
  Py_RETURN_NONE;
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr
PyMethodDef methods[] = {
    {"fwd", FAST(py_fwd)},
    {"bwd", FAST(py_bwd)},
    {"decode_step", FAST(py_decode_step)},
    {"gated_norm_fwd", FAST(py_gated_norm_fwd)},
    {"gated_norm_bwd", FAST(py_gated_norm_bwd)},
    {"conv_silu_fwd", FAST(py_conv_silu_fwd)},
    {"conv_silu_bwd", FAST(py_conv_silu_bwd)},
    {"status_word", py_status_word, METH_O, nullptr},
    {"set_error_class", py_set_error_class, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "native half of the M2RNN binding", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
