// CPython extension behind paper_2502_18394_b200/binding.py: argument marshalling of the per-step calls in native code.
//
// A ctypes call that builds its structures in Python spends 20 us of host time before the first kernel is launched, more
// than the kernels of a short call take (44 us for the gate and the mixer of a 1k sequence whose kernels take 18).  Here the
// tensors are unpacked, outputs and workspaces come from torch's allocator and the C ABI is called, without another Python
// object in between.  The C ABI is the only thing that touches the device.
#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <optional>
#include <string>
#include <vector>

#include "spectre.h"

namespace {

PyObject* g_error = nullptr;                       // binding.SpectreError

// dictionary keys, interned once
enum Key { kGamma, kBeta, kEps, kW1, kB1, kW2, kB2, kHidden, kModrelu, kToeplitz, kShared, kLevels, kLevelGates, kQbar, kWw1, kBw1,
           kWw2, kBw2, kSkip, kAttrB, kAttrH, kAttrD, kAttrN, kAttrSpec, kAttrV, kAttrQ, kAttrSum, kAttrStream, kKeys };
const char* const kNames[kKeys] = {"ln_gamma", "ln_beta", "ln_eps", "W1", "b1", "W2", "b2", "hidden", "modrelu_bias", "toeplitz",
                                   "shared_across_heads", "levels", "level_gates", "qbar", "Ww1", "bw1", "Ww2", "bw2", "skip",
                                   "B", "H", "D", "N_max", "prefix_fft", "V_buf", "Q_buf", "sum_q", "cuda_stream"};
PyObject* g_key[kKeys];

struct Failed {};                                  // a Python exception is set
[[noreturn]] void raise(PyObject* type, const char* text) {
  PyErr_SetString(type, text);
  throw Failed{};
}

void check(int status) {
  if (status == SPECTRE_OK) return;
  const std::string text = std::string(spectre_status_string(status)) + ": " + spectre_last_error();
  PyObject* e = PyObject_CallFunction(g_error, "is", status, text.c_str());
  if (e) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  throw Failed{};
}

bool none(PyObject* o) { return o == nullptr || o == Py_None; }

const at::Tensor& tensor(PyObject* o) {
  if (none(o) || !THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch.Tensor");
  return THPVariable_Unpack(o);
}
void* pointer(PyObject* o) { return none(o) ? nullptr : tensor(o).data_ptr(); }

int dtype_code(const at::Tensor& t) {
  switch (t.scalar_type()) {
    case at::kFloat: return SPECTRE_F32;
    case at::kBFloat16: return SPECTRE_BF16;
    case at::kHalf: return SPECTRE_F16;
    default: raise(PyExc_TypeError, (std::string("unsupported dtype ") + c10::toString(t.scalar_type())).c_str());
  }
}

spectre_act act(const at::Tensor& t) {
  if (t.dim() != 4 || t.stride(3) != 1) raise(PyExc_ValueError, "activation must be [B, L, H, D] with D contiguous");
  return spectre_act{t.data_ptr(), dtype_code(t), (int32_t)t.size(0), (int32_t)t.size(1), (int32_t)t.size(2), (int32_t)t.size(3),
                     t.stride(0), t.stride(1), t.stride(2)};
}

long long integer(PyObject* o) {
  if (PyLong_CheckExact(o)) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Failed{};
    return v;
  }
  PyObject* i = PyNumber_Long(o);                  // as int(o)
  if (!i) throw Failed{};
  const long long v = PyLong_AsLongLong(i);
  Py_DECREF(i);
  if (v == -1 && PyErr_Occurred()) throw Failed{};
  return v;
}
int32_t integer32(PyObject* o) { return (int32_t)integer(o); }
bool truth(PyObject* o) {
  const int t = PyObject_IsTrue(o);
  if (t < 0) throw Failed{};
  return t == 1;
}
double real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Failed{};
  return v;
}

PyObject* get(PyObject* dict, Key k) {             // borrowed, NULL if absent
  PyObject* v = PyDict_GetItemWithError(dict, g_key[k]);
  if (!v && PyErr_Occurred()) throw Failed{};
  return v;
}
PyObject* need(PyObject* dict, Key k) {
  PyObject* v = get(dict, k);
  if (!v) {
    PyErr_SetObject(PyExc_KeyError, g_key[k]);
    throw Failed{};
  }
  return v;
}
struct Attr {                                      // owned attribute
  PyObject* o;
  Attr(PyObject* from, Key k) : o(PyObject_GetAttr(from, g_key[k])) { if (!o) throw Failed{}; }
  ~Attr() { Py_DECREF(o); }
  Attr(const Attr&) = delete;
};

// The stream of a call: the current one, or the `cuda_stream` of the object given.  Outputs and workspaces of the call are
// allocated on it too: torch's allocator hands a freed block on in the order of the stream that it was allocated on.
struct Stream {
  std::optional<c10::cuda::CUDAStreamGuard> guard;
  void* st;
  Stream(PyObject* s, const at::Tensor& like) {
    if (none(s)) {
      st = c10::cuda::getCurrentCUDAStream().stream();
      return;
    }
    Attr a(s, kAttrStream);
    st = PyLong_AsVoidPtr(a.o);
    if (!st && PyErr_Occurred()) throw Failed{};
    if (like.is_cuda() && c10::cuda::getCurrentCUDAStream(like.get_device()).stream() != st)
      guard.emplace(c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(st), like.get_device()));
  }
};
spectre_ctx* context(PyObject* o) {
  if (none(o)) return nullptr;
  void* p = PyLong_AsVoidPtr(o);
  if (!p && PyErr_Occurred()) throw Failed{};
  return static_cast<spectre_ctx*>(p);
}

spectre_gate_params gate_params(PyObject* d) {
  if (!PyDict_Check(d)) raise(PyExc_TypeError, "gate parameters must be a dict");
  spectre_gate_params p = {};
  PyObject* tz = get(d, kToeplitz);
  if (!none(tz)) p.toeplitz_r = (int32_t)((tensor(tz).size(-2) - 1) / 2);
  const at::Tensor& w1 = tensor(need(d, kW1));
  p.wdtype = dtype_code(w1);
  p.hidden = integer32(need(d, kHidden));
  if (PyObject* s = get(d, kShared)) p.shared_across_heads = integer32(s);
  p.ln_gamma = (const float*)tensor(need(d, kGamma)).data_ptr();
  p.ln_beta = (const float*)tensor(need(d, kBeta)).data_ptr();
  p.ln_eps = (float)real(need(d, kEps));
  p.W1 = w1.data_ptr();
  p.b1 = (const float*)tensor(need(d, kB1)).data_ptr();
  p.W2 = tensor(need(d, kW2)).data_ptr();
  p.b2 = (const float*)tensor(need(d, kB2)).data_ptr();
  p.modrelu_bias = (const float*)pointer(get(d, kModrelu));
  p.toeplitz = (const float*)pointer(tz);
  return p;
}

spectre_wavelet wavelet(PyObject* d) {
  if (!PyDict_Check(d)) raise(PyExc_TypeError, "refinement parameters must be a dict");
  spectre_wavelet w = {};
  w.levels = integer32(need(d, kLevels));
  if (PyObject* h = get(d, kHidden)) w.hidden = integer32(h);
  PyObject* w1 = get(d, kWw1);
  w.wdtype = none(w1) ? SPECTRE_F32 : dtype_code(tensor(w1));
  if (PyObject* s = get(d, kShared)) w.shared_across_heads = integer32(s);
  w.level_gates = (const float*)pointer(get(d, kLevelGates));
  w.qbar = (const float*)pointer(get(d, kQbar));
  w.Ww1 = pointer(w1);
  w.bw1 = (const float*)pointer(get(d, kBw1));
  w.Ww2 = pointer(get(d, kWw2));
  w.bw2 = (const float*)pointer(get(d, kBw2));
  w.skip = (const int32_t*)pointer(get(d, kSkip));
  return w;
}

at::Tensor empty(at::IntArrayRef size, const at::Tensor& like, at::ScalarType t) { return at::empty(size, like.options().dtype(t)); }

// the caller's workspace, or one of the queried size
struct Workspace {
  at::Tensor own;
  void* ptr = nullptr;
  size_t bytes = 0;
  template <class Query>
  Workspace(PyObject* given, const at::Tensor& like, Query query) {
    if (!none(given)) {
      const at::Tensor& t = tensor(given);
      ptr = t.data_ptr();
      bytes = (size_t)t.numel();
    } else if (const size_t n = query()) {
      bytes = n < 16 ? 16 : n;
      own = empty({(int64_t)bytes}, like, at::kByte);
      ptr = own.data_ptr();
    }
  }
};

spectre_cache cache_state(PyObject* c, at::Tensor* v_buf) {
  spectre_cache s = {};
  { Attr a(c, kAttrB); s.B = integer32(a.o); }
  { Attr a(c, kAttrH); s.H = integer32(a.o); }
  { Attr a(c, kAttrD); s.D = integer32(a.o); }
  { Attr a(c, kAttrN); s.N_max = integer32(a.o); }
  { Attr a(c, kAttrSpec); s.prefix_fft = (float*)tensor(a.o).data_ptr(); }
  { Attr a(c, kAttrV); *v_buf = tensor(a.o); s.buf_dtype = dtype_code(*v_buf); s.V_buf = v_buf->data_ptr(); }
  { Attr a(c, kAttrQ); s.Q_buf = tensor(a.o).data_ptr(); }
  { Attr a(c, kAttrSum); s.sum_q = (float*)tensor(a.o).data_ptr(); }
  return s;
}

// A C ABI call with the interpreter released, as under ctypes.
template <class F> int released(F f) {
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f();
  Py_END_ALLOW_THREADS
  return rc;
}

// ARGS: the number of arguments F reads; the wrappers in binding.py pass every one
template <PyObject* (*F)(PyObject* const*), int ARGS>
PyObject* guarded(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != ARGS) return PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", ARGS, n);
  try {
    return F(a);
  } catch (const Failed&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// gate(ctx, params, n_fft, q, sum_q, inv_count, shift, shift_all, g_out, qbar_out, workspace, stream, static)
PyObject* gate(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  const spectre_gate_params p = gate_params(a[1]);
  const int32_t n = integer32(a[2]);
  const bool from_q = !none(a[3]), fixed = a[12] == Py_True;
  const at::Tensor& ref = tensor(from_q ? a[3] : a[4]);
  spectre_act q = {};
  int32_t B, H, D;
  if (from_q) {
    q = act(ref);
    B = q.B; H = q.H; D = q.D;
  } else {
    if (ref.dim() != 3) raise(PyExc_ValueError, "sum_q must be [B, H, D]");
    B = (int32_t)ref.size(0); H = (int32_t)ref.size(1); D = (int32_t)ref.size(2);
  }
  const float* sum_q = (const float*)pointer(a[4]);
  const float inv = (float)real(a[5]);
  const int64_t* shift = (const int64_t*)pointer(a[6]);
  const int64_t shift_all = integer(a[7]);
  const Stream on(a[11], ref);
  at::Tensor g = none(a[8]) ? empty({B, H, n / 2 + 1, 2}, ref, at::kFloat) : tensor(a[8]);
  float *out = (float*)g.data_ptr(), *qbar = (float*)pointer(a[9]);
  if (fixed) {
    check(released([&] { return spectre_gate_static(ctx, on.st, from_q ? &q : nullptr, sum_q, B, H, D, inv, &p, n, shift, shift_all, out, qbar); }));
  } else {
    const Workspace w(a[10], ref, [&] { return spectre_gate_workspace_bytes(ctx, B, H, D, n, p.toeplitz_r); });
    check(released([&] {
      return spectre_gate(ctx, on.st, from_q ? &q : nullptr, sum_q, B, H, D, inv, &p, n, shift, shift_all, out, qbar, w.ptr, w.bytes);
    }));
  }
  return THPVariable_Wrap(g);
}

// mixer_forward(ctx, v, g, y, n_fft, wrm, workspace, stream)
PyObject* mixer_forward(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  const at::Tensor& v = tensor(a[1]);
  const spectre_act av = act(v);
  const int32_t n = none(a[4]) ? av.L : integer32(a[4]);
  const Stream on(a[7], v);
  at::Tensor y = none(a[3]) ? at::empty_like(v) : tensor(a[3]);
  const spectre_act ay = act(y);
  const float* g = (const float*)pointer(a[2]);
  spectre_wavelet wrm = {};
  if (!none(a[5])) wrm = wavelet(a[5]);
  const Workspace w(a[6], v, [&] { return spectre_mixer_workspace_bytes(ctx, av.B, av.L, av.H, av.D, n, av.dtype); });
  check(released([&] { return spectre_mixer_forward(ctx, on.st, &av, g, &ay, n, none(a[5]) ? nullptr : &wrm, w.ptr, w.bytes); }));
  return THPVariable_Wrap(y);
}

// wavelet_refine(ctx, y_in, wrm, y_out, stream)
PyObject* wavelet_refine(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  const at::Tensor& x = tensor(a[1]);
  const Stream on(a[4], x);
  at::Tensor y = none(a[3]) ? at::empty_like(x) : tensor(a[3]);
  const spectre_wavelet w = wavelet(a[2]);
  const spectre_act ax = act(x), ay = act(y);
  check(released([&] { return spectre_wavelet_refine(ctx, on.st, &ax, &ay, &w); }));
  return THPVariable_Wrap(y);
}

// prefill(ctx, cache, q, v, workspace, stream)
PyObject* prefill(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  at::Tensor vb;
  const spectre_cache c = cache_state(a[1], &vb);
  const at::Tensor& v = tensor(a[3]);
  const spectre_act aq = act(tensor(a[2])), av = act(v);
  const Stream on(a[5], v);
  const Workspace w(a[4], v, [&] { return spectre_prefill_workspace_bytes(ctx, c.B, c.H, c.D, c.N_max); });
  check(released([&] { return spectre_prefix_cache_prefill(ctx, on.st, &c, &aq, &av, w.ptr, w.bytes); }));
  Py_RETURN_NONE;
}

void contiguous_tokens(const at::Tensor& q, const at::Tensor& v) {
  if (!(q.is_contiguous() && v.is_contiguous())) raise(PyExc_ValueError, "q_t and v_t must be contiguous [B, H, D]");
}

// append(ctx, cache, q_t, v_t, t, stream)
PyObject* append(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  const at::Tensor &q = tensor(a[2]), &v = tensor(a[3]);
  contiguous_tokens(q, v);
  const Stream on(a[5], q);
  at::Tensor vb;
  const spectre_cache c = cache_state(a[1], &vb);
  const int64_t t = integer(a[4]);
  check(released([&] { return spectre_prefix_cache_append(ctx, on.st, &c, q.data_ptr(), v.data_ptr(), t); }));
  Py_RETURN_NONE;
}

// decode_step(ctx, cache, q_t, v_t, t, params, rows, y_rows, g_out, workspace, stream)
PyObject* decode_step(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  const at::Tensor &q = tensor(a[2]), &v = tensor(a[3]);
  contiguous_tokens(q, v);
  std::vector<int32_t> rows;
  PyObject* seq = PySequence_Fast(a[6], "rows must be a sequence of integers");
  if (!seq) throw Failed{};
  try {
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(seq); ++i) rows.push_back(integer32(PySequence_Fast_GET_ITEM(seq, i)));
  } catch (...) {
    Py_DECREF(seq);
    throw;
  }
  Py_DECREF(seq);
  const int32_t nrows = (int32_t)rows.size();
  rows.push_back(0);                               // never an empty array
  const spectre_gate_params p = gate_params(a[5]);
  at::Tensor vb;
  const spectre_cache c = cache_state(a[1], &vb);
  const int64_t t = integer(a[4]);
  const Stream on(a[10], v);
  at::Tensor y = none(a[7]) ? empty({c.B, nrows, c.H, c.D}, v, v.scalar_type()) : tensor(a[7]);
  at::Tensor g = none(a[8]) ? empty({c.B, c.H, c.N_max / 2 + 1, 2}, v, at::kFloat) : tensor(a[8]);
  const Workspace w(a[9], v, [&] {
    const int32_t r = nrows < 1 ? 1 : (nrows > SPECTRE_DECODE_MAX_ROWS ? SPECTRE_DECODE_MAX_ROWS : nrows);
    return spectre_decode_workspace_bytes(ctx, c.B, c.H, c.D, c.N_max, r, p.toeplitz_r);
  });
  check(released([&] {
    return spectre_prefix_cache_decode_step(ctx, on.st, &c, q.data_ptr(), v.data_ptr(), t, &p, rows.data(), nrows, y.data_ptr(),
                                            (float*)g.data_ptr(), w.ptr, w.bytes);
  }));
  return Py_BuildValue("NN", THPVariable_Wrap(y), THPVariable_Wrap(g));
}

// readout(ctx, cache, g, y, workspace, stream)
PyObject* readout(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  at::Tensor vb;
  const spectre_cache c = cache_state(a[1], &vb);
  const at::Tensor& g = tensor(a[2]);
  const Stream on(a[5], g);
  at::Tensor y = none(a[3]) ? empty({c.B, c.N_max, c.H, c.D}, g, vb.scalar_type()) : tensor(a[3]);
  const spectre_act ay = act(y);
  const Workspace w(a[4], g, [&] { return spectre_readout_workspace_bytes(ctx, c.B, c.H, c.D, c.N_max); });
  check(released([&] { return spectre_prefix_cache_readout(ctx, on.st, &c, (const float*)g.data_ptr(), &ay, w.ptr, w.bytes); }));
  return THPVariable_Wrap(y);
}

// project_qv(ctx, x, Wq, Wv, q, v, sum_q, need_sum, workspace, stream)
PyObject* project_qv(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  const at::Tensor &x = tensor(a[1]), &wq = tensor(a[2]), &wv = tensor(a[3]);
  const spectre_act ax = act(x);
  if (wq.scalar_type() != wv.scalar_type() || !(wq.is_contiguous() && wv.is_contiguous()))
    raise(PyExc_ValueError, "Wq and Wv must be contiguous and of one dtype");
  const bool want_sum = none(a[6]) && truth(a[7]);
  const Stream on(a[9], x);
  at::Tensor q = none(a[4]) ? at::empty_like(x) : tensor(a[4]), v = none(a[5]) ? at::empty_like(x) : tensor(a[5]), sum;
  if (!none(a[6])) sum = tensor(a[6]);
  else if (want_sum) sum = empty({ax.B, ax.H, ax.D}, x, at::kFloat);
  const spectre_act aq = act(q), av = act(v);
  const Workspace w(a[8], x, [&] { return spectre_project_workspace_bytes(ctx, ax.H, ax.D); });
  float* s = sum.defined() ? (float*)sum.data_ptr() : nullptr;
  const int32_t wd = dtype_code(wq);
  check(released([&] { return spectre_project_qv(ctx, on.st, &ax, wq.data_ptr(), wv.data_ptr(), wd, &aq, &av, s, w.ptr, w.bytes); }));
  PyObject* so = sum.defined() ? THPVariable_Wrap(sum) : Py_NewRef(Py_None);
  return Py_BuildValue("NNN", THPVariable_Wrap(q), THPVariable_Wrap(v), so);
}

// mixer_backward(ctx, v, dy, g, n_fft, need_dv, need_dg, workspace, stream)
PyObject* mixer_backward(PyObject* const* a) {
  spectre_ctx* ctx = context(a[0]);
  const at::Tensor &v = tensor(a[1]), &dy = tensor(a[2]);
  const spectre_act av = act(v), ady = act(dy);
  const float* g = (const float*)pointer(a[3]);
  const int32_t n = none(a[4]) ? av.L : integer32(a[4]);
  const bool want_dv = truth(a[5]), want_dg = truth(a[6]);
  const Stream on(a[8], v);
  at::Tensor dv, dg;
  spectre_act adv = {};
  if (want_dv) {
    dv = at::empty_like(v);
    adv = act(dv);
  }
  if (want_dg) dg = empty({av.B, av.H, n / 2 + 1, 2}, v, at::kFloat);
  const Workspace w(a[7], v, [&] { return spectre_mixer_backward_workspace_bytes(ctx, av.B, av.L, av.H, av.D, n, av.dtype); });
  float* pg = want_dg ? (float*)dg.data_ptr() : nullptr;
  check(released([&] { return spectre_mixer_backward(ctx, on.st, &av, &ady, g, want_dv ? &adv : nullptr, pg, n, w.ptr, w.bytes); }));
  PyObject* ov = want_dv ? THPVariable_Wrap(dv) : Py_NewRef(Py_None);
  PyObject* og = want_dg ? THPVariable_Wrap(dg) : Py_NewRef(Py_None);
  return Py_BuildValue("NN", ov, og);
}

PyObject* set_error(PyObject*, PyObject* type) {
  Py_XDECREF(g_error);
  g_error = Py_NewRef(type);
  Py_RETURN_NONE;
}

#define SPECTRE_METHOD(name, args) {#name, (PyCFunction)(void (*)(void))guarded<name, args>, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {SPECTRE_METHOD(gate, 13), SPECTRE_METHOD(mixer_forward, 8), SPECTRE_METHOD(wavelet_refine, 5),
                           SPECTRE_METHOD(prefill, 6), SPECTRE_METHOD(append, 6), SPECTRE_METHOD(decode_step, 11),
                           SPECTRE_METHOD(readout, 6), SPECTRE_METHOD(project_qv, 10), SPECTRE_METHOD(mixer_backward, 9),
                           {"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
  for (int i = 0; i < kKeys; ++i)
    if (!(g_key[i] = PyUnicode_InternFromString(kNames[i]))) return nullptr;
  return PyModule_Create(&g_module);
}
