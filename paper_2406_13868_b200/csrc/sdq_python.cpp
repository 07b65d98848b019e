// Native half of the Python binding: the calls a program makes for every batch of activations (quantize, linear, grouped
// linear) or for every weight matrix (decompose, compact, channel norm), marshalled without ctypes.  Each function takes the
// arguments of its namesake in __init__.py, does what that does -- allocate what was not supplied, look up the current stream,
// call the C-ABI, raise SdqError -- and returns None where an argument is not what such a call has in the ordinary case (a CPU
// tensor, another type, another shape); the Python function then goes its own way, which checks and reports.
//
// Why it exists: the kernels of a one-token layer take ~11 us, and the same two calls through ctypes took the host 25 us,
// most of it argument conversion, torch.empty and the stream look-up from Python.
#include <Python.h>

#include <vector>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/sdq.h"

namespace {

PyTypeObject* act_type = nullptr;        // the ctypes structures of sdq_act_t, sdq_packed_t, sdq_config_t
PyTypeObject* packed_type = nullptr;
PyTypeObject* config_type = nullptr;
PyObject* quant_act = nullptr;           // class QuantAct
PyObject* packed_weight = nullptr;       // class PackedWeight
PyObject* sdq_error = nullptr;           // class SdqError
PyObject *s_desc, *s_buf, *s_N, *s_K, *s_cfg, *s_algo;

// memory of a ctypes structure, held for the lifetime of this object
class View {
 public:
  View() { v_.obj = nullptr; }
  ~View() { if (v_.obj) PyBuffer_Release(&v_); }
  View(const View&) = delete;
  View& operator=(const View&) = delete;
  void* open(PyObject* o, PyTypeObject* type) {
    if (!o || Py_TYPE(o) != type || PyObject_GetBuffer(o, &v_, PyBUF_SIMPLE) != 0) { PyErr_Clear(); v_.obj = nullptr; return nullptr; }
    return v_.buf;
  }
 private:
  Py_buffer v_;
};
// a strong reference that is given back
class Ref {
 public:
  explicit Ref(PyObject* o = nullptr) : o_(o) {}
  ~Ref() { Py_XDECREF(o_); }
  Ref(const Ref&) = delete;
  Ref& operator=(const Ref&) = delete;
  PyObject* get() const { return o_; }
  PyObject* release() { PyObject* o = o_; o_ = nullptr; return o; }
 private:
  PyObject* o_;
};
PyObject* attr(PyObject* o, PyObject* name) {
  PyObject* a = PyObject_GetAttr(o, name);
  if (!a) PyErr_Clear();
  return a;
}

void* current_stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

PyObject* raise(sdq_status_t st, const char* where) {
  Ref e(PyObject_CallFunction(sdq_error, "is", (int)st, where));
  if (e.get()) PyErr_SetObject(sdq_error, e.get());
  return nullptr;
}
bool is_cuda_matrix(PyObject* o, at::ScalarType type) {
  if (!THPVariable_Check(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.is_cuda() && t.scalar_type() == type && t.dim() == 2 && t.stride(1) == 1;
}
bool is_output(PyObject* o, at::ScalarType type, int64_t M, int64_t N) {
  if (!is_cuda_matrix(o, type)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.size(0) == M && t.size(1) == N;
}
at::Tensor new_output(int64_t M, int64_t N, at::ScalarType type, const at::Device& dev) {
  return at::empty({M, N}, at::TensorOptions().dtype(type).device(dev));
}
#define NOT_HERE Py_RETURN_NONE

PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 6 || !PyType_Check(a[0]) || !PyType_Check(a[1]) || !PyType_Check(a[2])) {
    PyErr_SetString(PyExc_TypeError, "bind(Act, Packed, Config, QuantAct, PackedWeight, SdqError)");
    return nullptr;
  }
  for (int i = 0; i < 6; ++i) Py_INCREF(a[i]);
  act_type = (PyTypeObject*)a[0]; packed_type = (PyTypeObject*)a[1]; config_type = (PyTypeObject*)a[2];
  quant_act = a[3]; packed_weight = a[4]; sdq_error = a[5];
  Py_RETURN_NONE;
}

// quantize_act(X, cfg, buf or None) -> QuantAct
PyObject* quantize_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 3 || !is_cuda_matrix(a[0], at::kBFloat16)) NOT_HERE;
  View vc;
  const sdq_config_t* cfg = (const sdq_config_t*)vc.open(a[1], config_type);
  if (!cfg) NOT_HERE;
  const at::Tensor& X = THPVariable_Unpack(a[0]);
  const int64_t M = X.size(0), K = X.size(1);
  at::Tensor buf;
  if (a[2] == Py_None) {
    size_t bytes = 0;
    const sdq_status_t st = sdq_act_size(M, K, cfg, &bytes);
    if (st != SDQ_OK) return raise(st, "sdq_act_size");
    buf = at::empty({(int64_t)bytes}, at::TensorOptions().dtype(at::kByte).device(X.device()));
  } else {
    if (!THPVariable_Check(a[2])) NOT_HERE;
    buf = THPVariable_Unpack(a[2]);
    if (!buf.is_cuda() || buf.scalar_type() != at::kByte) NOT_HERE;
  }
  Ref desc(PyObject_CallNoArgs((PyObject*)act_type));
  if (!desc.get()) return nullptr;
  {
    View vd;
    sdq_act_t* d = (sdq_act_t*)vd.open(desc.get(), act_type);
    if (!d) NOT_HERE;
    void* stream = current_stream();
    sdq_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = sdq_quantize_act(X.data_ptr(), M, K, X.stride(0), cfg, buf.data_ptr(), (size_t)buf.numel(), d, stream);
    Py_END_ALLOW_THREADS
    if (st != SDQ_OK) return raise(st, "sdq_quantize_act");
  }
  Ref b(a[2] == Py_None ? THPVariable_Wrap(std::move(buf)) : Py_NewRef(a[2])), m(PyLong_FromLongLong(M)), k(PyLong_FromLongLong(K));
  if (!b.get() || !m.get() || !k.get()) return nullptr;
  PyObject* args[5] = {b.get(), desc.get(), m.get(), k.get(), a[1]};
  return PyObject_Vectorcall(quant_act, args, 5, nullptr);
  END_HANDLE_TH_ERRORS
}

// linear(xq, p, out or None, f32, workspace or None) -> out
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 5) NOT_HERE;
  const int f32 = PyObject_IsTrue(a[3]);
  if (f32 < 0) { PyErr_Clear(); NOT_HERE; }
  Ref dx(attr(a[0], s_desc)), dp(attr(a[1], s_desc)), pb(attr(a[1], s_buf));
  View vx, vp;
  const sdq_act_t* x = (const sdq_act_t*)vx.open(dx.get(), act_type);
  const sdq_packed_t* p = (const sdq_packed_t*)vp.open(dp.get(), packed_type);
  if (!x || !p || !pb.get() || !THPVariable_Check(pb.get())) NOT_HERE;
  const at::ScalarType type = f32 ? at::kFloat : at::kBFloat16;
  at::Tensor out;
  if (a[2] == Py_None) out = new_output(x->M, p->N, type, THPVariable_Unpack(pb.get()).device());
  else if (is_output(a[2], type, x->M, p->N)) out = THPVariable_Unpack(a[2]);
  else NOT_HERE;
  void* ws = nullptr;
  size_t ws_bytes = 0;
  const bool has_ws = a[4] != Py_None;
  if (has_ws) {
    if (!THPVariable_Check(a[4])) NOT_HERE;
    const at::Tensor& w = THPVariable_Unpack(a[4]);
    if (!w.is_cuda() || w.scalar_type() != at::kByte) NOT_HERE;
    ws = w.data_ptr();
    ws_bytes = (size_t)w.numel();
  }
  void *y = out.data_ptr(), *stream = current_stream();
  const int64_t ldy = out.stride(0);
  sdq_status_t st;
  Py_BEGIN_ALLOW_THREADS
  if (has_ws) st = f32 ? sdq_linear_f32_ws(x, p, (float*)y, ldy, ws, ws_bytes, stream) : sdq_linear_ws(x, p, y, ldy, ws, ws_bytes, stream);
  else st = f32 ? sdq_linear_f32(x, p, (float*)y, ldy, stream) : sdq_linear(x, p, y, ldy, stream);
  Py_END_ALLOW_THREADS
  if (st != SDQ_OK) return raise(st, has_ws ? "sdq_linear_ws" : "sdq_linear");
  return a[2] == Py_None ? THPVariable_Wrap(std::move(out)) : Py_NewRef(a[2]);
  END_HANDLE_TH_ERRORS
}

// the layers of a grouped call, as the arrays the C-ABI takes
struct Group {
  std::vector<View> views;
  std::vector<Ref*> refs;
  std::vector<const sdq_act_t*> x;
  std::vector<const sdq_packed_t*> p;
  std::vector<void*> y;
  std::vector<int64_t> ldy;
  PyObject* outs = nullptr;              // new list of outputs, if they were not supplied
  ~Group() { for (Ref* r : refs) delete r; Py_XDECREF(outs); }
  // descriptor of layer i of the sequence `seq`
  void* desc(PyObject* o, PyTypeObject* type, View& v) {
    refs.push_back(new Ref(attr(o, s_desc)));
    return v.open(refs.back()->get(), type);
  }
};

// linear_group(xqs or None, X or None, ps, outs or None, f32): with X the fused-quantizer call, else xqs
PyObject* group(PyObject* xqs, PyObject* X, PyObject* ps, PyObject* outs, PyObject* f32_) {
  const int f32 = PyObject_IsTrue(f32_);
  if (f32 < 0) { PyErr_Clear(); NOT_HERE; }
  if (!PyList_Check(ps) && !PyTuple_Check(ps)) NOT_HERE;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(ps);
  if (n <= 0 || (xqs && ((!PyList_Check(xqs) && !PyTuple_Check(xqs)) || PySequence_Fast_GET_SIZE(xqs) != n))) NOT_HERE;
  if (outs != Py_None && ((!PyList_Check(outs) && !PyTuple_Check(outs)) || PySequence_Fast_GET_SIZE(outs) != n)) NOT_HERE;
  const at::ScalarType type = f32 ? at::kFloat : at::kBFloat16;
  Group g;
  g.views = std::vector<View>((size_t)(2 * n));
  g.refs.reserve((size_t)(2 * n));
  g.x.resize((size_t)n); g.p.resize((size_t)n); g.y.resize((size_t)n); g.ldy.resize((size_t)n);
  if (outs == Py_None) { g.outs = PyList_New(n); if (!g.outs) return nullptr; }
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* po = PySequence_Fast_GET_ITEM(ps, i);
    g.p[i] = (const sdq_packed_t*)g.desc(po, packed_type, g.views[2 * i]);
    if (!g.p[i]) NOT_HERE;
    int64_t M;
    if (xqs) {
      PyObject* xo = PySequence_Fast_GET_ITEM(xqs, i);
      // (the same quantized activations for several layers, the usual case, are opened once)
      if (i && xo == PySequence_Fast_GET_ITEM(xqs, i - 1)) g.x[i] = g.x[i - 1];
      else g.x[i] = (const sdq_act_t*)g.desc(xo, act_type, g.views[2 * i + 1]);
      if (!g.x[i]) NOT_HERE;
      M = g.x[i]->M;
    } else {
      M = THPVariable_Unpack(X).size(0);
    }
    if (outs == Py_None) {
      at::Device dev(at::kCUDA);
      if (X) dev = THPVariable_Unpack(X).device();
      else {
        Ref b(attr(po, s_buf));
        if (!b.get() || !THPVariable_Check(b.get())) NOT_HERE;
        dev = THPVariable_Unpack(b.get()).device();
      }
      at::Tensor t = new_output(M, g.p[i]->N, type, dev);
      g.y[i] = t.data_ptr(); g.ldy[i] = t.stride(0);
      PyObject* w = THPVariable_Wrap(std::move(t));
      if (!w) return nullptr;
      PyList_SET_ITEM(g.outs, i, w);
    } else {
      PyObject* o = PySequence_Fast_GET_ITEM(outs, i);
      if (!is_output(o, type, M, g.p[i]->N)) NOT_HERE;
      const at::Tensor& t = THPVariable_Unpack(o);
      g.y[i] = t.data_ptr(); g.ldy[i] = t.stride(0);
    }
  }
  void* stream = current_stream();
  const void* xp = nullptr;
  int64_t M = 0, K = 0, ldx = 0;
  at::Tensor ws;                         // the quantized activations, for the caching allocator to hand on in stream order
  if (X) {
    const at::Tensor& t = THPVariable_Unpack(X);
    xp = t.data_ptr(); M = t.size(0); K = t.size(1); ldx = t.stride(0);
    size_t bytes = 0;
    // (16 tokens of 4096: the call's range, anything else is refused; X on another device, whose streams the allocator would hand
    // the scratch on by, or no memory left: the form that needs none)
    if (M <= 16 && K <= 4096 && t.device().index() == c10::cuda::current_device() && sdq_act_size(M, K, &g.p[0]->cfg, &bytes) == SDQ_OK) {
      try {
        ws = at::empty({(int64_t)bytes}, at::TensorOptions().dtype(at::kByte).device(t.device()));
      } catch (const c10::OutOfMemoryError&) {
      }
    }
  }
  void* wp = ws.defined() ? ws.data_ptr() : nullptr;
  const size_t ws_bytes = ws.defined() ? (size_t)ws.numel() : 0;
  sdq_status_t st;
  Py_BEGIN_ALLOW_THREADS
  if (X) st = f32 ? sdq_linear_group_x_f32_ws((int)n, xp, M, K, ldx, g.p.data(), (float* const*)g.y.data(), g.ldy.data(), wp, ws_bytes, stream)
                  : sdq_linear_group_x_ws((int)n, xp, M, K, ldx, g.p.data(), g.y.data(), g.ldy.data(), wp, ws_bytes, stream);
  else st = f32 ? sdq_linear_group_f32((int)n, g.x.data(), g.p.data(), (float* const*)g.y.data(), g.ldy.data(), stream)
                : sdq_linear_group((int)n, g.x.data(), g.p.data(), g.y.data(), g.ldy.data(), stream);
  Py_END_ALLOW_THREADS
  if (st != SDQ_OK) return raise(st, X ? "sdq_linear_group_x" : "sdq_linear_group");
  if (outs != Py_None) return Py_NewRef(outs);
  PyObject* r = g.outs;
  g.outs = nullptr;
  return r;
}
// linear_group(xqs, ps, outs or None, f32) -> outputs
PyObject* linear_group(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 4) NOT_HERE;
  return group(a[0], nullptr, a[1], a[2], a[3]);
  END_HANDLE_TH_ERRORS
}
// linear_group_x(X, ps, outs or None, f32) -> outputs
PyObject* linear_group_x(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 4 || !is_cuda_matrix(a[0], at::kBFloat16)) NOT_HERE;
  return group(nullptr, a[0], a[1], a[2], a[3]);
  END_HANDLE_TH_ERRORS
}

// decompose(W, cfg, buf or None, col_weight or None) -> PackedWeight
PyObject* decompose(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 4 || !is_cuda_matrix(a[0], at::kBFloat16)) NOT_HERE;
  View vc;
  const sdq_config_t* cfg = (const sdq_config_t*)vc.open(a[1], config_type);
  if (!cfg) NOT_HERE;
  const at::Tensor& W = THPVariable_Unpack(a[0]);
  const int64_t N = W.size(0), K = W.size(1);
  const float* colw = nullptr;
  if (a[3] != Py_None) {
    if (!THPVariable_Check(a[3])) NOT_HERE;
    const at::Tensor& c = THPVariable_Unpack(a[3]);
    if (!c.is_cuda() || c.scalar_type() != at::kFloat || c.dim() != 1 || c.size(0) != K || !c.is_contiguous()) NOT_HERE;
    colw = (const float*)c.data_ptr();
  }
  size_t bytes = 0, algo = 0;
  sdq_status_t st = sdq_packed_size(N, K, cfg, &bytes, &algo);
  if (st != SDQ_OK) return raise(st, "sdq_packed_size");
  at::Tensor buf;
  if (a[2] == Py_None) {
    buf = at::empty({(int64_t)bytes}, at::TensorOptions().dtype(at::kByte).device(W.device()));
  } else {
    if (!THPVariable_Check(a[2])) NOT_HERE;
    buf = THPVariable_Unpack(a[2]);
    if (!buf.is_cuda() || buf.scalar_type() != at::kByte) NOT_HERE;
  }
  Ref desc(PyObject_CallNoArgs((PyObject*)packed_type));
  if (!desc.get()) return nullptr;
  {
    View vd;
    sdq_packed_t* d = (sdq_packed_t*)vd.open(desc.get(), packed_type);
    if (!d) NOT_HERE;
    void *stream = current_stream(), *w = W.data_ptr(), *b = buf.data_ptr();
    const int64_t ldw = W.stride(0);
    const size_t room = (size_t)buf.numel();
    Py_BEGIN_ALLOW_THREADS
    st = sdq_decompose_metric(w, N, K, ldw, cfg, colw, b, room, d, stream);
    Py_END_ALLOW_THREADS
    if (st != SDQ_OK) return raise(st, colw ? "sdq_decompose_metric" : "sdq_decompose");
  }
  Ref b(a[2] == Py_None ? THPVariable_Wrap(std::move(buf)) : Py_NewRef(a[2])), pn(PyLong_FromLongLong(N)), pk(PyLong_FromLongLong(K)), pa(PyLong_FromSize_t(algo));
  if (!b.get() || !pn.get() || !pk.get() || !pa.get()) return nullptr;
  PyObject* args[6] = {b.get(), desc.get(), pn.get(), pk.get(), a[1], pa.get()};
  return PyObject_Vectorcall(packed_weight, args, 6, nullptr);
  END_HANDLE_TH_ERRORS
}

// compact(p) -> PackedWeight
PyObject* compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 1) NOT_HERE;
  Ref dp(attr(a[0], s_desc)), pb(attr(a[0], s_buf)), pn(attr(a[0], s_N)), pk(attr(a[0], s_K)), pc(attr(a[0], s_cfg)), pa(attr(a[0], s_algo));
  View vp;
  const sdq_packed_t* p = (const sdq_packed_t*)vp.open(dp.get(), packed_type);
  if (!p || !pb.get() || !THPVariable_Check(pb.get()) || !pn.get() || !pk.get() || !pc.get() || !pa.get()) NOT_HERE;
  size_t bytes = 0;
  sdq_status_t st = sdq_packed_compact_size(p->N, p->K, &p->cfg, &bytes);
  if (st != SDQ_OK) return raise(st, "sdq_packed_compact_size");
  at::Tensor buf = at::empty({(int64_t)bytes}, at::TensorOptions().dtype(at::kByte).device(THPVariable_Unpack(pb.get()).device()));
  Ref desc(PyObject_CallNoArgs((PyObject*)packed_type));
  if (!desc.get()) return nullptr;
  {
    View vd;
    sdq_packed_t* d = (sdq_packed_t*)vd.open(desc.get(), packed_type);
    if (!d) NOT_HERE;
    void *stream = current_stream(), *b = buf.data_ptr();
    Py_BEGIN_ALLOW_THREADS
    st = sdq_packed_compact(p, b, bytes, d, stream);
    Py_END_ALLOW_THREADS
    if (st != SDQ_OK) return raise(st, "sdq_packed_compact");
  }
  Ref b(THPVariable_Wrap(std::move(buf)));
  if (!b.get()) return nullptr;
  PyObject* args[6] = {b.get(), desc.get(), pn.get(), pk.get(), pc.get(), pa.get()};
  return PyObject_Vectorcall(packed_weight, args, 6, nullptr);
  END_HANDLE_TH_ERRORS
}

// channel_norm(X) -> fp32 [K]
PyObject* channel_norm(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 1 || !is_cuda_matrix(a[0], at::kBFloat16)) NOT_HERE;
  const at::Tensor& X = THPVariable_Unpack(a[0]);
  at::Tensor c = at::empty({X.size(1)}, at::TensorOptions().dtype(at::kFloat).device(X.device()));
  void *stream = current_stream(), *x = X.data_ptr(), *y = c.data_ptr();
  const int64_t M = X.size(0), K = X.size(1), ldx = X.stride(0);
  sdq_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = sdq_channel_norm(x, M, K, ldx, (float*)y, stream);
  Py_END_ALLOW_THREADS
  if (st != SDQ_OK) return raise(st, "sdq_channel_norm");
  return THPVariable_Wrap(std::move(c));
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"decompose", (PyCFunction)(void (*)(void))decompose, METH_FASTCALL, nullptr},
                         {"compact", (PyCFunction)(void (*)(void))compact, METH_FASTCALL, nullptr},
                         {"channel_norm", (PyCFunction)(void (*)(void))channel_norm, METH_FASTCALL, nullptr},
                         {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, nullptr},
                         {"quantize_act", (PyCFunction)(void (*)(void))quantize_act, METH_FASTCALL, nullptr},
                         {"linear", (PyCFunction)(void (*)(void))linear, METH_FASTCALL, nullptr},
                         {"linear_group", (PyCFunction)(void (*)(void))linear_group, METH_FASTCALL, nullptr},
                         {"linear_group_x", (PyCFunction)(void (*)(void))linear_group_x, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
  s_desc = PyUnicode_InternFromString("desc");
  s_buf = PyUnicode_InternFromString("buf");
  s_N = PyUnicode_InternFromString("N");
  s_K = PyUnicode_InternFromString("K");
  s_cfg = PyUnicode_InternFromString("cfg");
  s_algo = PyUnicode_InternFromString("algorithmic_bytes");
  return PyModule_Create(&module);
}
