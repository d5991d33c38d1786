// CPython module behind the four tensor functions of the package: reads the tensors' pointers and
// sizes, allocates outputs and workspace from PyTorch's allocator, fills the ABI's structs and calls
// the library.  It computes nothing.  (The same in Python, over ctypes, took about 11 us of a call.)
//
// The library's functions are not linked: bind() receives their addresses from the ctypes handle that
// the package has loaded, so that there is one library in the process.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/types.h>

#include <optional>

#include "rodimus_ddts.h"

namespace {

decltype(&rodimus_ddts_fwd) g_fwd = nullptr;
decltype(&rodimus_ddts_fwd_workspace_bytes) g_fwd_ws = nullptr;
decltype(&rodimus_ddts_fwd_workspace_bytes_below) g_fwd_ws_below = nullptr;
decltype(&rodimus_ddts_step) g_step = nullptr;
decltype(&rodimus_ddts_bwd) g_bwd = nullptr;
decltype(&rodimus_ddts_bwd_workspace_bytes) g_bwd_ws = nullptr;
decltype(&rodimus_swska_fwd) g_swska = nullptr;

// A tensor argument: nullptr for None; anything that is neither is a TypeError.
struct Arg {
  const at::Tensor* t = nullptr;
  bool ok = true;
  explicit Arg(PyObject* o) {
    if (o == Py_None) return;
    if (!THPVariable_Check(o)) {
      PyErr_SetString(PyExc_TypeError, "expected a tensor");
      ok = false;
      return;
    }
    t = &THPVariable_Unpack(o);
  }
  void* ptr() const { return t ? t->data_ptr() : nullptr; }
};

bool on_device(std::initializer_list<const Arg*> args) {
  for (const Arg* a : args)
    if (a->t && !(a->t->is_cuda() && a->t->is_contiguous())) {
      PyErr_SetString(PyExc_ValueError, "tensors must be contiguous CUDA tensors");
      return false;
    }
  return true;
}
bool all_ok(std::initializer_list<const Arg*> args) {
  for (const Arg* a : args)
    if (!a->ok) return false;
  return true;
}
// The dtype code, or -1 (the caller reports RODIMUS_ERR_DTYPE).
int dtype_code(const at::Tensor& t) {
  return t.scalar_type() == at::kBFloat16 ? RODIMUS_BF16 : (t.scalar_type() == at::kFloat ? RODIMUS_F32 : -1);
}
bool rank_is(const Arg& a, int64_t n) {
  if (a.t && a.t->dim() == n) return true;
  PyErr_SetString(PyExc_ValueError, "a tensor has the wrong number of dimensions");
  return false;
}
void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
at::Tensor bytes_like(const at::Tensor& q, size_t n) {
  return at::empty({(int64_t)(n < 256 ? 256 : n)}, q.options().dtype(at::kByte));
}
// The prefill's workspace: what makes it fastest or, where that does not fit into the device's memory (it may
// be as large as the inputs), the next smaller size that it has a use for, down to the least it runs with.
at::Tensor fwd_workspace(const at::Tensor& q, const rodimus_ddts_fwd_params& p) {
  for (size_t n = g_fwd_ws(&p);;) {
    try {
      return bytes_like(q, n);
    } catch (const c10::OutOfMemoryError&) {
      const size_t less = g_fwd_ws_below(&p, n);
      if (less >= n) throw;
      n = less;
    }
  }
}
PyObject* wrap(const at::Tensor& t) { return THPVariable_Wrap(t); }

// The interpreter's lock is given up while tensors are allocated (which may wait for the device) and work is
// enqueued.
struct NoGil {
  PyThreadState* state = PyEval_SaveThread();
  NoGil() = default;
  NoGil(const NoGil&) = delete;
  ~NoGil() { PyEval_RestoreThread(state); }
};

// Every function returns an int - the status - where the library refused the call.  PyTorch's exceptions
// become the Python errors that its own functions raise (OutOfMemoryError among them).
#define RODIMUS_TRY try {
#define RODIMUS_CATCH                                                  \
  }                                                                    \
  catch (...) {                                                        \
    torch::translate_exception_to_python(std::current_exception());    \
    return nullptr;                                                    \
  }

// ddts_fwd(q, k, gate_x, temp_y, v, s0, cu_seqlens, cu_seqlens_host, scale, ingate, want_final_state, out,
//          final_state, workspace, beta_hat, feed_d, feed_x, value_decay) -> (o, sT | None)
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  RODIMUS_TRY
  if (n != 18) return PyErr_Format(PyExc_TypeError, "18 arguments expected");
  Arg q(a[0]), k(a[1]), x(a[2]), y(a[3]), v(a[4]), s0(a[5]), cu(a[6]), cu_h(a[7]), out(a[11]), fin(a[12]), ws(a[13]),
      beta(a[14]), fd(a[15]), fx(a[16]), vd(a[17]);
  if (!all_ok({&q, &k, &x, &y, &v, &s0, &cu, &cu_h, &out, &fin, &ws, &beta, &fd, &fx, &vd})) return nullptr;
  if (!on_device({&q, &k, &x, &y, &v, &s0, &cu, &beta, &fd, &fx, &vd})) return nullptr;
  if (!rank_is(q, 4) || !rank_is(v, 4)) return nullptr;
  const double scale = PyFloat_AsDouble(a[8]);
  const long ingate = PyLong_AsLong(a[9]);
  const int want = PyObject_IsTrue(a[10]);
  if (PyErr_Occurred()) return nullptr;
  rodimus_ddts_fwd_params p = {};
  p.struct_size = (int32_t)sizeof(p);
  p.dtype = dtype_code(*q.t);
  if (p.dtype < 0) return PyLong_FromLong(RODIMUS_ERR_DTYPE);
  p.ingate = (int32_t)ingate;
  p.B = (int32_t)q.t->size(0);
  p.H = (int32_t)v.t->size(1);
  p.T = (int32_t)q.t->size(2);
  p.dk = (int32_t)q.t->size(3);
  p.dv = (int32_t)v.t->size(3);
  p.scale = (float)scale;
  p.N = cu.t ? (int32_t)(cu.t->numel() - 1) : 0;
  p.shared_gates = q.t->size(1) == 1 && p.H > 1;
  std::optional<NoGil> no_gil(std::in_place);
  at::Tensor o = out.t ? *out.t : at::empty({p.B, p.H, p.T, p.dv}, q.t->options());
  at::Tensor sT;
  if (fin.t) sT = *fin.t;
  else if (want) sT = at::empty({cu.t ? p.N : p.B, p.H, p.dk, p.dv}, q.t->options().dtype(at::kFloat));
  p.q = q.ptr(); p.k = k.ptr(); p.gate_x = x.ptr(); p.temp_y = y.ptr(); p.v = v.ptr();
  p.o = o.data_ptr();
  p.s0 = (const float*)s0.ptr();
  p.sT = sT.defined() ? (float*)sT.data_ptr() : nullptr;
  p.cu_seqlens = (const int32_t*)cu.ptr();
  p.cu_seqlens_host = (const int32_t*)cu_h.ptr();
  p.beta_hat = beta.ptr(); p.feed_d = (const float*)fd.ptr(); p.feed_x = fx.ptr();
  p.value_decay = vd.ptr();
  p.stream = current_stream();
  at::Tensor w = ws.t ? *ws.t : fwd_workspace(*q.t, p);
  p.workspace = w.data_ptr();
  p.workspace_bytes = (size_t)w.numel() * w.element_size();
  const int rc = g_fwd(&p);
  no_gil.reset();
  if (rc != RODIMUS_OK) return PyLong_FromLong(rc);
  PyObject* r = PyTuple_New(2);
  if (!r) return nullptr;
  PyTuple_SET_ITEM(r, 0, wrap(o));
  if (sT.defined()) PyTuple_SET_ITEM(r, 1, wrap(sT));
  else { Py_INCREF(Py_None); PyTuple_SET_ITEM(r, 1, Py_None); }
  return r;
  RODIMUS_CATCH
}

// ddts_step(q, k, gate_x, temp_y, v, state, scale, ingate, out, beta_hat, feed_d, feed_x, value_decay) -> o
PyObject* step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  RODIMUS_TRY
  if (n != 13) return PyErr_Format(PyExc_TypeError, "13 arguments expected");
  Arg q(a[0]), k(a[1]), x(a[2]), y(a[3]), v(a[4]), state(a[5]), out(a[8]), beta(a[9]), fd(a[10]), fx(a[11]), vd(a[12]);
  if (!all_ok({&q, &k, &x, &y, &v, &state, &out, &beta, &fd, &fx, &vd})) return nullptr;
  if (!on_device({&q, &k, &x, &y, &v, &state, &beta, &fd, &fx, &vd})) return nullptr;
  if (!rank_is(q, 3) || !rank_is(v, 3)) return nullptr;
  const double scale = PyFloat_AsDouble(a[6]);
  const long ingate = PyLong_AsLong(a[7]);
  if (PyErr_Occurred()) return nullptr;
  rodimus_ddts_step_params p = {};
  p.struct_size = (int32_t)sizeof(p);
  p.dtype = dtype_code(*q.t);
  if (p.dtype < 0) return PyLong_FromLong(RODIMUS_ERR_DTYPE);
  p.ingate = (int32_t)ingate;
  p.Nseq = (int32_t)q.t->size(0);
  p.H = (int32_t)v.t->size(1);
  p.dk = (int32_t)q.t->size(2);
  p.dv = (int32_t)v.t->size(2);
  p.scale = (float)scale;
  p.shared_gates = q.t->size(1) == 1 && p.H > 1;
  std::optional<NoGil> no_gil(std::in_place);
  at::Tensor o = out.t ? *out.t : at::empty({p.Nseq, p.H, p.dv}, q.t->options());
  p.q = q.ptr(); p.k = k.ptr(); p.gate_x = x.ptr(); p.temp_y = y.ptr(); p.v = v.ptr();
  p.o = o.data_ptr();
  p.state = (float*)state.ptr();
  p.beta_hat = beta.ptr(); p.feed_d = (const float*)fd.ptr(); p.feed_x = fx.ptr();
  p.value_decay = vd.ptr();
  p.stream = current_stream();
  const int rc = g_step(&p);
  no_gil.reset();
  if (rc != RODIMUS_OK) return PyLong_FromLong(rc);
  return wrap(o);
  RODIMUS_CATCH
}

// ddts_bwd(q, k, gate_x, temp_y, v, d_o, s0, d_sT, cu_seqlens, cu_seqlens_host, scale, ingate, want_d_s0,
//          workspace) -> (d_q, d_k, d_gate_x, d_temp_y, d_v, d_s0 | None)
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  RODIMUS_TRY
  if (n != 14) return PyErr_Format(PyExc_TypeError, "14 arguments expected");
  Arg q(a[0]), k(a[1]), x(a[2]), y(a[3]), v(a[4]), d_o(a[5]), s0(a[6]), d_sT(a[7]), cu(a[8]), cu_h(a[9]), ws(a[13]);
  if (!all_ok({&q, &k, &x, &y, &v, &d_o, &s0, &d_sT, &cu, &cu_h, &ws})) return nullptr;
  if (!on_device({&q, &k, &x, &y, &v, &d_o, &s0, &d_sT, &cu})) return nullptr;
  if (!rank_is(q, 4) || !rank_is(v, 4)) return nullptr;
  const double scale = PyFloat_AsDouble(a[10]);
  const long ingate = PyLong_AsLong(a[11]);
  const int want = PyObject_IsTrue(a[12]);
  if (PyErr_Occurred()) return nullptr;
  rodimus_ddts_bwd_params p = {};
  p.struct_size = (int32_t)sizeof(p);
  p.dtype = dtype_code(*q.t);
  if (p.dtype < 0) return PyLong_FromLong(RODIMUS_ERR_DTYPE);
  p.ingate = (int32_t)ingate;
  p.B = (int32_t)q.t->size(0);
  p.H = (int32_t)q.t->size(1);
  p.T = (int32_t)q.t->size(2);
  p.dk = (int32_t)q.t->size(3);
  p.dv = (int32_t)v.t->size(3);
  p.scale = (float)scale;
  p.N = cu.t ? (int32_t)(cu.t->numel() - 1) : 0;
  std::optional<NoGil> no_gil(std::in_place);
  at::Tensor g[5];
  for (int i = 0; i < 4; ++i) g[i] = at::empty_like(*q.t);
  g[4] = at::empty_like(*v.t);
  at::Tensor g_s0;
  if (want) g_s0 = at::empty({cu.t ? p.N : p.B, p.H, p.dk, p.dv}, q.t->options().dtype(at::kFloat));
  p.q = q.ptr(); p.k = k.ptr(); p.gate_x = x.ptr(); p.temp_y = y.ptr(); p.v = v.ptr();
  p.s0 = (const float*)s0.ptr(); p.d_o = d_o.ptr(); p.d_sT = (const float*)d_sT.ptr();
  p.d_q = g[0].data_ptr(); p.d_k = g[1].data_ptr(); p.d_gate_x = g[2].data_ptr(); p.d_temp_y = g[3].data_ptr();
  p.d_v = g[4].data_ptr();
  p.d_s0 = want ? (float*)g_s0.data_ptr() : nullptr;
  p.cu_seqlens = (const int32_t*)cu.ptr();
  p.cu_seqlens_host = (const int32_t*)cu_h.ptr();
  p.stream = current_stream();
  at::Tensor w = ws.t ? *ws.t : bytes_like(*q.t, g_bwd_ws(&p));
  p.workspace = w.data_ptr();
  p.workspace_bytes = (size_t)w.numel() * w.element_size();
  const int rc = g_bwd(&p);
  no_gil.reset();
  if (rc != RODIMUS_OK) return PyLong_FromLong(rc);
  PyObject* r = PyTuple_New(6);
  if (!r) return nullptr;
  for (int i = 0; i < 5; ++i) PyTuple_SET_ITEM(r, i, wrap(g[i]));
  if (want) PyTuple_SET_ITEM(r, 5, wrap(g_s0));
  else { Py_INCREF(Py_None); PyTuple_SET_ITEM(r, 5, Py_None); }
  return r;
  RODIMUS_CATCH
}

// swska_fwd(q, k, v, window, scale | None, out | None) -> o
PyObject* swska(PyObject*, PyObject* const* a, Py_ssize_t n) {
  RODIMUS_TRY
  if (n != 6) return PyErr_Format(PyExc_TypeError, "6 arguments expected");
  Arg q(a[0]), k(a[1]), v(a[2]), out(a[5]);
  if (!all_ok({&q, &k, &v, &out}) || !on_device({&q, &k, &v})) return nullptr;
  if (!rank_is(q, 4)) return nullptr;
  const auto qs = q.t->sizes();
  if (!k.t || !v.t || k.t->sizes() != at::IntArrayRef({qs[0], qs[2], qs[3]}) || v.t->sizes() != qs)
    return PyErr_Format(PyExc_ValueError, "q, v must be [B,H,T,d] and k [B,T,d]");
  rodimus_swska_fwd_params p = {};
  p.struct_size = (int32_t)sizeof(p);
  p.dtype = dtype_code(*q.t);
  if (p.dtype < 0) return PyLong_FromLong(RODIMUS_ERR_DTYPE);
  p.B = (int32_t)qs[0]; p.H = (int32_t)qs[1]; p.T = (int32_t)qs[2]; p.d = (int32_t)qs[3];
  p.window = (int32_t)PyLong_AsLong(a[3]);
  p.scale = (float)(a[4] == Py_None ? 1.0 / std::sqrt((double)p.d) : PyFloat_AsDouble(a[4]));
  if (PyErr_Occurred()) return nullptr;
  std::optional<NoGil> no_gil(std::in_place);
  at::Tensor o = out.t ? *out.t : at::empty_like(*q.t);
  p.q = q.ptr(); p.k = k.ptr(); p.v = v.ptr();
  p.o = o.data_ptr();
  p.stream = current_stream();
  const int rc = g_swska(&p);
  no_gil.reset();
  if (rc != RODIMUS_OK) return PyLong_FromLong(rc);
  return wrap(o);
  RODIMUS_CATCH
}

// bind(addresses of rodimus_ddts_fwd, _fwd_workspace_bytes, _step, _bwd, _bwd_workspace_bytes, rodimus_swska_fwd,
//      rodimus_ddts_fwd_workspace_bytes_below)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 7) return PyErr_Format(PyExc_TypeError, "7 arguments expected");
  void* f[7];
  for (int i = 0; i < 7; ++i) {
    f[i] = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred()) return nullptr;
  }
  g_fwd = (decltype(g_fwd))f[0];
  g_fwd_ws = (decltype(g_fwd_ws))f[1];
  g_step = (decltype(g_step))f[2];
  g_bwd = (decltype(g_bwd))f[3];
  g_bwd_ws = (decltype(g_bwd_ws))f[4];
  g_swska = (decltype(g_swska))f[5];
  g_fwd_ws_below = (decltype(g_fwd_ws_below))f[6];
  Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"bind", (PyCFunction)(void*)bind, METH_FASTCALL, nullptr},
    {"ddts_fwd", (PyCFunction)(void*)fwd, METH_FASTCALL, nullptr},
    {"ddts_step", (PyCFunction)(void*)step, METH_FASTCALL, nullptr},
    {"ddts_bwd", (PyCFunction)(void*)bwd, METH_FASTCALL, nullptr},
    {"swska_fwd", (PyCFunction)(void*)swska, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&g_module); }
