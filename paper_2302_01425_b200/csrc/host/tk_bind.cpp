// tk_bind.cpp -- the argument marshalling of binding.py in C++: tensors and numbers in, one call of the C ABI out.
//
// A call of the C ABI takes 2-3 us of host time, most of it the launch; marshalling it through ctypes (an option
// structure filled field by field, five attribute calls per tensor, the current stream, ten argument conversions) took
// 8 us more, and a step on a router-sized batch is two calls around 10 us of kernels: 16384 x 64 forward + VJP 23 us
// through ctypes, 10.3 now (the kernels' time).  Here a tensor's checks are reads of its fields.
//
// Every function makes the checks that binding.py makes and returns the status of the call -- or None, without having
// called anything, when an argument is not a plain tensor of the expected kind (or too short, or a number of another
// type) or no library is bound: binding.py's own code then goes through it and raises the error.
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "tk.h"

namespace {

// The entry points of the bound library (addresses from the one that binding.py has loaded).
struct Entries {
  decltype(&tk_fwd) fwd;
  decltype(&tk_fwd_noalloc) fwd_noalloc;
  decltype(&tk_fwd_ex) fwd_ex;
  decltype(&tk_vjp) vjp;
  decltype(&tk_jvp) jvp;
  decltype(&tk_topk_loss) topk_loss;
  decltype(&tk_fwd_cols) fwd_cols;
  decltype(&tk_vjp_cols) vjp_cols;
  decltype(&tk_argsort) argsort;
  decltype(&tk_fwd_w) fwd_w;
  decltype(&tk_vjp_w) vjp_w;
};
Entries g_lib = {};
bool g_bound = false;

// The positional arguments of one call, converted one after the other; `ok` ends as false when one does not fit.
struct Args {
  PyObject* const* a;
  Py_ssize_t n, i = 0;
  bool ok = true;

  PyObject* next() {
    if (i >= n) { ok = false; return Py_None; }
    return a[i++];
  }
  long long integer() {
    PyObject* o = next();
    if (!ok || !PyLong_Check(o)) { ok = false; return 0; }
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    if (over || v > 0x7fffffffLL || v < -0x7fffffffLL) { ok = false; return 0; }     // (products of two cannot overflow)
    return v;
  }
  double number() {
    PyObject* o = next();
    if (ok && PyFloat_Check(o)) return PyFloat_AS_DOUBLE(o);
    if (ok && PyLong_Check(o)) {
      const double v = PyLong_AsDouble(o);
      if (PyErr_Occurred()) { PyErr_Clear(); ok = false; }
      return v;
    }
    ok = false;
    return 0.0;
  }
  // Address of a contiguous CUDA tensor of `need` elements or more; null for None where that is allowed.
  void* tensor(c10::ScalarType type, long long need, bool optional, long long* numel = nullptr) {
    PyObject* o = next();
    if (numel) *numel = 0;
    if (o == Py_None) { if (!optional) ok = false; return nullptr; }
    if (!ok || !THPVariable_Check(o)) { ok = false; return nullptr; }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.scalar_type() != type || !t.is_contiguous() || t.numel() < need) {
      ok = false;
      return nullptr;
    }
    if (numel) *numel = t.numel();
    return t.data_ptr();
  }
  float* f32(long long need, bool optional = false, long long* numel = nullptr) {
    return static_cast<float*>(tensor(c10::ScalarType::Float, need, optional, numel));
  }
  int32_t* i32(long long need, bool optional = false) {
    return static_cast<int32_t*>(tensor(c10::ScalarType::Int, need, optional));
  }
  tk_rowstate* state(long long rows, bool optional) {
    return static_cast<tk_rowstate*>(tensor(c10::ScalarType::Byte, rows * (long long)sizeof(tk_rowstate), optional));
  }
  void workspace(tk_opts* o) {
    long long bytes = 0;
    o->workspace = tensor(c10::ScalarType::Byte, 0, true, &bytes);
    o->workspace_bytes = (size_t)bytes;
  }
  bool all() const { return ok && i == n && g_bound; }
};

// one call of the library on torch's current stream, without the interpreter lock
template <class F>
PyObject* call(F f) {
  void* stream = c10::cuda::getCurrentCUDAStream().stream();
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f(stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

#define TK_TRY try {
#define TK_END                                   \
  }                                              \
  catch (...) {}                                 \
  PyErr_Clear();                                 \
  Py_RETURN_NONE;

// rows, n, k, p, lam, mode, theta, out
PyObject* b_fwd(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer(), k = g.integer();
  const double p = g.number(), lam = g.number();
  const int mode = (int)g.integer();
  const float* theta = g.f32(rows * n);
  float* out = g.f32(rows * n);
  if (g.all()) return call([&](void* st) { return g_lib.fwd(theta, rows, n, k, p, lam, mode, out, st); });
  TK_END
}

PyObject* b_fwd_noalloc(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer(), k = g.integer();
  const double p = g.number(), lam = g.number();
  const int mode = (int)g.integer();
  const float* theta = g.f32(rows * n);
  float* out = g.f32(rows * n);
  if (g.all()) return call([&](void* st) { return g_lib.fwd_noalloc(theta, rows, n, k, p, lam, mode, out, st); });
  TK_END
}

// rows, n, k, p, lam, mode, theta, out, solver, sweeps, perm_out, state_out, workspace, status_out, flags, tol
PyObject* b_fwd_ex(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer(), k = g.integer();
  const double p = g.number(), lam = g.number();
  const int mode = (int)g.integer();
  const float* theta = g.f32(rows * n);
  float* out = g.f32(rows * n);
  tk_opts o = {};
  o.solver = (int)g.integer();
  o.sweeps = (int)g.integer();
  o.perm_out = g.i32(rows * n, true);
  o.state_out = g.state(rows, true);
  g.workspace(&o);
  o.status_out = g.i32(1, true);
  o.flags = (int)g.integer();
  o.tol = (float)g.number();
  if (g.all()) return call([&](void* st) { return g_lib.fwd_ex(theta, rows, n, k, p, lam, mode, out, &o, st); });
  TK_END
}

// rows, n, k, p, lam, mode, theta, grad_out, grad_theta, state, workspace, status_out
PyObject* b_vjp(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer(), k = g.integer();
  const double p = g.number(), lam = g.number();
  const int mode = (int)g.integer();
  const float* theta = g.f32(rows * n);
  const float* gout = g.f32(rows * n);
  float* grad = g.f32(rows * n);
  tk_opts o = {};
  o.state_out = g.state(rows, true);
  g.workspace(&o);
  o.status_out = g.i32(1, true);
  if (g.all()) return call([&](void* st) { return g_lib.vjp(theta, gout, rows, n, k, p, lam, mode, grad, &o, st); });
  TK_END
}

// as b_vjp, with the tangent and its image
PyObject* b_jvp(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer(), k = g.integer();
  const double p = g.number(), lam = g.number();
  const int mode = (int)g.integer();
  const float* theta = g.f32(rows * n);
  const float* tangent = g.f32(rows * n);
  float* out = g.f32(rows * n);
  tk_opts o = {};
  o.state_out = g.state(rows, true);
  g.workspace(&o);
  o.status_out = g.i32(1, true);
  if (g.all()) return call([&](void* st) { return g_lib.jvp(theta, tangent, rows, n, k, p, lam, mode, out, &o, st); });
  TK_END
}

// rows, n, k, p, lam, theta, target, loss, grad, solver, sweeps, state_out, workspace, status_out
PyObject* b_topk_loss(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer(), k = g.integer();
  const double p = g.number(), lam = g.number();
  const float* theta = g.f32(rows * n);
  const int32_t* target = g.i32(rows, true);
  float* loss = g.f32(rows);
  float* grad = g.f32(rows * n);
  tk_opts o = {};
  o.solver = (int)g.integer();
  o.sweeps = (int)g.integer();
  o.state_out = g.state(rows, true);
  g.workspace(&o);
  o.status_out = g.i32(1, true);
  if (g.all()) return call([&](void* st) { return g_lib.topk_loss(theta, target, rows, n, k, p, lam, loss, grad, &o, st); });
  TK_END
}

long long cols_span(long long n, long long cols, long long ld) { return n > 0 ? (n - 1) * ld + cols : 0; }

// n, cols, ld, k, p, lam, mode, theta, out, solver, sweeps, perm_out, state_out, workspace, status_out, flags
PyObject* b_fwd_cols(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long n = g.integer(), cols = g.integer(), ld = g.integer(), k = g.integer();
  const double p = g.number(), lam = g.number();
  const int mode = (int)g.integer();
  const float* theta = g.f32(cols_span(n, cols, ld));
  float* out = g.f32(cols_span(n, cols, ld));
  tk_opts o = {};
  o.solver = (int)g.integer();
  o.sweeps = (int)g.integer();
  o.perm_out = g.i32(cols * n, true);
  o.state_out = g.state(cols, true);
  g.workspace(&o);
  o.status_out = g.i32(1, true);
  o.flags = (int)g.integer();
  if (g.all()) return call([&](void* st) { return g_lib.fwd_cols(theta, n, cols, ld, k, p, lam, mode, out, &o, st); });
  TK_END
}

// n, cols, ld, k, p, lam, mode, theta or None, grad_out, grad_theta, state, workspace, status_out
PyObject* b_vjp_cols(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long n = g.integer(), cols = g.integer(), ld = g.integer(), k = g.integer();
  const double p = g.number(), lam = g.number();
  const int mode = (int)g.integer();
  const float* theta = g.f32(cols_span(n, cols, ld), true);
  const float* gout = g.f32(cols_span(n, cols, ld));
  float* grad = g.f32(cols_span(n, cols, ld));
  tk_opts o = {};
  o.state_out = g.state(cols, true);
  g.workspace(&o);
  o.status_out = g.i32(1, true);
  if (g.all()) return call([&](void* st) { return g_lib.vjp_cols(theta, gout, n, cols, ld, k, p, lam, mode, grad, &o, st); });
  TK_END
}

// rows, n, mode, theta, perm_out, sorted_out, workspace, status_out
PyObject* b_argsort(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer();
  const int mode = (int)g.integer();
  const float* theta = g.f32(rows * n);
  int32_t* perm = g.i32(rows * n);
  float* sorted = g.f32(rows * n, true);
  tk_opts o = {};
  g.workspace(&o);
  o.status_out = g.i32(1, true);
  if (g.all()) return call([&](void* st) { return g_lib.argsort(theta, rows, n, mode, perm, sorted, &o, st); });
  TK_END
}

// w: [n] shared by every row or [rows, n]
long long w_rows_of(long long numel, long long rows, long long n) {
  if (numel == n && rows != 1) return 1;
  return numel >= rows * n ? rows : 1;
}

// rows, n, p, lam, theta, w, out, status_out
PyObject* b_fwd_w(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer();
  const double p = g.number(), lam = g.number();
  const float* theta = g.f32(rows * n);
  long long numel = 0;
  const float* w = g.f32(0, false, &numel);
  const long long w_rows = w_rows_of(numel, rows, n);
  float* out = g.f32(rows * n);
  tk_opts o = {};
  o.status_out = g.i32(1, true);
  if (g.all() && numel >= w_rows * n) return call([&](void* st) { return g_lib.fwd_w(theta, w, rows, n, w_rows, p, lam, out, &o, st); });
  TK_END
}

// rows, n, p, lam, theta, w, grad_out, grad_theta, grad_w, status_out
PyObject* b_vjp_w(PyObject*, PyObject* const* a, Py_ssize_t n_) {
  TK_TRY
  Args g{a, n_};
  const long long rows = g.integer(), n = g.integer();
  const double p = g.number(), lam = g.number();
  const float* theta = g.f32(rows * n);
  long long numel = 0;
  const float* w = g.f32(0, false, &numel);
  const long long w_rows = w_rows_of(numel, rows, n);
  const float* gout = g.f32(rows * n);
  float* grad = g.f32(rows * n);
  float* grad_w = g.f32(rows * n, true);
  tk_opts o = {};
  o.status_out = g.i32(1, true);
  if (g.all() && numel >= w_rows * n)
    return call([&](void* st) { return g_lib.vjp_w(theta, w, gout, rows, n, w_rows, p, lam, grad, grad_w, &o, st); });
  TK_END
}

// bind(addresses...) in the order of Entries; bind() unbinds
PyObject* b_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  constexpr Py_ssize_t N = sizeof(Entries) / sizeof(void*);
  g_bound = false;
  if (n == 0) Py_RETURN_NONE;
  if (n != N) { PyErr_SetString(PyExc_TypeError, "bind: wrong number of addresses"); return nullptr; }
  void* at[N];
  for (Py_ssize_t i = 0; i < N; ++i) {
    at[i] = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred()) return nullptr;
    if (!at[i]) { PyErr_SetString(PyExc_ValueError, "bind: null address"); return nullptr; }
  }
  std::memcpy(&g_lib, at, sizeof(g_lib));
  g_bound = true;
  Py_RETURN_NONE;
}

#define TK_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(b_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {TK_METHOD(bind), TK_METHOD(fwd), TK_METHOD(fwd_noalloc), TK_METHOD(fwd_ex), TK_METHOD(vjp),
                         TK_METHOD(jvp), TK_METHOD(topk_loss), TK_METHOD(fwd_cols), TK_METHOD(vjp_cols),
                         TK_METHOD(argsort), TK_METHOD(fwd_w), TK_METHOD(vjp_w), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tk_bind", "argument marshalling of the binding", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tk_bind() { return PyModule_Create(&module); }
