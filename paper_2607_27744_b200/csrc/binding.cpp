// Native half of binding.py: takes torch tensors apart and calls the C ABI of rocs.h.
//
// A call through ctypes spent 12-30 us of host time, most of it on attribute look-ups, argument conversion
// and torch.cuda.current_stream(); the GPU needs less than that for a small batch, so the host was what a
// small batch waited for.  Here a tensor is a C++ object, the stream comes from c10, and a call costs about
// a microsecond on top of its launches.  Nothing is kept between calls.  The GIL is released around the
// library call, as ctypes does.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>

#include "../../include/rocs.h"

namespace {

PyObject* g_error = nullptr;  // binding.RocsError, set once by binding.py

struct PyRaised {};  // a Python exception is already set

[[noreturn]] void raise(PyObject* type, const char* what) {
  PyErr_SetString(type, what);
  throw PyRaised{};
}
void require(bool ok, const char* what = "") {
  if (!ok) raise(PyExc_AssertionError, what);
}
void check(rocs_status_t code, const char* where) {
  if (code == ROCS_OK) return;
  PyObject* e = PyObject_CallFunction(g_error, "is", (int)code, where);
  if (e != nullptr) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  throw PyRaised{};
}

// One argument that is a tensor or None.
struct Arg {
  const at::Tensor* t = nullptr;
  PyObject* obj = nullptr;
  explicit Arg(PyObject* o) : obj(o) {
    if (o == Py_None) return;
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch.Tensor");
    t = &THPVariable_Unpack(o);
  }
  explicit operator bool() const { return t != nullptr; }
  const at::Tensor* operator->() const {
    if (t == nullptr) raise(PyExc_AttributeError, "a required tensor is None");
    return t;
  }
  const void* ptr() const { return t ? t->const_data_ptr() : nullptr; }
  void* mut() const { return t ? t->mutable_data_ptr() : nullptr; }  // written to: a lazy clone gets memory of its own first
  int64_t size(int64_t d) const { return (*this)->size(d); }
  // row stride of a row-major 2-D CUDA tensor
  int64_t ld() const {
    require((*this)->dim() == 2 && t->stride(1) == 1 && t->is_cuda(), "expect a row-major 2-D CUDA tensor");
    return t->size(0) > 1 ? t->stride(0) : std::max(t->stride(0), t->size(1));
  }
  rocs_dtype_t dtype() const {
    if ((*this)->scalar_type() == at::kBFloat16) return ROCS_BF16;
    if (t->scalar_type() != at::kFloat) raise(PyExc_TypeError, "unsupported dtype: bfloat16 or float32 expected");
    return ROCS_F32;
  }
  size_t bytes() const { return t ? (size_t)t->numel() : 0; }  // of a uint8 workspace
  void need_dims(int64_t n) const {
    if ((*this)->dim() != n) {
      PyErr_Format(PyExc_ValueError, "expected a tensor of %d dimensions, got %d", (int)n, (int)t->dim());
      throw PyRaised{};
    }
  }
};

// The caller's tensor, or a new one with `like`'s device.
struct Out {
  at::Tensor made;
  Arg given;
  explicit Out(PyObject* o) : given(o) {}
  void or_empty(at::IntArrayRef shape, const Arg& like, at::ScalarType type) {
    if (!given) {
      made = at::empty(shape, at::TensorOptions().dtype(type).device(like->device()));
      given.t = &made;
    }
  }
  PyObject* release() {
    if (made.defined()) return THPVariable_Wrap(made);
    return Py_NewRef(given.obj);
  }
};

int32_t i32(PyObject* o) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) throw PyRaised{};
  return (int32_t)v;
}
float f32(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyRaised{};
  return (float)v;
}
bool truth(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw PyRaised{};
  return v != 0;
}
struct PlanArg {
  const rocs_plan_t* handle;
  int64_t R, N;
  // handle (an int, None once closed), R, N
  explicit PlanArg(PyObject* const* a) : handle(nullptr) {
    if (a[0] != Py_None) handle = static_cast<const rocs_plan_t*>(PyLong_AsVoidPtr(a[0]));
    R = PyLong_AsLongLong(a[1]);
    N = PyLong_AsLongLong(a[2]);
    if (PyErr_Occurred()) throw PyRaised{};
  }
};
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
rocs_act_t act(PyObject* relu) { return truth(relu) ? ROCS_ACT_RELU : ROCS_ACT_NONE; }

template <typename F>
rocs_status_t call(F&& f) {
  rocs_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = f();
  Py_END_ALLOW_THREADS
  return st;
}

PyObject* plan_create(PyObject* const* a) {
  const Arg off(a[0]), host(a[1]);
  require(off->is_cuda() && off->scalar_type() == at::kInt && off->is_contiguous());
  require(host->is_cpu() && host->scalar_type() == at::kInt && host->is_contiguous());
  const int64_t n = host->numel(), R = off->numel() - 1;
  const int32_t* h = static_cast<const int32_t*>(host.ptr());
  const int64_t N = n ? h[n - 1] : 0;
  void* st = stream();
  rocs_plan_t* plan = nullptr;
  check(call([&] { return rocs_plan_create(&plan, (int32_t)R, N, static_cast<const int32_t*>(off.ptr()), h, st); }),
        "rocs_plan_create");
  return Py_BuildValue("NLL", PyLong_FromVoidPtr(plan), (long long)R, (long long)N);
}

PyObject* plan_destroy(PyObject* const* a) {
  rocs_plan_t* plan = static_cast<rocs_plan_t*>(PyLong_AsVoidPtr(a[0]));
  call([&] { return rocs_plan_destroy(plan); });
  Py_RETURN_NONE;
}

// plan (3), XR, XC, W_CR, W_CC, bias, relu, out, workspace
PyObject* ikbo_linear(PyObject* const* a) {
  const PlanArg plan(a);
  const Arg XR(a[3]), XC(a[4]), W_CR(a[5]), W_CC(a[6]), bias(a[7]);
  const int32_t d_req = XR ? (int32_t)XR.size(1) : 0, d_cand = (int32_t)XC.size(1), d_out = (int32_t)W_CC.size(0);
  require(XC.size(0) == plan.N);
  Out out(a[9]), ws(a[10]);
  out.or_empty({plan.N, d_out}, XC, XC->scalar_type());
  const size_t need = d_req > 0 ? rocs_ikbo_linear_workspace(plan.handle, d_out) : 0;
  if (need) ws.or_empty({(int64_t)need}, XC, at::kByte);
  if (bias) require(bias->scalar_type() == at::kFloat && bias->is_contiguous());
  const rocs_dtype_t dt = XC.dtype();
  const int64_t ld_xr = d_req ? XR.ld() : 0, ld_xc = XC.ld(), ld_wcr = d_req ? W_CR.ld() : 0, ld_wcc = W_CC.ld(),
                ld_y = out.given.ld();
  const rocs_act_t ac = act(a[8]);
  void* st = stream();
  check(call([&] {
          return rocs_ikbo_linear(plan.handle, dt, d_req, d_cand, d_out, XR.ptr(), ld_xr, XC.ptr(), ld_xc,
                                  d_req ? W_CR.ptr() : nullptr, ld_wcr, W_CC.ptr(), ld_wcc,
                                  static_cast<const float*>(bias.ptr()), ac, out.given.mut(), ld_y, ws.given.mut(),
                                  ws.given.bytes(), st);
        }),
        "rocs_ikbo_linear");
  return out.release();
}

// plan (3), XR, XC, W_CR, W_CC, bias, relu, out, row_stats, workspace
PyObject* ikbo_linear_stats(PyObject* const* a) {
  const PlanArg plan(a);
  const Arg XR(a[3]), XC(a[4]), W_CR(a[5]), W_CC(a[6]), bias(a[7]);
  const int32_t d_req = (int32_t)XR.size(1), d_cand = (int32_t)XC.size(1), d_out = (int32_t)W_CC.size(0);
  require(XC.size(0) == plan.N);
  Out out(a[9]), stats(a[10]), ws(a[11]);
  out.or_empty({plan.N, d_out}, XC, XC->scalar_type());
  stats.or_empty({plan.N, 2}, XC, at::kFloat);
  if (!ws.given) ws.or_empty({(int64_t)rocs_ikbo_linear_stats_workspace(plan.handle, d_out)}, XC, at::kByte);
  const rocs_dtype_t dt = XC.dtype();
  const int64_t ld_xr = XR.ld(), ld_xc = XC.ld(), ld_wcr = W_CR.ld(), ld_wcc = W_CC.ld(), ld_y = out.given.ld();
  const rocs_act_t ac = act(a[8]);
  void* st = stream();
  check(call([&] {
          return rocs_ikbo_linear_stats(plan.handle, dt, d_req, d_cand, d_out, XR.ptr(), ld_xr, XC.ptr(), ld_xc, W_CR.ptr(),
                                        ld_wcr, W_CC.ptr(), ld_wcc, static_cast<const float*>(bias.ptr()), ac,
                                        out.given.mut(), ld_y, static_cast<float*>(stats.given.mut()), ws.given.mut(),
                                        ws.given.bytes(), st);
        }),
        "rocs_ikbo_linear_stats");
  return Py_BuildValue("NN", out.release(), stats.release());
}

// W, out
PyObject* weight_row_sums(PyObject* const* a) {
  const Arg W(a[0]);
  Out out(a[1]);
  W.need_dims(2);
  out.or_empty({W.size(0)}, W, at::kFloat);
  const rocs_dtype_t dt = W.dtype();
  const int64_t ld = W.ld();
  void* st = stream();
  check(call([&] {
          return rocs_weight_row_sums(dt, (int32_t)W.size(0), (int32_t)W.size(1), W.ptr(), ld,
                                      static_cast<float*>(out.given.mut()), st);
        }),
        "rocs_weight_row_sums");
  return out.release();
}

// X, row_stats, W, wbar, bias, eps, kind, relu, out
PyObject* linear_normed(PyObject* const* a) {
  const Arg X(a[0]), stats(a[1]), W(a[2]), wbar(a[3]), bias(a[4]);
  X.need_dims(2);
  const int64_t M = X.size(0);
  const int32_t d_in = (int32_t)X.size(1), d_out = (int32_t)W.size(0);
  require(stats->scalar_type() == at::kFloat && stats->dim() == 2 && stats.size(0) == M && stats.size(1) == 2 &&
          stats->is_contiguous());
  Out out(a[8]);
  out.or_empty({M, d_out}, X, X->scalar_type());
  const rocs_dtype_t dt = X.dtype();
  const int64_t ld_x = X.ld(), ld_w = W.ld(), ld_y = out.given.ld();
  const float eps = f32(a[5]);
  const auto kind = (rocs_norm_t)i32(a[6]);
  const rocs_act_t ac = act(a[7]);
  void* st = stream();
  check(call([&] {
          return rocs_linear_normed(dt, kind, M, d_in, d_out, X.ptr(), ld_x, static_cast<const float*>(stats.ptr()), eps,
                                    W.ptr(), ld_w, static_cast<const float*>(wbar.ptr()),
                                    static_cast<const float*>(bias.ptr()), ac, out.given.mut(), ld_y, st);
        }),
        "rocs_linear_normed");
  return out.release();
}

// X, W, bias, relu, out
PyObject* linear(PyObject* const* a) {
  const Arg X(a[0]), W(a[1]), bias(a[2]);
  X.need_dims(2);
  const int64_t M = X.size(0);
  const int32_t d_in = (int32_t)X.size(1), d_out = (int32_t)W.size(0);
  Out out(a[4]);
  out.or_empty({M, d_out}, X, X->scalar_type());
  const rocs_dtype_t dt = X.dtype();
  const int64_t ld_x = X.ld(), ld_w = W.ld(), ld_y = out.given.ld();
  const rocs_act_t ac = act(a[3]);
  void* st = stream();
  check(call([&] {
          return rocs_linear(dt, M, d_in, d_out, X.ptr(), ld_x, W.ptr(), ld_w, static_cast<const float*>(bias.ptr()), ac,
                             out.given.mut(), ld_y, st);
        }),
        "rocs_linear");
  return out.release();
}

// plan (3), Q, K, V, seq_offsets, scale, out
PyObject* dca_attention(PyObject* const* a) {
  const PlanArg plan(a);
  const Arg Q(a[3]), K(a[4]), V(a[5]), seq(a[6]);
  Q.need_dims(4);
  require(Q.size(0) == plan.N && Q->is_contiguous() && K->is_contiguous() && V->is_contiguous());
  require(seq->scalar_type() == at::kInt && seq->is_cuda() && seq->numel() == plan.R + 1);
  const int32_t n_q = (int32_t)Q.size(1), H = (int32_t)Q.size(2), dh = (int32_t)Q.size(3);
  Out out(a[8]), ws(Py_None);
  out.or_empty(Q->sizes(), Q, Q->scalar_type());
  const size_t need = rocs_dca_attention_workspace(plan.handle, n_q, H, dh);
  if (need) ws.or_empty({(int64_t)need}, Q, at::kByte);
  const rocs_dtype_t dt = Q.dtype();
  const float scale = f32(a[7]);
  const int64_t T = K.size(0);
  void* st = stream();
  check(call([&] {
          return rocs_dca_attention(plan.handle, dt, n_q, H, dh, scale, Q.ptr(), K.ptr(), V.ptr(), T,
                                    static_cast<const int32_t*>(seq.ptr()), out.given.mut(), ws.given.mut(), need, st);
        }),
        "rocs_dca_attention");
  return out.release();
}

// plan (3), XR, XC, W, n_ro, n_co, YR, YC, OR, OC, workspace
PyObject* glm_interaction(PyObject* const* a) {
  const PlanArg plan(a);
  const Arg XR(a[3]), XC(a[4]), W(a[5]), YR(a[8]), YC(a[9]), OR_(a[10]), OC(a[11]);
  XR.need_dims(3);
  XC.need_dims(3);
  require(XR.size(0) == plan.R && XC.size(0) == plan.N && XR->is_contiguous() && XC->is_contiguous());
  const int32_t n_r = (int32_t)XR.size(1), d = (int32_t)XR.size(2), n_c = (int32_t)XC.size(1);
  const int32_t n_ro = i32(a[6]), n_co = i32(a[7]);
  if (W) require(W->dim() == 2 && W.size(0) == n_ro + n_co && W.size(1) == n_r + n_c && W->is_contiguous());
  Out ws(a[12]);
  const size_t need = W ? rocs_glm_interaction_workspace(plan.handle, n_r, n_c, n_co) : 0;
  if (need) ws.or_empty({(int64_t)need}, XC, at::kByte);
  const rocs_dtype_t dt = XC.dtype();
  void* st = stream();
  check(call([&] {
          return rocs_glm_interaction(plan.handle, dt, n_r, n_c, d, XR.ptr(), XC.ptr(), W.ptr(), n_ro, n_co, YR.mut(), YC.mut(),
                                      OR_.mut(), OC.mut(), ws.given.mut(), ws.given.bytes(), st);
        }),
        "rocs_glm_interaction");
  Py_RETURN_NONE;
}

// plan (3), XR, XC, P, FR, FC, workspace
PyObject* glm_fm_projection(PyObject* const* a) {
  const PlanArg plan(a);
  const Arg XR(a[3]), XC(a[4]), P(a[5]), FR(a[6]), FC(a[7]);
  XR.need_dims(3);
  XC.need_dims(3);
  require(XR.size(0) == plan.R && XC.size(0) == plan.N && XR->is_contiguous() && XC->is_contiguous());
  const int32_t n_r = (int32_t)XR.size(1), d = (int32_t)XR.size(2), n_c = (int32_t)XC.size(1);
  require(P->dim() == 2 && P.size(0) == n_r + n_c && P->is_contiguous() && P->scalar_type() == XC->scalar_type());
  const int32_t k = (int32_t)P.size(1);
  Out ws(a[8]);
  if (!ws.given) ws.or_empty({(int64_t)rocs_glm_fm_projection_workspace(plan.handle, d, k)}, XC, at::kByte);
  const rocs_dtype_t dt = XC.dtype();
  void* st = stream();
  check(call([&] {
          return rocs_glm_fm_projection(plan.handle, dt, n_r, n_c, d, k, XR.ptr(), XC.ptr(), P.ptr(), FR.mut(), FC.mut(),
                                        ws.given.mut(), ws.given.bytes(), st);
        }),
        "rocs_glm_fm_projection");
  Py_RETURN_NONE;
}

// X, gamma, beta, eps, kind, out
PyObject* group_norm(PyObject* const* a) {
  const Arg X(a[0]), gamma(a[1]), beta(a[2]);
  require(X->dim() == 2 && X->stride(1) == 1);
  Out out(a[5]);
  out.or_empty({X.size(0), X.size(1)}, X, X->scalar_type());
  const rocs_dtype_t dt = X.dtype();
  const int64_t ld_x = X.ld(), ld_y = out.given.ld();
  const float eps = f32(a[3]);
  const auto kind = (rocs_norm_t)i32(a[4]);
  void* st = stream();
  check(call([&] {
          return rocs_group_norm(dt, kind, X.size(0), (int32_t)X.size(1), X.ptr(), ld_x, gamma.ptr(), beta.ptr(), eps,
                                 out.given.mut(), ld_y, st);
        }),
        "rocs_group_norm");
  return out.release();
}

// cand_offsets, XR, XC, W_CR, W_CC, out, bias, relu
PyObject* ikbo_linear_static(PyObject* const* a) {
  const Arg off(a[0]), XR(a[1]), XC(a[2]), W_CR(a[3]), W_CC(a[4]), out(a[5]), bias(a[6]);
  const rocs_dtype_t dt = XC.dtype();
  const int64_t ld_xr = XR.ld(), ld_xc = XC.ld(), ld_wcr = W_CR.ld(), ld_wcc = W_CC.ld(), ld_y = out.ld();
  const rocs_act_t ac = act(a[7]);
  void* st = stream();
  check(call([&] {
          return rocs_ikbo_linear_static(dt, (int32_t)(off->numel() - 1), XC.size(0), static_cast<const int32_t*>(off.ptr()),
                                         (int32_t)XR.size(1), (int32_t)XC.size(1), (int32_t)W_CC.size(0), XR.ptr(), ld_xr,
                                         XC.ptr(), ld_xc, W_CR.ptr(), ld_wcr, W_CC.ptr(), ld_wcc,
                                         static_cast<const float*>(bias.ptr()), ac, out.mut(), ld_y, st);
        }),
        "rocs_ikbo_linear_static");
  return Py_NewRef(a[5]);
}

PyObject* set_error_type(PyObject* const* a) {
  Py_XSETREF(g_error, Py_NewRef(a[0]));
  Py_RETURN_NONE;
}

// Argument count, and C++ exceptions as the Python ones that torch raises for them (running out of memory has a type of
// its own, which callers catch to score a smaller batch).
template <PyObject* (*F)(PyObject* const*), Py_ssize_t N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", N, n);
    return nullptr;
  }
  try {
    return F(args);
  } catch (const PyRaised&) {
    return nullptr;
  }
  END_HANDLE_TH_ERRORS
}

#define ENTRY(name, n) {#name, (PyCFunction)(void (*)(void))entry<name, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY(plan_create, 2),
                         ENTRY(plan_destroy, 1),
                         ENTRY(ikbo_linear, 11),
                         ENTRY(ikbo_linear_stats, 12),
                         ENTRY(weight_row_sums, 2),
                         ENTRY(linear_normed, 9),
                         ENTRY(linear, 5),
                         ENTRY(dca_attention, 9),
                         ENTRY(glm_interaction, 13),
                         ENTRY(glm_fm_projection, 9),
                         ENTRY(group_norm, 6),
                         ENTRY(ikbo_linear_static, 8),
                         ENTRY(set_error_type, 1),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
