// The binding's short calls in native code (module _calls).  A kernel-level call is a launch of two or three microseconds; from
// Python, allocating its result and marshalling a dozen arguments through ctypes took three to six more, so that a chain of
// them ran at the speed of the host (score, selection, LayerNorm and fill of 16 x 256 rows: 30 us of host time for 16 us of
// kernels).  Each function here takes the tensors as they are, checks them, allocates the results from torch's allocator and
// calls the C ABI with the interpreter lock released, as ctypes does: those four calls 30 -> 14 us of host time; with inputs
// that come from HBM each time the chain is the GPU's again, 30.2 -> 25.8 us.
//
// They serve plain CUDA tensors only.  Whatever is not that -- another type, device or layout, a subclass, a functorch wrapper,
// an active torch-function or dispatch mode, a number that is no int -- is answered with None, and binding.py goes its
// general way, which raises the errors.  An int is the status of a call that the library refused.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/TensorSubclassLikeUtils.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/fvar.h"

// Read from the file by build.py: the symbols below are those of one torch and one Python.
extern "C" __attribute__((used)) const char fvar_calls_built_for[] = FVAR_BUILT_FOR;

namespace {

bool modes_active() { return at::impl::torch_function_mode_enabled() || c10::impl::TorchDispatchModeTLS::any_modes_set(); }

// The tensor behind `o` if it is a plain one, else nullptr.
const at::Tensor *plain(PyObject *o) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor &t = THPVariable_Unpack(o);
  if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || at::isTensorSubclassLike(t)) return nullptr;
  return &t;
}
const at::Tensor *plain(PyObject *o, at::ScalarType type, int64_t dims) {
  const at::Tensor *t = plain(o);
  return t && t->scalar_type() == type && (dims < 0 || t->dim() == dims) && t->is_contiguous() ? t : nullptr;
}
bool as_int(PyObject *o, int *v) {
  if (!PyLong_CheckExact(o)) return false;
  int over = 0;
  const long long x = PyLong_AsLongLongAndOverflow(o, &over);
  if (over || x != static_cast<int>(x)) return false;
  *v = static_cast<int>(x);
  return true;
}
bool as_pair(PyObject *o, int *a, int *b) {
  return PyTuple_CheckExact(o) && PyTuple_GET_SIZE(o) == 2 && as_int(PyTuple_GET_ITEM(o, 0), a) && as_int(PyTuple_GET_ITEM(o, 1), b);
}
bool fits(int64_t v) { return v == static_cast<int>(v); }

at::Tensor empty_like_device(const at::Tensor &t, at::IntArrayRef sizes, at::ScalarType type) {
  return at::detail::empty_cuda(sizes, type, t.device(), std::nullopt);
}
void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
PyObject *none() { Py_RETURN_NONE; }
PyObject *wrap(const at::Tensor &t) { return THPVariable_Wrap(t); }
PyObject *pair_of(PyObject *a, PyObject *b) {
  PyObject *r = a && b ? PyTuple_New(2) : nullptr;
  if (!r) { Py_XDECREF(a); Py_XDECREF(b); return nullptr; }
  PyTuple_SET_ITEM(r, 0, a);
  PyTuple_SET_ITEM(r, 1, b);
  return r;
}

// Runs f (a call of the C ABI) without the interpreter lock.
template <typename F>
fvar_status unlocked(F f) {
  PyThreadState *save = PyEval_SaveThread();
  const fvar_status s = f();
  PyEval_RestoreThread(save);
  return s;
}
// A C++ exception (an allocation that failed) leaves as None: the general way meets it again and raises it as torch does.
template <typename F>
PyObject *guarded(F f) {
  if (modes_active()) return none();
  try {
    return f();
  } catch (...) {
    return none();
  }
}

PyObject *row_scores(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    const at::Tensor *x = n == 1 ? plain(a[0], at::kFloat, 3) : nullptr;
    if (!x || !fits(x->size(0)) || !fits(x->size(1)) || !fits(x->size(2))) return none();
    const int B = x->size(0), M = x->size(1), C = x->size(2);
    at::Tensor s = empty_like_device(*x, {B, M}, at::kFloat);
    const float *xp = static_cast<const float *>(x->data_ptr());
    float *sp = static_cast<float *>(s.data_ptr());
    void *st = stream();
    const fvar_status r = unlocked([&] { return fvar_row_scores(xp, B, M, C, sp, st); });
    return r == FVAR_OK ? wrap(s) : PyLong_FromLong(r);
  });
}

PyObject *select_topr(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    const at::Tensor *s = n == 2 ? plain(a[0], at::kFloat, 2) : nullptr;
    int r = 0;
    if (!s || !as_int(a[1], &r) || r < 0 || !fits(s->size(0)) || !fits(s->size(1))) return none();
    const int B = s->size(0), M = s->size(1);
    at::Tensor idx = empty_like_device(*s, {B, r}, at::kInt), inv = empty_like_device(*s, {B, M}, at::kInt);
    const float *sp = static_cast<const float *>(s->data_ptr());
    int *ip = static_cast<int *>(idx.data_ptr()), *vp = static_cast<int *>(inv.data_ptr());
    void *st = stream();
    const fvar_status e = unlocked([&] { return fvar_select_topr(sp, B, M, r, ip, vp, st); });
    return e == FVAR_OK ? pair_of(wrap(idx), wrap(inv)) : PyLong_FromLong(e);
  });
}

PyObject *ln_modulate(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    const at::Tensor *x = n == 4 ? plain(a[0], at::kFloat, 3) : nullptr;
    const at::Tensor *sh = x ? plain(a[1], at::kFloat, -1) : nullptr, *sc = sh ? plain(a[2], at::kFloat, -1) : nullptr;
    if (!sc || !PyFloat_CheckExact(a[3]) || !fits(x->size(0) * x->size(1)) || !fits(x->size(2))) return none();
    const int B = x->size(0), rows = x->size(1), C = x->size(2);
    const float eps = static_cast<float>(PyFloat_AS_DOUBLE(a[3]));
    at::Tensor y = empty_like_device(*x, {B, rows, C}, at::kBFloat16);
    const float *xp = static_cast<const float *>(x->data_ptr()), *hp = static_cast<const float *>(sh->data_ptr()), *cp = static_cast<const float *>(sc->data_ptr());
    void *yp = y.data_ptr(), *st = stream();
    const fvar_status e = unlocked([&] { return fvar_ln_modulate(xp, B * rows, C, rows, hp, cp, C, eps, yp, st); });
    return e == FVAR_OK ? wrap(y) : PyLong_FromLong(e);
  });
}

PyObject *rtr_fill(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    const at::Tensor *prev = n == 5 ? plain(a[0], at::kFloat, 3) : nullptr, *out = prev ? plain(a[4], at::kFloat, -1) : nullptr;
    int h0 = 0, w0 = 0, h1 = 0, w1 = 0;
    if (!out || !as_pair(a[1], &h0, &w0) || !as_pair(a[2], &h1, &w1) || !fits(prev->size(0)) || !fits(prev->size(2))) return none();
    const int *ip = nullptr;
    if (a[3] != Py_None) {
      const at::Tensor *inv = plain(a[3]);
      if (!inv) return none();
      ip = static_cast<const int *>(inv->data_ptr());
    }
    const int B = prev->size(0), C = prev->size(2);
    const float *pp = static_cast<const float *>(prev->data_ptr());
    float *op = static_cast<float *>(out->data_ptr());
    void *st = stream();
    const fvar_status e = unlocked([&] { return fvar_rtr_fill(pp, B, h0, w0, h1, w1, C, ip, op, st); });
    if (e != FVAR_OK) return PyLong_FromLong(e);
    Py_INCREF(a[4]);
    return a[4];
  });
}

PyObject *cfg_combine(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    const at::Tensor *p = n == 2 ? plain(a[0], at::kBFloat16, -1) : nullptr;
    if (!p || p->dim() < 1 || p->size(0) < 1 || !fits(p->size(0)) || !PyFloat_CheckExact(a[1])) return none();
    const int B = p->size(0);
    const long long per = p->numel() / B;
    const float s = static_cast<float>(PyFloat_AS_DOUBLE(a[1]));
    c10::SmallVector<int64_t, 6> sizes(p->sizes().begin(), p->sizes().end());
    sizes[0] = B / 2;
    at::Tensor out = empty_like_device(*p, sizes, at::kBFloat16);
    const void *pp = p->data_ptr();
    void *op = out.data_ptr(), *st = stream();
    const fvar_status e = unlocked([&] { return fvar_cfg_combine(pp, B, per, s, op, st); });
    return e == FVAR_OK ? wrap(out) : PyLong_FromLong(e);
  });
}

// (ctx address, fo, scale, tokens of the next scale or 0, pairs?) -> (codes, next tokens or None)
PyObject *scale_transition(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    const at::Tensor *fo = n == 5 && PyLong_CheckExact(a[0]) ? plain(a[1], at::kBFloat16, 3) : nullptr;
    int k = 0, next = 0;
    if (!fo || !as_int(a[2], &k) || !as_int(a[3], &next) || next < 0 || !PyBool_Check(a[4]) || !fits(fo->size(0))) return none();
    fvar_ctx *ctx = static_cast<fvar_ctx *>(PyLong_AsVoidPtr(a[0]));
    const bool pairs = a[4] == Py_True;
    const int64_t B = fo->size(0);
    at::Tensor codes = empty_like_device(*fo, {B, fo->size(1)}, at::kInt), nxt;
    if (next > 0) nxt = empty_like_device(*fo, {pairs ? 2 * B : B, next, fo->size(2)}, at::kBFloat16);
    const void *fp = fo->data_ptr();
    int *cp = static_cast<int *>(codes.data_ptr());
    void *np = next > 0 ? nxt.data_ptr() : nullptr;
    const fvar_status e = unlocked([&] {
      return pairs ? fvar_scale_transition_pairs(ctx, fp, k, static_cast<int>(B), cp, np) : fvar_scale_transition(ctx, fp, k, static_cast<int>(B), cp, np);
    });
    if (e != FVAR_OK) return PyLong_FromLong(e);
    if (next > 0) return pair_of(wrap(codes), wrap(nxt));
    Py_INCREF(Py_None);
    return pair_of(wrap(codes), Py_None);
  });
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(row_scores), FAST(select_topr), FAST(ln_modulate), FAST(rtr_fill), FAST(cfg_combine), FAST(scale_transition), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&module); }
