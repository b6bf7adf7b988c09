// The way from a Python call on torch tensors to the C ABI (include/linattn.h, include/tconv.h) for the calls a model makes per layer.
//
// With few tokens a call's time is the time its arguments take: in Python, tensor by tensor and through ctypes, 9.4 us a call, of which the
// launch is 2.6.  Here the same checks read the tensors' fields.  Only the plain case is taken: exact torch.Tensor arguments, dense memory
// on a CUDA device, no mode or transform that wants to see torch functions.  Anything else answers NotImplemented before the library is called,
// and the caller goes the general way, which says what is wrong.  Time to issue a call, before and after, us:
// forward of 192 tokens 9.4 -> 5.1, cached step 9.7 -> 5.9, rotary read-only step 10.3 -> 5.4, temporal convolution step 9.0 -> 4.6 (which is then
// all that one of a few hundred positions takes: 9.0 -> 4.3).
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/ops/empty_like.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>

#include "linattn.h"
#include "tconv.h"

namespace {

// The library's entry points, from the library that the package has loaded.
decltype(&linattn_forward) p_forward;
decltype(&linattn_forward_rope) p_forward_rope;
decltype(&blocklin_step) p_step;
decltype(&blocklin_peek) p_peek;
decltype(&blocklin_step_rope) p_step_rope;
decltype(&blocklin_peek_rope) p_peek_rope;
decltype(&tconv_forward) p_tconv_forward;
decltype(&tconv_block_step) p_tconv_step;
PyObject* p_failed;   // failed(status, where): raises what the library's status means

PyObject* general() { Py_RETURN_NOTIMPLEMENTED; }

bool watched() { return at::impl::torch_function_mode_enabled() || c10::impl::TorchDispatchModeTLS::any_modes_set(); }

// The tensor in `o`, or null: not exactly a torch.Tensor, or none whose memory is simply there.
const at::Tensor* plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  using c10::DispatchKey;
  constexpr c10::DispatchKeySet odd({DispatchKey::Python, DispatchKey::PythonTLSSnapshot, DispatchKey::FuncTorchBatched, DispatchKey::FuncTorchGradWrapper,
                                     DispatchKey::Functionalize, DispatchKey::ZeroTensor, DispatchKey::Conjugate, DispatchKey::Negative});
  if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || t.key_set().has_any(odd) || !t.has_storage()) return nullptr;
  return &t;
}

int dtype_of(const at::Tensor& t) { return t.scalar_type() == at::kBFloat16 ? LINATTN_BF16 : t.scalar_type() == at::kFloat ? LINATTN_F32 : -1; }

bool fits(int64_t n) { return n <= INT32_MAX; }   // (a descriptor's numbers; of an expanded tensor they may not)

bool same(const at::Tensor& a, const at::Tensor& b) {
  return a.sizes() == b.sizes() && a.strides() == b.strides() && a.scalar_type() == b.scalar_type() && a.get_device() == b.get_device();
}

// [B, N, H, d] tensors of one layout: the descriptor.
bool describe(const at::Tensor& t, linattn_desc* d) {
  if (t.dim() != 4 || t.stride(3) != 1 || dtype_of(t) < 0 || !fits(t.size(0)) || !fits(t.size(2)) || !fits(t.size(3))) return false;
  d->B = (int32_t)t.size(0); d->H = (int32_t)t.size(2); d->d = (int32_t)t.size(3); d->dtype = dtype_of(t);
  d->stride_b = t.stride(0); d->stride_n = t.stride(1); d->stride_h = t.stride(2);
  return true;
}

bool is_table(const at::Tensor& t, const at::Tensor& q, int64_t rows) {
  return t.dim() == 3 && t.size(0) == rows && t.size(1) == q.size(3) / 2 && t.size(2) == 2 && t.scalar_type() == at::kHalf && t.is_contiguous() &&
         t.get_device() == q.get_device();
}

void* stream_of(const at::Tensor& t) { return c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)t.get_device()).stream(); }

// `out`, or a new tensor like `like` where it is None; false: not a plain one of that layout.
bool output(PyObject* out, const at::Tensor& like, at::Tensor* o) {
  if (out == Py_None) {
    *o = at::empty_like(like);
    return same(*o, like);
  }
  const at::Tensor* t = plain(out);
  if (!t || !same(*t, like)) return false;
  *o = *t;
  return true;
}

// What the library answered.  It has been called, and is not called again: a call that commits a block and takes several launches may
// have done so before it failed.
PyObject* answer(int status, const char* where, PyObject* out, at::Tensor&& o) {
  if (status != LINATTN_OK) {
    PyObject* none = PyObject_CallFunction(p_failed, "is", status, where);
    if (!none) return nullptr;
    Py_DECREF(none);
    return PyErr_Format(PyExc_SystemError, "%s: status %d", where, status);
  }
  if (out != Py_None) { Py_INCREF(out); return out; }
  return THPVariable_Wrap(std::move(o));
}

// In the calls below pointers and streams are taken before the interpreter's lock is let go: taking them may throw, and what is thrown becomes a
// Python error.

// forward(q, k, v, eps, out, workspace)
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 6 || !p_forward || !PyFloat_CheckExact(a[3]) || watched()) return general();
  const at::Tensor *q = plain(a[0]), *k = plain(a[1]), *v = plain(a[2]), *ws = plain(a[5]);
  linattn_desc d;
  at::Tensor o;
  if (!q || !k || !v || !ws || !describe(*q, &d) || !same(*k, *q) || !same(*v, *q) || ws->scalar_type() != at::kByte || !output(a[4], *q, &o)) return general();
  const float eps = (float)PyFloat_AS_DOUBLE(a[3]);
  const int64_t N = q->size(1);
  const void *pq = q->data_ptr(), *pk = k->data_ptr(), *pv = v->data_ptr();
  void *po = o.data_ptr(), *pw = ws->data_ptr(), *stream = stream_of(*q);
  const size_t room = (size_t)ws->numel();
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = p_forward(&d, N, pq, pk, pv, po, eps, pw, room, stream);
  Py_END_ALLOW_THREADS
  return answer(st, "linattn_forward", a[4], std::move(o));
  END_HANDLE_TH_ERRORS
}

// forward_rope(q, k, v, table, eps, out, workspace)
PyObject* forward_rope(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 7 || !p_forward_rope || !PyFloat_CheckExact(a[4]) || watched()) return general();
  const at::Tensor *q = plain(a[0]), *k = plain(a[1]), *v = plain(a[2]), *table = plain(a[3]), *ws = plain(a[6]);
  linattn_desc d;
  at::Tensor o;
  if (!q || !k || !v || !table || !ws || !describe(*q, &d) || !same(*k, *q) || !same(*v, *q) || !is_table(*table, *q, q->size(1)) ||
      ws->scalar_type() != at::kByte || !output(a[5], *q, &o))
    return general();
  const float eps = (float)PyFloat_AS_DOUBLE(a[4]);
  const int64_t N = q->size(1);
  const void *pq = q->data_ptr(), *pk = k->data_ptr(), *pv = v->data_ptr(), *pt = table->data_ptr();
  void *po = o.data_ptr(), *pw = ws->data_ptr(), *stream = stream_of(*q);
  const size_t room = (size_t)ws->numel();
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = p_forward_rope(&d, N, pq, pk, pv, po, eps, pt, pw, room, stream);
  Py_END_ALLOW_THREADS
  return answer(st, "linattn_forward_rope", a[5], std::move(o));
  END_HANDLE_TH_ERRORS
}

// step(commit, handle, B, H, d, dtype code, q, k, v, table or None, out): a cache of dense blocks, queries given
PyObject* step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 11 || !p_step || !PyLong_Check(a[1]) || watched()) return general();   // (a closed cache has None)
  const at::Tensor *q = plain(a[6]), *k = plain(a[7]), *v = plain(a[8]), *table = a[9] == Py_None ? nullptr : plain(a[9]);
  linattn_desc d;
  at::Tensor o;
  if (!q || !k || !v || (a[9] != Py_None && !table) || !describe(*k, &d) || !k->is_contiguous() || !same(*q, *k) || !same(*v, *k)) return general();
  if (d.B != PyLong_AsLong(a[2]) || d.H != PyLong_AsLong(a[3]) || d.d != PyLong_AsLong(a[4]) || d.dtype != PyLong_AsLong(a[5])) return general();
  if ((table && !is_table(*table, *k, k->size(1))) || !output(a[10], *q, &o)) return general();
  auto* cache = static_cast<blocklin_cache*>(PyLong_AsVoidPtr(a[1]));
  const bool commit = a[0] == Py_True;
  const int64_t T = k->size(1);
  const void *pq = q->data_ptr(), *pk = k->data_ptr(), *pv = v->data_ptr(), *pt = table ? table->data_ptr() : nullptr;
  void *po = o.data_ptr(), *stream = stream_of(*k);
  int st;
  Py_BEGIN_ALLOW_THREADS
  if (table) st = (commit ? p_step_rope : p_peek_rope)(cache, T, pq, pk, pv, po, pt, stream);
  else st = (commit ? p_step : p_peek)(cache, T, pq, pk, pv, po, stream);
  Py_END_ALLOW_THREADS
  return answer(st, table ? (commit ? "blocklin_step_rope" : "blocklin_peek_rope") : commit ? "blocklin_step" : "blocklin_peek", a[10], std::move(o));
  END_HANDLE_TH_ERRORS
}

// conv(x, w, out, frame or None, commit): dense [B, T, HW, D]; with a frame a block step on that cache
PyObject* conv(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 5 || !p_tconv_forward || watched()) return general();
  const at::Tensor *x = plain(a[0]), *w = plain(a[1]), *frame = a[3] == Py_None ? nullptr : plain(a[3]);
  at::Tensor y;
  if (!x || !w || (a[3] != Py_None && !frame) || x->dim() != 4 || dtype_of(*x) < 0 || !x->is_contiguous() || !fits(x->size(0)) ||
      !fits(x->size(2)) || !fits(x->size(3)))
    return general();
  if (w->scalar_type() != at::kFloat || w->dim() != 2 || w->size(0) != 3 || w->size(1) != x->size(3) || !w->is_contiguous()) return general();
  if (frame && (frame->dim() != 3 || frame->size(0) != x->size(0) || frame->size(1) != x->size(2) || frame->size(2) != x->size(3) ||
                frame->scalar_type() != x->scalar_type() || !frame->is_contiguous()))
    return general();
  if (!output(a[2], *x, &y)) return general();
  const tconv_desc d{(int32_t)x->size(0), (int32_t)x->size(2), (int32_t)x->size(3), dtype_of(*x), 0, 0};
  const int commit = a[4] == Py_True;
  const int64_t T = x->size(1);
  const void* px = x->data_ptr();
  const float* taps = w->data_ptr<float>();
  void *pf = frame ? frame->data_ptr() : nullptr, *py = y.data_ptr(), *stream = stream_of(*x);
  int st;
  Py_BEGIN_ALLOW_THREADS
  if (frame) st = p_tconv_step(&d, T, px, taps, pf, py, commit, stream);
  else st = p_tconv_forward(&d, T, px, taps, py, stream);
  Py_END_ALLOW_THREADS
  return answer(st, frame ? "tconv_block_step" : "tconv_forward", a[2], std::move(y));
  END_HANDLE_TH_ERRORS
}

// bind(failed, addresses of forward, forward_rope, step, peek, step_rope, peek_rope, tconv_forward, tconv_block_step)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 9 || !PyCallable_Check(a[0])) return PyErr_Format(PyExc_TypeError, "what raises an error, and eight addresses");
  void* p[8];
  for (int i = 0; i < 8; ++i)
    if (!(p[i] = PyLong_AsVoidPtr(a[1 + i]))) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_ValueError, "an address is null");
  Py_INCREF(a[0]);
  Py_XSETREF(p_failed, a[0]);
  p_forward = reinterpret_cast<decltype(p_forward)>(p[0]);
  p_forward_rope = reinterpret_cast<decltype(p_forward_rope)>(p[1]);
  p_step = reinterpret_cast<decltype(p_step)>(p[2]);
  p_peek = reinterpret_cast<decltype(p_peek)>(p[3]);
  p_step_rope = reinterpret_cast<decltype(p_step_rope)>(p[4]);
  p_peek_rope = reinterpret_cast<decltype(p_peek_rope)>(p[5]);
  p_tconv_forward = reinterpret_cast<decltype(p_tconv_forward)>(p[6]);
  p_tconv_step = reinterpret_cast<decltype(p_tconv_step)>(p[7]);
  Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(forward), FAST(forward_rope), FAST(step), FAST(conv), FAST(bind), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

#ifndef BUILT_AGAINST
#error "the version of the torch that this is built against"
#endif
PyMODINIT_FUNC PyInit__binding() {
  PyObject* m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "built_against", BUILT_AGAINST) < 0) Py_CLEAR(m);
  return m;
}
