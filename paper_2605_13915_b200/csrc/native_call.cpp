// Argument marshalling of the hot entry points in native code (the module paper_2605_13915_b200._native): a call takes torch
// tensors, checks them, and passes their addresses, sizes and the current CUDA stream to the C ABI of msd.h.
//
// Why: through ctypes a decode-sized linear layer cost 18 us of host time, of which the library itself (argument checks,
// tensor maps, two kernel launches) is 5; looking up the stream alone took 3.4 us.  The kernels of such a layer run for
// 12 to 20 us, so it was the host that set the pace.  Only marshalling lives here: every call returns the status code of
// the C function and binding.py turns it into an exception, allocates outputs and workspaces, and documents the arguments.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <vector>

#include "msd.h"

namespace {

// One call's arguments, taken off the array in order; the first problem sets a Python exception and every later take
// returns an empty value.
class Args {
 public:
  Args(PyObject* const* a, Py_ssize_t n) : a_(a), n_(n) {}
  bool ok() const { return ok_; }

  const at::Tensor* tensor(bool nullable = false) { return take(nullable, false); }
  // written by the kernels: a contiguous CUDA tensor, or page-locked host memory that they can reach
  const at::Tensor* buffer(bool nullable = false) { return take(nullable, true); }
  int64_t integer() {
    PyObject* o = next();
    if (!o) return 0;
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) ok_ = false;
    return v;
  }
  double number() {
    PyObject* o = next();
    if (!o) return 0.0;
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) ok_ = false;
    return v;
  }
  void fail(PyObject* type, const char* what) {
    if (ok_) PyErr_SetString(type, what);
    ok_ = false;
  }

 private:
  const at::Tensor* take(bool nullable, bool pinned) {
    PyObject* o = next();
    if (!o) return nullptr;
    if (o == Py_None && nullable) return nullptr;
    if (!THPVariable_Check(o)) {
      fail(PyExc_TypeError, "expected a tensor");
      return nullptr;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!(t.is_cuda() || (pinned && t.is_pinned())) || !t.is_contiguous()) {
      fail(PyExc_ValueError, "expected contiguous CUDA tensors");
      return nullptr;
    }
    return &t;
  }
  PyObject* next() {
    if (!ok_) return nullptr;
    if (i_ >= n_) {
      fail(PyExc_TypeError, "too few arguments");
      return nullptr;
    }
    return a_[i_++];
  }
  PyObject* const* a_;
  Py_ssize_t n_, i_ = 0;
  bool ok_ = true;
};

void* addr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
template <typename T>
T* addr_as(const at::Tensor* t) { return static_cast<T*>(addr(t)); }
msd_out_t out_type(const at::Tensor* y) { return y->scalar_type() == at::kBFloat16 ? MSD_OUT_BF16 : MSD_OUT_FP32; }
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The workspace a tensor offers: its bytes from the first 1024-byte boundary on, none where it ends before that.
struct Workspace {
  void* p;
  size_t bytes;
  explicit Workspace(const at::Tensor* t) {
    const uintptr_t base = reinterpret_cast<uintptr_t>(t->data_ptr()), al = (base + 1023) / 1024 * 1024;
    p = reinterpret_cast<void*>(al);
    bytes = t->nbytes() > al - base ? t->nbytes() - (al - base) : 0;
  }
};

// Calls into the library without the interpreter's lock: a launch waits where the stream's queue is full, and what is ahead in
// the queue may need a Python thread to go on.  Everything the call needs has been read off the arguments by then (the
// caller's frame keeps the tensors).
template <typename Call>
PyObject* status_of(const Call& call) {
  PyThreadState* lock = PyEval_SaveThread();
  const msd_status_t s = call();
  PyEval_RestoreThread(lock);
  return PyLong_FromLong(static_cast<long>(s));
}

// (-n: at least n; the sizes past them are not asked for)
bool dims(Args& a, std::initializer_list<std::pair<const at::Tensor*, int>> want) {
  if (!a.ok()) return false;
  for (const auto& w : want)
    if (w.second < 0 ? w.first->dim() < -w.second : w.first->dim() != w.second) {
      a.fail(PyExc_ValueError, "a tensor has the wrong number of dimensions");
      return false;
    }
  return true;
}

// (x, w, w_scale, ws, y, acc or None, scaling); None for a pointer that the library requires is passed on, and refused there
PyObject* gemm_w8a16(PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  const at::Tensor *x = a.tensor(), *w = a.tensor(), *s = a.tensor(true), *ws = a.buffer(), *y = a.buffer(),
                   *acc = a.buffer(true);
  const int64_t scaling = a.integer();
  if (!dims(a, {{x, 2}, {w, -1}})) return nullptr;
  const Workspace k(ws);
  const int64_t M = x->size(0), N = w->size(0), K = x->size(1);
  void *xp = addr(x), *yp = addr(y), *st = stream();
  const auto *wp = addr_as<int8_t>(w);
  const auto *sp = addr_as<float>(s);
  auto *ap = addr_as<int32_t>(acc);
  const msd_out_t yt = out_type(y);
  return status_of([&] { return msd_gemm_w8a16_ex(xp, wp, sp, M, N, K, yp, yt, ap, static_cast<msd_scaling_t>(scaling), k.p, k.bytes, st); });
}

// (x, w_fp4, scales, prepared, ws, y)
PyObject* gemm_w4a16(PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  const at::Tensor *x = a.tensor(), *w = a.tensor(), *s = a.tensor(true);
  const bool prepared = a.integer() != 0;
  const at::Tensor *ws = a.buffer(), *y = a.buffer();
  if (!dims(a, {{x, 2}, {w, -1}})) return nullptr;
  const Workspace k(ws);
  const auto fn = prepared ? msd_gemm_w4a16_prepared : msd_gemm_w4a16;
  const int64_t M = x->size(0), N = w->size(0), K = x->size(1);
  void *xp = addr(x), *yp = addr(y), *st = stream();
  const auto *wp = addr_as<uint8_t>(w), *sp = addr_as<uint8_t>(s);
  const msd_out_t yt = out_type(y);
  return status_of([&] { return fn(xp, wp, sp, M, N, K, yp, yt, k.p, k.bytes, st); });
}

// Rows per expert from a Python sequence; their sum must be the number of rows of x.
bool group_sizes(Args& a, PyObject* seq, int64_t E, int64_t rows, std::vector<int32_t>& out) {
  const THPObjectPtr fast(PySequence_Fast(seq, "group_sizes: expected a sequence"));
  if (!fast) return false;
  int64_t sum = 0;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast.get());
  out.reserve(static_cast<size_t>(E));
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* item = PySequence_Fast_GET_ITEM(fast.get(), i);
    THPObjectPtr as_int;
    if (!PyLong_Check(item)) {                   // whatever int() takes
      as_int = PyNumber_Long(item);
      if (!as_int) return false;
      item = as_int.get();
    }
    const long v = PyLong_AsLong(item);
    if (v == -1 && PyErr_Occurred()) return false;
    out.push_back(static_cast<int32_t>(v));
    sum += v;
  }
  if (n != E || sum != rows) {
    a.fail(PyExc_AssertionError, "group_sizes: one per expert, adding up to the rows of x");
    return false;
  }
  return true;
}

// (x, w, w_scale, group_sizes, ws, y)
PyObject* grouped_gemm_w8a16(PyObject* const* args, Py_ssize_t n) {
  if (n != 6) return PyErr_Format(PyExc_TypeError, "expected 6 arguments");
  Args t(args, 3), u(args + 4, 2);
  const at::Tensor *x = t.tensor(), *w = t.tensor(), *s = t.tensor(true);
  if (!dims(t, {{x, 2}, {w, 3}})) return nullptr;
  const at::Tensor *ws = u.buffer(), *y = u.buffer();
  std::vector<int32_t> sizes;
  if (!u.ok() || !group_sizes(u, args[3], w->size(0), x->size(0), sizes)) return nullptr;
  if (x->size(1) != w->size(2)) return PyErr_Format(PyExc_AssertionError, "x and w differ in K");
  const Workspace k(ws);
  const int32_t E = static_cast<int32_t>(w->size(0));
  const int64_t N = w->size(1), K = w->size(2);
  void *xp = addr(x), *yp = addr(y), *st = stream();
  const auto *wp = addr_as<int8_t>(w);
  const auto *sp = addr_as<float>(s);
  const msd_out_t yt = out_type(y);
  return status_of([&] { return msd_grouped_gemm_w8a16(xp, wp, sp, sizes.data(), E, N, K, yp, yt, k.p, k.bytes, st); });
}

// (x, w_fp4, scales, group_sizes, prepared, ws, y)
PyObject* grouped_gemm_w4a16(PyObject* const* args, Py_ssize_t n) {
  if (n != 7) return PyErr_Format(PyExc_TypeError, "expected 7 arguments");
  Args t(args, 3), u(args + 4, 3);
  const at::Tensor *x = t.tensor(), *w = t.tensor(), *s = t.tensor(true);
  if (!dims(t, {{x, 2}, {w, 3}})) return nullptr;
  const bool prepared = u.integer() != 0;
  const at::Tensor *ws = u.buffer(), *y = u.buffer();
  std::vector<int32_t> sizes;
  if (!u.ok() || !group_sizes(u, args[3], w->size(0), x->size(0), sizes)) return nullptr;
  if (x->size(1) != 2 * w->size(2)) return PyErr_Format(PyExc_AssertionError, "x and w_fp4 differ in K");
  const Workspace k(ws);
  const auto fn = prepared ? msd_grouped_gemm_w4a16_prepared : msd_grouped_gemm_w4a16;
  const int32_t E = static_cast<int32_t>(w->size(0));
  const int64_t N = w->size(1), K = 2 * w->size(2);
  void *xp = addr(x), *yp = addr(y), *st = stream();
  const auto *wp = addr_as<uint8_t>(w), *sp = addr_as<uint8_t>(s);
  const msd_out_t yt = out_type(y);
  return status_of([&] { return fn(xp, wp, sp, sizes.data(), E, N, K, yp, yt, k.p, k.bytes, st); });
}

// (q, k, v or None, k_scale, v_scale or None, cu_seqlens, max_seqlen, softmax_scale, Dv, ws, out, lse or None);
// q is [B, Hq, D], or with `spec` (several query tokens) [B, q_len, Hq, D]
template <bool spec>
PyObject* attn_decode(PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  const at::Tensor *q = a.tensor(), *k = a.tensor(), *v = a.tensor(true), *ks = a.tensor(true), *vs = a.tensor(true), *cu = a.tensor(true);
  const int32_t max_seqlen = static_cast<int32_t>(a.integer());
  const float scale = static_cast<float>(a.number());
  const int32_t Dv = static_cast<int32_t>(a.integer());
  const at::Tensor *ws = a.buffer(), *out = a.buffer(), *lse = a.buffer(true);
  constexpr int rank = spec ? 4 : 3;
  if (!dims(a, {{q, rank}, {k, -2}})) return nullptr;
  const Workspace w(ws);
  const int32_t B = static_cast<int32_t>(q->size(0)), Hq = static_cast<int32_t>(q->size(rank - 2)), D = static_cast<int32_t>(q->size(rank - 1));
  const int32_t Hkv = static_cast<int32_t>(k->size(1)), q_len = spec ? static_cast<int32_t>(q->size(1)) : 1;
  const int64_t T = k->size(0);
  void *qp = addr(q), *op = addr(out), *st = stream();
  const auto *kp = addr_as<int8_t>(k), *vp = addr_as<int8_t>(v);
  const auto *ksp = addr_as<float>(ks), *vsp = addr_as<float>(vs);
  const auto *cup = addr_as<int32_t>(cu);
  auto *lp = addr_as<float>(lse);
  return status_of([&] {
    if constexpr (spec)
      return msd_attn_decode_int8kv_spec(qp, kp, vp, ksp, vsp, cup, T, max_seqlen, B, q_len, Hq, Hkv, D, Dv, scale, op, lp, w.p, w.bytes, st);
    else
      return msd_attn_decode_int8kv(qp, kp, vp, ksp, vsp, cup, T, max_seqlen, B, Hq, Hkv, D, Dv, scale, op, lp, w.p, w.bytes, st);
  });
}

// (q, k, v or None, k_scale, v_scale or None, block_table, seqlens, page_size, max_seqlen, softmax_scale, Dv, ws, out, lse or None)
PyObject* attn_decode_int8kv_paged(PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  const at::Tensor *q = a.tensor(), *k = a.tensor(), *v = a.tensor(true), *ks = a.tensor(true), *vs = a.tensor(true), *table = a.tensor(),
                   *len = a.tensor(true);
  const int32_t page = static_cast<int32_t>(a.integer()), max_seqlen = static_cast<int32_t>(a.integer());
  const float scale = static_cast<float>(a.number());
  const int32_t Dv = static_cast<int32_t>(a.integer());
  const at::Tensor *ws = a.buffer(), *out = a.buffer(), *lse = a.buffer(true);
  if (!dims(a, {{q, 3}, {k, -2}, {table, -2}})) return nullptr;
  const Workspace w(ws);
  const int32_t B = static_cast<int32_t>(q->size(0)), Hq = static_cast<int32_t>(q->size(1)), D = static_cast<int32_t>(q->size(2));
  const int32_t Hkv = static_cast<int32_t>(k->size(1)), max_blocks = static_cast<int32_t>(table->size(1));
  const int64_t blocks = page > 0 ? k->size(0) / page : 0;      // (the library refuses other pages)
  void *qp = addr(q), *op = addr(out), *st = stream();
  const auto *kp = addr_as<int8_t>(k), *vp = addr_as<int8_t>(v);
  const auto *ksp = addr_as<float>(ks), *vsp = addr_as<float>(vs);
  const auto *tp = addr_as<int32_t>(table), *np = addr_as<int32_t>(len);
  auto *lp = addr_as<float>(lse);
  return status_of([&] {
    return msd_attn_decode_int8kv_paged(qp, kp, vp, ksp, vsp, tp, np, blocks, page, max_blocks, max_seqlen, B, Hq, Hkv, D, Dv, scale, op, lp,
                                        w.p, w.bytes, st);
  });
}

// What the interpreter calls: C++ exceptions (a tensor without storage or with another layout, no memory) become Python's.
template <PyObject* (*fn)(PyObject* const*, Py_ssize_t)>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  return fn(args, n);
  END_HANDLE_TH_ERRORS
}

template <PyObject* (*fn)(PyObject* const*, Py_ssize_t)>
PyMethodDef method(const char* name) {
  return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(entry<fn>)), METH_FASTCALL, nullptr};
}

PyMethodDef methods[] = {
    method<gemm_w8a16>("gemm_w8a16"), method<gemm_w4a16>("gemm_w4a16"), method<grouped_gemm_w8a16>("grouped_gemm_w8a16"),
    method<grouped_gemm_w4a16>("grouped_gemm_w4a16"), method<attn_decode<false>>("attn_decode_int8kv"),
    method<attn_decode<true>>("attn_decode_int8kv_spec"), method<attn_decode_int8kv_paged>("attn_decode_int8kv_paged"),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (build.py looks for it: a module built for another torch is built again)
extern "C" __attribute__((used, visibility("default"))) const char msd_call_module_built_for[] = MSD_BUILT_FOR;

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
