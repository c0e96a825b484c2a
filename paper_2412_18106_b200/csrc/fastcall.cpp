// Native form of the binding's per-step calls: checks the tensors' types, shapes and strides, picks
// their pointers and the current stream and calls the C entry points (addresses handed over by
// binding.py, which owns the library).  A Python call through ctypes costs 12 - 15 us of attribute
// lookups and conversions for `run`, as much as the kernels of a small batch; this takes about 1 us
// (two steps of a four-request batch, planned and run: 108 -> 43 us; two steps of 13 decode requests over
// eight layers 554 -> 387 us, which is the device's time).
// A call whose arguments do not pass returns None: the Python form then raises what is wrong.  So does one
// whose arguments throw when they are looked at (guarded); no C++ exception leaves an entry point.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <cstdint>
#include <new>
#include <vector>

#include "xy_attn.h"
#include "xy_gemm.h"

namespace {

decltype(&xy_attn_plan) f_plan = nullptr;
decltype(&xy_attn_run) f_run = nullptr;
decltype(&xy_attn_run_fp8kv) f_run_fp8 = nullptr;
decltype(&xy_attn_append_kv) f_append = nullptr;
decltype(&xy_gemm_run_ws) f_gemm = nullptr;

PyObject* none() { Py_RETURN_NONE; }

template <class F>
bool addr(PyObject* o, F& f) {
  f = reinterpret_cast<F>(PyLong_AsVoidPtr(o));
  return f != nullptr && !PyErr_Occurred();
}

// bind(plan, run, run_fp8kv, append_kv, gemm_run_ws): addresses of the C entry points
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 5 || !addr(a[0], f_plan) || !addr(a[1], f_run) || !addr(a[2], f_run_fp8) || !addr(a[3], f_append) ||
      !addr(a[4], f_gemm)) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "bind takes five function addresses");
    return nullptr;
  }
  return none();
}

template <class Body>
PyObject* guarded(Body body) {
  try {
    return body();
  } catch (const std::bad_alloc&) {
    return PyErr_NoMemory();
  } catch (...) {
    PyErr_Clear();  // (an exception of a Python tensor subclass is a set Python error too)
    return none();
  }
}

// A CUDA tensor of the given type and number of dimensions whose last one is contiguous.
const at::Tensor* cuda_tensor(PyObject* o, at::ScalarType type, int64_t dim) {
  if (!THPVariable_Check(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_cuda() || t.layout() != at::kStrided || t.scalar_type() != type || t.dim() != dim || t.stride(dim - 1) != 1) return nullptr;
  return &t;
}

// None: the current stream of the current device; else an integer handle.
bool stream_of(PyObject* o, void*& s) {
  if (o == Py_None) {
    s = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  s = PyLong_AsVoidPtr(o);
  return !PyErr_Occurred();
}

// Calls into the library without the GIL: `call` only passes on pointers and numbers that it holds.
template <class Call>
PyObject* status(Call call) {
  struct Unlocked {  // the lock is taken again on every way out
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
  };
  int rc;
  {
    Unlocked u;
    rc = call();
  }
  return PyLong_FromLong(rc);
}

struct Pools {
  const at::Tensor *k, *v, *bt;
};
bool pools(PyObject* k, PyObject* v, PyObject* bt, at::ScalarType type, Pools& p) {
  p.k = cuda_tensor(k, type, 4);
  p.v = cuda_tensor(v, type, 4);
  p.bt = cuda_tensor(bt, at::kInt, 2);
  return p.k && p.v && p.bt && p.k->strides() == p.v->strides();
}

// run(ctx, head_dim, q, k_pool, v_pool, block_table, sm_scale, o, lse, tree_mask, stream [, k_scale, v_scale])
PyObject* run(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 11 && n != 13) return none();
  const bool fp8 = n == 13;
  xy_attn_ctx* ctx = static_cast<xy_attn_ctx*>(PyLong_AsVoidPtr(a[0]));
  const int64_t D = PyLong_AsLongLong(a[1]);
  const double scale = PyFloat_AsDouble(a[6]);
  if (PyErr_Occurred()) return nullptr;
  Pools p;
  const at::Tensor* q = cuda_tensor(a[2], at::kBFloat16, 3);
  const at::Tensor* o = cuda_tensor(a[7], at::kBFloat16, 3);
  if (!q || !o || !pools(a[3], a[4], a[5], fp8 ? at::kByte : at::kBFloat16, p) || !THPVariable_Check(a[8])) return none();
  const at::Tensor& lse = THPVariable_Unpack(a[8]);
  if (!lse.is_cuda() || lse.layout() != at::kStrided || lse.scalar_type() != at::kFloat || !lse.is_contiguous()) return none();
  if (q->stride(1) != D || o->stride(1) != D) return none();
  const uint64_t* mask = nullptr;
  if (a[9] != Py_None) {
    if (!THPVariable_Check(a[9])) return none();
    mask = static_cast<const uint64_t*>(THPVariable_Unpack(a[9]).data_ptr());
  }
  void* s;
  if (!stream_of(a[10], s)) return nullptr;
  const at::Tensor &k = *p.k, &bt = *p.bt;
  const void *qp = q->data_ptr(), *kp = k.data_ptr(), *vp = p.v->data_ptr();
  void* op = o->data_ptr();
  auto* lp = static_cast<float*>(lse.data_ptr());
  auto* btp = static_cast<const int32_t*>(bt.data_ptr());
  const int64_t qs = q->stride(0), os = o->stride(0), pages = k.size(0), ps = k.stride(0), hs = k.stride(1), ts = k.stride(2);
  const auto bts = static_cast<int32_t>(bt.stride(0));
  const auto sc = static_cast<float>(scale);
  if (!fp8) return status([=] { return f_run(ctx, qp, qs, kp, vp, pages, ps, hs, ts, btp, bts, mask, sc, op, os, lp, s); });
  const at::Tensor *ks = cuda_tensor(a[11], at::kFloat, 2), *vs = cuda_tensor(a[12], at::kFloat, 2);
  if (!ks || !vs || !ks->is_contiguous() || !vs->is_contiguous() || ks->sizes() != vs->sizes() || ks->size(0) != k.size(0) ||
      ks->size(1) != k.size(1))
    return none();
  auto *ksp = static_cast<const float*>(ks->data_ptr()), *vsp = static_cast<const float*>(vs->data_ptr());
  return status([=] { return f_run_fp8(ctx, qp, qs, kp, vp, ksp, vsp, pages, ps, hs, ts, btp, bts, mask, sc, op, os, lp, s); });
}

// append_kv(ctx, head_dim, qkv, k_pool, v_pool, block_table, stream)
PyObject* append_kv(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 7) return none();
  xy_attn_ctx* ctx = static_cast<xy_attn_ctx*>(PyLong_AsVoidPtr(a[0]));
  const int64_t D = PyLong_AsLongLong(a[1]);
  if (PyErr_Occurred()) return nullptr;
  Pools p;
  const at::Tensor* qkv = cuda_tensor(a[2], at::kBFloat16, 3);
  if (!qkv || qkv->stride(1) != D || !pools(a[3], a[4], a[5], at::kBFloat16, p)) return none();
  void* s;
  if (!stream_of(a[6], s)) return nullptr;
  const void* src = qkv->data_ptr();
  void *kp = p.k->data_ptr(), *vp = p.v->data_ptr();
  auto* btp = static_cast<const int32_t*>(p.bt->data_ptr());
  const int64_t ss = qkv->stride(0), pages = p.k->size(0), ps = p.k->stride(0), hs = p.k->stride(1), ts = p.k->stride(2);
  const auto bts = static_cast<int32_t>(p.bt->stride(0));
  return status([=] { return f_append(ctx, src, ss, kp, vp, pages, ps, hs, ts, btp, bts, s); });
}

// gemm(a, w, c, tile_n, stream, workspace)
PyObject* gemm(PyObject*, PyObject* const* x, Py_ssize_t n) {
  if (n != 6) return none();
  const at::Tensor *a = cuda_tensor(x[0], at::kBFloat16, 2), *w = cuda_tensor(x[1], at::kBFloat16, 2),
                   *c = cuda_tensor(x[2], at::kBFloat16, 2);
  const long tile_n = PyLong_AsLong(x[3]);
  if (PyErr_Occurred()) return nullptr;
  if (!a || !w || !c) return none();
  const int64_t M = a->size(0), K = a->size(1), N = w->size(0);
  if (w->size(1) != K || c->size(0) != M || c->size(1) != N || M > INT32_MAX || N > INT32_MAX || K > INT32_MAX) return none();
  void* ws = nullptr;
  int64_t ws_bytes = 0;
  if (x[5] != Py_None) {
    const at::Tensor* t = cuda_tensor(x[5], at::kByte, 1);
    if (!t) return none();
    ws = t->data_ptr();
    ws_bytes = t->numel();
  }
  void* s;
  if (!stream_of(x[4], s)) return nullptr;
  // the row stride of a single row says nothing
  const int64_t lda = M > 1 ? a->stride(0) : std::max(K, a->stride(0)), ldc = M > 1 ? c->stride(0) : std::max(N, c->stride(0));
  const void *ap = a->data_ptr(), *wp = w->data_ptr();
  void* cp = c->data_ptr();
  const int64_t ldw = w->stride(0);
  const auto m32 = static_cast<int32_t>(M), n32 = static_cast<int32_t>(N), k32 = static_cast<int32_t>(K),
             tn = static_cast<int32_t>(tile_n);
  return status([=] { return f_gemm(ap, lda, wp, ldw, cp, ldc, m32, n32, k32, tn, ws, ws_bytes, s); });
}

// Contiguous one-dimensional int32 buffer (a numpy array).
struct Ints {
  Py_buffer b{};
  bool held = false;
  bool take(PyObject* o) {
    if (!PyObject_CheckBuffer(o)) return false;
    if (PyObject_GetBuffer(o, &b, PyBUF_FORMAT | PyBUF_ND | PyBUF_C_CONTIGUOUS) != 0) {
      PyErr_Clear();
      return false;
    }
    held = true;
    return b.ndim == 1 && b.itemsize == 4 && b.format != nullptr && b.format[0] == 'i' && b.format[1] == 0;
  }
  const int32_t* data() const { return static_cast<const int32_t*>(b.buf); }
  Py_ssize_t size() const { return b.shape[0]; }
  ~Ints() {
    if (held) PyBuffer_Release(&b);
  }
};

// plan(ctx, q_len, kv_len, mask_kind, parent_off, parents, stream, address of the plan info)
PyObject* plan(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 8) return none();
  xy_attn_ctx* ctx = static_cast<xy_attn_ctx*>(PyLong_AsVoidPtr(a[0]));
  auto* info = static_cast<xy_attn_plan_info*>(PyLong_AsVoidPtr(a[7]));
  if (PyErr_Occurred()) return nullptr;
  Ints q, kv, kind, off, par;
  if (!q.take(a[1]) || !kv.take(a[2]) || !kind.take(a[3]) || !off.take(a[4])) return none();
  const bool trees = a[5] != Py_None;
  if (trees && !par.take(a[5])) return none();
  const Py_ssize_t R = q.size();
  if (kv.size() != R || kind.size() != R || off.size() != R || R > INT32_MAX) return none();
  void* s;
  if (!stream_of(a[6], s)) return nullptr;
  const int32_t np = trees ? static_cast<int32_t>(par.size()) : 0;
  std::vector<xy_attn_request> reqs(static_cast<size_t>(R > 0 ? R : 1));
  for (Py_ssize_t r = 0; r < R; ++r) reqs[r] = xy_attn_request{q.data()[r], kv.data()[r], kind.data()[r], off.data()[r]};
  const int32_t* parents = np > 0 ? par.data() : nullptr;
  return status([&] { return f_plan(ctx, reqs.data(), static_cast<int32_t>(R), parents, np, s, info); });
}

// the entry points: a body behind guarded()
template <PyObject* (*body)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* entry(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  return guarded([&] { return body(self, a, n); });
}

PyMethodDef methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<bind>)), METH_FASTCALL, nullptr},
    {"plan", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<plan>)), METH_FASTCALL, nullptr},
    {"run", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<run>)), METH_FASTCALL, nullptr},
    {"append_kv", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<append_kv>)), METH_FASTCALL, nullptr},
    {"gemm", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<gemm>)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() { return PyModule_Create(&module); }
