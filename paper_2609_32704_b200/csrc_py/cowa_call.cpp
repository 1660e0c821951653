// Native argument path of the Python binding: checks a call's tensors, fills in sizes, strides and the current stream
// and calls the C entry point.  The same steps in Python and ctypes take 10 to 20 us, more than a small call's kernels
// (one decode step over 8K of cache: 16.3 us to enqueue, 5.9 with this path; forward and backward at 1K 47, 18.8).
//
// Every function returns the C entry point's status, or None when it did not call it because something about the arguments
// is not plain (another type, a subclass, a wrong dtype or layout, a torch function mode): the caller then takes the Python
// path, which handles or refuses it.  So nothing is accepted or refused here that is not there.
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/version.h>

#include <climits>
#include <initializer_list>

#include "cowa.h"

namespace {

PyTypeObject* g_params = nullptr;  // binding.Params
decltype(&cowa_fwd) g_fwd;
decltype(&cowa_prefill) g_prefill;
decltype(&cowa_prefill_varlen) g_prefill_varlen;
decltype(&cowa_bwd) g_bwd;
decltype(&cowa_bwd_varlen) g_bwd_varlen;
decltype(&cowa_decode) g_decode;
decltype(&cowa_decode_multi) g_decode_multi;
decltype(&cowa_decode_paged) g_decode_paged;

enum Layout { kAnyStrides, kContiguous };

// A plain tensor of this dtype, layout and dimension count on a CUDA device, or nullptr.
const at::Tensor* tensor(PyObject* o, at::ScalarType type, Layout layout, int dim) {
  if (!THPVariable_CheckTypeExact(Py_TYPE(o))) return nullptr;
  const at::Tensor& x = THPVariable_Unpack(o);
  if (!x.defined() || !x.is_cuda() || x.scalar_type() != type || x.layout() != at::kStrided || !x.has_storage()) return nullptr;
  if (x.key_set().has(c10::DispatchKey::Python) || (dim >= 0 && x.dim() != dim)) return nullptr;
  for (int64_t n : x.sizes())
    if (n > INT_MAX) return nullptr;
  if (layout == kContiguous ? !x.is_contiguous() : x.dim() < 3 || !(x.stride(-1) == 1 || x.size(-1) == 1)) return nullptr;
  return &x;
}
const at::Tensor* bf16(PyObject* o, Layout layout, int dim) { return tensor(o, at::kBFloat16, layout, dim); }
const at::Tensor* f32(PyObject* o) { return tensor(o, at::kFloat, kContiguous, -1); }
const at::Tensor* i32(PyObject* o, int dim) { return tensor(o, at::kInt, kContiguous, dim); }

bool same_layout(const at::Tensor* a, const at::Tensor* b) { return a->sizes() == b->sizes() && a->strides() == b->strides(); }

struct Workspace {
  void* ptr = nullptr;
  size_t bytes = 0;
  bool set(PyObject* o) {
    if (!THPVariable_CheckTypeExact(Py_TYPE(o))) return false;
    const at::Tensor& x = THPVariable_Unpack(o);
    if (!x.defined() || !x.has_storage() || x.key_set().has(c10::DispatchKey::Python)) return false;
    ptr = x.data_ptr();
    bytes = (size_t)x.numel() * x.element_size();
    return true;
  }
};

// The caller's cowa_params_t, or a copy that holds the tensors' strides when one of them is not contiguous.
struct CallParams {
  Py_buffer view = {};
  cowa_params_t own;
  const cowa_params_t* p = nullptr;
  ~CallParams() { if (view.obj) PyBuffer_Release(&view); }
  bool set(PyObject* o) {
    if (Py_TYPE(o) != g_params) return false;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) { PyErr_Clear(); view.obj = nullptr; return false; }
    p = static_cast<const cowa_params_t*>(view.buf);
    return view.len == (Py_ssize_t)sizeof(cowa_params_t);
  }
  void strides(const at::Tensor* q, const at::Tensor* k, const at::Tensor* v, const at::Tensor* o) {
    bool all = true;
    for (const at::Tensor* t : {q, k, v, o}) all = all && (!t || t->is_contiguous());
    if (all) return;
    own = *p;
    p = &own;
    auto put = [](int64_t* s, const at::Tensor* t) {
      for (int i = 0; t && i < 3; ++i) s[i] = t->stride(i);
    };
    put(own.q_strides, q); put(own.k_strides, k); put(own.v_strides, v); put(own.o_strides, o);
  }
};

const at::Tensor* const kNone = nullptr;
int I(int64_t n) { return (int)n; }
template <class T>
T* at_ptr(const at::Tensor* t) { return t ? static_cast<T*>(t->data_ptr()) : nullptr; }

// Runs `call` without the GIL, as ctypes does.
template <class F>
PyObject* enqueue(F call) {
  void* st = c10::cuda::getCurrentCUDAStream().stream();
  struct Released {
    PyThreadState* s = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(s); }
  };
  int rc;
  {
    Released r;
    rc = call(st);
  }
  return PyLong_FromLong(rc);
}

#define COWA_PLAIN(cond) \
  if (!(cond)) Py_RETURN_NONE
#define COWA_ENTRY(name, nargs)                                                            \
  PyObject* name##_body(PyObject* const* x);                                               \
  PyObject* name(PyObject*, PyObject* const* x, Py_ssize_t n) {                            \
    if (n != nargs || at::impl::torch_function_mode_enabled()) Py_RETURN_NONE;             \
    try {                                                                                  \
      return name##_body(x);                                                               \
    } catch (...) {                                                                        \
      Py_RETURN_NONE; /* raised before the entry point ran: the Python path raises its own */ \
    }                                                                                      \
  }                                                                                        \
  PyObject* name##_body(PyObject* const* x)

PyObject* fwd_like(PyObject* const* x, bool prefill) {
  const at::Tensor *q = bf16(x[0], kAnyStrides, 4), *k = bf16(x[1], kAnyStrides, 4), *v = bf16(x[2], kAnyStrides, 4),
                   *o = bf16(x[3], kAnyStrides, 4), *lse = f32(x[4]);
  CallParams p;
  COWA_PLAIN(q && k && v && o && lse && p.set(x[5]));
  p.strides(q, k, v, o);
  const int B = I(q->size(0)), Hq = I(q->size(1)), Nq = I(q->size(2)), D = I(q->size(3)), Hkv = I(k->size(1)), Nk = I(k->size(2));
  void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr(), *op = o->data_ptr();
  float* lp = at_ptr<float>(lse);
  return enqueue([&](void* st) {
    return prefill ? g_prefill(qp, kp, vp, op, lp, B, Nq, Nk, Hq, Hkv, D, p.p, st)
                   : g_fwd(qp, kp, vp, op, lp, B, Nq, Hq, Hkv, D, p.p, st);
  });
}
COWA_ENTRY(fwd, 6) { return fwd_like(x, false); }
COWA_ENTRY(prefill, 6) { return fwd_like(x, true); }

COWA_ENTRY(prefill_varlen, 8) {
  const at::Tensor *q = bf16(x[0], kContiguous, 3), *k = bf16(x[1], kContiguous, 3), *v = bf16(x[2], kContiguous, 3),
                   *o = bf16(x[3], kContiguous, -1), *lse = f32(x[4]), *cq = i32(x[5], -1), *ck = i32(x[6], -1);
  CallParams p;
  COWA_PLAIN(q && k && v && o && lse && cq && ck && cq->numel() == ck->numel() && cq->numel() >= 2 && p.set(x[7]));
  const int B = I(cq->numel() - 1), Hq = I(q->size(0)), tq = I(q->size(1)), D = I(q->size(2)), Hkv = I(k->size(0)), tk = I(k->size(1));
  void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr(), *op = o->data_ptr();
  float* lp = at_ptr<float>(lse);
  const int32_t *cqp = at_ptr<int32_t>(cq), *ckp = at_ptr<int32_t>(ck);
  return enqueue([&](void* st) { return g_prefill_varlen(qp, kp, vp, op, lp, cqp, ckp, B, tq, tk, Hq, Hkv, D, p.p, st); });
}

COWA_ENTRY(bwd, 11) {
  const at::Tensor* t[9];
  for (int i = 0; i < 9; ++i) {
    t[i] = i == 4 ? f32(x[4]) : bf16(x[i], kAnyStrides, 4);
    COWA_PLAIN(t[i]);
  }
  CallParams p;
  Workspace ws;
  COWA_PLAIN(same_layout(t[5], t[3]) && same_layout(t[6], t[0]) && same_layout(t[7], t[1]) && same_layout(t[8], t[2]));
  COWA_PLAIN(p.set(x[9]) && ws.set(x[10]));
  p.strides(t[0], t[1], t[2], t[3]);
  const int B = I(t[0]->size(0)), Hq = I(t[0]->size(1)), T = I(t[0]->size(2)), D = I(t[0]->size(3)), Hkv = I(t[1]->size(1));
  void* a[9];
  for (int i = 0; i < 9; ++i) a[i] = t[i]->data_ptr();
  return enqueue([&](void* st) {
    return g_bwd(a[0], a[1], a[2], a[3], static_cast<float*>(a[4]), a[5], a[6], a[7], a[8], B, T, Hq, Hkv, D, p.p, ws.ptr, ws.bytes, st);
  });
}

COWA_ENTRY(bwd_varlen, 12) {
  const at::Tensor* t[9];
  for (int i = 0; i < 9; ++i) {
    t[i] = i == 4 ? f32(x[4]) : bf16(x[i], kContiguous, i < 2 ? 3 : -1);
    COWA_PLAIN(t[i]);
  }
  const at::Tensor* cu = i32(x[9], -1);
  CallParams p;
  Workspace ws;
  COWA_PLAIN(cu && p.set(x[10]) && ws.set(x[11]));
  const int B = I(cu->numel() - 1), Hq = I(t[0]->size(0)), total = I(t[0]->size(1)), D = I(t[0]->size(2)), Hkv = I(t[1]->size(0));
  void* a[9];
  for (int i = 0; i < 9; ++i) a[i] = t[i]->data_ptr();
  const int32_t* cup = at_ptr<int32_t>(cu);
  return enqueue([&](void* st) {
    return g_bwd_varlen(a[0], a[1], a[2], a[3], static_cast<float*>(a[4]), a[5], a[6], a[7], a[8], cup, B, total, Hq, Hkv, D, p.p,
                        ws.ptr, ws.bytes, st);
  });
}

COWA_ENTRY(decode, 8) {
  const at::Tensor *q = bf16(x[0], kContiguous, 3), *k = bf16(x[1], kAnyStrides, 4), *v = bf16(x[2], kAnyStrides, 4),
                   *lens = i32(x[3], -1), *o = bf16(x[4], kContiguous, -1), *lse = x[5] == Py_None ? kNone : f32(x[5]);
  CallParams p;
  Workspace ws;
  COWA_PLAIN(q && k && v && lens && o && (lse || x[5] == Py_None) && p.set(x[6]) && ws.set(x[7]));
  p.strides(nullptr, k, v, nullptr);
  const int B = I(q->size(0)), Hq = I(q->size(1)), D = I(q->size(2)), Hkv = I(k->size(1)), Tmax = I(k->size(2));
  void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr(), *op = o->data_ptr();
  const int32_t* np = at_ptr<int32_t>(lens);
  float* lp = at_ptr<float>(lse);
  return enqueue([&](void* st) { return g_decode(qp, kp, vp, np, op, lp, B, Tmax, Hq, Hkv, D, p.p, ws.ptr, ws.bytes, st); });
}

COWA_ENTRY(decode_multi, 8) {
  const at::Tensor *q = bf16(x[0], kContiguous, 4), *k = bf16(x[1], kContiguous, 4), *v = bf16(x[2], kContiguous, -1),
                   *lens = i32(x[3], -1), *o = bf16(x[4], kContiguous, -1), *lse = x[5] == Py_None ? kNone : f32(x[5]);
  CallParams p;
  Workspace ws;
  COWA_PLAIN(q && k && v && lens && o && (lse || x[5] == Py_None) && p.set(x[6]) && ws.set(x[7]));
  const int B = I(q->size(0)), Nq = I(q->size(1)), Hq = I(q->size(2)), D = I(q->size(3)), Hkv = I(k->size(1)), Tmax = I(k->size(2));
  void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr(), *op = o->data_ptr();
  const int32_t* np = at_ptr<int32_t>(lens);
  float* lp = at_ptr<float>(lse);
  return enqueue([&](void* st) { return g_decode_multi(qp, kp, vp, np, op, lp, B, Nq, Tmax, Hq, Hkv, D, p.p, ws.ptr, ws.bytes, st); });
}

COWA_ENTRY(decode_paged, 9) {
  const at::Tensor *q = bf16(x[0], kContiguous, 4), *k = bf16(x[1], kContiguous, 4), *v = bf16(x[2], kContiguous, -1),
                   *tab = i32(x[3], 2), *lens = i32(x[4], -1), *o = bf16(x[5], kContiguous, -1),
                   *lse = x[6] == Py_None ? kNone : f32(x[6]);
  CallParams p;
  Workspace ws;
  COWA_PLAIN(q && k && v && tab && lens && o && (lse || x[6] == Py_None) && p.set(x[7]) && ws.set(x[8]));
  const int B = I(q->size(0)), Nq = I(q->size(1)), Hq = I(q->size(2)), D = I(q->size(3)), Hkv = I(k->size(1)), page = I(k->size(2)),
            pages = I(tab->size(1));
  void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr(), *op = o->data_ptr();
  const int32_t *tp = at_ptr<int32_t>(tab), *np = at_ptr<int32_t>(lens);
  float* lp = at_ptr<float>(lse);
  return enqueue([&](void* st) {
    return g_decode_paged(qp, kp, vp, tp, np, op, lp, B, Nq, pages, page, Hq, Hkv, D, p.p, ws.ptr, ws.bytes, st);
  });
}

// bind(Params, [addresses of the entry points, in the order below])
PyObject* bind(PyObject*, PyObject* args) {
  PyObject *type, *list;
  if (!PyArg_ParseTuple(args, "O!O!", &PyType_Type, &type, &PyList_Type, &list)) return nullptr;
  void* fn[8];
  if (PyList_GET_SIZE(list) != 8) { PyErr_SetString(PyExc_ValueError, "eight addresses"); return nullptr; }
  for (int i = 0; i < 8; ++i) {
    fn[i] = PyLong_AsVoidPtr(PyList_GET_ITEM(list, i));
    if (!fn[i] && PyErr_Occurred()) return nullptr;
  }
  g_fwd = reinterpret_cast<decltype(g_fwd)>(fn[0]);
  g_prefill = reinterpret_cast<decltype(g_prefill)>(fn[1]);
  g_prefill_varlen = reinterpret_cast<decltype(g_prefill_varlen)>(fn[2]);
  g_bwd = reinterpret_cast<decltype(g_bwd)>(fn[3]);
  g_bwd_varlen = reinterpret_cast<decltype(g_bwd_varlen)>(fn[4]);
  g_decode = reinterpret_cast<decltype(g_decode)>(fn[5]);
  g_decode_multi = reinterpret_cast<decltype(g_decode_multi)>(fn[6]);
  g_decode_paged = reinterpret_cast<decltype(g_decode_paged)>(fn[7]);
  Py_INCREF(type);
  g_params = reinterpret_cast<PyTypeObject*>(type);
  Py_RETURN_NONE;
}

#define COWA_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {COWA_METHOD(fwd), COWA_METHOD(prefill), COWA_METHOD(prefill_varlen), COWA_METHOD(bwd), COWA_METHOD(bwd_varlen),
                         COWA_METHOD(decode), COWA_METHOD(decode_multi), COWA_METHOD(decode_paged),
                         {"bind", bind, METH_VARARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_cowa_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__cowa_call() {
  PyObject* m = PyModule_Create(&module);
  if (m) PyModule_AddStringConstant(m, "torch_version", TORCH_VERSION);  // built against; tensors of another one are not read
  return m;
}
