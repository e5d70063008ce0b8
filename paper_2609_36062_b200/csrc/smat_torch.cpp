// Python entry points of the passes as a native extension: argument checks, output allocation, the current stream and
// the call into libsmat, for the methods of binding.SmatPlan.  It holds no state besides the plan handle and shape it
// is given; the Python form of the same checks (attribute look-ups, shape tuples, ctypes conversions) cost about 8 us a
// decoding step and 25 us a forward + backward, more than the kernels of a small problem.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>
#include <initializer_list>
#include <string>

#include "../../include/smat.h"

namespace {

struct Plan {
  PyObject_HEAD
  const smat_plan* handle;
  int64_t b, h, T, dk, dv, n, m;
  at::ScalarType dtype;
};

PyObject* smat_error = nullptr;   // binding.SmatError

bool fail_status(int code, const char* what) {
  if (code == SMAT_OK) return true;
  PyObject* e = PyObject_CallFunction(smat_error, "is", code, what);
  if (e) {
    PyErr_SetObject(smat_error, e);
    Py_DECREF(e);
  }
  return false;
}

std::string shape_text(at::IntArrayRef s) {
  std::string t = "(";
  for (size_t i = 0; i < s.size(); ++i) t += (i ? ", " : "") + std::to_string(s[i]);
  return t + ")";
}

// The tensor behind `o`, checked: CUDA, dtype, contiguous, exactly this shape.
const at::Tensor* tensor(PyObject* o, const char* name, at::ScalarType dtype, at::IntArrayRef shape) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_ValueError, "%s: expected a tensor", name);
    return nullptr;
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_cuda()) {
    PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor", name);
    return nullptr;
  }
  if (t.scalar_type() != dtype || t.sizes() != shape || !t.is_contiguous()) {
    PyErr_Format(PyExc_ValueError, "%s: expected a contiguous CUDA tensor of %s and shape %s, got %s %s", name,
                 c10::toString(dtype), shape_text(shape).c_str(), c10::toString(t.scalar_type()),
                 shape_text(t.sizes()).c_str());
    return nullptr;
  }
  return &t;
}

bool workspace(PyObject* o, const char* name, void** ptr, size_t* bytes) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_ValueError, "%s: expected a tensor", name);
    return false;
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  *ptr = t.data_ptr();
  *bytes = (size_t)t.numel();
  return true;
}

bool stream(PyObject* o, void** st) {
  if (o == Py_None) {
    *st = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
  if (!v) return false;
  *st = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

// The interpreter lock is released for a call into the library (a full launch queue may block it).  The library throws
// nothing; what can throw, the data pointers of tensors without storage among it, is asked for before.
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};
template <typename F>
int unlocked(F call) {
  Unlocked lock;
  return call();
}

// Anything int() takes (a position kept as a float or as an array scalar among it).
bool token_index(PyObject* o, long long* t) {
  if (PyLong_CheckExact(o)) {
    *t = PyLong_AsLongLong(o);
    return !(*t == -1 && PyErr_Occurred());
  }
  PyObject* n = PyNumber_Long(o);
  if (!n) return false;
  *t = PyLong_AsLongLong(n);
  Py_DECREF(n);
  return !(*t == -1 && PyErr_Occurred());
}

bool arity(Py_ssize_t got, Py_ssize_t want, const char* name) {
  if (got == want) return true;
  PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, got %zd", name, want, got);
  return false;
}

// An output: the caller's tensor, or a new one like `like`.  A tensor handed in has the same element type, is contiguous
// and holds at least as many elements: another view of the same rows, or a larger buffer whose first part is written.
bool output(PyObject* o, const char* name, const at::Tensor& like, at::Tensor* out) {
  if (o == Py_None) {
    *out = at::empty_like(like);
    return true;
  }
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.is_cuda() && t.scalar_type() == like.scalar_type() && t.numel() >= like.numel() && t.is_contiguous()) {
      *out = t;
      return true;
    }
  }
  PyErr_Format(PyExc_ValueError, "%s: expected a contiguous CUDA tensor of %s that holds shape %s", name,
               c10::toString(like.scalar_type()), shape_text(like.sizes()).c_str());
  return false;
}

PyObject* wrap(const at::Tensor& t) { return THPVariable_Wrap(t); }

PyObject* wrap_all(std::initializer_list<at::Tensor> ts) {
  PyObject* tuple = PyTuple_New((Py_ssize_t)ts.size());
  if (!tuple) return nullptr;
  Py_ssize_t i = 0;
  for (const at::Tensor& t : ts) PyTuple_SET_ITEM(tuple, i++, wrap(t));
  return tuple;
}

// The exception in flight as the one torch raises for it (an exhausted device: torch.OutOfMemoryError).
PyObject* raise() {
  torch::translate_exception_to_python(std::current_exception());
  return nullptr;
}

// forward(kind, Q, K, V, log_a, O, workspace, stream, prof, type): kind 0 plain or routed, 1 gated, 2 normalised
PyObject* plan_forward(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  try {
    if (!arity(n, 10, "forward")) return nullptr;
    const Plan& p = *reinterpret_cast<Plan*>(self);
    const long kind = PyLong_AsLong(a[0]);
    const int64_t sk[4] = {p.b, p.h, p.T, p.dk}, sv[4] = {p.b, p.h, p.T, p.dv};
    const at::Tensor *Q = tensor(a[1], "Q", p.dtype, sk), *K = Q ? tensor(a[2], "K", p.dtype, sk) : nullptr;
    const at::Tensor* V = K ? tensor(a[3], "V", p.dtype, sv) : nullptr;
    if (!V) return nullptr;
    const int64_t sg[2] = {p.b * p.h, p.T};
    const at::Tensor* la = kind == 1 ? tensor(a[4], "log_a", at::kFloat, sg) : nullptr;
    if (kind == 1 && !la) return nullptr;
    at::Tensor O;
    void *ws, *st;
    size_t bytes;
    if (kind == 0 && a[5] != Py_None && !tensor(a[5], "O", p.dtype, sv)) return nullptr;
    if (!output(a[5], "O", *V, &O) || !workspace(a[6], "workspace", &ws, &bytes) || !stream(a[7], &st)) return nullptr;
    const void *q = Q->data_ptr(), *k = K->data_ptr(), *v = V->data_ptr();
    void* o = O.data_ptr();
    int rc;
    const char* what;
    if (kind == 1) {
      what = "smat_forward_gated";
      const float* log_a = la->data_ptr<float>();
      rc = unlocked([&] { return smat_forward_gated(p.handle, q, k, v, log_a, o, ws, bytes, st); });
    } else if (kind == 2) {
      what = "smat_forward_normalized";
      rc = unlocked([&] { return smat_forward_normalized(p.handle, q, k, v, o, ws, bytes, st); });
    } else if (a[8] != Py_None || a[9] != Py_None) {
      const int64_t sp[2] = {p.b * p.h, p.n}, stp[2] = {p.b * p.h, p.m};
      const at::Tensor *prof = tensor(a[8], "prof", at::kInt, sp), *type = prof ? tensor(a[9], "type", at::kInt, stp) : nullptr;
      if (!type) return nullptr;
      what = "smat_forward_routed";
      const int32_t *cells = prof->data_ptr<int>(), *types = type->data_ptr<int>();
      rc = unlocked([&] { return smat_forward_routed(p.handle, q, k, v, o, cells, types, ws, bytes, st); });
    } else {
      what = "smat_forward";
      rc = unlocked([&] { return smat_forward(p.handle, q, k, v, o, ws, bytes, st); });
    }
    return fail_status(rc, what) ? wrap(O) : nullptr;
  } catch (...) {
    return raise();
  }
}

// backward(kind, Q, K, V, log_a, O, dO, dQ, dK, dV, dlog_a, workspace, stream, prof, type)
PyObject* plan_backward(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  try {
    if (!arity(n, 15, "backward")) return nullptr;
    const Plan& p = *reinterpret_cast<Plan*>(self);
    const long kind = PyLong_AsLong(a[0]);
    const int64_t sk[4] = {p.b, p.h, p.T, p.dk}, sv[4] = {p.b, p.h, p.T, p.dv};
    const at::Tensor *Q = tensor(a[1], "Q", p.dtype, sk), *K = Q ? tensor(a[2], "K", p.dtype, sk) : nullptr;
    const at::Tensor* V = K ? tensor(a[3], "V", p.dtype, sv) : nullptr;
    const at::Tensor* O = V && kind == 2 ? tensor(a[5], "O", p.dtype, sv) : V;
    const at::Tensor* dO = O ? tensor(a[6], "dO", p.dtype, sv) : nullptr;
    if (!dO) return nullptr;
    const int64_t sg[2] = {p.b * p.h, p.T};
    const at::Tensor* la = kind == 1 ? tensor(a[4], "log_a", at::kFloat, sg) : nullptr;
    if (kind == 1 && !la) return nullptr;
    at::Tensor dQ, dK, dV, dla;
    void *ws, *st;
    size_t bytes;
    if (!output(a[7], "dQ", *Q, &dQ) || !output(a[8], "dK", *K, &dK) || !output(a[9], "dV", *V, &dV) ||
        (la && !output(a[10], "dlog_a", *la, &dla)) || !workspace(a[11], "workspace", &ws, &bytes) || !stream(a[12], &st))
      return nullptr;
    const void *q = Q->data_ptr(), *k = K->data_ptr(), *v = V->data_ptr(), *go = dO->data_ptr();
    void *gq = dQ.data_ptr(), *gk = dK.data_ptr(), *gv = dV.data_ptr();
    int rc;
    const char* what;
    if (kind == 1) {
      what = "smat_backward_gated";
      const float* log_a = la->data_ptr<float>();
      float* glog_a = dla.data_ptr<float>();
      rc = unlocked([&] { return smat_backward_gated(p.handle, q, k, v, log_a, go, gq, gk, gv, glog_a, ws, bytes, st); });
    } else if (kind == 2) {
      what = "smat_backward_normalized";
      const void* o = O->data_ptr();
      rc = unlocked([&] { return smat_backward_normalized(p.handle, q, k, v, o, go, gq, gk, gv, ws, bytes, st); });
    } else if (a[13] != Py_None || a[14] != Py_None) {
      const int64_t sp[2] = {p.b * p.h, p.n}, stp[2] = {p.b * p.h, p.m};
      const at::Tensor *prof = tensor(a[13], "prof", at::kInt, sp), *type = prof ? tensor(a[14], "type", at::kInt, stp) : nullptr;
      if (!type) return nullptr;
      what = "smat_backward_routed";
      const int32_t *cells = prof->data_ptr<int>(), *types = type->data_ptr<int>();
      rc = unlocked([&] { return smat_backward_routed(p.handle, q, k, v, go, gq, gk, gv, cells, types, ws, bytes, st); });
    } else {
      what = "smat_backward";
      rc = unlocked([&] { return smat_backward(p.handle, q, k, v, go, gq, gk, gv, ws, bytes, st); });
    }
    if (!fail_status(rc, what)) return nullptr;
    return la ? wrap_all({dQ, dK, dV, dla}) : wrap_all({dQ, dK, dV});
  } catch (...) {
    return raise();
  }
}

// decode_step(q, k, v, log_a_t, t, cache, o, stream): log_a_t None for the ungated step
PyObject* plan_decode_step(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  try {
    if (!arity(n, 8, "decode_step")) return nullptr;
    const Plan& p = *reinterpret_cast<Plan*>(self);
    const int64_t sk[3] = {p.b, p.h, p.dk}, sv[3] = {p.b, p.h, p.dv};
    const at::Tensor *q = tensor(a[0], "q", p.dtype, sk), *k = q ? tensor(a[1], "k", p.dtype, sk) : nullptr;
    const at::Tensor* v = k ? tensor(a[2], "v", p.dtype, sv) : nullptr;
    if (!v) return nullptr;
    const at::Tensor* la = nullptr;
    if (a[3] != Py_None) {
      if (!THPVariable_Check(a[3])) {
        PyErr_SetString(PyExc_ValueError, "log_a_t: expected a tensor");
        return nullptr;
      }
      la = &THPVariable_Unpack(a[3]);
      if (!la->is_cuda() || !la->is_contiguous() || la->scalar_type() != at::kFloat || la->numel() != p.b * p.h) {
        PyErr_Format(PyExc_ValueError, "log_a_t: expected a contiguous CUDA fp32 tensor of %lld log-gates", (long long)(p.b * p.h));
        return nullptr;
      }
    }
    long long t;
    if (!token_index(a[4], &t)) return nullptr;
    at::Tensor o;
    void *cache, *st;
    size_t bytes;
    if (!workspace(a[5], "cache", &cache, &bytes) || !output(a[6], "o", *v, &o) || !stream(a[7], &st)) return nullptr;
    const void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr();
    void* op = o.data_ptr();
    const float* log_a = la ? la->data_ptr<float>() : nullptr;
    const int rc = unlocked([&] {
      return la ? smat_decode_step_gated(p.handle, qp, kp, vp, log_a, t, op, cache, bytes, st)
                : smat_decode_step(p.handle, qp, kp, vp, t, op, cache, bytes, st);
    });
    return fail_status(rc, la ? "smat_decode_step_gated" : "smat_decode_step") ? wrap(o) : nullptr;
  } catch (...) {
    return raise();
  }
}

// Plan(handle, batch, heads, T, d_k, d_v, bf16)
PyObject* plan_new(PyTypeObject* type, PyObject* args, PyObject*) {
  unsigned long long handle;
  long long b, h, T, dk, dv;
  int bf16;
  if (!PyArg_ParseTuple(args, "KLLLLLi", &handle, &b, &h, &T, &dk, &dv, &bf16)) return nullptr;
  smat_geometry g;
  const smat_plan* plan = reinterpret_cast<const smat_plan*>(handle);
  if (!fail_status(smat_get_geometry(plan, &g), "smat_get_geometry")) return nullptr;
  Plan* p = reinterpret_cast<Plan*>(type->tp_alloc(type, 0));
  if (!p) return nullptr;
  p->handle = plan;
  p->b = b; p->h = h; p->T = T; p->dk = dk; p->dv = dv; p->n = g.n; p->m = g.m;
  p->dtype = bf16 ? at::kBFloat16 : at::kFloat;
  return reinterpret_cast<PyObject*>(p);
}

PyMethodDef plan_methods[] = {
    {"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(plan_forward)), METH_FASTCALL, nullptr},
    {"backward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(plan_backward)), METH_FASTCALL, nullptr},
    {"decode_step", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(plan_decode_step)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyTypeObject plan_type = {PyVarObject_HEAD_INIT(nullptr, 0)};

PyObject* set_error(PyObject*, PyObject* cls) {
  Py_INCREF(cls);
  Py_XSETREF(smat_error, cls);
  Py_RETURN_NONE;
}

PyMethodDef module_methods[] = {{"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_smat_torch", nullptr, -1, module_methods};

}  // namespace

PyMODINIT_FUNC PyInit__smat_torch(void) {
  plan_type.tp_name = "_smat_torch.Plan";
  plan_type.tp_basicsize = sizeof(Plan);
  plan_type.tp_flags = Py_TPFLAGS_DEFAULT;
  plan_type.tp_new = plan_new;
  plan_type.tp_methods = plan_methods;
  if (PyType_Ready(&plan_type) < 0) return nullptr;
  PyObject* m = PyModule_Create(&module_def);
  if (!m) return nullptr;
  Py_INCREF(&plan_type);
  if (PyModule_AddObject(m, "Plan", reinterpret_cast<PyObject*>(&plan_type)) < 0) {
    Py_DECREF(&plan_type);
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
