// Python extension module _step: the calls that a model makes per layer and token (and a prefill), from tensors to the C
// entry points.  The same checks as binding.py makes, without the interpreter between them: through ctypes a call's
// checks and argument conversions took 2 to 3 us of its 6 (append, decode, one after the other), more than the kernels of a
// short context take.  Whatever does not pass the checks (a subclass, another device, a stream that was given) is left to
// binding.py's general forms, which accept or refuse it.  Nothing is remembered from call to call; the GIL is released
// around the library's calls, as ctypes does.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

constexpr long kNotHandled = 1;      // status of a call that binding.py has to make (the library's are 0 and below)

using Fn3 = int (*)(void*, const void*, const void*, void*);                                         // append
using FnDecode = int (*)(void*, const void*, void*, void*);
using FnPrefill = int (*)(void*, const void*, const void*, int32_t, void*);
using FnHost = int (*)(void*, const void*, const void*, const void*, void*, void*, void*);

struct Steps {
  PyObject_HEAD
  void* handle;
  int device;
  int64_t kv[3], q[3];
  Fn3 append;
  FnDecode decode;
  FnPrefill prefill;
  FnHost host;
};

// The tensor behind a plain torch.Tensor of fp16 values, else null.
const at::Tensor* plain_half(PyObject* o) {
  if (Py_TYPE(o) != reinterpret_cast<PyTypeObject*>(THPVariableClass)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.defined() && t.scalar_type() == at::kHalf && t.layout() == at::kStrided ? &t : nullptr;
}
bool is_shape(const at::Tensor& t, const int64_t* shape) { return t.sizes().equals(c10::IntArrayRef(shape, 3)) && t.is_contiguous(); }

void* device_ptr(const Steps* s, PyObject* o, const int64_t* shape) {
  const at::Tensor* t = plain_half(o);
  if (!t || !t->is_cuda() || t->get_device() != s->device || !is_shape(*t, shape)) return nullptr;
  return t->data_ptr();
}
void* host_ptr(PyObject* o, const int64_t* shape) {
  const at::Tensor* t = plain_half(o);
  if (!t || !t->is_cpu() || !is_shape(*t, shape)) return nullptr;
  return t->data_ptr();
}
bool current(const Steps* s) { return c10::cuda::current_device() == s->device; }
void* stream_of(const Steps* s) { return c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)s->device).stream(); }

// f's status; exceptions (of its checks: a tensor without storage, say) leave the call to binding.py
template <typename F> PyObject* guarded(F f) {
  long st = kNotHandled;
  try {
    st = f();
  } catch (...) {
    PyErr_Clear();
    st = kNotHandled;
  }
  return PyLong_FromLong(st);
}
// f's status with the GIL released; it is held again whether f returns or throws
template <typename F> long without_gil(F f) {
  struct Released {
    PyThreadState* state = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(state); }
  } released;
  return f();
}

PyObject* steps_append(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  const Steps* s = reinterpret_cast<Steps*>(self);
  return guarded([&]() -> long {
    if (n != 2 || !current(s)) return kNotHandled;
    const void *k = device_ptr(s, a[0], s->kv), *v = device_ptr(s, a[1], s->kv);
    if (!k || !v) return kNotHandled;
    void* st = stream_of(s);
    return without_gil([&] { return s->append(s->handle, k, v, st); });
  });
}

PyObject* steps_prefill(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  const Steps* s = reinterpret_cast<Steps*>(self);
  return guarded([&]() -> long {
    if (n != 2 || !current(s)) return kNotHandled;
    const at::Tensor *k = plain_half(a[0]), *v = plain_half(a[1]);
    if (!k || !v || k->dim() != 4 || k->size(2) <= 0 || k->size(2) > INT32_MAX) return kNotHandled;
    const int64_t shape[4] = {s->kv[0], s->kv[1], k->size(2), s->kv[2]};
    for (const at::Tensor* t : {k, v})
      if (!t->is_cuda() || t->get_device() != s->device || !t->sizes().equals(c10::IntArrayRef(shape, 4)) || !t->is_contiguous())
        return kNotHandled;
    const void *kp = k->data_ptr(), *vp = v->data_ptr();
    void* st = stream_of(s);
    return without_gil([&] { return s->prefill(s->handle, kp, vp, (int32_t)shape[2], st); });
  });
}

// decode(q, out or None): the result, or a status
PyObject* steps_decode(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  const Steps* s = reinterpret_cast<Steps*>(self);
  PyObject* result = nullptr;
  PyObject* status = guarded([&]() -> long {
    if (n != 2 || !current(s)) return kNotHandled;
    const void* q = device_ptr(s, a[0], s->q);
    if (!q) return kNotHandled;
    at::Tensor fresh;
    void* out;
    if (a[1] == Py_None) {
      fresh = at::empty(c10::IntArrayRef(s->q, 3), at::TensorOptions().dtype(at::kHalf).device(at::kCUDA, (c10::DeviceIndex)s->device));
      out = fresh.data_ptr();
    } else {
      out = device_ptr(s, a[1], s->q);
      if (!out) return kNotHandled;
    }
    void* st = stream_of(s);
    const long r = without_gil([&] { return s->decode(s->handle, q, out, st); });
    if (r == 0) {
      if (a[1] == Py_None) result = THPVariable_Wrap(fresh);
      else { result = a[1]; Py_INCREF(result); }
    }
    return r;
  });
  if (!result) return status;
  Py_DECREF(status);
  return result;
}

// step_host(k, v, q, out, address of the staging buffer)
PyObject* steps_host(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  const Steps* s = reinterpret_cast<Steps*>(self);
  return guarded([&]() -> long {
    if (n != 5 || !current(s)) return kNotHandled;
    const void *k = host_ptr(a[0], s->kv), *v = host_ptr(a[1], s->kv), *q = host_ptr(a[2], s->q);
    void *out = host_ptr(a[3], s->q), *staging = PyLong_AsVoidPtr(a[4]);
    if (!k || !v || !q || !out || !staging) { PyErr_Clear(); return kNotHandled; }
    void* st = stream_of(s);
    return without_gil([&] { return s->host(s->handle, k, v, q, out, staging, st); });
  });
}

// Steps(handle, device, kv shape, q shape, addresses of the four entry points)
int steps_init(PyObject* self, PyObject* args, PyObject*) {
  Steps* s = reinterpret_cast<Steps*>(self);
  unsigned long long h, fa, fd, fp, fh;
  long long kv[3], q[3];
  if (!PyArg_ParseTuple(args, "Ki(LLL)(LLL)KKKK", &h, &s->device, &kv[0], &kv[1], &kv[2], &q[0], &q[1], &q[2], &fa, &fd, &fp, &fh)) return -1;
  for (int i = 0; i < 3; ++i) { s->kv[i] = kv[i]; s->q[i] = q[i]; }
  s->handle = reinterpret_cast<void*>(h);
  s->append = reinterpret_cast<Fn3>(fa);
  s->decode = reinterpret_cast<FnDecode>(fd);
  s->prefill = reinterpret_cast<FnPrefill>(fp);
  s->host = reinterpret_cast<FnHost>(fh);
  return 0;
}

template <typename F> PyCFunction as_method(F f) { return reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(f)); }
PyMethodDef steps_methods[] = {{"append", as_method(steps_append), METH_FASTCALL, nullptr},
                               {"decode", as_method(steps_decode), METH_FASTCALL, nullptr},
                               {"prefill", as_method(steps_prefill), METH_FASTCALL, nullptr},
                               {"step_host", as_method(steps_host), METH_FASTCALL, nullptr},
                               {nullptr, nullptr, 0, nullptr}};
PyTypeObject steps_type = {PyVarObject_HEAD_INIT(nullptr, 0)};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_step", nullptr, -1, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__step() {
  steps_type.tp_name = "_step.Steps";
  steps_type.tp_basicsize = sizeof(Steps);
  steps_type.tp_flags = Py_TPFLAGS_DEFAULT;
  steps_type.tp_new = PyType_GenericNew;
  steps_type.tp_init = steps_init;
  steps_type.tp_methods = steps_methods;
  if (PyType_Ready(&steps_type) < 0) return nullptr;
  PyObject* m = PyModule_Create(&module_def);
  if (!m) return nullptr;
  Py_INCREF(&steps_type);
  if (PyModule_AddObject(m, "Steps", reinterpret_cast<PyObject*>(&steps_type)) < 0) return nullptr;
  return m;
}
