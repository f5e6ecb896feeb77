// The calls of the token loop, as a CPython extension: tensor checks, output allocation, the current stream and the call
// itself in native code.  What bounds a small cache or a block-by-block loop is how fast the host issues: the same steps in
// Python over ctypes took longer than the launch itself (issue of one block append + attention: 22 us, 10.6 us here; of a decode
// step of one block: 22 us, 12 us here).  Rarer calls stay on ctypes.
// Every function does what its Python twin in binding.py documents; the library call runs without the interpreter lock.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/Functions.h>
#include <c10/cuda/CUDAStream.h>

#include "../../include/pmkvq.h"

namespace {

// what this was compiled against, read by build.py from the file
__attribute__((used)) const char kBuiltFor[] = HOST_FOR;

PyObject *g_error = nullptr;     // PmkvqError(status, what)
PyObject *g_stream_attr = nullptr;  // "cuda_stream"

PyObject *fail(pmkvq_status st, const char *what) {
  if (PyObject *e = PyObject_CallFunction(g_error, "is", (int)st, what)) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  return nullptr;
}
PyObject *value_error(const char *what) {
  PyErr_SetString(PyExc_ValueError, what);
  return nullptr;
}

bool int_arg(PyObject *o, int64_t &v) {  // any integer; the library checks the range
  PyObject *i = PyNumber_Index(o);
  if (!i) return false;
  v = (int64_t)PyLong_AsUnsignedLongLongMask(i);
  Py_DECREF(i);
  return !(v == -1 && PyErr_Occurred());
}
bool handle_arg(PyObject *o, pmkvq_cache *&h) {
  int64_t v = 0;
  if (!int_arg(o, v)) return false;
  h = reinterpret_cast<pmkvq_cache *>(v);
  return true;
}
// a stream object, or None for the current stream of the current device
bool stream_arg(PyObject *o, void *&st) {
  if (o == Py_None) {
    st = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  PyObject *p = PyObject_GetAttr(o, g_stream_attr);
  int64_t v = 0;
  const bool ok = p && int_arg(p, v);
  Py_XDECREF(p);
  st = reinterpret_cast<void *>(v);
  return ok;
}
const at::Tensor *tensor_arg(PyObject *o, at::ScalarType dtype, const char *what) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s must be a tensor", what);
    return nullptr;
  }
  const at::Tensor &t = THPVariable_Unpack(o);
  if (!t.is_cuda() || !t.is_contiguous() || t.scalar_type() != dtype) {
    PyErr_Format(PyExc_ValueError, "%s must be a contiguous CUDA tensor of torch.%s", what, dtype == at::kFloat ? "float32" : "bfloat16");
    return nullptr;
  }
  return &t;
}
bool arg_count(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "%zd arguments, %zd wanted", n, want);
  return false;
}

// (handle, layer, k, v, numbers of one token's K, stream) -> status
PyObject *append(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  pmkvq_cache *h;
  void *st;
  int64_t layer, token;
  if (!arg_count(n, 6) || !handle_arg(a[0], h) || !int_arg(a[1], layer) || !int_arg(a[4], token)) return nullptr;
  const at::Tensor *k = tensor_arg(a[2], at::kBFloat16, "k"), *v = k ? tensor_arg(a[3], at::kBFloat16, "v") : nullptr;
  if (!v) return nullptr;
  if (k->dim() == 0) {
    PyErr_SetString(PyExc_IndexError, "K has no dimensions");
    return nullptr;
  }
  const int64_t n_new = k->dim() == 3 ? 1 : k->size(0);
  if (k->numel() != n_new * token || v->numel() != k->numel()) return value_error("bad K/V shape");
  if (!stream_arg(a[5], st)) return nullptr;
  const void *kp = k->data_ptr(), *vp = v->data_ptr();
  pmkvq_status s;
  Py_BEGIN_ALLOW_THREADS
  s = pmkvq_append(h, (int32_t)layer, kp, vp, (int32_t)n_new, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(s);
  END_HANDLE_TH_ERRORS
}

// (handle, layer, q, batch, q_heads, out or None, stream) -> out
PyObject *decode_attention(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  pmkvq_cache *h;
  void *st;
  int64_t layer, batch, heads;
  if (!arg_count(n, 7) || !handle_arg(a[0], h) || !int_arg(a[1], layer) || !int_arg(a[3], batch) || !int_arg(a[4], heads)) return nullptr;
  const at::Tensor *q = tensor_arg(a[2], at::kBFloat16, "q");
  if (!q) return nullptr;
  if (q->numel() != batch * heads * 128) return value_error("bad Q shape");
  at::Tensor made;
  const at::Tensor *out = &made;
  if (a[5] == Py_None) made = at::empty({batch, heads, 128}, q->options().dtype(at::kFloat));
  else if (!(out = tensor_arg(a[5], at::kFloat, "out"))) return nullptr;
  if (out->numel() < q->numel()) return value_error("bad out shape");  // (a larger one has always been taken: its head is written)
  if (!stream_arg(a[6], st)) return nullptr;
  const void *qp = q->data_ptr();
  float *op = static_cast<float *>(out->data_ptr());
  pmkvq_status s;
  Py_BEGIN_ALLOW_THREADS
  s = pmkvq_decode_attention(h, (int32_t)layer, qp, op, st);
  Py_END_ALLOW_THREADS
  if (s != PMKVQ_OK) return fail(s, "pmkvq_decode_attention");
  if (made.defined()) return THPVariable_Wrap(made);
  Py_INCREF(a[5]);
  return a[5];
  END_HANDLE_TH_ERRORS
}

// (handle, k, v, q, layers, batch, kv_heads, q_heads, out or None, stream) -> out
PyObject *decode_step(PyObject *, PyObject *const *a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  pmkvq_cache *h;
  void *st;
  int64_t layers, batch, kv_heads, heads;
  if (!arg_count(n, 10) || !handle_arg(a[0], h) || !int_arg(a[4], layers) || !int_arg(a[5], batch) || !int_arg(a[6], kv_heads) ||
      !int_arg(a[7], heads))
    return nullptr;
  const at::Tensor *k = tensor_arg(a[1], at::kBFloat16, "k"), *v = k ? tensor_arg(a[2], at::kBFloat16, "v") : nullptr;
  const at::Tensor *q = v ? tensor_arg(a[3], at::kBFloat16, "q") : nullptr;
  if (!q) return nullptr;
  if (k->numel() != layers * batch * kv_heads * 128 || v->numel() != k->numel() || q->numel() != layers * batch * heads * 128)
    return value_error("bad K/V/Q shape");
  at::Tensor made;
  const at::Tensor *out = &made;
  if (a[8] == Py_None) made = at::empty({layers, batch, heads, 128}, q->options().dtype(at::kFloat));
  else if (!(out = tensor_arg(a[8], at::kFloat, "out"))) return nullptr;
  if (out->numel() != q->numel()) return value_error("bad out shape");
  if (!stream_arg(a[9], st)) return nullptr;
  const void *kp = k->data_ptr(), *vp = v->data_ptr(), *qp = q->data_ptr();
  float *op = static_cast<float *>(out->data_ptr());
  pmkvq_status s;
  Py_BEGIN_ALLOW_THREADS
  s = pmkvq_decode_step(h, kp, vp, qp, op, st);
  Py_END_ALLOW_THREADS
  if (s != PMKVQ_OK) return fail(s, "pmkvq_decode_step");
  if (made.defined()) return THPVariable_Wrap(made);
  Py_INCREF(a[8]);
  return a[8];
  END_HANDLE_TH_ERRORS
}

// (handle, layer, n_tokens, cur_bits)
PyObject *restore_layer_state(PyObject *, PyObject *const *a, Py_ssize_t n) {
  pmkvq_cache *h;
  int64_t layer, tokens, bits;
  if (!arg_count(n, 4) || !handle_arg(a[0], h) || !int_arg(a[1], layer) || !int_arg(a[2], tokens) || !int_arg(a[3], bits)) return nullptr;
  const pmkvq_status s = pmkvq_restore_layer_state(h, (int32_t)layer, (int32_t)tokens, (int32_t)bits);
  if (s != PMKVQ_OK) return fail(s, "pmkvq_restore_layer_state");
  Py_RETURN_NONE;
}

// the current stream of the current device, as an integer
PyObject *current_stream(PyObject *, PyObject *) {
  HANDLE_TH_ERRORS
  return PyLong_FromVoidPtr(c10::cuda::getCurrentCUDAStream().stream());
  END_HANDLE_TH_ERRORS
}

PyObject *set_error(PyObject *, PyObject *type) {
  Py_INCREF(type);
  Py_XSETREF(g_error, type);
  Py_RETURN_NONE;
}

#define FAST(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {FAST(append), FAST(decode_attention), FAST(decode_step), FAST(restore_layer_state),
                          {"current_stream", current_stream, METH_NOARGS, nullptr}, {"set_error", set_error, METH_O, nullptr},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_host_calls", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_calls() {
  if (!(g_stream_attr = PyUnicode_InternFromString("cuda_stream"))) return nullptr;
  return PyModule_Create(&kModule);
}
