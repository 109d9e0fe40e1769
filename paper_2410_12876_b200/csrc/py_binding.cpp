// Argument marshalling of the calls in ag.h for Python, as an extension module.
//
// A decode step of a short cache takes the GPU 4-8 us.  Marshalled in Python (ctypes conversions, a
// current_stream() object, is_contiguous() and data_ptr() per tensor) one call cost the host 11-12 us, so
// a loop of decode steps and every prompt of a few hundred tokens ran at the host's speed.  Here a call
// reads the tensors' pointers through torch's C++ API and the structs through the buffer protocol.
// Nothing but marshalling: each function returns the ag_status of its C counterpart.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/ag.h"

namespace {

// Reads the positional arguments of one call in order.  The first failure sets the Python error and
// makes every later read return zero; the caller looks at done() once.
class Args {
 public:
  Args(PyObject *const *args, Py_ssize_t n) : a_(args), n_(n) {}
  // After the last argument: whether all were read and none is left over.
  bool done() {
    if (ok_ && i_ < n_) {
      PyErr_SetString(PyExc_TypeError, "too many arguments");
      ok_ = false;
    }
    return ok_;
  }

  const ag_layer_desc *desc() {
    PyObject *o = next();
    return o ? static_cast<const ag_layer_desc *>(buffer(o, sizeof(ag_layer_desc))) : nullptr;
  }
  // RaggedCache: its `struct` is the ctypes ag_cache the tensors' addresses were put into
  ag_cache *cache() {
    PyObject *o = next();
    if (!o) return nullptr;
    static PyObject *const name = PyUnicode_InternFromString("struct");
    PyObject *s = PyObject_GetAttr(o, name);
    if (!s) return fail<ag_cache *>();
    ag_cache *c = static_cast<ag_cache *>(buffer(s, sizeof(ag_cache)));   // the cache keeps its struct alive
    Py_DECREF(s);
    return c;
  }
  // None, an address, or a contiguous tensor
  void *ptr() {
    PyObject *o = next();
    if (!o || o == Py_None) return nullptr;
    if (THPVariable_Check(o)) {
      const at::Tensor &t = THPVariable_Unpack(o);
      if (!t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "tensor must be contiguous");
        return fail<void *>();
      }
      return t.data_ptr();
    }
    void *p = PyLong_AsVoidPtr(o);
    return !p && PyErr_Occurred() ? fail<void *>() : p;
  }
  // workspace tensor (or None): address and size in bytes
  void *workspace(size_t *bytes) {
    *bytes = 0;
    PyObject *o = next();
    if (!o || o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) {
      PyErr_SetString(PyExc_TypeError, "workspace must be a tensor or None");
      return fail<void *>();
    }
    const at::Tensor &t = THPVariable_Unpack(o);
    *bytes = t.nbytes();
    return t.data_ptr();
  }
  float real() {
    PyObject *o = next();
    if (!o) return 0.f;
    const double v = PyFloat_AsDouble(o);
    return v == -1.0 && PyErr_Occurred() ? fail<float>() : static_cast<float>(v);
  }
  // None (the current stream of the current device), a cudaStream_t as an integer, or a torch stream
  void *stream() {
    PyObject *o = next();
    if (!o) return nullptr;
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *s = PyLong_Check(o) ? Py_NewRef(o) : PyObject_GetAttrString(o, "cuda_stream");
    if (!s) return fail<void *>();
    void *p = PyLong_AsVoidPtr(s);
    Py_DECREF(s);
    return !p && PyErr_Occurred() ? fail<void *>() : p;
  }

 private:
  PyObject *next() {
    if (!ok_) return nullptr;
    if (i_ >= n_) {
      PyErr_SetString(PyExc_TypeError, "too few arguments");
      return fail<PyObject *>();
    }
    return a_[i_++];
  }
  void *buffer(PyObject *o, size_t size) {
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return fail<void *>();
    void *p = b.buf;
    const bool fits = static_cast<size_t>(b.len) == size;
    PyBuffer_Release(&b);                    // `o` stays referenced by the caller's frame
    if (!fits) {
      PyErr_SetString(PyExc_TypeError, "a struct of another size");
      return fail<void *>();
    }
    return p;
  }
  template <typename T> T fail() { ok_ = false; return T(); }
  PyObject *const *a_;
  Py_ssize_t n_, i_ = 0;
  bool ok_ = true;
};

// Runs the C call without the interpreter lock (a launch may block on a full queue).
template <typename F>
PyObject *finish(Args &a, F &&call) {
  if (!a.done()) return nullptr;
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

// A C++ exception (torch's, for a device that cannot be used) becomes a Python error.
template <PyObject *(*F)(Args &)>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n) {
  try {
    Args a(args, n);
    return F(a);
  } catch (const std::exception &e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyObject *gate_forward(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *X = a.ptr(), *Wq = a.ptr(), *Wk = a.ptr(), *Wv = a.ptr(), *Wo = a.ptr(), *gamma = a.ptr(), *scores = a.ptr(),
       *flags = a.ptr();
  size_t wb;
  void *ws = a.workspace(&wb), *st = a.stream();
  return finish(a, [&] {
    return ag_gate_forward(d, X, Wq, Wk, Wv, Wo, static_cast<float *>(gamma), static_cast<float *>(scores),
                           static_cast<uint8_t *>(flags), ws, wb, st);
  });
}
PyObject *gate_linear_forward(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *X = a.ptr(), *W = a.ptr(), *gamma = a.ptr(), *scores = a.ptr(), *flags = a.ptr(), *st = a.stream();
  return finish(a, [&] {
    return ag_gate_linear_forward(d, X, W, static_cast<float *>(gamma), static_cast<float *>(scores),
                                  static_cast<uint8_t *>(flags), st);
  });
}
PyObject *compact_kv(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *K = a.ptr(), *V = a.ptr(), *flags = a.ptr();
  ag_cache *c = a.cache();
  void *prefix = a.ptr(), *idx = a.ptr(), *status = a.ptr();
  size_t wb;
  void *ws = a.workspace(&wb), *st = a.stream();
  return finish(a, [&] {
    return ag_compact_kv(d, K, V, static_cast<uint8_t *>(flags), c, static_cast<int32_t *>(prefix),
                         static_cast<int32_t *>(idx), static_cast<int32_t *>(status), ws, wb, st);
  });
}
PyObject *kv_project_cache(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *X = a.ptr(), *Wk = a.ptr(), *Wv = a.ptr(), *flags = a.ptr();
  ag_cache *c = a.cache();
  void *prefix = a.ptr(), *idx = a.ptr(), *K = a.ptr(), *V = a.ptr(), *status = a.ptr(), *st = a.stream();
  return finish(a, [&] {
    return ag_kv_project_cache(d, X, Wk, Wv, static_cast<uint8_t *>(flags), c, static_cast<int32_t *>(prefix),
                               static_cast<int32_t *>(idx), K, V, static_cast<int32_t *>(status), st);
  });
}
PyObject *qkv_project_cache(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *X = a.ptr(), *Wq = a.ptr(), *Wk = a.ptr(), *Wv = a.ptr(), *flags = a.ptr();
  ag_cache *c = a.cache();
  void *prefix = a.ptr(), *idx = a.ptr(), *Q = a.ptr(), *K = a.ptr(), *V = a.ptr(), *status = a.ptr(),
       *st = a.stream();
  return finish(a, [&] {
    return ag_qkv_project_cache(d, X, Wq, Wk, Wv, static_cast<uint8_t *>(flags), c, static_cast<int32_t *>(prefix),
                                static_cast<int32_t *>(idx), Q, K, V, static_cast<int32_t *>(status), st);
  });
}
PyObject *prefill_attn(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *Q = a.ptr(), *K = a.ptr(), *V = a.ptr(), *flags = a.ptr();
  ag_cache *c = a.cache();
  void *prefix = a.ptr();
  const float scale = a.real();
  void *O = a.ptr();
  size_t wb;
  void *ws = a.workspace(&wb), *st = a.stream();
  return finish(a, [&] {
    return ag_prefill_attn(d, Q, K, V, static_cast<uint8_t *>(flags), c, static_cast<int32_t *>(prefix), scale, O, ws,
                           wb, st);
  });
}
PyObject *out_project(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *O = a.ptr(), *Wo = a.ptr(), *X = a.ptr(), *Y = a.ptr(), *st = a.stream();
  return finish(a, [&] { return ag_out_project(d, O, Wo, X, Y, st); });
}
PyObject *decode_attn(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *q = a.ptr(), *k = a.ptr(), *v = a.ptr();
  ag_cache *c = a.cache();
  const float scale = a.real();
  void *o = a.ptr();
  size_t wb;
  void *ws = a.workspace(&wb), *st = a.stream();
  return finish(a, [&] { return ag_decode_attn(d, q, k, v, c, scale, o, ws, wb, st); });
}
PyObject *decode_attn_noalloc(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *q = a.ptr(), *k = a.ptr(), *v = a.ptr();
  ag_cache *c = a.cache();
  const float scale = a.real();
  void *o = a.ptr(), *st = a.stream();
  return finish(a, [&] { return ag_decode_attn_noalloc(d, q, k, v, c, scale, o, st); });
}
PyObject *decode_step(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *q = a.ptr(), *k = a.ptr(), *v = a.ptr(), *f = a.ptr();
  ag_cache *c = a.cache();
  const float scale = a.real();
  void *o = a.ptr(), *status = a.ptr();
  size_t wb;
  void *ws = a.workspace(&wb), *st = a.stream();
  return finish(a, [&] {
    return ag_decode_step(d, q, k, v, static_cast<uint8_t *>(f), c, scale, o, static_cast<int32_t *>(status), ws, wb,
                          st);
  });
}
PyObject *cache_append(Args &a) {
  const ag_layer_desc *d = a.desc();
  void *k = a.ptr(), *v = a.ptr(), *f = a.ptr();
  ag_cache *c = a.cache();
  void *status = a.ptr(), *st = a.stream();
  return finish(a, [&] {
    return ag_cache_append(d, k, v, static_cast<uint8_t *>(f), c, static_cast<int32_t *>(status), st);
  });
}

template <PyObject *(*F)(Args &)>
PyMethodDef method(const char *name) {
  return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(&entry<F>)), METH_FASTCALL, nullptr};
}

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void) {
  static PyMethodDef methods[] = {
      method<gate_forward>("gate_forward"), method<gate_linear_forward>("gate_linear_forward"),
      method<compact_kv>("compact_kv"), method<kv_project_cache>("kv_project_cache"),
      method<qkv_project_cache>("qkv_project_cache"), method<prefill_attn>("prefill_attn"),
      method<out_project>("out_project"), method<decode_attn>("decode_attn"),
      method<decode_attn_noalloc>("decode_attn_noalloc"), method<decode_step>("decode_step"),
      method<cache_append>("cache_append"), {nullptr, nullptr, 0, nullptr}};
  static PyModuleDef def = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};
  PyObject *m = PyModule_Create(&def);
  if (m && PyModule_AddStringConstant(m, "tag", AG_MARSHAL_TAG) != 0) Py_CLEAR(m);
  return m;
}
