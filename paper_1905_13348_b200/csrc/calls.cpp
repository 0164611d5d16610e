// The per-window calls of the binding as a Python extension module: tensors, counts and stream to the C ABI.
//
// What bounds such a call is the host.  Through ctypes infaas_select_batch took 5.0 us, of which the launch
// itself is 2.5: 1.0 went into asking four tensors for their device, layout, type and address one attribute
// at a time and 0.7 into ctypes.  Here a tensor is looked at in C++: 2.9 us.  Anything but a plain contiguous
// CUDA tensor of the wanted width goes through the binding's own `_dev_ptr` (subclasses, objects that only look
// like tensors, None) or gets its error from there.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>

#include "infaas.h"

namespace {

PyObject *g_dev_ptr = nullptr, *g_length = nullptr;      // binding._dev_ptr, binding._length
PyObject *s_handle = nullptr, *s_value = nullptr, *s_width[2] = {nullptr, nullptr};
enum Width { U16, U32 };

// The arguments of one call; the first that cannot be converted leaves a Python error and ok = false.
struct Args {
  PyObject *const *v;
  bool ok = true;

  infaas_catalog *catalog(int i) {
    void *p = nullptr;
    PyObject *h = ok ? PyObject_GetAttr(v[i], s_handle) : nullptr;
    PyObject *a = h ? PyObject_GetAttr(h, s_value) : nullptr;      // a ctypes.c_void_p's: an int, or None
    ok = a != nullptr;
    if (ok && a != Py_None) {
      p = PyLong_AsVoidPtr(a);
      ok = !PyErr_Occurred();
    }
    Py_XDECREF(a);
    Py_XDECREF(h);
    return static_cast<infaas_catalog *>(p);
  }
  void *tensor(int i, Width w) {
    if (!ok || v[i] == Py_None) return nullptr;
    if (THPVariable_CheckExact(v[i])) {
      const at::Tensor &t = THPVariable_Unpack(v[i]);
      const at::ScalarType s = t.scalar_type();
      const bool fits = w == U16 ? s == at::kShort || s == at::kUInt16 : s == at::kInt || s == at::kUInt32;
      if (fits && t.is_cuda() && t.is_contiguous()) return t.mutable_data_ptr();
    }
    PyObject *a = PyObject_CallFunctionObjArgs(g_dev_ptr, v[i], s_width[w], nullptr);
    ok = a != nullptr;
    void *p = ok && a != Py_None ? PyLong_AsVoidPtr(a) : nullptr;
    ok = ok && !PyErr_Occurred();
    Py_XDECREF(a);
    return p;
  }
  unsigned long long number(PyObject *o) {                         // int(o), wrapped to 64 bits as ctypes does
    PyObject *a = ok ? PyNumber_Long(o) : nullptr;
    const unsigned long long x = a ? PyLong_AsUnsignedLongLongMask(a) : 0;
    ok = a != nullptr && !PyErr_Occurred();
    Py_XDECREF(a);
    return x;
  }
  uint32_t u32(int i) { return (uint32_t)number(v[i]); }
  // A count, or (None) the length of the tensor at `of`.
  uint64_t count(int i, int of) {
    if (!ok || v[i] != Py_None) return number(v[i]);
    if (THPVariable_CheckExact(v[of])) {
      const at::Tensor &t = THPVariable_Unpack(v[of]);
      if (t.dim() > 0) return (uint64_t)t.size(0);
    }
    PyObject *a = PyObject_CallFunctionObjArgs(g_length, v[of], nullptr);
    ok = a != nullptr;
    const uint64_t n = ok ? number(a) : 0;
    Py_XDECREF(a);
    return n;
  }
  void *stream(int i) {                                            // the address binding._stream_ptr gives, or None
    if (!ok || v[i] == Py_None) return nullptr;
    return reinterpret_cast<void *>(number(v[i]));
  }
};

// `call` returns the C ABI's code with the interpreter lock released.
template <class F>
PyObject *finish(const Args &a, F call) {
  if (!a.ok) return nullptr;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// `body(args)` for calls of exactly N arguments; C++ exceptions (torch's) become RuntimeError.
template <int N, class F>
PyObject *entry(PyObject *const *v, Py_ssize_t n, F body) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
    return nullptr;
  }
  try {
    Args a{v};
    return body(a);
  } catch (const std::exception &e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyObject *setup(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return entry<2>(v, n, [](Args &a) -> PyObject * {
    Py_XSETREF(g_dev_ptr, Py_NewRef(a.v[0]));
    Py_XSETREF(g_length, Py_NewRef(a.v[1]));
    Py_RETURN_NONE;
  });
}

// catalog, task, slo, min_acc, decision, n, stream
PyObject *select_batch(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return entry<7>(v, n, [](Args &a) {
    const uint64_t m = a.count(5, 1);
    infaas_catalog *c = a.catalog(0);
    const auto *task = static_cast<const uint16_t *>(a.tensor(1, U16));
    const auto *slo = static_cast<const uint32_t *>(a.tensor(2, U32));
    const auto *acc = static_cast<const uint16_t *>(a.tensor(3, U16));
    auto *dec = static_cast<uint32_t *>(a.tensor(4, U32));
    void *s = a.stream(6);
    return finish(a, [=] { return infaas_select_batch(c, task, slo, acc, m, dec, s); });
  });
}

// catalog, task, slo, min_acc, decision, n, window_us, stream
PyObject *select_update(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return entry<8>(v, n, [](Args &a) {
    const uint64_t m = a.count(5, 1);
    infaas_catalog *c = a.catalog(0);
    const auto *task = static_cast<const uint16_t *>(a.tensor(1, U16));
    const auto *slo = static_cast<const uint32_t *>(a.tensor(2, U32));
    const auto *acc = static_cast<const uint16_t *>(a.tensor(3, U16));
    auto *dec = static_cast<uint32_t *>(a.tensor(4, U32));
    const uint32_t us = a.u32(6);
    void *s = a.stream(7);
    return finish(a, [=] { return infaas_select_update(c, task, slo, acc, m, dec, us, s); });
  });
}

// catalog, decision, n, window_us, stream
PyObject *load_update(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return entry<5>(v, n, [](Args &a) {
    const uint64_t m = a.count(2, 1);
    infaas_catalog *c = a.catalog(0);
    const auto *dec = static_cast<const uint32_t *>(a.tensor(1, U32));
    const uint32_t us = a.u32(3);
    void *s = a.stream(4);
    return finish(a, [=] { return infaas_load_update(c, dec, m, us, s); });
  });
}

// catalog, decision, n, stream
PyObject *tally(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return entry<4>(v, n, [](Args &a) {
    const uint64_t m = a.count(2, 1);
    infaas_catalog *c = a.catalog(0);
    const auto *dec = static_cast<const uint32_t *>(a.tensor(1, U32));
    void *s = a.stream(3);
    return finish(a, [=] { return infaas_tally(c, dec, m, s); });
  });
}

// catalog, window_us, stream
PyObject *advance(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return entry<3>(v, n, [](Args &a) {
    infaas_catalog *c = a.catalog(0);
    const uint32_t us = a.u32(1);
    void *s = a.stream(2);
    return finish(a, [=] { return infaas_advance(c, us, s); });
  });
}

// catalog, window_us, slack_pct, lambda_milli, variant, delta, stream
PyObject *autoscale_step(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return entry<7>(v, n, [](Args &a) {
    infaas_catalog *c = a.catalog(0);
    const uint32_t us = a.u32(1), slack = a.u32(2), lambda = a.u32(3);
    auto *variant = static_cast<uint32_t *>(a.tensor(4, U32)), *delta = static_cast<uint32_t *>(a.tensor(5, U32));
    void *s = a.stream(6);
    return finish(a, [=] { return infaas_autoscale_step(c, us, slack, lambda, variant, delta, s); });
  });
}

// catalog, decision, n, worker, stream
PyObject *assign_workers(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return entry<5>(v, n, [](Args &a) {
    const uint64_t m = a.count(2, 1);
    infaas_catalog *c = a.catalog(0);
    const auto *dec = static_cast<const uint32_t *>(a.tensor(1, U32));
    auto *worker = static_cast<uint32_t *>(a.tensor(3, U32));
    void *s = a.stream(4);
    return finish(a, [=] { return infaas_assign_workers(c, dec, m, worker, s); });
  });
}

#define CALL(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {CALL(setup), CALL(select_batch), CALL(select_update), CALL(load_update), CALL(tally),
                         CALL(advance), CALL(autoscale_step), CALL(assign_workers), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void) {
  s_handle = PyUnicode_InternFromString("handle");
  s_value = PyUnicode_InternFromString("value");
  s_width[U16] = PyUnicode_InternFromString("u16");
  s_width[U32] = PyUnicode_InternFromString("u32");
  if (!s_handle || !s_value || !s_width[U16] || !s_width[U32]) return nullptr;
  return PyModule_Create(&module);
}
