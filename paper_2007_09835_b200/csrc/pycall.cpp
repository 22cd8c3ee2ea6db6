// Python extension module `_pycall`: one convolution call on torch tensors without the interpreter's share of it.
//
// Describing two tensors, filling the parameter structures and going through ctypes takes 8 to 10 us of Python for a call
// whose library part takes 1 to 3; here the tensors' fields are read through the C API (about 1 us for a call).  The
// library's functions are reached through addresses that the binding hands over, so this module links to nothing.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>

#include "rt3d.h"

namespace {

PyObject *g_float32, *g_bfloat16, *g_raw_stream, *g_get_device;      // owned
PyObject *s_shape, *s_stride, *s_dtype, *s_data_ptr;

typedef rt3d_status (*ConvFn)(const rt3d_tensor*, const rt3d_packed*, const float*, const rt3d_conv_params*, rt3d_tensor*, void*);
typedef rt3d_status (*FusedFn)(const rt3d_tensor*, const rt3d_packed*, const float*, const rt3d_conv_params*,
                               const rt3d_fusion*, rt3d_tensor*, void*);

PyObject* setup(PyObject*, PyObject* args) {
  PyObject *f32, *bf16, *raw, *dev;
  if (!PyArg_ParseTuple(args, "OOOO", &f32, &bf16, &raw, &dev)) return nullptr;
  Py_INCREF(f32); Py_INCREF(bf16); Py_INCREF(raw); Py_INCREF(dev);
  Py_XSETREF(g_float32, f32); Py_XSETREF(g_bfloat16, bf16); Py_XSETREF(g_raw_stream, raw); Py_XSETREF(g_get_device, dev);
  Py_RETURN_NONE;
}

bool as_pointer(PyObject* v, uintptr_t* out) {
  if (v == Py_None) { *out = 0; return true; }
  *out = reinterpret_cast<uintptr_t>(PyLong_AsVoidPtr(v));
  return !(*out == 0 && PyErr_Occurred());
}

bool data_ptr(PyObject* t, uintptr_t* out) {
  PyObject* r = PyObject_CallMethodNoArgs(t, s_data_ptr);
  if (!r) return false;
  const bool ok = as_pointer(r, out);
  Py_DECREF(r);
  return ok;
}

// Dense in (n, t, h, w) with the last dimension as pitch, as strides say (extents of 1 included).
int strides_are_dense(PyObject* t, const int64_t (&e)[5]) {
  PyObject* st = PyObject_CallMethodNoArgs(t, s_stride);
  if (!st) return -1;
  int ok = PyTuple_Check(st) && PyTuple_GET_SIZE(st) == 5;
  int64_t want = 1;
  for (int i = 4; i >= 0 && ok; --i) {
    ok = PyLong_AsLongLong(PyTuple_GET_ITEM(st, i)) == want;
    want *= e[i];
  }
  Py_DECREF(st);
  return PyErr_Occurred() ? -1 : ok;
}

// The descriptor that binding.tensor_desc makes, with the same refusals.
bool describe(PyObject* t, PyObject* channels, rt3d_tensor* d) {
  PyObject* shape = PyObject_GetAttr(t, s_shape);
  if (!shape) return false;
  if (!PyTuple_Check(shape) || PyTuple_GET_SIZE(shape) != 5) {
    Py_DECREF(shape);
    PyErr_SetString(PyExc_ValueError, "expected a 5-D NDHWC tensor with unit channel stride");
    return false;
  }
  int64_t e[5];
  for (int i = 0; i < 5; ++i) e[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(shape, i));
  Py_DECREF(shape);
  if (PyErr_Occurred()) return false;
  const int dense = strides_are_dense(t, e);
  if (dense < 0) return false;
  if (!dense) {
    PyErr_SetString(PyExc_ValueError, "tensor must be dense in (n,t,h,w) with pitch = size of last dimension");
    return false;
  }
  PyObject* dt = PyObject_GetAttr(t, s_dtype);
  if (!dt) return false;
  const int code = dt == g_float32 ? RT3D_F32 : dt == g_bfloat16 ? RT3D_BF16 : -1;
  if (code < 0) PyErr_SetObject(PyExc_KeyError, dt);
  Py_DECREF(dt);
  if (code < 0) return false;
  uintptr_t data;
  if (!data_ptr(t, &data)) return false;
  const long c = PyLong_AsLong(channels);
  if (c == -1 && PyErr_Occurred()) return false;
  d->data = reinterpret_cast<void*>(data);
  d->n = int32_t(e[0]); d->t = int32_t(e[1]); d->h = int32_t(e[2]); d->w = int32_t(e[3]);
  d->c = int32_t(c); d->c_stride = int32_t(e[4]); d->dtype = code;
  return true;
}

bool stream_of(PyObject* v, uintptr_t* out) {
  if (v != Py_None) return as_pointer(v, out);
  PyObject* dev = PyObject_CallNoArgs(g_get_device);
  if (!dev) return false;
  PyObject* st = PyObject_CallOneArg(g_raw_stream, dev);
  Py_DECREF(dev);
  if (!st) return false;
  const bool ok = as_pointer(st, out);
  Py_DECREF(st);
  return ok;
}

bool tensor_or_none(PyObject* t, uintptr_t* out) {
  *out = 0;
  return t == Py_None || data_ptr(t, out);
}

bool ints(PyObject* const* a, int n, int* out) {
  for (int i = 0; i < n; ++i) {
    const long v = PyLong_AsLong(a[i]);
    if (v == -1 && PyErr_Occurred()) return false;
    out[i] = int(v);
  }
  return true;
}

bool want(Py_ssize_t n, Py_ssize_t expected) {
  if (n != expected) PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
  return n == expected;
}

// A library call with the interpreter released, as ctypes makes it: a launch may have to wait for room in its stream.
template <typename F>
PyObject* released(const F& call) {
  rt3d_status s;
  Py_BEGIN_ALLOW_THREADS
  s = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(long(s));
}

// The three calls of the pruning step, with the arguments of their binding functions behind the library's address.
PyObject* group_norms(PyObject*, PyObject* const* a, Py_ssize_t n) {   // address, w, g_m, g_n, norm, norms, stream
  uintptr_t fn, w, norms, stream;
  int v[3], e[5];
  if (!want(n, 7) || !as_pointer(a[0], &fn) || !data_ptr(a[1], &w) || !ints(a + 2, 3, v) || !data_ptr(a[5], &norms) ||
      !stream_of(a[6], &stream))
    return nullptr;
  PyObject* shape = PyObject_GetAttr(a[1], s_shape);
  if (!shape) return nullptr;
  bool ok = PyTuple_Check(shape) && PyTuple_GET_SIZE(shape) == 5;
  if (!ok) PyErr_SetString(PyExc_ValueError, "expected a 5-D weight tensor");
  for (int i = 0; ok && i < 5; ++i) {
    PyObject* item = PyTuple_GET_ITEM(shape, i);
    ok = ints(&item, 1, e + i);
  }
  Py_DECREF(shape);
  if (!ok) return nullptr;
  return released([&] {
    return reinterpret_cast<decltype(&rt3d_kgs_group_norms)>(fn)(
        reinterpret_cast<const float*>(w), e[0], e[1], e[2], e[3], e[4], v[0], v[1], v[2], reinterpret_cast<float*>(norms),
        reinterpret_cast<void*>(stream));
  });
}

PyObject* reweight(PyObject*, PyObject* const* a, Py_ssize_t n) {      // address, norms, count, eps, threshold, penalty, keep, stream
  uintptr_t fn, norms, penalty, keep, stream;
  if (!want(n, 8) || !as_pointer(a[0], &fn) || !data_ptr(a[1], &norms)) return nullptr;
  const long long count = PyLong_AsLongLong(a[2]);
  const double eps = PyFloat_AsDouble(a[3]), threshold = PyFloat_AsDouble(a[4]);
  if (PyErr_Occurred() || !tensor_or_none(a[5], &penalty) || !tensor_or_none(a[6], &keep) || !stream_of(a[7], &stream)) return nullptr;
  return released([&] {
    return reinterpret_cast<decltype(&rt3d_kgs_reweight)>(fn)(
        reinterpret_cast<const float*>(norms), count, float(eps), float(threshold), reinterpret_cast<float*>(penalty),
        reinterpret_cast<uint8_t*>(keep), reinterpret_cast<void*>(stream));
  });
}

PyObject* expand_mask(PyObject*, PyObject* const* a, Py_ssize_t n) {   // address, group mask, M, N, Kt, Kh, Kw, g_m, g_n, mask, stream
  uintptr_t fn, g, mask, stream;
  int v[7];
  if (!want(n, 11) || !as_pointer(a[0], &fn) || !data_ptr(a[1], &g) || !ints(a + 2, 7, v) || !data_ptr(a[9], &mask) ||
      !stream_of(a[10], &stream))
    return nullptr;
  return released([&] {
    return reinterpret_cast<decltype(&rt3d_kgs_expand_mask)>(fn)(
        reinterpret_cast<const uint8_t*>(g), v[0], v[1], v[2], v[3], v[4], v[5], v[6], reinterpret_cast<uint8_t*>(mask),
        reinterpret_cast<void*>(stream));
  });
}

// pointers_are(tensors, addresses): whether every tensor of a tuple still has its address of a bytes object (8 bytes each).
PyObject* pointers_are(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!want(n, 2)) return nullptr;
  if (!PyTuple_Check(a[0]) || !PyBytes_Check(a[1]) || PyBytes_GET_SIZE(a[1]) != PyTuple_GET_SIZE(a[0]) * Py_ssize_t(sizeof(uintptr_t))) {
    PyErr_SetString(PyExc_TypeError, "a tuple of tensors and their addresses");
    return nullptr;
  }
  for (Py_ssize_t i = 0; i < PyTuple_GET_SIZE(a[0]); ++i) {
    uintptr_t now, then;
    if (!data_ptr(PyTuple_GET_ITEM(a[0], i), &now)) return nullptr;
    __builtin_memcpy(&then, PyBytes_AS_STRING(a[1]) + i * sizeof(then), sizeof(then));
    if (now != then) Py_RETURN_FALSE;
  }
  Py_RETURN_TRUE;
}

// conv(address, x, c_in, handle, bias, params, y, c_out, stream[, residual, (pool_t, pool_h, pool_w)]) -> status.
// With the last two the address is rt3d_conv3d_sparse_fused's, else rt3d_conv3d_sparse's or _dense's.
PyObject* conv(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 9 && n != 11) {
    PyErr_SetString(PyExc_TypeError, "conv takes 9 or 11 arguments");
    return nullptr;
  }
  uintptr_t fn, handle, bias = 0, stream = 0;
  rt3d_tensor x{}, y{}, r{};
  if (!as_pointer(a[0], &fn) || !describe(a[1], a[2], &x) || !as_pointer(a[3], &handle)) return nullptr;
  if (a[4] != Py_None && !data_ptr(a[4], &bias)) return nullptr;
  if (!describe(a[6], a[7], &y)) return nullptr;
  if (!stream_of(a[8], &stream)) return nullptr;
  rt3d_fusion fz{};
  if (n == 11) {
    if (a[9] != Py_None) {
      if (!describe(a[9], a[7], &r)) return nullptr;
      fz.residual = &r;
    }
    int32_t* pool[3] = {&fz.pool_t, &fz.pool_h, &fz.pool_w};
    for (int i = 0; i < 3; ++i) {
      PyObject* v = PySequence_GetItem(a[10], i);
      if (!v) return nullptr;
      *pool[i] = int32_t(PyLong_AsLong(v));
      Py_DECREF(v);
    }
    if (PyErr_Occurred()) return nullptr;
  }
  Py_buffer p;
  if (PyObject_GetBuffer(a[5], &p, PyBUF_SIMPLE) != 0) return nullptr;
  if (p.len != Py_ssize_t(sizeof(rt3d_conv_params))) {
    PyBuffer_Release(&p);
    PyErr_SetString(PyExc_ValueError, "not a parameter structure");
    return nullptr;
  }
  rt3d_conv_params params;
  __builtin_memcpy(&params, p.buf, sizeof(params));
  PyBuffer_Release(&p);
  return released([&] {
    const auto* w = reinterpret_cast<const rt3d_packed*>(handle);
    const auto* b = reinterpret_cast<const float*>(bias);
    void* st = reinterpret_cast<void*>(stream);
    return n == 11 ? reinterpret_cast<FusedFn>(fn)(&x, w, b, &params, &fz, &y, st)
                   : reinterpret_cast<ConvFn>(fn)(&x, w, b, &params, &y, st);
  });
}

PyMethodDef methods[] = {
    {"setup", setup, METH_VARARGS, "setup(float32, bfloat16, raw_stream, get_device): torch objects the calls need"},
    {"conv", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(conv)), METH_FASTCALL,
     "conv(address, x, c_in, handle, bias, params, y, c_out, stream[, residual, pool]) -> status"},
    {"group_norms", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(group_norms)), METH_FASTCALL, ""},
    {"reweight", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(reweight)), METH_FASTCALL, ""},
    {"expand_mask", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(expand_mask)), METH_FASTCALL, ""},
    {"pointers_are", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(pointers_are)), METH_FASTCALL,
     "pointers_are(tensors, addresses) -> bool"},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pycall(void) {
  s_shape = PyUnicode_InternFromString("shape");
  s_stride = PyUnicode_InternFromString("stride");
  s_dtype = PyUnicode_InternFromString("dtype");
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  return PyModule_Create(&module);
}
