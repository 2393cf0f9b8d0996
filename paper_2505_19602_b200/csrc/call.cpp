// The hot calls of the C ABI for Python callers: tensors are read through PyTorch's C++ interface and handed to the function
// whose address the binding passes, in one native call.  A step of a small map costs the host 5.9 us this way; with four ctypes
// structures built for every call (and the launches and events that a step made then) it was 14.5 us, twice what the GPU takes.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>
#include <vector>

#include "../../include/scalekv.h"

namespace {

// A C++ exception (a sparse tensor has no strides, a wrapped one no memory) becomes the Python one that the tensor's own method
// raises: none may cross the interpreter's C frames.
template <typename F> bool guarded(F read) {
  try {
    return read();
  } catch (...) {
    torch::translate_exception_to_python(std::current_exception());
    return false;
  }
}

// obj.name() or, with an index, obj.name(index)
bool ask(PyObject *obj, const char *name, int index, long long *out) {
  PyObject *r = index < 0 ? PyObject_CallMethod(obj, name, nullptr) : PyObject_CallMethod(obj, name, "i", index);
  if (!r) return false;
  *out = (long long)(intptr_t)PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return !PyErr_Occurred();
}

bool bad_shape() {
  PyErr_SetString(PyExc_AssertionError, "expected [B, H, n, d] with contiguous head_dim");
  return false;
}

// [B, H, n, d] tensor -> view with element strides; the last axis must be contiguous.  Anything else that has a tensor's dim(),
// stride(i) and data_ptr() is asked for them (a subclass of Tensor may have its own).
bool view(PyObject *obj, scalekv_tensor *out) {
  if (!THPVariable_CheckExact(obj)) {
    long long dim, last, ptr, sb, sh, st;
    if (!ask(obj, "dim", -1, &dim)) return false;
    if (dim != 4) return bad_shape();
    if (!ask(obj, "stride", 3, &last)) return false;
    if (last != 1) return bad_shape();
    if (!ask(obj, "data_ptr", -1, &ptr) || !ask(obj, "stride", 0, &sb) || !ask(obj, "stride", 1, &sh) || !ask(obj, "stride", 2, &st)) return false;
    *out = {reinterpret_cast<const void *>((intptr_t)ptr), sb, sh, st};
    return true;
  }
  return guarded([&] {
    const at::Tensor &t = THPVariable_Unpack(obj);
    if (t.dim() != 4 || t.stride(3) != 1) return bad_shape();
    out->ptr = t.data_ptr();
    out->stride_b = t.stride(0);
    out->stride_h = t.stride(1);
    out->stride_t = t.stride(2);
    return true;
  });
}

// None or a tensor of floats
bool floats(PyObject *obj, float **out) {
  *out = nullptr;
  if (obj == Py_None) return true;
  if (!THPVariable_CheckExact(obj)) {
    long long ptr;
    if (!ask(obj, "data_ptr", -1, &ptr)) return false;
    *out = reinterpret_cast<float *>((intptr_t)ptr);
    return true;
  }
  return guarded([&] {
    *out = static_cast<float *>(THPVariable_Unpack(obj).data_ptr());
    return true;
  });
}

template <typename T> T address(PyObject *obj) { return reinterpret_cast<T>(PyLong_AsVoidPtr(obj)); }

bool arguments(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return false;
}

#define CALL(expr)            \
  int st;                     \
  if (PyErr_Occurred()) return nullptr; \
  Py_BEGIN_ALLOW_THREADS      \
  st = (int)(expr);           \
  Py_END_ALLOW_THREADS        \
  return PyLong_FromLong(st)

// step(function, ctx, layer, scale, Q, K, V, O, lse, w, window address)
PyObject *step(PyObject *, PyObject *const *a, Py_ssize_t n) {
  scalekv_tensor q, k, v, o;
  float *lse;
  if (!arguments(n, 11) || !view(a[4], &q) || !view(a[5], &k) || !view(a[6], &v) || !view(a[7], &o) || !floats(a[8], &lse)) return nullptr;
  const auto fn = address<decltype(&scalekv_step)>(a[0]);
  const auto ctx = address<scalekv_ctx *>(a[1]);
  const int layer = (int)PyLong_AsLong(a[2]), scale = (int)PyLong_AsLong(a[3]), w = (int)PyLong_AsLong(a[9]);
  const auto window = address<const int32_t *>(a[10]);
  CALL(fn(ctx, layer, scale, q, k, v, o, lse, w, window));
}

// step_ex(function, ctx, layer, scale, Q, K, V, O, lse, compress, w, window address, options address)
PyObject *step_ex(PyObject *, PyObject *const *a, Py_ssize_t n) {
  scalekv_tensor q, k, v, o;
  float *lse;
  if (!arguments(n, 13) || !view(a[4], &q) || !view(a[5], &k) || !view(a[6], &v) || !view(a[7], &o) || !floats(a[8], &lse)) return nullptr;
  const auto fn = address<decltype(&scalekv_step_ex)>(a[0]);
  const auto ctx = address<scalekv_ctx *>(a[1]);
  const int layer = (int)PyLong_AsLong(a[2]), scale = (int)PyLong_AsLong(a[3]), compress = (int)PyLong_AsLong(a[9]), w = (int)PyLong_AsLong(a[10]);
  const auto window = address<const int32_t *>(a[11]);
  const auto opts = address<const scalekv_select_opts *>(a[12]);
  CALL(fn(ctx, layer, scale, q, k, v, o, lse, compress, w, window, opts));
}

// append(function, ctx, layer, scale, K, V)
PyObject *append(PyObject *, PyObject *const *a, Py_ssize_t n) {
  scalekv_tensor k, v;
  if (!arguments(n, 6) || !view(a[4], &k) || !view(a[5], &v)) return nullptr;
  const auto fn = address<decltype(&scalekv_append)>(a[0]);
  const auto ctx = address<scalekv_ctx *>(a[1]);
  const int layer = (int)PyLong_AsLong(a[2]), scale = (int)PyLong_AsLong(a[3]);
  CALL(fn(ctx, layer, scale, k, v));
}

// attend(function, ctx, layer, Q, O, lse)
PyObject *attend(PyObject *, PyObject *const *a, Py_ssize_t n) {
  scalekv_tensor q, o;
  float *lse;
  if (!arguments(n, 6) || !view(a[3], &q) || !view(a[4], &o) || !floats(a[5], &lse)) return nullptr;
  const auto fn = address<decltype(&scalekv_attend)>(a[0]);
  const auto ctx = address<scalekv_ctx *>(a[1]);
  const int layer = (int)PyLong_AsLong(a[2]);
  CALL(fn(ctx, layer, q, o, lse));
}

// compress_ex(function, ctx, layer, Qw or None, w, window address, full map, options address)
PyObject *compress_ex(PyObject *, PyObject *const *a, Py_ssize_t n) {
  scalekv_tensor q = {nullptr, 0, 0, 0};
  if (!arguments(n, 8) || (a[3] != Py_None && !view(a[3], &q))) return nullptr;
  const auto fn = address<decltype(&scalekv_compress_ex)>(a[0]);
  const auto ctx = address<scalekv_ctx *>(a[1]);
  const int layer = (int)PyLong_AsLong(a[2]), w = (int)PyLong_AsLong(a[4]), full = (int)PyLong_AsLong(a[6]);
  const auto window = address<const int32_t *>(a[5]);
  const auto opts = address<const scalekv_select_opts *>(a[7]);
  CALL(fn(ctx, layer, q, w, window, full, opts));
}

// [batch][heads] of floats, as lists of lists
PyObject *lists(const std::vector<double> &x, Py_ssize_t batch, Py_ssize_t heads) {
  PyObject *out = PyList_New(batch);
  for (Py_ssize_t b = 0; out && b < batch; ++b) {
    PyObject *row = PyList_New(heads);
    for (Py_ssize_t h = 0; row && h < heads; ++h) {
      PyObject *v = PyFloat_FromDouble(x[(size_t)(b * heads + h)]);
      if (!v) Py_CLEAR(row);
      else PyList_SET_ITEM(row, h, v);
    }
    if (!row) Py_CLEAR(out);
    else PyList_SET_ITEM(out, b, row);
  }
  return out;
}

// layer_stats_ex(function, ctx, layer, Q, topk_prime, query_stride, batch, heads) -> (status, car, htk and the three per slice)
PyObject *layer_stats_ex(PyObject *, PyObject *const *a, Py_ssize_t n) {
  scalekv_tensor q;
  if (!arguments(n, 8) || !view(a[3], &q)) return nullptr;
  const auto fn = address<decltype(&scalekv_layer_stats_ex)>(a[0]);
  const auto ctx = address<scalekv_ctx *>(a[1]);
  const int layer = (int)PyLong_AsLong(a[2]), topk = (int)PyLong_AsLong(a[4]), stride = (int)PyLong_AsLong(a[5]);
  const Py_ssize_t batch = PyLong_AsSsize_t(a[6]), heads = PyLong_AsSsize_t(a[7]);
  if (PyErr_Occurred()) return nullptr;
  double car = 0.0, htk = 0.0;
  int st = 0;
  std::vector<double> cs, ts, ns;
  if (!guarded([&] {
        cs.resize((size_t)(batch * heads)); ts.resize(cs.size()); ns.resize(cs.size());
        return true;
      })) return nullptr;
  Py_BEGIN_ALLOW_THREADS
  st = (int)fn(ctx, layer, q, topk, stride, &car, &htk, cs.data(), ts.data(), ns.data());
  Py_END_ALLOW_THREADS
  PyObject *c = lists(cs, batch, heads), *t = lists(ts, batch, heads), *m = lists(ns, batch, heads);
  if (c && t && m) return Py_BuildValue("(iddNNN)", st, car, htk, c, t, m);
  Py_XDECREF(c); Py_XDECREF(t); Py_XDECREF(m);
  return nullptr;
}

#define METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(step), METHOD(step_ex), METHOD(append), METHOD(attend), METHOD(compress_ex), METHOD(layer_stats_ex),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_scalekv_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__scalekv_call() { return PyModule_Create(&module); }
