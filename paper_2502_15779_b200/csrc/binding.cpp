// Argument marshalling of the calls a decode step makes once per layer, in native code: type, device, layout and shape
// checks of the tensors, their pointers, the current stream, the call. Marshalled by ctypes these calls cost the host 11
// to 13 us each, 6.6 of them outside the library (a Python stream object, an argument object per pointer), more than the
// GPU needs for a small layer. No computation here; the library's entry points are handed over by address
// (bind), so that the same module serves whichever build of it is loaded.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/rcp.h"

namespace {

struct Entry {
  decltype(&rcp_quantize_act) quantize_act = nullptr;
  decltype(&rcp_gemv_w2a4_variant) gemv = nullptr;
  decltype(&rcp_gemv_w2a4_grouped_variant) gemv_grouped = nullptr;
  decltype(&rcp_gemv_w2a16_checked) gemv_w2a16 = nullptr;
  decltype(&rcp_gemv_w3a4) gemv_w3a4 = nullptr;
  decltype(&rcp_linear_w2a4_checked) linear = nullptr;
  decltype(&rcp_linear_w2a4_host) linear_host = nullptr;
} g_fn;


// A contiguous CUDA tensor of the given type, or a TypeError.
const at::Tensor* dev(PyObject* o, at::ScalarType type, const char* name) {
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.is_cuda() && t.scalar_type() == type && t.is_contiguous()) return &t;
  }
  PyErr_Format(PyExc_TypeError, "%s: expected a contiguous CUDA tensor of dtype torch.%s", name,
               type == at::kHalf ? "float16" : type == at::kInt ? "int32" : "uint8");
  return nullptr;
}
// The data pointer of an optional tensor (None: null).
bool ptr(PyObject* o, const char* name, void** out) {
  *out = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s: expected a tensor or None", name);
    return false;
  }
  *out = THPVariable_Unpack(o).data_ptr();
  return true;
}
bool has_shape(const at::Tensor& t, std::initializer_list<int64_t> want) { return t.sizes() == at::IntArrayRef(want); }
bool bad_shapes(const char* what) {
  PyErr_Format(PyExc_ValueError, "shape mismatch between %s", what);
  return false;
}
// What int(o) and float(o) take: whole-numbered floats, numpy scalars, one-element tensors as well.
bool integer(PyObject* o, int* out) {
  PyObject* v = PyNumber_Long(o);
  if (!v) return false;
  const long x = PyLong_AsLong(v);
  Py_DECREF(v);
  if (x == -1 && PyErr_Occurred()) return false;
  *out = (int)x;
  return true;
}
bool real(PyObject* o, float* out) {
  PyObject* v = PyNumber_Float(o);
  if (!v) return false;
  const double x = PyFloat_AS_DOUBLE(v);
  Py_DECREF(v);
  *out = (float)x;
  return true;
}
// What a call returns to Python: its status (0: done).
PyObject* status(int rc) { return PyLong_FromLong(rc); }

// Runs `call(stream)` with t's device current and its current stream, without the interpreter lock.
template <typename Call>
PyObject* on_device(const at::Tensor& t, Call call) {
  int rc;
  const c10::cuda::CUDAGuard guard(t.device());
  void* const stream = c10::cuda::getCurrentCUDAStream(t.device().index()).stream();
  Py_BEGIN_ALLOW_THREADS
  rc = call(stream);
  Py_END_ALLOW_THREADS
  return status(rc);
}
bool count(Py_ssize_t have, Py_ssize_t want) {
  if (have == want) return true;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, have);
  return false;
}

// C++ exceptions of the tensor library become RuntimeErrors
template <typename F>
PyObject* guarded(F f) {
  try {
    return f();
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// bind({name: address}): the loaded library's entry points
PyObject* bind(PyObject*, PyObject* table) {
  if (!PyDict_Check(table)) {
    PyErr_SetString(PyExc_TypeError, "bind: a dict of addresses is expected");
    return nullptr;
  }
  auto take = [&](const char* name, auto& fn) {
    PyObject* v = PyDict_GetItemString(table, name);   // borrowed
    if (!v) {
      PyErr_Format(PyExc_KeyError, "bind: %s is missing", name);
      return false;
    }
    void* const p = PyLong_AsVoidPtr(v);
    if (PyErr_Occurred()) return false;
    fn = reinterpret_cast<std::decay_t<decltype(fn)>>(p);
    return true;
  };
  if (!take("rcp_quantize_act", g_fn.quantize_act) || !take("rcp_gemv_w2a4_variant", g_fn.gemv) ||
      !take("rcp_gemv_w2a4_grouped_variant", g_fn.gemv_grouped) || !take("rcp_gemv_w2a16_checked", g_fn.gemv_w2a16) ||
      !take("rcp_gemv_w3a4", g_fn.gemv_w3a4) || !take("rcp_linear_w2a4_checked", g_fn.linear) ||
      !take("rcp_linear_w2a4_host", g_fn.linear_host))
    return nullptr;
  Py_RETURN_NONE;
}

// (x, had_block, clip_ratio, xq, scale)
PyObject* quantize_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    int B;
    float clip;
    void *xq, *scale;
    if (!count(n, 5)) return nullptr;
    const at::Tensor* x = dev(a[0], at::kHalf, "x");
    if (!x || !integer(a[1], &B) || !real(a[2], &clip) || !ptr(a[3], "xq", &xq) || !ptr(a[4], "scale", &scale)) return nullptr;
    if (x->dim() != 2) { bad_shapes("x and [M][K]"); return nullptr; }
    const int M = (int)x->size(0), K = (int)x->size(1);
    const void* const xp = x->data_ptr();
    return on_device(*x, [&](void* st) { return g_fn.quantize_act(xp, M, K, B, clip, static_cast<uint8_t*>(xq), scale, st); });
  });
}

// (variant, words, lut, group, xq, scale, y, workspace, S_dbg); group 0: one grid per row
PyObject* gemv_w2a4(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    int variant, group;
    void *y, *ws, *S;
    if (!count(n, 9) || !integer(a[0], &variant) || !integer(a[3], &group)) return nullptr;
    const at::Tensor* words = dev(a[1], at::kInt, "words");
    if (!words) return nullptr;
    const at::Tensor* lut = dev(a[2], at::kHalf, "lut");
    if (!lut) return nullptr;
    const at::Tensor* xq = dev(a[4], at::kByte, "xq");
    if (!xq) return nullptr;
    const at::Tensor* scale = dev(a[5], at::kHalf, "scale");
    if (!scale || !ptr(a[6], "y", &y) || !ptr(a[7], "workspace", &ws) || !ptr(a[8], "S_dbg", &S)) return nullptr;
    const bool two = words->dim() == 2 && xq->dim() == 2;
    const int64_t N = two ? words->size(0) : 0, K = two ? 16 * words->size(1) : 0, M = two ? xq->size(0) : 0;
    const bool grid = group == 0 ? has_shape(*lut, {N, 4}) : group > 0 && K % group == 0 && has_shape(*lut, {N, K / group, 4});
    if (!two || !grid || !has_shape(*xq, {M, K / 2}) || !has_shape(*scale, {M})) {
      bad_shapes(group == 0 ? "words, lut, xq and scale" : "words, lut, group, xq and scale");
      return nullptr;
    }
    const uint32_t* const wp = static_cast<const uint32_t*>(words->data_ptr());
    const void *lp = lut->data_ptr(), *sp = scale->data_ptr();
    const uint8_t* const qp = static_cast<const uint8_t*>(xq->data_ptr());
    return on_device(*words, [&](void* st) {
      return group == 0 ? g_fn.gemv(variant, wp, lp, qp, sp, (int)M, (int)N, (int)K, y, ws, static_cast<int32_t*>(S), st)
                        : g_fn.gemv_grouped(variant, wp, lp, group, qp, sp, (int)M, (int)N, (int)K, y, ws, static_cast<int32_t*>(S), st);
    });
  });
}

// (words, lut, x, y, digits, unit, workspace, S_dbg)
PyObject* gemv_w2a16(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    void *y, *digits, *unit, *ws, *S;
    if (!count(n, 8)) return nullptr;
    const at::Tensor* words = dev(a[0], at::kInt, "words");
    if (!words) return nullptr;
    const at::Tensor* lut = dev(a[1], at::kHalf, "lut");
    if (!lut) return nullptr;
    const at::Tensor* x = dev(a[2], at::kHalf, "x");
    if (!x || !ptr(a[3], "y", &y) || !ptr(a[4], "digits", &digits) || !ptr(a[5], "unit", &unit) || !ptr(a[6], "workspace", &ws) ||
        !ptr(a[7], "S_dbg", &S))
      return nullptr;
    const bool two = words->dim() == 2 && x->dim() == 2;
    const int64_t N = two ? words->size(0) : 0, K = two ? 16 * words->size(1) : 0, M = two ? x->size(0) : 0;
    if (!two || !has_shape(*x, {M, K}) || !has_shape(*lut, {N, 4})) { bad_shapes("words, lut and x"); return nullptr; }
    const uint32_t* const wp = static_cast<const uint32_t*>(words->data_ptr());
    const void *lp = lut->data_ptr(), *xp = x->data_ptr();
    return on_device(*words, [&](void* st) {
      return g_fn.gemv_w2a16(wp, lp, xp, (int)M, (int)N, (int)K, y, static_cast<int8_t*>(digits), static_cast<float*>(unit), ws,
                             static_cast<int32_t*>(S), st);
    });
  });
}

// (words2, words1, lut, group, xq, scale, y, S_dbg)
PyObject* gemv_w3a4(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    int group;
    void *y, *S;
    if (!count(n, 8) || !integer(a[3], &group)) return nullptr;
    const at::Tensor* words2 = dev(a[0], at::kInt, "words2");
    if (!words2) return nullptr;
    const at::Tensor* words1 = dev(a[1], at::kInt, "words1");
    if (!words1) return nullptr;
    const at::Tensor* lut = dev(a[2], at::kHalf, "lut");
    if (!lut) return nullptr;
    const at::Tensor* xq = dev(a[4], at::kByte, "xq");
    if (!xq) return nullptr;
    const at::Tensor* scale = dev(a[5], at::kHalf, "scale");
    if (!scale || !ptr(a[6], "y", &y) || !ptr(a[7], "S_dbg", &S)) return nullptr;
    const bool two = words2->dim() == 2 && xq->dim() == 2;
    const int64_t N = two ? words2->size(0) : 0, K = two ? 16 * words2->size(1) : 0, M = two ? xq->size(0) : 0;
    const bool grid = group == 0 ? has_shape(*lut, {N, 8}) : has_shape(*lut, {N, K / std::max(group, 1), 8});
    if (!two || !grid || !has_shape(*words1, {N, K / 32}) || !has_shape(*xq, {M, K / 2}) || !has_shape(*scale, {M})) {
      bad_shapes("words2, words1, lut, group, xq and scale");
      return nullptr;
    }
    const uint32_t *w2 = static_cast<const uint32_t*>(words2->data_ptr()), *w1 = static_cast<const uint32_t*>(words1->data_ptr());
    const void *lp = lut->data_ptr(), *sp = scale->data_ptr();
    const uint8_t* const qp = static_cast<const uint8_t*>(xq->data_ptr());
    return on_device(*words2, [&](void* st) {
      return g_fn.gemv_w3a4(w2, w1, lp, group, qp, sp, (int)M, (int)N, (int)K, y, static_cast<int32_t*>(S), st);
    });
  });
}

// (x, had_block, clip_ratio, words, lut, group, y, xq, scale, workspace, S_dbg)
PyObject* linear_w2a4(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    int B, group;
    float clip;
    void *y, *xq, *scale, *ws, *S;
    if (!count(n, 11)) return nullptr;
    const at::Tensor* x = dev(a[0], at::kHalf, "x");
    if (!x) return nullptr;
    const at::Tensor* words = dev(a[3], at::kInt, "words");
    if (!words) return nullptr;
    const at::Tensor* lut = dev(a[4], at::kHalf, "lut");
    if (!lut || !integer(a[1], &B) || !real(a[2], &clip) || !integer(a[5], &group) || !ptr(a[6], "y", &y) || !ptr(a[7], "xq", &xq) ||
        !ptr(a[8], "scale", &scale) || !ptr(a[9], "workspace", &ws) || !ptr(a[10], "S_dbg", &S))
      return nullptr;
    const bool two = words->dim() == 2 && x->dim() == 2;
    const int64_t N = two ? words->size(0) : 0, K = two ? x->size(1) : 0, M = two ? x->size(0) : 0;
    const bool grid = group == 0 ? has_shape(*lut, {N, 4}) : has_shape(*lut, {N, K / std::max(group, 1), 4});
    if (!two || words->size(1) * 16 != K || !grid) { bad_shapes("x, words, lut and group"); return nullptr; }
    const uint32_t* const wp = static_cast<const uint32_t*>(words->data_ptr());
    const void *lp = lut->data_ptr(), *xp = x->data_ptr();
    return on_device(*words, [&](void* st) {
      return g_fn.linear(xp, (int)M, (int)K, B, clip, wp, lp, group, (int)N, y, static_cast<uint8_t*>(xq), scale, ws,
                         static_cast<int32_t*>(S), st);
    });
  });
}

// (x_host, had_block, clip_ratio, words, lut, y_host, x_dev, xq_dev, scale_dev, y_dev, workspace)
PyObject* linear_w2a4_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    int B;
    float clip;
    void *lut, *xd, *xq, *scale, *yd, *ws;
    if (!count(n, 11)) return nullptr;
    if (!THPVariable_Check(a[0]) || !THPVariable_Check(a[5]) || !THPVariable_Check(a[3])) {
      PyErr_SetString(PyExc_TypeError, "x_host, words and y_host must be tensors");
      return nullptr;
    }
    const at::Tensor &x = THPVariable_Unpack(a[0]), &y = THPVariable_Unpack(a[5]), &words = THPVariable_Unpack(a[3]);
    if (x.is_cuda() || y.is_cuda() || x.scalar_type() != at::kHalf || y.scalar_type() != at::kHalf) {
      PyErr_SetString(PyExc_TypeError, "x_host / y_host must be fp16 host tensors");
      return nullptr;
    }
    if (!integer(a[1], &B) || !real(a[2], &clip) || !ptr(a[4], "lut", &lut) || !ptr(a[6], "x_dev", &xd) || !ptr(a[7], "xq_dev", &xq) ||
        !ptr(a[8], "scale_dev", &scale) || !ptr(a[9], "y_dev", &yd) || !ptr(a[10], "workspace", &ws))
      return nullptr;
    if (x.dim() != 2 || !words.is_cuda()) { bad_shapes("x_host and [M][K]"); return nullptr; }
    const int M = (int)x.size(0), K = (int)x.size(1), N = (int)words.size(0);
    const void* const xp = x.data_ptr();
    void* const yp = y.data_ptr();
    const uint32_t* const wp = static_cast<const uint32_t*>(words.data_ptr());
    return on_device(words, [&](void* st) {
      return g_fn.linear_host(xp, M, K, B, clip, wp, lut, N, yp, xd, static_cast<uint8_t*>(xq), scale, yd, ws, st);
    });
  });
}

#define RCP_FAST(fn) {#fn, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fn)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {{"bind", bind, METH_O, nullptr}, RCP_FAST(quantize_act), RCP_FAST(gemv_w2a4), RCP_FAST(gemv_w2a16),
                          RCP_FAST(gemv_w3a4), RCP_FAST(linear_w2a4), RCP_FAST(linear_w2a4_host), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&kModule); }
