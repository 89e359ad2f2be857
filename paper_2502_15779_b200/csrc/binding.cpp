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

#ifndef RCP_HEADER_ID
#define RCP_HEADER_ID 0ull
#endif

namespace {

struct Entry {
  decltype(&rcp_quantize_act) quantize_act = nullptr;
  decltype(&rcp_gemv_w2a4_variant) gemv = nullptr;
  decltype(&rcp_gemv_w2a4_grouped_variant) gemv_grouped = nullptr;
  decltype(&rcp_gemv_w2a16_checked) gemv_w2a16 = nullptr;
  decltype(&rcp_gemv_w3a4) gemv_w3a4 = nullptr;
  decltype(&rcp_linear_w2a4_checked) linear = nullptr;
  decltype(&rcp_linear_w2a4_host) linear_host = nullptr;
  decltype(&rcp_gemv_workspace_bytes) workspace_bytes = nullptr;
} g_fn;


const char* type_name(at::ScalarType t) {
  return t == at::kHalf ? "float16" : t == at::kInt ? "int32" : t == at::kFloat ? "float32" : t == at::kChar ? "int8" : "uint8";
}
bool on_other_device(const char* name) {
  PyErr_Format(PyExc_ValueError, "%s: not on the device of the call's first tensor", name);
  return false;
}
// A contiguous CUDA tensor of the given type (on the device of `like`), or a TypeError.
const at::Tensor* dev(PyObject* o, at::ScalarType type, const char* name, const at::Tensor* like = nullptr) {
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.is_cuda() && t.scalar_type() == type && t.is_contiguous()) {
      if (like && t.device() != like->device()) { on_other_device(name); return nullptr; }
      return &t;
    }
  }
  PyErr_Format(PyExc_TypeError, "%s: expected a contiguous CUDA tensor of dtype torch.%s", name, type_name(type));
  return nullptr;
}
// The address of an optional buffer (None: null) that the library knows nothing else of: at least `need` elements of the given
// type (kByte: or int8; kAny: bytes of any type), contiguous, on the device of `like` or in page-locked host memory, which
// the device reaches as well.
constexpr at::ScalarType kAny = at::ScalarType::Undefined;
bool buffer(PyObject* o, const char* name, at::ScalarType type, const at::Tensor& like, int64_t need, void** out) {
  *out = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s: expected a tensor or None", name);
    return false;
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  const at::ScalarType have = t.scalar_type();
  if (have == type && t.is_cuda() && t.numel() >= need && t.is_contiguous() && t.get_device() == like.get_device()) {   // as a rule
    *out = t.data_ptr();
    return true;
  }
  const bool fits = type == kAny || have == type || ((type == at::kByte || type == at::kChar) && (have == at::kByte || have == at::kChar));
  if (!fits || !t.is_contiguous() || !(t.is_cuda() || t.is_pinned())) {
    PyErr_Format(PyExc_TypeError, "%s: expected a contiguous CUDA tensor%s%s", name, type == kAny ? "" : " of dtype torch.",
                 type == kAny ? "" : type_name(type));
    return false;
  }
  if (t.is_cuda() && t.device() != like.device()) return on_other_device(name);
  if ((type == kAny ? (int64_t)t.nbytes() : t.numel()) < need) {
    PyErr_Format(PyExc_ValueError, "%s: %lld %s, %lld are needed", name, (long long)(type == kAny ? (int64_t)t.nbytes() : t.numel()),
                 type == kAny ? "bytes" : "elements", (long long)need);
    return false;
  }
  *out = t.data_ptr();
  return true;
}
// bytes of workspace the library wants (0 for shapes it refuses)
int64_t workspace_bytes(int64_t M, int64_t N, int64_t K) { return (int64_t)g_fn.workspace_bytes((int)M, (int)N, (int)K); }
bool has_shape(const at::Tensor& t, std::initializer_list<int64_t> want) { return t.sizes() == at::IntArrayRef(want); }
bool bad_shapes(const char* what) {
  PyErr_Format(PyExc_ValueError, "shape mismatch between %s", what);
  return false;
}
// What int(o) and float(o) take: whole-numbered floats, numpy scalars, one-element tensors as well.
bool integer(PyObject* o, int* out) {
  long x;
  if (PyLong_CheckExact(o)) {
    x = PyLong_AsLong(o);
  } else {
    PyObject* v = PyNumber_Long(o);
    if (!v) return false;
    x = PyLong_AsLong(v);
    Py_DECREF(v);
  }
  if (x == -1 && PyErr_Occurred()) return false;
  *out = (int)x;
  return true;
}
bool real(PyObject* o, float* out) {
  if (PyFloat_CheckExact(o)) {
    *out = (float)PyFloat_AS_DOUBLE(o);
    return true;
  }
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
      !take("rcp_linear_w2a4_host", g_fn.linear_host) || !take("rcp_gemv_workspace_bytes", g_fn.workspace_bytes))
    return nullptr;
  decltype(&rcp_header_id) header_id = nullptr;
  if (!take("rcp_header_id", header_id)) return nullptr;
  if (header_id() != RCP_HEADER_ID) {
    g_fn = {};
    PyErr_SetString(PyExc_RuntimeError, "the library and its marshalling module were not built from the same include/rcp.h: build both anew "
                                        "with `python -m paper_2502_15779_b200.build`");
    return nullptr;
  }
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
    if (!x || !integer(a[1], &B) || !real(a[2], &clip)) return nullptr;
    if (x->dim() != 2) { bad_shapes("x and [M][K]"); return nullptr; }
    const int M = (int)x->size(0), K = (int)x->size(1);
    if (!buffer(a[3], "xq", at::kByte, *x, x->size(0) * (x->size(1) / 2), &xq) || !buffer(a[4], "scale", at::kHalf, *x, x->size(0), &scale))
      return nullptr;
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
    const at::Tensor* lut = dev(a[2], at::kHalf, "lut", words);
    if (!lut) return nullptr;
    const at::Tensor* xq = dev(a[4], at::kByte, "xq", words);
    if (!xq) return nullptr;
    const at::Tensor* scale = dev(a[5], at::kHalf, "scale", words);
    if (!scale) return nullptr;
    const bool two = words->dim() == 2 && xq->dim() == 2;
    const int64_t N = two ? words->size(0) : 0, K = two ? 16 * words->size(1) : 0, M = two ? xq->size(0) : 0;
    const bool grid = group == 0 ? has_shape(*lut, {N, 4}) : group > 0 && K % group == 0 && has_shape(*lut, {N, K / group, 4});
    if (!two || !grid || !has_shape(*xq, {M, K / 2}) || !has_shape(*scale, {M})) {
      bad_shapes(group == 0 ? "words, lut, xq and scale" : "words, lut, group, xq and scale");
      return nullptr;
    }
    if (!buffer(a[6], "y", at::kHalf, *words, M * N, &y) || !buffer(a[7], "workspace", kAny, *words, workspace_bytes(M, N, K), &ws) ||
        !buffer(a[8], "S_dbg", at::kInt, *words, M * N * (group ? K / group : 1) * 4, &S))
      return nullptr;
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
    const at::Tensor* lut = dev(a[1], at::kHalf, "lut", words);
    if (!lut) return nullptr;
    const at::Tensor* x = dev(a[2], at::kHalf, "x", words);
    if (!x) return nullptr;
    const bool two = words->dim() == 2 && x->dim() == 2;
    const int64_t N = two ? words->size(0) : 0, K = two ? 16 * words->size(1) : 0, M = two ? x->size(0) : 0;
    if (!two || !has_shape(*x, {M, K}) || !has_shape(*lut, {N, 4})) { bad_shapes("words, lut and x"); return nullptr; }
    if (!buffer(a[3], "y", at::kHalf, *words, M * N, &y) || !buffer(a[4], "digits", at::kChar, *words, M * 4 * K, &digits) ||
        !buffer(a[5], "unit", at::kFloat, *words, M * 4, &unit) ||
        !buffer(a[6], "workspace", kAny, *words, workspace_bytes(M, N, K), &ws) || !buffer(a[7], "S_dbg", at::kInt, *words, 4 * M * N * 4, &S))
      return nullptr;
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
    const at::Tensor* words1 = dev(a[1], at::kInt, "words1", words2);
    if (!words1) return nullptr;
    const at::Tensor* lut = dev(a[2], at::kHalf, "lut", words2);
    if (!lut) return nullptr;
    const at::Tensor* xq = dev(a[4], at::kByte, "xq", words2);
    if (!xq) return nullptr;
    const at::Tensor* scale = dev(a[5], at::kHalf, "scale", words2);
    if (!scale) return nullptr;
    const bool two = words2->dim() == 2 && xq->dim() == 2;
    const int64_t N = two ? words2->size(0) : 0, K = two ? 16 * words2->size(1) : 0, M = two ? xq->size(0) : 0;
    const bool grid = group == 0 ? has_shape(*lut, {N, 8}) : has_shape(*lut, {N, K / std::max(group, 1), 8});
    if (!two || !grid || !has_shape(*words1, {N, K / 32}) || !has_shape(*xq, {M, K / 2}) || !has_shape(*scale, {M})) {
      bad_shapes("words2, words1, lut, group, xq and scale");
      return nullptr;
    }
    if (!buffer(a[6], "y", at::kHalf, *words2, M * N, &y) ||
        !buffer(a[7], "S_dbg", at::kInt, *words2, M * N * (group ? K / std::max(group, 1) : 1) * 8, &S))
      return nullptr;
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
    const at::Tensor* words = dev(a[3], at::kInt, "words", x);
    if (!words) return nullptr;
    const at::Tensor* lut = dev(a[4], at::kHalf, "lut", x);
    if (!lut || !integer(a[1], &B) || !real(a[2], &clip) || !integer(a[5], &group)) return nullptr;
    const bool two = words->dim() == 2 && x->dim() == 2;
    const int64_t N = two ? words->size(0) : 0, K = two ? x->size(1) : 0, M = two ? x->size(0) : 0;
    const bool grid = group == 0 ? has_shape(*lut, {N, 4}) : has_shape(*lut, {N, K / std::max(group, 1), 4});
    if (!two || words->size(1) * 16 != K || !grid) { bad_shapes("x, words, lut and group"); return nullptr; }
    if (!buffer(a[6], "y", at::kHalf, *x, M * N, &y) || !buffer(a[7], "xq", at::kByte, *x, M * (K / 2), &xq) ||
        !buffer(a[8], "scale", at::kHalf, *x, M, &scale) || !buffer(a[9], "workspace", kAny, *x, workspace_bytes(M, N, K), &ws) ||
        !buffer(a[10], "S_dbg", at::kInt, *x, M * N * (group ? K / std::max(group, 1) : 1) * 4, &S))
      return nullptr;
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
    void *xd, *xq, *scale, *yd, *ws;
    if (!count(n, 11)) return nullptr;
    if (!THPVariable_Check(a[0]) || !THPVariable_Check(a[5])) {
      PyErr_SetString(PyExc_TypeError, "x_host and y_host must be tensors");
      return nullptr;
    }
    const at::Tensor &x = THPVariable_Unpack(a[0]), &y = THPVariable_Unpack(a[5]);
    if (!x.is_cpu() || !y.is_cpu() || x.scalar_type() != at::kHalf || y.scalar_type() != at::kHalf || !x.is_contiguous() ||
        !y.is_contiguous()) {
      PyErr_SetString(PyExc_TypeError, "x_host / y_host must be contiguous fp16 host tensors");
      return nullptr;
    }
    const at::Tensor* words = dev(a[3], at::kInt, "words");
    if (!words) return nullptr;
    const at::Tensor* lut = dev(a[4], at::kHalf, "lut", words);
    if (!lut || !integer(a[1], &B) || !real(a[2], &clip)) return nullptr;
    const bool two = words->dim() == 2 && x.dim() == 2;
    const int64_t N = two ? words->size(0) : 0, K = two ? x.size(1) : 0, M = two ? x.size(0) : 0;
    if (!two || words->size(1) * 16 != K || lut->numel() != 4 * N || y.numel() < M * N) {
      bad_shapes("x_host, words, lut and y_host");
      return nullptr;
    }
    if (!buffer(a[6], "x_dev", at::kHalf, *words, M * K, &xd) || !buffer(a[7], "xq_dev", at::kByte, *words, M * (K / 2), &xq) ||
        !buffer(a[8], "scale_dev", at::kHalf, *words, M, &scale) || !buffer(a[9], "y_dev", at::kHalf, *words, M * N, &yd) ||
        !buffer(a[10], "workspace", kAny, *words, workspace_bytes(M, N, K), &ws))
      return nullptr;
    const void *const xp = x.data_ptr(), *const lp = lut->data_ptr();
    void* const yp = y.data_ptr();
    const uint32_t* const wp = static_cast<const uint32_t*>(words->data_ptr());
    return on_device(*words, [&](void* st) {
      return g_fn.linear_host(xp, (int)M, (int)K, B, clip, wp, lp, (int)N, yp, xd, static_cast<uint8_t*>(xq), scale, yd, ws, st);
    });
  });
}

#define RCP_FAST(fn) {#fn, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fn)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {{"bind", bind, METH_O, nullptr}, RCP_FAST(quantize_act), RCP_FAST(gemv_w2a4), RCP_FAST(gemv_w2a16),
                          RCP_FAST(gemv_w3a4), RCP_FAST(linear_w2a4), RCP_FAST(linear_w2a4_host), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&kModule); }
