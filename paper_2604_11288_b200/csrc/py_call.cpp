// Native argument marshalling for the entry points of libta.so that a program calls once per layer or per generated token.
// CPython module _ta_call: ctypes spends about 8 us converting the 19 arguments of ta_compress, as much as the call itself
// takes; this takes about 2 us. Function addresses come from the ctypes-loaded library (set_function), so that there is one
// copy of it and one place that decides which. Marshalling only: every check of the values is the library's.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "ta.h"

namespace {

PyObject* g_void_p = nullptr;       // ctypes.c_void_p
PyObject* g_view = nullptr;         // the ctypes structures of the binding
PyObject* g_policy = nullptr;
PyObject* g_batch = nullptr;
PyObject* g_stream = nullptr;
PyObject* g_data_ptr = nullptr;     // interned names
PyObject* g_stride = nullptr;
PyObject* g_ctypes = nullptr;
PyObject* g_data = nullptr;

enum Fn { kCompress, kCompressLse, kCompressScores, kStreamStep, kDetect, kMaskConf, kFns };
void* g_fn[kFns];

// The memory of a ctypes object of type `cls`. The object outlives the call: the caller's argument list holds it.
bool ctypes_memory(PyObject* o, PyObject* cls, size_t size, void** out) {
  if (!PyObject_TypeCheck(o, reinterpret_cast<PyTypeObject*>(cls))) {
    PyErr_Format(PyExc_TypeError, "expected %s, got %s", reinterpret_cast<PyTypeObject*>(cls)->tp_name, Py_TYPE(o)->tp_name);
    return false;
  }
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
  const bool fits = (size_t)b.len >= size;
  *out = b.buf;
  PyBuffer_Release(&b);
  if (!fits) PyErr_SetString(PyExc_TypeError, "structure is too small");
  return fits;
}

// Address of a tensor, a numpy array, an int, a ctypes pointer or None.
bool pointer(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = nullptr;
    return true;
  }
  if (PyLong_Check(o)) {
    *out = PyLong_AsVoidPtr(o);
    return !PyErr_Occurred();
  }
  if (PyObject_TypeCheck(o, reinterpret_cast<PyTypeObject*>(g_void_p))) {
    void* at = nullptr;
    if (!ctypes_memory(o, g_void_p, sizeof(void*), &at)) return false;
    memcpy(out, at, sizeof(void*));
    return true;
  }
  PyObject* v = PyObject_VectorcallMethod(g_data_ptr, &o, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, nullptr);
  if (!v && PyErr_ExceptionMatches(PyExc_AttributeError)) {  // numpy
    PyErr_Clear();
    PyObject* c = PyObject_GetAttr(o, g_ctypes);
    v = c ? PyObject_GetAttr(c, g_data) : nullptr;
    Py_XDECREF(c);
  }
  if (!v) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

bool integer(PyObject* o, long long* out) {
  *out = PyLong_AsLongLong(o);
  return !(*out == -1 && PyErr_Occurred());
}

struct Args {  // reads the arguments in order; `ok` turns false with a Python error set
  PyObject* const* v;
  bool ok = true;
  template <class T>
  T* ptr() {
    void* p = nullptr;
    if (ok) ok = pointer(*v, &p);
    ++v;
    return static_cast<T*>(p);
  }
  template <class T>
  T* object(PyObject* cls) {
    void* p = nullptr;
    if (ok) ok = ctypes_memory(*v, cls, sizeof(T), &p);
    ++v;
    return static_cast<T*>(p);
  }
  ta_bf16_view view() {
    ta_bf16_view r = {};
    const void* p = object<const ta_bf16_view>(g_view);
    if (ok) memcpy(&r, p, sizeof r);
    return r;
  }
  long long num() {
    long long n = 0;
    if (ok) ok = integer(*v, &n);
    ++v;
    return n;
  }
  uint64_t word() {
    uint64_t n = 0;
    if (ok) {
      n = PyLong_AsUnsignedLongLongMask(*v);
      ok = !(n == (uint64_t)-1 && PyErr_Occurred());
    }
    ++v;
    return n;
  }
  float real() {
    double d = 0.0;
    if (ok) {
      d = PyFloat_AsDouble(*v);
      ok = !(d == -1.0 && PyErr_Occurred());
    }
    ++v;
    return (float)d;
  }
};

bool count_is(Py_ssize_t n, Py_ssize_t want) {
  if (n != want) PyErr_Format(PyExc_TypeError, "%zd arguments, %zd expected", n, want);
  return n == want;
}

template <class F>
PyObject* run(bool ok, F f) {
  if (!ok) return nullptr;
  ta_status s;
  Py_BEGIN_ALLOW_THREADS
  s = f();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)s);
}

PyObject* compress(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 18)) return nullptr;
  Args a{v};
  auto* ctx = a.ptr<ta_ctx>();
  auto* pats = a.ptr<ta_patterns>();
  auto* pol = a.object<ta_policy>(g_policy);
  auto* batch = a.object<ta_batch>(g_batch);
  const int Hq = (int)a.num(), Hkv = (int)a.num(), d = (int)a.num(), K = (int)a.num();
  auto* ids = a.ptr<int32_t>();
  const ta_bf16_view q = a.view(), k = a.view(), vv = a.view();
  const uint64_t epoch = a.word();
  auto *ko = a.ptr<void>(), *vo = a.ptr<void>();
  auto *idx = a.ptr<int32_t>(), *cnt = a.ptr<int32_t>();
  auto* st = a.ptr<void>();
  return run(a.ok, [&] {
    return reinterpret_cast<decltype(&ta_compress)>(g_fn[kCompress])(ctx, pats, pol, batch, Hq, Hkv, d, K, ids, q, k, vv, epoch,
                                                                    ko, vo, idx, cnt, st);
  });
}

PyObject* compress_lse(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 19)) return nullptr;
  Args a{v};
  auto* ctx = a.ptr<ta_ctx>();
  auto* pats = a.ptr<ta_patterns>();
  auto* pol = a.object<ta_policy>(g_policy);
  auto* batch = a.object<ta_batch>(g_batch);
  const int Hq = (int)a.num(), Hkv = (int)a.num(), d = (int)a.num(), K = (int)a.num();
  auto* ids = a.ptr<int32_t>();
  const ta_bf16_view q = a.view(), k = a.view(), vv = a.view();
  auto* lse = a.ptr<float>();
  const uint64_t epoch = a.word();
  auto *ko = a.ptr<void>(), *vo = a.ptr<void>();
  auto *idx = a.ptr<int32_t>(), *cnt = a.ptr<int32_t>();
  auto* st = a.ptr<void>();
  return run(a.ok, [&] {
    return reinterpret_cast<decltype(&ta_compress_lse)>(g_fn[kCompressLse])(ctx, pats, pol, batch, Hq, Hkv, d, K, ids, q, k, vv,
                                                                           lse, epoch, ko, vo, idx, cnt, st);
  });
}

PyObject* compress_scores(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 18)) return nullptr;
  Args a{v};
  auto* ctx = a.ptr<ta_ctx>();
  auto* pats = a.ptr<ta_patterns>();
  auto* pol = a.object<ta_policy>(g_policy);
  auto* batch = a.object<ta_batch>(g_batch);
  const int Hkv = (int)a.num(), d = (int)a.num(), K = (int)a.num();
  auto* ids = a.ptr<int32_t>();
  auto *score = a.ptr<float>(), *score2 = a.ptr<float>();
  const ta_bf16_view k = a.view(), vv = a.view();
  const uint64_t epoch = a.word();
  auto *ko = a.ptr<void>(), *vo = a.ptr<void>();
  auto *idx = a.ptr<int32_t>(), *cnt = a.ptr<int32_t>();
  auto* st = a.ptr<void>();
  return run(a.ok, [&] {
    return reinterpret_cast<decltype(&ta_compress_scores)>(g_fn[kCompressScores])(ctx, pats, pol, batch, Hkv, d, K, ids, score,
                                                                                 score2, k, vv, epoch, ko, vo, idx, cnt, st);
  });
}

PyObject* stream_step(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 8)) return nullptr;
  Args a{v};
  auto* ctx = a.ptr<ta_ctx>();
  auto* pats = a.ptr<ta_patterns>();
  auto* pol = a.object<ta_policy>(g_policy);
  auto* s = a.object<ta_stream>(g_stream);
  auto* ids = a.ptr<int32_t>();
  auto* attn = a.ptr<float>();
  auto* ev = a.ptr<int32_t>();
  auto* st = a.ptr<void>();
  return run(a.ok, [&] {
    return reinterpret_cast<decltype(&ta_stream_step)>(g_fn[kStreamStep])(ctx, pats, pol, s, ids, attn, ev, st);
  });
}

PyObject* detect(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 9)) return nullptr;
  Args a{v};
  auto* ctx = a.ptr<ta_ctx>();
  const long long total = a.num();
  auto* emb = a.ptr<void>();
  const long long stride = a.num();
  const int D = (int)a.num();
  auto* concepts = a.ptr<void>();
  const int C = (int)a.num();
  auto* conf = a.ptr<float>();
  auto* st = a.ptr<void>();
  return run(a.ok, [&] {
    return reinterpret_cast<decltype(&ta_detect_embedding)>(g_fn[kDetect])(ctx, total, emb, stride, D, concepts, C, conf, st);
  });
}

PyObject* mask_conf(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 13)) return nullptr;
  Args a{v};
  auto* ctx = a.ptr<ta_ctx>();
  auto* pol = a.object<ta_policy>(g_policy);
  auto* batch = a.object<ta_batch>(g_batch);
  auto* ids = a.ptr<int32_t>();
  auto* conf = a.ptr<float>();
  const float threshold = a.real(), budget = a.real();
  const int span = (int)a.num(), rank = (int)a.num();
  auto* flags = a.ptr<uint8_t>();
  auto *voucher = a.ptr<float>(), *u = a.ptr<float>();
  auto* st = a.ptr<void>();
  return run(a.ok, [&] {
    return reinterpret_cast<decltype(&ta_sponsor_mask_conf)>(g_fn[kMaskConf])(ctx, pol, batch, ids, conf, threshold, budget, span,
                                                                             rank, flags, voucher, u, st);
  });
}

// view(tensor, ragged): strides and address of a [L, B, H, n, d] or ragged [L, H, total, d] tensor as a ta_bf16_view
PyObject* view(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 2)) return nullptr;
  const int ragged = PyObject_IsTrue(v[1]);
  if (ragged < 0) return nullptr;
  ta_bf16_view r = {};
  if (v[0] != Py_None) {
    PyObject* t = v[0];
    PyObject* s = PyObject_VectorcallMethod(g_stride, &t, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, nullptr);
    if (!s) return nullptr;
    long long x[5] = {};
    const Py_ssize_t dims = PyTuple_Check(s) ? PyTuple_GET_SIZE(s) : -1;
    bool ok = dims == (ragged ? 4 : 5);
    if (!ok) PyErr_Format(PyExc_AssertionError, "a tensor of %d dimensions is needed", ragged ? 4 : 5);
    for (Py_ssize_t i = 0; ok && i < dims; ++i) ok = integer(PyTuple_GET_ITEM(s, i), &x[i]);
    Py_DECREF(s);
    if (!ok) return nullptr;
    if (x[dims - 1] != 1) {
      PyErr_SetString(PyExc_AssertionError, "head_dim must be contiguous");
      return nullptr;
    }
    void* p = nullptr;
    if (!pointer(t, &p)) return nullptr;
    r.ptr = p;
    r.stride_l = x[0];
    r.stride_b = ragged ? 0 : x[1];
    r.stride_h = x[ragged ? 1 : 2];
    r.stride_n = x[ragged ? 2 : 3];
  }
  PyObject* o = PyObject_CallNoArgs(g_view);
  void* at = nullptr;
  if (!o || !ctypes_memory(o, g_view, sizeof r, &at)) {
    Py_XDECREF(o);
    return nullptr;
  }
  memcpy(at, &r, sizeof r);
  return o;
}

PyObject* set_types(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 5)) return nullptr;
  PyObject** to[5] = {&g_void_p, &g_view, &g_policy, &g_batch, &g_stream};
  for (int i = 0; i < 5; ++i) {
    if (!PyType_Check(v[i])) {
      PyErr_SetString(PyExc_TypeError, "types are needed");
      return nullptr;
    }
    Py_INCREF(v[i]);
    Py_XDECREF(*to[i]);
    *to[i] = v[i];
  }
  Py_RETURN_NONE;
}

PyObject* set_function(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (!count_is(n, 2)) return nullptr;
  static const char* names[kFns] = {"ta_compress", "ta_compress_lse", "ta_compress_scores", "ta_stream_step",
                                    "ta_detect_embedding", "ta_sponsor_mask_conf"};
  const char* name = PyUnicode_AsUTF8(v[0]);
  if (!name) return nullptr;
  for (int i = 0; i < kFns; ++i)
    if (!strcmp(name, names[i])) {
      if (!pointer(v[1], &g_fn[i])) return nullptr;
      Py_RETURN_NONE;
    }
  PyErr_Format(PyExc_KeyError, "%s", name);
  return nullptr;
}

#define TA_METHOD(name, f, doc) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)), METH_FASTCALL, doc}
PyMethodDef methods[] = {
    TA_METHOD("set_types", set_types, "c_void_p and the structures view, policy, batch, stream"),
    TA_METHOD("set_function", set_function, "name and address of an entry point"),
    TA_METHOD("view", view, "ta_bf16_view of a tensor"),
    TA_METHOD("ta_compress", compress, "status of the call"),
    TA_METHOD("ta_compress_lse", compress_lse, "status of the call"),
    TA_METHOD("ta_compress_scores", compress_scores, "status of the call"),
    TA_METHOD("ta_stream_step", stream_step, "status of the call"),
    TA_METHOD("ta_detect_embedding", detect, "status of the call"),
    TA_METHOD("ta_sponsor_mask_conf", mask_conf, "status of the call"),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_ta_call", "argument marshalling for libta.so", -1, methods, nullptr, nullptr,
                      nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__ta_call() {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  g_stride = PyUnicode_InternFromString("stride");
  g_ctypes = PyUnicode_InternFromString("ctypes");
  g_data = PyUnicode_InternFromString("data");
  return PyModule_Create(&module);
}
