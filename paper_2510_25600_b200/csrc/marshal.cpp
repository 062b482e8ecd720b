// Argument marshalling of the hot entry points for Python (the module `_marshal`): each function takes device pointers as
// integers, descriptors and host arrays as objects with the buffer protocol (ctypes structures, numpy arrays), calls the C
// entry point of the same name with the GIL released and returns its status.  No step of the method runs here.
// A call through ctypes with numpy's pointer conversion cost 12-25 us of host time, several times the kernel behind it for
// one decode step; this way it is the launch itself (about 3 us) and 1-2 us of Python.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "purekv.h"

namespace {

// The positional arguments of one call, read in order; `ok` goes false (with a Python error set) at the first that does not fit.
class Args {
 public:
  Args(const char* name, PyObject* const* v, Py_ssize_t n, Py_ssize_t want) : v_(v), n_(n) {
    if (n != want) {
      PyErr_Format(PyExc_TypeError, "%s: %zd arguments, got %zd", name, want, n);
      ok = false;
    }
  }
  ~Args() {
    for (int i = 0; i < n_buf_; ++i) PyBuffer_Release(&buf_[i]);
  }
  Args(const Args&) = delete;
  Args& operator=(const Args&) = delete;

  void* ptr() {  // an address, or None
    PyObject* o = next();
    if (!ok || o == Py_None) return nullptr;
    void* p = PyLong_AsVoidPtr(o);
    if (p == nullptr && PyErr_Occurred()) ok = false;
    return p;
  }
  long long integer() {
    PyObject* o = next();
    if (!ok) return 0;
    const long long x = PyLong_AsLongLong(o);
    if (x == -1 && PyErr_Occurred()) ok = false;
    return x;
  }
  int32_t i32() {
    const long long x = integer();
    if (ok && (x < INT32_MIN || x > INT32_MAX)) {
      PyErr_SetString(PyExc_OverflowError, "value does not fit 32 bits");
      ok = false;
    }
    return (int32_t)x;
  }
  float f32() {
    PyObject* o = next();
    if (!ok) return 0.f;
    const double x = PyFloat_AsDouble(o);
    if (x == -1.0 && PyErr_Occurred()) ok = false;
    return (float)x;
  }
  // a contiguous host object of at least `bytes` bytes
  const void* host(size_t bytes) {
    PyObject* o = next();
    if (!ok) return nullptr;
    if (PyObject_GetBuffer(o, &buf_[n_buf_], PyBUF_SIMPLE) != 0) {
      ok = false;
      return nullptr;
    }
    const Py_buffer& b = buf_[n_buf_++];
    if ((size_t)b.len < bytes) {
      PyErr_Format(PyExc_ValueError, "host array of %zd bytes, need %zu", b.len, bytes);
      ok = false;
      return nullptr;
    }
    return b.buf;
  }
  const purekv_batch* batch() { return static_cast<const purekv_batch*>(host(sizeof(purekv_batch))); }
  const int32_t* ints(int64_t n) { return static_cast<const int32_t*>(host((size_t)(n > 0 ? n : 0) * sizeof(int32_t))); }

  bool ok = true;

 private:
  PyObject* next() { return ok && at_ < n_ ? v_[at_++] : (ok = false, nullptr); }
  PyObject* const* v_;
  Py_ssize_t n_, at_ = 0;
  Py_buffer buf_[4];
  int n_buf_ = 0;
};

template <typename F>
PyObject* call(F f) {
  purekv_status st;
  Py_BEGIN_ALLOW_THREADS;
  st = f();
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong((long)st);
}

PyObject* prefill(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("st_sparse_prefill", v, n, 17);
  const void *q = a.ptr(), *k = a.ptr(), *vv = a.ptr();
  void* o = a.ptr();
  float* lse = (float*)a.ptr();
  const purekv_batch* b = a.batch();
  void* plan = a.ptr();
  const purekv_plan_info* info = (const purekv_plan_info*)a.host(sizeof(purekv_plan_info));
  const int32_t h = a.i32(), hkv = a.i32(), d = a.i32(), dt = a.i32();
  const float scale = a.f32();
  void* ws = a.ptr();
  const size_t ws_bytes = (size_t)a.integer();
  int32_t* status = (int32_t*)a.ptr();
  void* stream = a.ptr();
  if (!a.ok) return nullptr;
  return call([&] {
    return purekv_st_sparse_prefill(q, k, vv, o, lse, b, plan, info, h, hkv, d, (purekv_dtype)dt, scale, ws, ws_bytes, status,
                                    stream);
  });
}

PyObject* prefill_layers(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("st_sparse_prefill_layers", v, n, 22);
  const void *q = a.ptr(), *k = a.ptr(), *vv = a.ptr();
  void* o = a.ptr();
  float* lse = (float*)a.ptr();
  const int64_t qs = a.integer(), ks = a.integer(), os = a.integer(), ls = a.integer();
  const int32_t layers = a.i32();
  const purekv_batch* b = a.batch();
  void* plan = a.ptr();
  const purekv_plan_info* info = (const purekv_plan_info*)a.host(sizeof(purekv_plan_info));
  const int32_t h = a.i32(), hkv = a.i32(), d = a.i32(), dt = a.i32();
  const float scale = a.f32();
  void* ws = a.ptr();
  const size_t ws_bytes = (size_t)a.integer();
  int32_t* status = (int32_t*)a.ptr();
  void* stream = a.ptr();
  if (!a.ok) return nullptr;
  return call([&] {
    return purekv_st_sparse_prefill_layers(q, k, vv, o, lse, qs, ks, os, ls, layers, b, plan, info, h, hkv, d, (purekv_dtype)dt,
                                           scale, ws, ws_bytes, status, stream);
  });
}

PyObject* score(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("lowlayer_score", v, n, 13);
  const void *q = a.ptr(), *k = a.ptr();
  float* c = (float*)a.ptr();
  const purekv_batch* b = a.batch();
  const int32_t window = a.i32(), h = a.i32(), hkv = a.i32(), d = a.i32(), dt = a.i32();
  const float scale = a.f32();
  void* ws = a.ptr();
  const size_t ws_bytes = (size_t)a.integer();
  void* stream = a.ptr();
  if (!a.ok) return nullptr;
  return call([&] { return purekv_lowlayer_score(q, k, c, b, window, h, hkv, d, (purekv_dtype)dt, scale, ws, ws_bytes, stream); });
}

PyObject* score_lse(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("lowlayer_score_lse", v, n, 13);
  const void *q = a.ptr(), *k = a.ptr();
  const float* lse = (const float*)a.ptr();
  float* c = (float*)a.ptr();
  const purekv_batch* b = a.batch();
  const int32_t window = a.i32(), h = a.i32(), hkv = a.i32(), d = a.i32(), dt = a.i32();
  const float scale = a.f32();
  int32_t* status = (int32_t*)a.ptr();
  void* stream = a.ptr();
  if (!a.ok) return nullptr;
  return call([&] { return purekv_lowlayer_score_lse(q, k, lse, c, b, window, h, hkv, d, (purekv_dtype)dt, scale, status, stream); });
}

PyObject* score_ex(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("lowlayer_score_ex", v, n, 15);
  const void *q = a.ptr(), *k = a.ptr();
  float* c = (float*)a.ptr();
  const purekv_batch* b = a.batch();
  const int32_t window = a.i32(), obs = a.i32(), pool = a.i32(), h = a.i32(), hkv = a.i32(), d = a.i32(), dt = a.i32();
  const float scale = a.f32();
  void* ws = a.ptr();
  const size_t ws_bytes = (size_t)a.integer();
  void* stream = a.ptr();
  if (!a.ok) return nullptr;
  return call([&] {
    return purekv_lowlayer_score_ex(q, k, c, b, window, obs, pool, h, hkv, d, (purekv_dtype)dt, scale, ws, ws_bytes, stream);
  });
}

PyObject* select_topk(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("select_topk", v, n, 18);
  const float* c = (const float*)a.ptr();
  const void* vv = a.ptr();
  const int64_t stride = a.integer();
  const int32_t layers = a.i32();
  const purekv_batch* b = a.batch();
  const int32_t window = a.i32();
  const int32_t* keep = (const int32_t*)a.ptr();
  const int32_t* h_keep = a.ints(b ? b->n_req : 0);
  const int32_t* cu = (const int32_t*)a.ptr();
  const int32_t* h_cu = a.ints(b ? (int64_t)b->n_req + 1 : 0);
  const int32_t hkv = a.i32(), d = a.i32(), dt = a.i32();
  int32_t* idx = (int32_t*)a.ptr();
  float* s = (float*)a.ptr();
  void* ws = a.ptr();
  const size_t ws_bytes = (size_t)a.integer();
  void* stream = a.ptr();
  if (!a.ok) return nullptr;
  return call([&] {
    return purekv_select_topk(c, vv, stride, layers, b, window, keep, h_keep, cu, h_cu, hkv, d, (purekv_dtype)dt, idx, s, ws,
                              ws_bytes, stream);
  });
}

PyObject* compact_kv(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("compact_kv", v, n, 15);
  const void *k = a.ptr(), *vv = a.ptr();
  const int64_t stride = a.integer();
  const int32_t layers = a.i32();
  const int32_t* idx = (const int32_t*)a.ptr();
  const purekv_batch* b = a.batch();
  const int32_t* cu = (const int32_t*)a.ptr();
  const int32_t* h_cu = a.ints(b ? (int64_t)b->n_req + 1 : 0);
  const int32_t hkv = a.i32(), d = a.i32(), dt = a.i32();
  void *ko = a.ptr(), *vo = a.ptr();
  const int64_t out_stride = a.integer();
  void* stream = a.ptr();
  if (!a.ok) return nullptr;
  return call([&] {
    return purekv_compact_kv(k, vv, stride, layers, idx, b, cu, h_cu, hkv, d, (purekv_dtype)dt, ko, vo, out_stride, stream);
  });
}

PyObject* decode(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("decode_attention", v, n, 16);
  const void *q = a.ptr(), *k = a.ptr(), *vv = a.ptr();
  void* o = a.ptr();
  float* lse = (float*)a.ptr();
  const int32_t* cu = (const int32_t*)a.ptr();
  const int32_t n_req = a.i32();
  const int32_t* h_cu = a.ints((int64_t)n_req + 1);
  const int32_t h = a.i32(), hkv = a.i32(), d = a.i32(), dt = a.i32();
  const float scale = a.f32();
  void* ws = a.ptr();
  const size_t ws_bytes = (size_t)a.integer();
  void* stream = a.ptr();
  if (!a.ok) return nullptr;
  return call([&] {
    return purekv_decode_attention(q, k, vv, o, lse, cu, h_cu, n_req, h, hkv, d, (purekv_dtype)dt, scale, ws, ws_bytes, stream);
  });
}

PyObject* plan_build_host(PyObject*, PyObject* const* v, Py_ssize_t n) {
  Args a("plan_build_layers_host", v, n, 11);
  const purekv_batch* b = a.batch();
  const purekv_st_params* p = (const purekv_st_params*)a.host(sizeof(purekv_st_params));
  const int32_t dt = a.i32(), d = a.i32(), h = a.i32(), hkv = a.i32(), n_ctas = a.i32(), layers = a.i32();
  void* out = a.ptr();
  const size_t bytes = (size_t)a.integer();
  purekv_plan_info* info = (purekv_plan_info*)a.host(sizeof(purekv_plan_info));  // (a ctypes structure: written in place)
  if (!a.ok) return nullptr;
  return call([&] { return purekv_plan_build_layers_host(b, p, (purekv_dtype)dt, d, h, hkv, n_ctas, layers, out, bytes, info); });
}

#define PK_METHOD(name, f) {name, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PK_METHOD("purekv_st_sparse_prefill", prefill), PK_METHOD("purekv_st_sparse_prefill_layers", prefill_layers),
                         PK_METHOD("purekv_lowlayer_score", score),
                         PK_METHOD("purekv_lowlayer_score_lse", score_lse), PK_METHOD("purekv_lowlayer_score_ex", score_ex),
                         PK_METHOD("purekv_select_topk", select_topk), PK_METHOD("purekv_compact_kv", compact_kv),
                         PK_METHOD("purekv_decode_attention", decode),
                         PK_METHOD("purekv_plan_build_layers_host", plan_build_host), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void) { return PyModule_Create(&module); }
