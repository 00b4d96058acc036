// Native call path of the Python binding for the entry points that run once per layer, block or token: argument
// conversion and the call itself, without ctypes. A call takes tensor addresses, sizes and torch's stride tuples and returns
// the status. One decoded token through 32 layers whose kernels take 5 us each was bound by the host at 8.2 us a layer.
// What ctypes takes is taken: for a number whatever says that it is an integer (__index__: numpy's integers, tensors of one element),
// modulo the width of the parameter, for a pointer an int; the interpreter lock is released during the call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>

#include "../../include/laser_kv.h"

namespace {

decltype(&laser_kv_select_block) f_select_block;
decltype(&laser_kv_select_tail) f_select_tail;
decltype(&laser_kv_decode_attention) f_decode_attention;
decltype(&laser_kv_two_stage_topk) f_two_stage_topk;
decltype(&laser_kv_gather_append) f_gather_append;
decltype(&laser_kv_window_scores) f_window_scores;
decltype(&laser_kv_collision_counts) f_collision_counts;
decltype(&laser_kv_consensus_accumulate) f_consensus_accumulate;

// The arguments of one call, taken in order; a failed conversion leaves a Python error.
struct Args {
  PyObject* const* p;
  bool ok = true;
  long long integer(PyObject* o) {
    if (!ok) return 0;
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) ok = false;
    return (long long)v;
  }
  long long i64() { return integer(*p++); }
  int32_t i32() { return (int32_t)i64(); }
  void* ptr() {
    PyObject* o = *p++;
    if (ok && !PyLong_Check(o)) {
      PyErr_Format(PyExc_TypeError, "address expected as int instead of %s", Py_TYPE(o)->tp_name);
      ok = false;
    }
    return reinterpret_cast<void*>(integer(o));
  }
  float f32() {
    PyObject* o = *p++;
    if (!ok) return 0.f;
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) ok = false;
    return (float)v;
  }
  template <int N>
  void strides(int64_t (&s)[N]) {
    PyObject* t = *p++;
    if (!PyTuple_Check(t) || PyTuple_GET_SIZE(t) < N) {
      if (ok) PyErr_Format(PyExc_ValueError, "expected at least %d strides", N);
      ok = false;
      return;
    }
    for (int i = 0; i < N; ++i) s[i] = integer(PyTuple_GET_ITEM(t, i));
  }
};

bool count_is(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return false;
}

template <typename F>
PyObject* call(const Args& a, F&& f) {
  if (!a.ok) return nullptr;
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = (int)f();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(status);
}

template <typename F>
PyObject* select(F f, PyObject* const* argv, Py_ssize_t n) {
  if (!count_is(n, 9)) return nullptr;
  Args a{argv};
  auto h = static_cast<laser_kv_handle_t>(a.ptr());
  const int32_t layer = a.i32();
  void *k = a.ptr(), *v = a.ptr(), *q = a.ptr();
  int64_t ks[3] = {0, 0, 0}, qs[3] = {0, 0, 0};
  a.strides(ks);
  a.strides(qs);
  const int32_t count = a.i32();
  void* stream = a.ptr();
  return call(a, [&] { return f(h, layer, k, v, q, ks, qs, count, stream); });
}
PyObject* py_select_block(PyObject*, PyObject* const* argv, Py_ssize_t n) { return select(f_select_block, argv, n); }
PyObject* py_select_tail(PyObject*, PyObject* const* argv, Py_ssize_t n) { return select(f_select_tail, argv, n); }

PyObject* py_decode_attention(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  if (!count_is(n, 9)) return nullptr;
  Args a{argv};
  auto h = static_cast<laser_kv_handle_t>(a.ptr());
  const int32_t layer = a.i32();
  void* q = a.ptr();
  int64_t qs[2] = {0, 0};
  a.strides(qs);
  const float scale = a.f32();
  float* out = static_cast<float*>(a.ptr());
  void* scratch = a.ptr();
  const size_t bytes = (size_t)a.i64();
  void* stream = a.ptr();
  return call(a, [&] { return f_decode_attention(h, layer, q, qs, scale, out, scratch, bytes, stream); });
}

PyObject* py_two_stage_topk(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  if (!count_is(n, 9)) return nullptr;
  Args a{argv};
  auto s = static_cast<const float*>(a.ptr());
  auto c = static_cast<const uint32_t*>(a.ptr());
  const int32_t n_seg = a.i32(), S = a.i32(), anchors = a.i32(), ke = a.i32(), kl = a.i32();
  auto idx = static_cast<int32_t*>(a.ptr());
  void* stream = a.ptr();
  return call(a, [&] { return f_two_stage_topk(s, c, n_seg, S, anchors, ke, kl, idx, stream); });
}

PyObject* py_gather_append(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  if (!count_is(n, 18)) return nullptr;
  Args a{argv};
  void *k = a.ptr(), *v = a.ptr();
  const int64_t seg = a.i64(), row = a.i64();
  const int32_t rows = a.i32();
  auto idx = static_cast<const int32_t*>(a.ptr());
  const int32_t n_seg = a.i32(), keep = a.i32();
  void *kd = a.ptr(), *vd = a.ptr();
  const int64_t dseg = a.i64(), cap = a.i64();
  auto pos = static_cast<int32_t*>(a.ptr());
  const int64_t pseg = a.i64(), off = a.i64();
  const int32_t base = a.i32();
  auto status = static_cast<int32_t*>(a.ptr());
  void* stream = a.ptr();
  return call(a, [&] { return f_gather_append(k, v, seg, row, rows, idx, n_seg, keep, kd, vd, dseg, cap, pos, pseg, off, base, status, stream); });
}

PyObject* py_window_scores(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  if (!count_is(n, 15)) return nullptr;
  Args a{argv};
  void *k = a.ptr(), *q = a.ptr();
  int64_t ks[3] = {0, 0, 0}, qs[3] = {0, 0, 0};
  a.strides(ks);
  a.strides(qs);
  const int32_t batch = a.i32(), hq = a.i32(), hkv = a.i32(), S = a.i32(), w = a.i32(), nb = a.i32();
  const float scale = a.f32();
  void* scratch = a.ptr();
  const size_t bytes = (size_t)a.i64();
  float* out = static_cast<float*>(a.ptr());
  void* stream = a.ptr();
  return call(a, [&] { return f_window_scores(k, q, ks, qs, batch, hq, hkv, S, w, nb, scale, scratch, bytes, out, stream); });
}

PyObject* py_collision_counts(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  if (!count_is(n, 17)) return nullptr;
  Args a{argv};
  void *k = a.ptr(), *q = a.ptr(), *planes = a.ptr();
  int64_t ks[3] = {0, 0, 0}, qs[3] = {0, 0, 0};
  a.strides(ks);
  a.strides(qs);
  const int32_t batch = a.i32(), hq = a.i32(), hkv = a.i32(), S = a.i32(), w = a.i32(), nb = a.i32(), bits = a.i32(), tables = a.i32();
  void* scratch = a.ptr();
  const size_t bytes = (size_t)a.i64();
  auto out = static_cast<uint32_t*>(a.ptr());
  void* stream = a.ptr();
  return call(a, [&] { return f_collision_counts(k, q, planes, ks, qs, batch, hq, hkv, S, w, nb, bits, tables, scratch, bytes, out, stream); });
}

PyObject* py_consensus_accumulate(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  if (!count_is(n, 10)) return nullptr;
  Args a{argv};
  auto s = static_cast<const float*>(a.ptr());
  auto c = static_cast<const uint32_t*>(a.ptr());
  const int32_t batch = a.i32(), heads = a.i32(), nb = a.i32(), S = a.i32(), carry = a.i32();
  auto sa = static_cast<float*>(a.ptr());
  auto ca = static_cast<uint32_t*>(a.ptr());
  void* stream = a.ptr();
  return call(a, [&] { return f_consensus_accumulate(s, c, batch, heads, nb, S, carry, sa, ca, stream); });
}

template <typename F>
bool resolve(void* lib, const char* name, F& f) {
  f = reinterpret_cast<F>(dlsym(lib, name));
  if (f) return true;
  PyErr_Format(PyExc_OSError, "%s not found in the library", name);
  return false;
}

// setup(path): the library whose functions are called (already loaded by then).
PyObject* py_setup(PyObject*, PyObject* path) {
  const char* name = PyUnicode_AsUTF8(path);
  if (!name) return nullptr;
  void* lib = dlopen(name, RTLD_NOW);
  if (!lib) return PyErr_Format(PyExc_OSError, "%s", dlerror());
  if (!resolve(lib, "laser_kv_select_block", f_select_block) || !resolve(lib, "laser_kv_select_tail", f_select_tail) ||
      !resolve(lib, "laser_kv_decode_attention", f_decode_attention) || !resolve(lib, "laser_kv_two_stage_topk", f_two_stage_topk) ||
      !resolve(lib, "laser_kv_gather_append", f_gather_append) || !resolve(lib, "laser_kv_window_scores", f_window_scores) ||
      !resolve(lib, "laser_kv_collision_counts", f_collision_counts) ||
      !resolve(lib, "laser_kv_consensus_accumulate", f_consensus_accumulate))
    return nullptr;
  Py_RETURN_NONE;
}

#define LKV_FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {{"setup", py_setup, METH_O, nullptr},
                         LKV_FAST(select_block),
                         LKV_FAST(select_tail),
                         LKV_FAST(decode_attention),
                         LKV_FAST(two_stage_topk),
                         LKV_FAST(gather_append),
                         LKV_FAST(window_scores),
                         LKV_FAST(collision_counts),
                         LKV_FAST(consensus_accumulate),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pycall(void) { return PyModule_Create(&module); }
