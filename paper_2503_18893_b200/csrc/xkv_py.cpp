// CPython module over the C ABI for the calls of a decode step and the other per-prompt calls (argument marshalling
// only).  A decode step is a handful of kernels of a few microseconds each, so what a call costs on the host is part
// of its latency: through ctypes and torch.cuda.current_stream() a call spent 4.5 us before its first launch, here
// 0.7 us.  The quantiser's calls, whose kernels take as long as their launches, allocate their results here too (10.5 us of
// host time for a pair of torch.empty and a launch through Python, 5 us here).  Tensor arguments are anything with a
// data_ptr() method (or None, or an integer address); a stream is None (torch's current one), an object with a
// cuda_stream attribute, or something that int() takes.  Every function returns the status.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "xkv.h"

namespace {

PyObject *s_data_ptr, *s_cuda_stream;      // interned attribute names
PyObject *g_get_device, *g_get_stream;     // torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream

// Cursor over the arguments of a call; `bad` is set (with a Python exception) by the first one that does not convert.
struct Args {
  PyObject* const* v;
  Py_ssize_t n, at;
  bool bad;
  Args(PyObject* const* args, Py_ssize_t have, Py_ssize_t want) : v(args), n(have), at(0), bad(false) {
    if (have != want) {
      PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, have);
      bad = true;
    }
  }
  PyObject* next() { return bad ? nullptr : v[at++]; }
  void* address(PyObject* o) {
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) bad = true;
    return p;
  }
  void* ptr() {
    PyObject* o = next();
    if (!o || o == Py_None) return nullptr;
    if (PyLong_Check(o)) return address(o);
    PyObject* r = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!r) { bad = true; return nullptr; }
    void* p = address(r);
    Py_DECREF(r);
    return p;
  }
  long long i64() {
    PyObject* o = next();
    if (!o) return 0;
    const long long x = PyLong_AsLongLong(o);
    if (x == -1 && PyErr_Occurred()) bad = true;
    return x;
  }
  int i32() {
    const long long x = i64();
    if (!bad && (x < INT32_MIN || x > INT32_MAX)) {
      PyErr_SetString(PyExc_OverflowError, "integer argument does not fit 32 bits");
      bad = true;
    }
    return (int)x;
  }
  void* stream() {
    PyObject* o = next();
    if (!o) return nullptr;
    if (PyLong_Check(o)) return address(o);
    PyObject* r;
    if (o == Py_None) {
      PyObject* dev = PyObject_CallNoArgs(g_get_device);
      if (!dev) { bad = true; return nullptr; }
      r = PyObject_CallOneArg(g_get_stream, dev);
      Py_DECREF(dev);
    } else {
      r = PyObject_GetAttr(o, s_cuda_stream);
      if (!r && PyErr_ExceptionMatches(PyExc_AttributeError)) {      // anything int() takes, such as numpy's integers
        PyErr_Clear();
        r = PyNumber_Long(o);
      }
    }
    if (!r) { bad = true; return nullptr; }
    void* p = address(r);
    Py_DECREF(r);
    return p;
  }
};

#define XKV_PY(name, want) \
  PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs) { \
    Args a(args, nargs, want);
#define XKV_PY_END(call) \
    if (a.bad) return nullptr; \
    int st; \
    Py_BEGIN_ALLOW_THREADS st = call; \
    Py_END_ALLOW_THREADS \
    return PyLong_FromLong(st); \
  }

XKV_PY(sr_select, 8)
  xkv_group* g = (xkv_group*)a.ptr();
  const int l0 = a.i32(), l1 = a.i32();
  void* q = a.ptr();
  const int k = a.i32();
  int32_t* idx = (int32_t*)a.ptr();
  int32_t* cnt = (int32_t*)a.ptr();
  void* s = a.stream();
XKV_PY_END(xkv_sr_select(g, l0, l1, q, k, idx, cnt, s))

XKV_PY(sr_select_static, 15)
  xkv_select_static_config cfg;
  cfg.struct_size = sizeof(cfg);
  cfg.G = a.i32(); cfg.batch = a.i32(); cfg.T = a.i32(); cfg.H_kv = a.i32(); cfg.H_q = a.i32(); cfg.d_h = a.i32();
  cfg.chunk = a.i32();
  cfg.landmarks = a.ptr();
  const int l0 = a.i32(), l1 = a.i32();
  void* q = a.ptr();
  const int k = a.i32();
  int32_t* idx = (int32_t*)a.ptr();
  int32_t* cnt = (int32_t*)a.ptr();
  void* s = a.stream();
XKV_PY_END(xkv_sr_select_static(&cfg, l0, l1, q, k, idx, cnt, s))

XKV_PY(sr_reconstruct_attend, 10)
  xkv_group* g = (xkv_group*)a.ptr();
  const int l0 = a.i32(), l1 = a.i32();
  void* q = a.ptr();
  const int32_t* idx = (const int32_t*)a.ptr();
  const int32_t* cnt = (const int32_t*)a.ptr();
  const int k_cap = a.i32();
  void* out = a.ptr();
  float* lse = (float*)a.ptr();
  void* s = a.stream();
XKV_PY_END(xkv_sr_reconstruct_attend(g, l0, l1, q, idx, cnt, k_cap, out, lse, s))

XKV_PY(sr_reconstruct_attend_tail, 16)
  xkv_group* g = (xkv_group*)a.ptr();
  const int l0 = a.i32(), l1 = a.i32();
  void* q = a.ptr();
  const int32_t* idx = (const int32_t*)a.ptr();
  const int32_t* cnt = (const int32_t*)a.ptr();
  const int k_cap = a.i32();
  void* tk = a.ptr();
  void* tv = a.ptr();
  const int32_t* len = (const int32_t*)a.ptr();
  const int cap = a.i32();
  void* ws = a.ptr();
  const uint64_t ws_bytes = (uint64_t)a.i64();
  void* out = a.ptr();
  float* lse = (float*)a.ptr();
  void* s = a.stream();
XKV_PY_END(xkv_sr_reconstruct_attend_tail(g, l0, l1, q, idx, cnt, k_cap, tk, tv, len, cap, ws, ws_bytes, out, lse, s))

XKV_PY(dense_attend, 13)
  xkv_group* g = (xkv_group*)a.ptr();
  const int l0 = a.i32(), l1 = a.i32();
  void* q = a.ptr();
  void* K = a.ptr();
  void* V = a.ptr();
  const int32_t* len = (const int32_t*)a.ptr();
  const int cap = a.i32();
  void* ws = a.ptr();
  const uint64_t ws_bytes = (uint64_t)a.i64();
  void* out = a.ptr();
  float* lse = (float*)a.ptr();
  void* s = a.stream();
XKV_PY_END(xkv_dense_attend(g, l0, l1, q, K, V, len, cap, ws, ws_bytes, out, lse, s))

// The interpreter lock is given back for a scope: an allocation or a launch may wait for the device (a full launch queue),
// and the device for another Python thread.
struct WithoutGil {
  PyThreadState* state = PyEval_SaveThread();
  WithoutGil() = default;
  WithoutGil(const WithoutGil&) = delete;
  WithoutGil& operator=(const WithoutGil&) = delete;
  ~WithoutGil() { PyEval_RestoreThread(state); }
};

// An uninitialised tensor of x's device with x's leading sizes and `last` columns.
at::Tensor like(const at::Tensor& x, int64_t last, at::ScalarType type) {
  c10::DimVector sizes(x.sizes().begin(), x.sizes().end());
  sizes.back() = last;
  return at::empty(sizes, x.options().dtype(type));
}
const at::Tensor* tensor(PyObject* o) {
  if (!THPVariable_Check(o) || THPVariable_Unpack(o).dim() < 1) {
    PyErr_SetString(PyExc_TypeError, "expected a tensor of at least one dimension");
    return nullptr;
  }
  return &THPVariable_Unpack(o);
}

// quantize_rtn(x, bits, stream) -> (status, codes, meta or None)
PyObject* quantize_rtn(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  Args a(args, nargs, 3);
  const at::Tensor* x = a.bad ? nullptr : tensor(a.next());
  if (!x) return nullptr;
  const int bits = a.i32();
  void* s = a.stream();
  if (a.bad) return nullptr;
  HANDLE_TH_ERRORS
  at::Tensor codes, meta;
  int st;
  {
    const WithoutGil no_gil;
    const int64_t cols = x->size(-1), rows = cols ? x->numel() / cols : 0;
    codes = like(*x, cols / 2, at::kByte);
    // 4 bits: one scale/offset word per group beside the codes; 3 bits: the 16-byte records hold them
    if (bits == 4) meta = like(*x, cols / 32, at::kInt);
    st = xkv_quantize_rtn(x->const_data_ptr(), rows, cols > INT32_MAX ? 0 : (int)cols, bits, codes.mutable_data_ptr(),
                          bits == 4 ? meta.mutable_data_ptr() : nullptr, s);
  }
  return Py_BuildValue("iNN", st, THPVariable_Wrap(codes), bits == 4 ? THPVariable_Wrap(meta) : Py_NewRef(Py_None));
  END_HANDLE_TH_ERRORS
}

// dequantize_rtn(codes, meta, bits, stream) -> (status, x)
PyObject* dequantize_rtn(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  Args a(args, nargs, 4);
  const at::Tensor* codes = a.bad ? nullptr : tensor(a.next());
  if (!codes) return nullptr;
  void* meta = a.ptr();
  const int bits = a.i32();
  void* s = a.stream();
  if (a.bad) return nullptr;
  HANDLE_TH_ERRORS
  at::Tensor x;
  int st;
  {
    const WithoutGil no_gil;
    const int64_t half = codes->size(-1), rows = half ? codes->numel() / half : 0;
    x = like(*codes, half * 2, at::kBFloat16);
    st = xkv_dequantize_rtn(codes->const_data_ptr(), meta, rows, half > INT32_MAX / 2 ? 0 : (int)(half * 2), bits,
                            x.mutable_data_ptr(), s);
  }
  return Py_BuildValue("iN", st, THPVariable_Wrap(x));
  END_HANDLE_TH_ERRORS
}

// torch_hooks(get_device, get_current_raw_stream): how "the current stream" is found.
PyObject* torch_hooks(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs != 2) { PyErr_SetString(PyExc_TypeError, "expected 2 arguments"); return nullptr; }
  Py_INCREF(args[0]);
  Py_INCREF(args[1]);
  Py_XSETREF(g_get_device, args[0]);
  Py_XSETREF(g_get_stream, args[1]);
  Py_RETURN_NONE;
}

#define XKV_DEF(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {XKV_DEF(sr_select), XKV_DEF(sr_select_static), XKV_DEF(sr_reconstruct_attend),
                         XKV_DEF(sr_reconstruct_attend_tail), XKV_DEF(dense_attend), XKV_DEF(quantize_rtn),
                         XKV_DEF(dequantize_rtn), XKV_DEF(torch_hooks), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_xkv", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__xkv(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_data_ptr || !s_cuda_stream) return nullptr;
  return PyModule_Create(&module);
}
