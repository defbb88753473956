// Host path of the calls a decode or prefill loop makes once per linear: argument checks, output and workspace allocation,
// the current stream, and the call into libstb.so, without the interpreter.  (Through ctypes a GEMV call cost 17 us on the
// host, twice what its kernel takes.)
//
// Every function takes the Python function's arguments by position and either does the whole call or, where an argument is
// not the plain case, hands all of them to the Python form it was given at start-up (which takes every case, and raises
// what it always raised).
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/stb.h"

namespace {

// entry points of libstb.so, by address (the library is loaded by the Python side)
decltype(&stb_gemv) f_gemv;
decltype(&stb_gemm_workspace) f_gemm_workspace;
decltype(&stb_gemm) f_gemm;
decltype(&stb_gemm_f16_workspace) f_gemm_f16_workspace;
decltype(&stb_gemm_f16) f_gemm_f16;
decltype(&stb_layer_stack) f_layer_stack;
decltype(&stb_layer_stack_resident) f_layer_stack_resident;
PyObject* on_error;                   // callable(status, where): raises
PyObject *s_n, *s_m, *s_N, *s_buf, *s_dev_status, *s_cuda_stream;

struct Layer {
  int n, m, N;
  const void* buf;
  int* dev_status;
};

bool int_attr(PyObject* o, PyObject* name, int& out) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (!v) return false;
  const long x = PyLong_Check(v) ? PyLong_AsLong(v) : -1;
  Py_DECREF(v);
  out = (int)x;
  return x >= 0 && x <= 0x7FFFFFFF;
}
// false (no Python error left behind) where the object is not the plain case
bool layer_of(PyObject* o, Layer& l) {
  bool ok = int_attr(o, s_n, l.n) && int_attr(o, s_m, l.m) && int_attr(o, s_N, l.N);
  PyObject* b = ok ? PyObject_GetAttr(o, s_buf) : nullptr;
  PyObject* d = b ? PyObject_GetAttr(o, s_dev_status) : nullptr;
  ok = d && THPVariable_Check(b) && (d == Py_None || THPVariable_Check(d));
  if (ok) {
    l.buf = THPVariable_Unpack(b).data_ptr();
    l.dev_status = d == Py_None ? nullptr : static_cast<int*>(THPVariable_Unpack(d).data_ptr());
  }
  Py_XDECREF(b);
  Py_XDECREF(d);
  PyErr_Clear();
  return ok;
}
// the stream argument, or the current stream of the current device
bool stream_of(PyObject* o, void*& s) {
  if (o == Py_None) {
    s = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  PyObject* v = PyObject_GetAttr(o, s_cuda_stream);
  if (!v) { PyErr_Clear(); return false; }
  s = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  if (PyErr_Occurred()) { PyErr_Clear(); return false; }
  return true;
}
bool rows_of(PyObject* o, at::ScalarType t, bool vector_too, at::Tensor& x) {
  if (!THPVariable_Check(o)) return false;
  x = THPVariable_Unpack(o);
  return x.scalar_type() == t && x.is_cuda() && ((x.dim() == 2 && x.stride(1) == 1) || (vector_too && x.dim() == 1 && x.stride(0) == 1));
}
// A tensor that the call makes for itself, on the launch stream: its memory belongs to that stream's pool, so that nothing else is
// given it while the call still runs.  `kept`: one that the caller gets, and reads as a rule on the current stream.
at::Tensor make(at::IntArrayRef size, const at::TensorOptions& options, void* s, bool kept) {
  const c10::DeviceIndex dev = options.device().index();
  const c10::cuda::CUDAStream current = c10::cuda::getCurrentCUDAStream(dev);
  if (current.stream() == static_cast<cudaStream_t>(s)) return at::empty(size, options);
  const c10::cuda::CUDAStreamGuard guard(c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(s), dev));
  at::Tensor t = at::empty(size, options);
  if (kept) c10::cuda::CUDACachingAllocator::recordStream(t.storage().data_ptr(), current);
  return t;
}
// output: the given tensor (two-dimensional, of type 32 or 16), or a new one of the asked type
bool output_of(PyObject* out, PyObject* out_dtype, at::ScalarType t16, int64_t rows, int64_t n, const at::Tensor& like, void* s, at::Tensor& y) {
  if (out != Py_None) {
    if (!THPVariable_Check(out)) return false;
    y = THPVariable_Unpack(out);
    return y.dim() == 2 && (y.scalar_type() == at::kFloat || y.scalar_type() == t16);
  }
  at::ScalarType t = at::kFloat;
  if (out_dtype != Py_None) {
    if (!THPDtype_Check(out_dtype)) return false;
    t = reinterpret_cast<THPDtype*>(out_dtype)->scalar_type;
    if (t != at::kFloat && t != t16) return false;
  }
  y = make({rows, n}, like.options().dtype(t), s, true);
  return true;
}
stb_dtype dtype_code(at::ScalarType t) { return t == at::kFloat ? STB_F32 : (t == at::kHalf ? STB_F16 : STB_BF16); }

// the call itself runs without the interpreter's lock (a launch can wait for room in the stream's queue)
template <class F>
int unlocked(F call) {
  PyThreadState* t = PyEval_SaveThread();
  const int rc = call();
  PyEval_RestoreThread(t);
  return rc;
}

PyObject* failed(int rc, const char* where) {
  PyObject* r = PyObject_CallFunction(on_error, "is", rc, where);
  Py_XDECREF(r);
  if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, where);
  return nullptr;
}
PyObject* wrap(const at::Tensor& t) { return THPVariable_Wrap(t); }

// what the Python forms are called with where the plain case does not hold
PyObject* slow[5];
PyObject* pass_on(int which, PyObject* const* args, Py_ssize_t n) { return PyObject_Vectorcall(slow[which], args, (size_t)n, nullptr); }
// where torch threw (no device, no memory, a tensor without storage; nothing was launched): the Python form raises what it raises
PyObject* threw(int which, PyObject* const* args, Py_ssize_t n) {
  PyErr_Clear();
  return pass_on(which, args, n);
}

// gemv(layer, x, out, out_dtype, stream): 17.0 us of host time per call through ctypes, 6.6 us here (1024 x 8192), of which the launch is the larger part
PyObject* bind_gemv(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Layer l;
  at::Tensor x, y;
  void* s;
  if (n != 5) return pass_on(0, a, n);
  try {
    if (!layer_of(a[0], l) || !rows_of(a[1], at::kHalf, true, x)) return pass_on(0, a, n);
    const bool vec = x.dim() == 1;
    const int64_t batch = vec ? 1 : x.size(0);
    if (!stream_of(a[4], s) || !output_of(a[2], a[3], at::kHalf, batch, l.n, x, s, y)) return pass_on(0, a, n);
    const void* xp = x.data_ptr();
    void* yp = y.data_ptr();
    const size_t ldx = (size_t)(vec ? x.size(0) : x.stride(0)), ldy = (size_t)y.stride(0);
    const stb_dtype dt = dtype_code(y.scalar_type());
    const int rc = unlocked([&] { return f_gemv(l.buf, l.n, l.m, l.N, xp, (int)batch, ldx, yp, dt, ldy, l.dev_status, s); });
    if (rc != STB_OK) return failed(rc, "stb_gemv");
    if (vec) return wrap(y.select(0, 0));
    if (a[2] != Py_None) { Py_INCREF(a[2]); return a[2]; }
    return wrap(y);
  } catch (const std::exception&) {
    return threw(0, a, n);
  }
}

// gemm(layer, X, out, out_dtype, ws, stream) and gemm_f16
template <bool kF16>
PyObject* bind_gemm(PyObject*, PyObject* const* a, Py_ssize_t n) {
  constexpr int which = kF16 ? 2 : 1;
  constexpr at::ScalarType t16 = kF16 ? at::kHalf : at::kBFloat16;
  Layer l;
  at::Tensor x, y, ws;
  void* s;
  if (n != 6) return pass_on(which, a, n);
  try {
    if (!layer_of(a[0], l) || !rows_of(a[1], t16, false, x) || !stream_of(a[5], s)) return pass_on(which, a, n);
    const int64_t T = x.size(0);
    size_t need = 0;
    if ((kF16 ? f_gemm_f16_workspace : f_gemm_workspace)(l.n, l.m, l.N, (int)T, &need) != STB_OK) return pass_on(which, a, n);
    if (a[4] != Py_None) {
      if (!THPVariable_Check(a[4])) return pass_on(which, a, n);
      ws = THPVariable_Unpack(a[4]);
    }
    if (!output_of(a[2], a[3], t16, T, l.n, x, s, y)) return pass_on(which, a, n);
    if (!ws.defined() || (size_t)ws.nbytes() < need) ws = make({(int64_t)(need < 256 ? 256 : need)}, x.options().dtype(at::kByte), s, false);
    const void* xp = x.data_ptr();
    void *yp = y.data_ptr(), *wp = ws.data_ptr();
    const size_t ldx = (size_t)x.stride(0), ldy = (size_t)y.stride(0), wb = (size_t)ws.nbytes();
    const stb_dtype dt = dtype_code(y.scalar_type());
    const int rc = unlocked([&] { return (kF16 ? f_gemm_f16 : f_gemm)(l.buf, l.n, l.m, l.N, xp, (int)T, ldx, yp, dt, ldy, wp, wb, l.dev_status, s); });
    if (rc != STB_OK) return failed(rc, kF16 ? "stb_gemm_f16" : "stb_gemm");
    if (a[2] != Py_None) { Py_INCREF(a[2]); return a[2]; }
    return wrap(y);
  } catch (const std::exception&) {
    return threw(which, a, n);
  }
}

bool status_of(PyObject* o, int*& p) {
  p = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) return false;
  p = static_cast<int*>(THPVariable_Unpack(o).data_ptr());
  return true;
}
// The marshalled steps of a list call (a ctypes array of stb_step).
struct Steps {
  Py_buffer b;
  const stb_step* data = nullptr;
  int count = 0;
  explicit Steps(PyObject* o) {
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) { PyErr_Clear(); return; }
    if (b.len % sizeof(stb_step)) { PyBuffer_Release(&b); return; }
    data = static_cast<const stb_step*>(b.buf);
    count = (int)(b.len / sizeof(stb_step));
    held = true;
  }
  ~Steps() { if (held) PyBuffer_Release(&b); }
  bool held = false;
};
// layer_stack(steps, dev_status, stream, marshalled)
PyObject* bind_layer_stack(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void* s;
  int* st;
  try {
    if (n != 4 || a[3] == Py_None || !stream_of(a[2], s) || !status_of(a[1], st)) return pass_on(3, a, n);
    const Steps steps(a[3]);
    if (!steps.held) return pass_on(3, a, n);
    const int rc = unlocked([&] { return f_layer_stack(steps.data, steps.count, st, s); });
    if (rc != STB_OK) return failed(rc, "stb_layer_stack");
    Py_RETURN_NONE;
  } catch (const std::exception&) {
    return threw(3, a, n);
  }
}
// layer_stack_resident(steps, ws, dev_status, stream, marshalled, selftest)
PyObject* bind_layer_stack_resident(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void* s;
  int* st;
  try {
    if (n != 6 || a[4] == Py_None || a[5] != Py_False || !THPVariable_Check(a[1]) || !stream_of(a[3], s) || !status_of(a[2], st)) return pass_on(4, a, n);
    const at::Tensor& ws = THPVariable_Unpack(a[1]);
    void* wp = ws.data_ptr();
    const size_t wb = (size_t)ws.numel();
    const Steps steps(a[4]);
    if (!steps.held) return pass_on(4, a, n);
    const int rc = unlocked([&] { return f_layer_stack_resident(steps.data, steps.count, wp, wb, st, s); });
    if (rc != STB_OK) return failed(rc, "stb_layer_stack_resident");
    Py_RETURN_NONE;
  } catch (const std::exception&) {
    return threw(4, a, n);
  }
}

// start(addresses of the seven entry points in the order above, on_error, the five Python forms)
PyObject* bind_start(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 13) { PyErr_SetString(PyExc_TypeError, "start takes 13 arguments"); return nullptr; }
  void* p[7];
  for (int i = 0; i < 7; ++i) p[i] = PyLong_AsVoidPtr(a[i]);
  if (PyErr_Occurred()) return nullptr;
  f_gemv = reinterpret_cast<decltype(f_gemv)>(p[0]);
  f_gemm_workspace = reinterpret_cast<decltype(f_gemm_workspace)>(p[1]);
  f_gemm = reinterpret_cast<decltype(f_gemm)>(p[2]);
  f_gemm_f16_workspace = reinterpret_cast<decltype(f_gemm_f16_workspace)>(p[3]);
  f_gemm_f16 = reinterpret_cast<decltype(f_gemm_f16)>(p[4]);
  f_layer_stack = reinterpret_cast<decltype(f_layer_stack)>(p[5]);
  f_layer_stack_resident = reinterpret_cast<decltype(f_layer_stack_resident)>(p[6]);
  Py_INCREF(a[7]);
  on_error = a[7];
  for (int i = 0; i < 5; ++i) { Py_INCREF(a[8 + i]); slow[i] = a[8 + i]; }
  Py_RETURN_NONE;
}

#define FAST(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fn)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST("start", bind_start), FAST("gemv", bind_gemv), FAST("gemm", bind_gemm<false>), FAST("gemm_f16", bind_gemm<true>),
                         FAST("layer_stack", bind_layer_stack), FAST("layer_stack_resident", bind_layer_stack_resident), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_stb_bind", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__stb_bind(void) {
  s_n = PyUnicode_InternFromString("n"); s_m = PyUnicode_InternFromString("m"); s_N = PyUnicode_InternFromString("N");
  s_buf = PyUnicode_InternFromString("buf"); s_dev_status = PyUnicode_InternFromString("dev_status"); s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  return PyModule_Create(&module);
}
