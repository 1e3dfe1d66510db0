// The usual call of binding.py in native code: tensors checked, the output allocated, the argument struct filled and the
// library entered without the interpreter in between.  What is not the usual call, or lacks a workspace, returns None and goes through
// binding.py, which checks, reports and provides one; nothing has been launched then.  What the library refuses otherwise is
// raised from here: entered again, a call could succeed and an error of CUDA's that the first entry took would be lost.
//
// A call of one head of 256 x 256 takes its kernel 4.9 us and took the host 7.1: the interpreter's part of that, attribute by attribute,
// was 3.3 us and is under 1 here (loop of calls: 7.3 -> 5.3 us; small row softmax 5.3 -> 3.5).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/jit/frontend/tracer.h>

#include <limits>

#include "attn.h"
#include "gemm.h"

namespace {

int (*g_attn)(const attn_call*) = nullptr;
int (*g_gemm)(const gemm_call*) = nullptr;
int (*g_softmax)(const softmax_call*) = nullptr;
PyObject* g_refused = nullptr;   // binding.py's: raises for (status, entry point)

// Someone looks at or stands in for the operations of a call: those are binding.py's to make.
bool watched() {
  return c10::impl::TorchDispatchModeTLS::any_modes_set() || at::impl::torch_function_mode_enabled() || torch::jit::tracer::isTracing();
}

// A plain contiguous bf16 tensor on the current CUDA device, or null.
const at::Tensor* plain(PyObject* obj, c10::DeviceIndex device) {
  if (!THPVariable_CheckExact(obj)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(obj);
  if (!t.defined()) return nullptr;
  const c10::DispatchKeySet keys = t.unsafeGetTensorImpl()->key_set();
  if (keys.has_any(c10::DispatchKeySet({c10::DispatchKey::Python, c10::DispatchKey::Functionalize, c10::DispatchKey::FuncTorchBatched,
                                        c10::DispatchKey::FuncTorchGradWrapper, c10::DispatchKey::Negative, c10::DispatchKey::Conjugate,
                                        c10::DispatchKey::ZeroTensor})))
    return nullptr;
  if (t.layout() != c10::kStrided || !t.is_cuda() || t.scalar_type() != at::kBFloat16 || t.get_device() != device || !t.has_storage() ||
      !t.is_contiguous())
    return nullptr;
  for (const int64_t n : t.sizes())
    if (n < 1 || n > std::numeric_limits<int>::max()) return nullptr;
  return &t;
}

// The current device if the first tensor of a call is on one, else -1 (no tensor is on that; without a GPU there is nothing to ask).
c10::DeviceIndex device_of_call(PyObject* first) {
  return THPVariable_CheckExact(first) && THPVariable_Unpack(first).is_cuda() ? c10::cuda::current_device() : c10::DeviceIndex(-1);
}

// Enters the library without the interpreter's lock, as ctypes does.
template <class C>
int enter(int (*fn)(const C*), const C& call) {
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = fn(&call);
  Py_END_ALLOW_THREADS
  return rc;
}
PyObject* answer(int rc, const char* where, PyObject* given, at::Tensor& made) {
  if (rc == ATTN_ERR_NEED_WORKSPACE) Py_RETURN_NONE;
  if (rc != ATTN_OK) {
    Py_XDECREF(PyObject_CallFunction(g_refused, "is", rc, where));
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, where);
    return nullptr;
  }
  if (given != Py_None) return Py_NewRef(given);
  return THPVariable_Wrap(std::move(made));
}

// attn(q, k, v, o or None, causal, whether q may have another length than k and v)
PyObject* py_attn(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 6 || !g_attn || watched()) Py_RETURN_NONE;
  const c10::DeviceIndex device = device_of_call(args[0]);
  const at::Tensor *q = plain(args[0], device), *k = plain(args[1], device), *v = plain(args[2], device);
  if (!q || !k || !v || q->dim() != 4 || k->dim() != 4 || v->dim() != 4) Py_RETURN_NONE;
  const int causal = PyObject_IsTrue(args[4]);
  if (causal < 0) return nullptr;
  const bool other_length = args[5] == Py_True;
  const auto qs = q->sizes(), ks = k->sizes();
  if (ks != v->sizes() || qs[0] != ks[0] || qs[1] != ks[1] || qs[3] != ks[3] || (!other_length && qs[2] != ks[2])) Py_RETURN_NONE;
  at::Tensor made;
  void* out;
  if (args[3] == Py_None) {
    made = at::empty_like(*q);
    out = made.data_ptr();
  } else {
    const at::Tensor* o = plain(args[3], device);
    if (!o || o->sizes() != qs) Py_RETURN_NONE;
    out = o->data_ptr();
  }
  attn_call c = {};
  c.q = q->data_ptr();
  c.k = k->data_ptr();
  c.v = v->data_ptr();
  c.o = out;
  c.cuda_stream = c10::cuda::getCurrentCUDAStream(device).stream();
  c.B = (int)qs[0];
  c.H = (int)qs[1];
  c.Lq = (int)qs[2];
  c.Lk = (int)ks[2];
  c.d = (int)qs[3];
  c.causal = causal;
  return answer(enter(g_attn, c), other_length ? "attn_forward_qk" : causal ? "attn_forward_causal" : "attn_forward", args[3], made);
  END_HANDLE_TH_ERRORS
}

// gemm(a, b, c or None, "kn" or "nk")
PyObject* py_gemm(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 4 || !g_gemm || watched()) Py_RETURN_NONE;
  const c10::DeviceIndex device = device_of_call(args[0]);
  const at::Tensor *a = plain(args[0], device), *b = plain(args[1], device);
  if (!a || !b || (a->dim() != 2 && a->dim() != 3) || (b->dim() != 2 && b->dim() != 3) || !PyUnicode_Check(args[3])) Py_RETURN_NONE;
  const bool kn = PyUnicode_CompareWithASCIIString(args[3], "kn") == 0;
  if (!kn && PyUnicode_CompareWithASCIIString(args[3], "nk") != 0) Py_RETURN_NONE;
  const auto as = a->sizes(), bs = b->sizes();
  const int64_t batch = as.size() == 3 ? as[0] : 1, M = as[as.size() - 2], K = as[as.size() - 1];
  const int64_t rows = bs[bs.size() - 2], cols = bs[bs.size() - 1], N = kn ? cols : rows;
  if ((bs.size() == 3 ? bs[0] : 1) != batch || (kn ? rows : cols) != K) Py_RETURN_NONE;
  at::Tensor made;
  void* out;
  if (args[2] == Py_None) {
    made = as.size() == 3 ? at::empty({batch, M, N}, a->options()) : at::empty({M, N}, a->options());
    out = made.data_ptr();
  } else {
    const at::Tensor* c = plain(args[2], device);
    if (!c || c->numel() != batch * M * N) Py_RETURN_NONE;
    out = c->data_ptr();
  }
  gemm_call g = {};
  g.a = a->data_ptr();
  g.b = b->data_ptr();
  g.c = out;
  g.cuda_stream = c10::cuda::getCurrentCUDAStream(device).stream();
  g.batch = (int)batch;
  g.M = (int)M;
  g.N = (int)N;
  g.K = (int)K;
  g.b_layout = kn ? 0 : 1;
  return answer(enter(g_gemm, g), "gemm_forward", args[2], made);
  END_HANDLE_TH_ERRORS
}

// softmax(s, scale, out or None)
PyObject* py_softmax(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 3 || !g_softmax || watched() || !PyFloat_Check(args[1])) Py_RETURN_NONE;
  const c10::DeviceIndex device = device_of_call(args[0]);
  const at::Tensor* s = plain(args[0], device);
  if (!s || s->dim() < 1) Py_RETURN_NONE;
  at::Tensor made;
  void* out;
  if (args[2] == Py_None) {
    made = at::empty_like(*s);
    out = made.data_ptr();
  } else {
    const at::Tensor* o = plain(args[2], device);
    if (!o || o->sizes() != s->sizes()) Py_RETURN_NONE;
    out = o->data_ptr();
  }
  softmax_call c = {};
  c.s = s->data_ptr();
  c.p = out;
  c.cuda_stream = c10::cuda::getCurrentCUDAStream(device).stream();
  c.cols = (int)s->sizes().back();
  c.rows = s->numel() / c.cols;
  c.scale = PyFloat_AS_DOUBLE(args[1]);
  return answer(enter(g_softmax, c), "softmax_rows_forward", args[2], made);
  END_HANDLE_TH_ERRORS
}

// bind(addresses of attn_forward_call, gemm_forward_call, softmax_rows_forward_call, a callable that raises for a status and an entry point)
PyObject* py_bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != 4 || !PyCallable_Check(args[3])) {
    PyErr_SetString(PyExc_TypeError, "bind takes three addresses and a callable");
    return nullptr;
  }
  void* p[3];
  for (int i = 0; i < 3; ++i) {
    p[i] = PyLong_AsVoidPtr(args[i]);
    if (!p[i]) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "no address");
      return nullptr;
    }
  }
  g_attn = reinterpret_cast<decltype(g_attn)>(p[0]);
  g_gemm = reinterpret_cast<decltype(g_gemm)>(p[1]);
  g_softmax = reinterpret_cast<decltype(g_softmax)>(p[2]);
  Py_XSETREF(g_refused, Py_NewRef(args[3]));
  Py_RETURN_NONE;
}

PyMethodDef kMethods[] = {{"bind", reinterpret_cast<PyCFunction>(py_bind), METH_FASTCALL, nullptr},
                          {"attn", reinterpret_cast<PyCFunction>(py_attn), METH_FASTCALL, nullptr},
                          {"gemm", reinterpret_cast<PyCFunction>(py_gemm), METH_FASTCALL, nullptr},
                          {"softmax", reinterpret_cast<PyCFunction>(py_softmax), METH_FASTCALL, nullptr},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_fast", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fast() { return PyModule_Create(&kModule); }
