// The marshalling of the whole-layer calls in native code (a CPython extension).  A layer of a few tokens takes the GPU
// 6 us, its two kernel launches take the host 4.2 (both measured); checking seven tensors, reading their addresses and
// converting fifteen arguments in Python took another 5.7.  Nothing is computed here, and nothing is kept between calls
// but the addresses of the library's entry points.
//
//   set_entry(kind, address)   kind 0..3: torq_rotated_linear, _mxint4, _structured, _nvfp4
//   layer(kind, X, R, R_intra, Wq, Ws, Y, workspace, dbg_codes, dbg_scales, stream[, x_scale, w_scale])
//     -> the library's status, or -1 when an operand is not what the call takes (the caller then finds out which).
// Operands that may be missing are None; stream is None (the current one) or a cudaStream_t as an integer.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/torq.h"

namespace {

using LayerFn = decltype(&torq_rotated_linear);
using LayerNvFn = decltype(&torq_rotated_linear_nvfp4);
constexpr int kNv = 3, kKinds = 4;
void* g_entry[kKinds] = {};

// Address of a contiguous CUDA tensor of `dtype`; None gives NULL where that is allowed.
bool operand(PyObject* o, at::ScalarType dtype, bool optional, void** out) {
  *out = nullptr;
  if (o == Py_None) return optional;
  if (!THPVariable_Check(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (t.scalar_type() != dtype || !t.is_cuda() || !t.is_contiguous()) return false;
  *out = t.data_ptr();
  return true;
}

// Scratch: any dtype; the caller counts a byte for each element.
bool scratch(PyObject* o, void** out, size_t* bytes) {
  if (!THPVariable_Check(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_cuda() || !t.is_contiguous()) return false;
  *out = t.data_ptr();
  *bytes = (size_t)t.numel();
  return true;
}

PyObject* set_entry(PyObject*, PyObject* const* a, Py_ssize_t n) {
  const long kind = n == 2 ? PyLong_AsLong(a[0]) : -1;
  if (kind < 0 || kind >= kKinds) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "set_entry(kind, address)");
    return nullptr;
  }
  void* p = PyLong_AsVoidPtr(a[1]);
  if (PyErr_Occurred()) return nullptr;
  g_entry[kind] = p;
  Py_RETURN_NONE;
}

PyObject* layer(PyObject*, PyObject* const* a, Py_ssize_t n) try {
  const long kind = n >= 11 ? PyLong_AsLong(a[0]) : -1;
  if (kind < 0 || kind >= kKinds || n != (kind == kNv ? 13 : 11) || !g_entry[kind]) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "layer(): wrong arguments");
    return nullptr;
  }
  void *X, *R, *Ri, *Wq, *Ws, *ws, *dc, *ds;
  size_t ws_bytes;
  if (!operand(a[1], at::kBFloat16, false, &X) || !operand(a[2], at::kBFloat16, true, &R) ||
      !operand(a[3], at::kBFloat16, true, &Ri) || !operand(a[4], at::kByte, false, &Wq) || !operand(a[5], at::kByte, false, &Ws) ||
      !scratch(a[7], &ws, &ws_bytes) || !operand(a[8], at::kByte, true, &dc) || !operand(a[9], at::kByte, true, &ds) ||
      !THPVariable_Check(a[6]))
    return PyLong_FromLong(-1);
  const at::Tensor &x = THPVariable_Unpack(a[1]), &w = THPVariable_Unpack(a[4]), &y = THPVariable_Unpack(a[6]);
  const bool f32 = y.scalar_type() == at::kFloat;
  if (x.dim() != 2 || w.dim() < 1 || !y.is_cuda() || !y.is_contiguous() || (!f32 && y.scalar_type() != at::kBFloat16) ||
      y.numel() < x.size(0) * w.size(0))
    return PyLong_FromLong(-1);
  void* stream = a[10] == Py_None ? (void*)c10::cuda::getCurrentCUDAStream().stream() : PyLong_AsVoidPtr(a[10]);
  if (PyErr_Occurred()) return nullptr;
  const int64_t M = x.size(0), d = x.size(1), N = w.size(0);
  const torq_dtype dt = f32 ? TORQ_F32 : TORQ_BF16;
  void* yp = y.data_ptr();
  torq_status rc;
  if (kind == kNv) {
    const double xs = PyFloat_AsDouble(a[11]), wsc = PyFloat_AsDouble(a[12]);
    if (PyErr_Occurred()) return nullptr;
    Py_BEGIN_ALLOW_THREADS;                              // a launch may wait for room in the stream's queue
    rc = reinterpret_cast<LayerNvFn>(g_entry[kind])(X, R, Ri, (float)xs, Wq, Ws, (float)wsc, M, d, N, yp, dt, ws, ws_bytes, dc, ds, stream);
    Py_END_ALLOW_THREADS;
  } else {
    Py_BEGIN_ALLOW_THREADS;
    rc = reinterpret_cast<LayerFn>(g_entry[kind])(X, R, Ri, Wq, Ws, M, d, N, yp, dt, ws, ws_bytes, dc, ds, stream);
    Py_END_ALLOW_THREADS;
  }
  return PyLong_FromLong((long)rc);
} catch (const std::exception&) {                        // a tensor without storage, for instance
  return PyLong_FromLong(-1);
}

PyMethodDef methods[] = {
    {"set_entry", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(set_entry)), METH_FASTCALL, "address of a library entry point"},
    {"layer", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(layer)), METH_FASTCALL, "one whole-layer call"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_torq_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__torq_binding() { return PyModule_Create(&module); }
