// Calls of the C ABI straight from PyTorch tensors: the regular call of binding.py's entry points in one native function each.
//
// A call through ctypes spends 10 to 12 us of host time on checks, conversions and torch.empty, as long as the kernels of
// small problems run.  Here the same checks, the output's allocation and the call take about 4.  Every function returns None for
// anything that is not the regular case -- a tensor of another type, device or layout, an explicit stream, formats of other
// types, an active torch-function or dispatch mode, an exception -- and has then done nothing that a caller can see: binding.py
// goes on as it would without this module, and raises what it raises.  A status other than 0 is returned as an integer.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/ops/empty.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>
#include <optional>

#include "lba.h"

namespace {

PyObject* g_format_type = nullptr;     // formats.LbaFormat
PyObject* g_parameter_type = nullptr;  // torch.nn.Parameter: a tensor like any other here, as weights, scales and biases often are
PyObject* g_field[5];               // its attribute names, interned

struct NotRegular {};

[[noreturn]] void not_regular() { throw NotRegular(); }

int as_int(PyObject* o) {
  if (!PyLong_CheckExact(o)) not_regular();
  int overflow = 0;
  const long v = PyLong_AsLongAndOverflow(o, &overflow);
  if (overflow || v < INT_MIN || v > INT_MAX) not_regular();
  return (int)v;
}

lba_fmt as_format(PyObject* o) {
  int32_t v[5];
  if (Py_TYPE(o) == (PyTypeObject*)g_format_type) {
    for (int i = 0; i < 5; ++i) {
      PyObject* const a = PyObject_GetAttr(o, g_field[i]);
      if (!a) {
        PyErr_Clear();
        not_regular();
      }
      const bool plain = PyLong_CheckExact(a);
      int overflow = 0;
      const long x = plain ? PyLong_AsLongAndOverflow(a, &overflow) : 0;
      Py_DECREF(a);
      if (!plain || overflow || x < INT_MIN || x > INT_MAX) not_regular();
      v[i] = (int32_t)x;
    }
  } else if (PyTuple_CheckExact(o) && PyTuple_GET_SIZE(o) == 5) {
    for (int i = 0; i < 5; ++i) v[i] = as_int(PyTuple_GET_ITEM(o, i));
  } else {
    not_regular();
  }
  lba_fmt f;
  f.man_bits = v[0];
  f.exp_bits = v[1];
  f.bias = v[2];
  f.rounding = v[3];
  f.flags = v[4];
  return f;
}

// a contiguous tensor of `dtype` on the current device
const at::Tensor& as_tensor(PyObject* o, c10::ScalarType dtype, int dim, int device) {
  if (Py_TYPE(o) != (PyTypeObject*)THPVariableClass && Py_TYPE(o) != (PyTypeObject*)g_parameter_type) not_regular();  // no other subclass
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || !t.is_cuda() || t.get_device() != device || t.scalar_type() != dtype || !t.is_contiguous() ||
      (dim >= 0 && t.dim() != dim))
    not_regular();
  return t;
}

void pair_of(PyObject* o, int (&v)[2]) {
  if (!PyTuple_CheckExact(o) || PyTuple_GET_SIZE(o) != 2) not_regular();
  v[0] = as_int(PyTuple_GET_ITEM(o, 0));
  v[1] = as_int(PyTuple_GET_ITEM(o, 1));
}

struct Call {
  int device;
  void* stream;
  explicit Call(PyObject* stream_arg) {
    if (stream_arg != Py_None || at::impl::PythonTorchFunctionTLS::stack_len() > 0 || c10::impl::TorchDispatchModeTLS::any_modes_set())
      not_regular();
    device = c10::cuda::current_device();
    stream = (void*)c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)device).stream();
  }
  at::Tensor fresh(at::IntArrayRef sizes, c10::ScalarType dtype) const {
    return at::empty(sizes, at::TensorOptions().dtype(dtype).device(c10::Device(c10::kCUDA, (c10::DeviceIndex)device)));
  }
};

// scales and bias, as every forward entry point takes them
struct Scales {
  const float *a, *b, *bias;
  int a_len, b_len;
  Scales(PyObject* sa, PyObject* sb, PyObject* bi, int device) {
    const at::Tensor &ta = as_tensor(sa, at::kFloat, -1, device), &tb = as_tensor(sb, at::kFloat, -1, device);
    if (ta.numel() > INT_MAX || tb.numel() > INT_MAX) not_regular();
    a = (const float*)ta.data_ptr();
    b = (const float*)tb.data_ptr();
    a_len = (int)ta.numel();
    b_len = (int)tb.numel();
    bias = bi == Py_None ? nullptr : (const float*)as_tensor(bi, at::kFloat, -1, device).data_ptr();
  }
};

// the output a caller passed, or a new one
at::Tensor output(PyObject* out, const Call& call, at::IntArrayRef sizes, c10::ScalarType dtype) {
  return out == Py_None ? call.fresh(sizes, dtype) : as_tensor(out, dtype, -1, call.device);
}

PyObject* result(int status, PyObject* given, const at::Tensor& out) {
  if (status != 0) return PyLong_FromLong(status);
  if (given != Py_None) return Py_NewRef(given);
  return THPVariable_Wrap(out);
}

template <typename F>
int without_gil(F f) {
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = f();
  Py_END_ALLOW_THREADS
  return status;
}

template <typename F>
PyObject* regular_or_none(Py_ssize_t n, Py_ssize_t want, F f) {
  if (n != want) Py_RETURN_NONE;
  try {
    return f();
  } catch (...) {  // NotRegular, or an error that the caller's own path runs into and reports
    PyErr_Clear();
    Py_RETURN_NONE;
  }
}

// A, B, scale_a, scale_b, bias, prod_fmt, acc_fmt, order, chunk, out, stream
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return regular_or_none(n, 11, [&]() -> PyObject* {
    const Call call(a[10]);
    const at::Tensor &A = as_tensor(a[0], at::kByte, 2, call.device), &B = as_tensor(a[1], at::kByte, 2, call.device);
    const int64_t M = A.size(0), N = B.size(0), K = A.size(1);
    if (B.size(1) != K) not_regular();
    const Scales s(a[2], a[3], a[4], call.device);
    const lba_fmt pf = as_format(a[5]), af = as_format(a[6]);
    const int order = as_int(a[7]), chunk = as_int(a[8]);
    const at::Tensor out = output(a[9], call, {M, N}, at::kFloat);
    const uint8_t *const pa = (const uint8_t*)A.data_ptr(), *const pb = (const uint8_t*)B.data_ptr();
    float* const po = (float*)out.data_ptr();
    return result(without_gil([&] {
                    return lba_gemm(pa, pb, s.a, s.a_len, s.b, s.b_len, s.bias, M, N, K, &pf, &af, order, chunk, po, call.stream);
                  }), a[9], out);
  });
}

// the same with A [Z][M][K], B [Z][N][K] or [N][K]
PyObject* gemm_batched(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return regular_or_none(n, 11, [&]() -> PyObject* {
    const Call call(a[10]);
    const at::Tensor &A = as_tensor(a[0], at::kByte, 3, call.device), &B = as_tensor(a[1], at::kByte, -1, call.device);
    const int64_t Z = A.size(0), M = A.size(1), K = A.size(2);
    const bool shared = B.dim() == 2;
    if (!shared && (B.dim() != 3 || B.size(0) != Z)) not_regular();
    const int64_t N = B.size(shared ? 0 : 1);
    if (B.size(shared ? 1 : 2) != K) not_regular();
    const Scales s(a[2], a[3], a[4], call.device);
    const lba_fmt pf = as_format(a[5]), af = as_format(a[6]);
    const int order = as_int(a[7]), chunk = as_int(a[8]);
    const at::Tensor out = output(a[9], call, {Z, M, N}, at::kFloat);
    const uint8_t *const pa = (const uint8_t*)A.data_ptr(), *const pb = (const uint8_t*)B.data_ptr();
    float* const po = (float*)out.data_ptr();
    return result(without_gil([&] {
                    return lba_gemm_batched(pa, pb, s.a, s.a_len, s.b, s.b_len, s.bias, Z, M, N, K, M * K, shared ? 0 : N * K, M * N, &pf,
                                            &af, order, chunk, po, call.stream);
                  }), a[9], out);
  });
}

// x, w, scale_x, scale_w, bias, stride, pad, prod_fmt, acc_fmt, order, chunk, out, stream
PyObject* conv2d(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return regular_or_none(n, 13, [&]() -> PyObject* {
    const Call call(a[12]);
    const at::Tensor &x = as_tensor(a[0], at::kByte, 4, call.device), &w = as_tensor(a[1], at::kByte, 4, call.device);
    int64_t d[7] = {x.size(0), x.size(1), x.size(2), x.size(3), w.size(0), w.size(1), w.size(2)};
    int stride[2], pad[2];
    pair_of(a[5], stride);
    pair_of(a[6], pad);
    if (w.size(3) != d[3] || stride[0] < 1 || stride[1] < 1 || pad[0] < 0 || pad[1] < 0) not_regular();
    for (int64_t v : d)
      if (v < 1 || v > INT_MAX / 4) not_regular();
    if (pad[0] > INT_MAX / 4 || pad[1] > INT_MAX / 4) not_regular();
    const int64_t h = d[1] + 2 * (int64_t)pad[0] - d[5], v = d[2] + 2 * (int64_t)pad[1] - d[6];
    if (h < 0 || v < 0) not_regular();
    const Scales s(a[2], a[3], a[4], call.device);
    const lba_fmt pf = as_format(a[7]), af = as_format(a[8]);
    const int order = as_int(a[9]), chunk = as_int(a[10]);
    const at::Tensor out = output(a[11], call, {d[0], h / stride[0] + 1, v / stride[1] + 1, d[4]}, at::kFloat);
    const uint8_t *const px = (const uint8_t*)x.data_ptr(), *const pw = (const uint8_t*)w.data_ptr();
    float* const po = (float*)out.data_ptr();
    return result(without_gil([&] {
                    return lba_conv2d(px, pw, s.a, s.a_len, s.b, s.b_len, s.bias, (int)d[0], (int)d[1], (int)d[2], (int)d[3], (int)d[4],
                                      (int)d[5], (int)d[6], stride[0], stride[1], pad[0], pad[1], &pf, &af, order, chunk, po, call.stream);
                  }), a[11], out);
  });
}

PyObject* init_module(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 2) {
    PyErr_SetString(PyExc_TypeError, "init takes the format class and the parameter class");
    return nullptr;
  }
  static const char* const names[5] = {"man_bits", "exp_bits", "bias", "rounding", "flags"};
  for (int i = 0; i < 5; ++i)
    if (!g_field[i] && !(g_field[i] = PyUnicode_InternFromString(names[i]))) return nullptr;
  Py_XSETREF(g_format_type, Py_NewRef(a[0]));
  Py_XSETREF(g_parameter_type, Py_NewRef(a[1]));
  Py_RETURN_NONE;
}

PyMethodDef kMethods[] = {
    {"init", (PyCFunction)(void (*)(void))init_module, METH_FASTCALL, "the format class whose instances are read by attribute, and the parameter class"},
    {"gemm", (PyCFunction)(void (*)(void))gemm, METH_FASTCALL, nullptr},
    {"gemm_batched", (PyCFunction)(void (*)(void))gemm_batched, METH_FASTCALL, nullptr},
    {"conv2d", (PyCFunction)(void (*)(void))conv2d, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "lba_torch", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_lba_torch() {
  PyObject* const m = PyModule_Create(&kModule);
  if (m && PyModule_AddStringConstant(m, "built_for", LBA_TORCH_TAG) != 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
