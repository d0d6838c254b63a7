// The calls that a program makes once per token, as functions of a Python extension module: check the
// tensors, allocate the outputs, call the C ABI.  Marshalling only.
//
// What it is for: with the kernel of a one-token call at 5 us, the caller's side was what a call
// took: three allocations through Python 4.8 us, the ctypes call 3.5, the rest 1.8.
//
// The functions take the entry points' addresses (bind), so that this module needs no link to the
// CUDA library; they return (status, outputs...) and leave the exception to the Python side.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "gsi.h"

namespace {

decltype(&gsi_forward_n) forward_n = nullptr;
decltype(&gsi_extend_basis) extend_basis = nullptr;
decltype(&gsi_forward_static) forward_static = nullptr;

struct NoGil {
  PyThreadState* state = PyEval_SaveThread();
  ~NoGil() { PyEval_RestoreThread(state); }
};

// The handle of a stream argument that is not None: an int or an object with cuda_stream.
bool stream_of(PyObject* o, bool* given, void** out) {
  *given = o != Py_None;
  *out = nullptr;
  if (!*given) return true;
  PyObject* number = PyObject_GetAttrString(o, "cuda_stream");
  if (!number) {
    if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
    PyErr_Clear();
    number = Py_NewRef(o);
  }
  PyObject* value = PyNumber_Long(number);
  Py_DECREF(number);
  if (!value) return false;
  *out = PyLong_AsVoidPtr(value);
  Py_DECREF(value);
  return !PyErr_Occurred();
}

const at::Tensor* tensor_of(PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_SetString(PyExc_TypeError, "a tensor is expected");
    return nullptr;
  }
  return &THPVariable_Unpack(o);
}
// The input of a call.
const at::Tensor* input_of(PyObject* o) {
  const at::Tensor* x = tensor_of(o);
  if (x && !(x->is_cuda() && x->scalar_type() == at::kFloat && x->is_contiguous())) {
    PyErr_SetString(PyExc_AssertionError, "x must be a contiguous float32 tensor on a CUDA device");
    return nullptr;
  }
  return x;
}
// An output that the caller gave, or one that is allocated here.
bool output_of(PyObject* o, at::Tensor* t) {
  if (o == Py_None) return true;
  const at::Tensor* given = tensor_of(o);
  if (given) *t = *given;
  return given != nullptr;
}
bool enough(Py_ssize_t given, Py_ssize_t wanted) {
  if (given == wanted) return true;
  PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
  return false;
}

void allocate(const at::Tensor& x, int64_t n, int64_t O, at::Tensor* y, at::Tensor* gate, at::Tensor* rho) {
  if (!y->defined()) *y = at::empty({n, O}, x.options());
  if (!gate->defined()) *gate = at::empty({n}, x.options().dtype(at::kByte));
  if (!rho->defined()) *rho = at::empty({n}, x.options());
}

// forward(handle, O, x, y, gate, rho, stream) -> (status, y, gate, rho)
PyObject* py_forward(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  HANDLE_TH_ERRORS
  if (!enough(n_args, 7)) return nullptr;
  auto handle = static_cast<gsi_handle_t>(PyLong_AsVoidPtr(args[0]));
  const int64_t O = PyLong_AsLongLong(args[1]);
  if (PyErr_Occurred()) return nullptr;
  const at::Tensor* x = input_of(args[2]);
  at::Tensor y, gate, rho;
  bool given;
  void* stream;
  if (!x || !output_of(args[3], &y) || !output_of(args[4], &gate) || !output_of(args[5], &rho) ||
      !stream_of(args[6], &given, &stream))
    return nullptr;
  int status;
  {
    NoGil no_gil;
    const int64_t n = x->size(0);
    allocate(*x, n, O, &y, &gate, &rho);
    if (!given) stream = c10::cuda::getCurrentCUDAStream().stream();
    status = forward_n(handle, static_cast<const float*>(x->data_ptr()), (int)n, static_cast<float*>(y.data_ptr()),
                       static_cast<unsigned char*>(gate.data_ptr()), static_cast<float*>(rho.data_ptr()),
                       static_cast<gsi_stream_t>(stream));
  }
  return Py_BuildValue("iNNN", status, THPVariable_Wrap(y), THPVariable_Wrap(gate), THPVariable_Wrap(rho));
  END_HANDLE_TH_ERRORS
}

// extend(handle, x, tau, k_active, stream) -> (status, appended, rho)
PyObject* py_extend(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  HANDLE_TH_ERRORS
  if (!enough(n_args, 5)) return nullptr;
  auto handle = static_cast<gsi_handle_t>(PyLong_AsVoidPtr(args[0]));
  const double tau = PyFloat_AsDouble(args[2]);
  if (PyErr_Occurred()) return nullptr;
  const at::Tensor* x = input_of(args[1]);
  const at::Tensor* k_active = x ? tensor_of(args[3]) : nullptr;
  bool given;
  void* stream;
  if (!k_active || !stream_of(args[4], &given, &stream)) return nullptr;
  if (!(k_active->is_cuda() && k_active->scalar_type() == at::kInt && k_active->numel() == 1)) {
    PyErr_SetString(PyExc_AssertionError, "k_active must be one int32 on a CUDA device");
    return nullptr;
  }
  at::Tensor appended, rho;
  int status;
  {
    NoGil no_gil;
    appended = at::empty({1}, x->options().dtype(at::kInt));
    rho = at::empty({1}, x->options());
    if (!given) stream = c10::cuda::getCurrentCUDAStream().stream();
    status = extend_basis(handle, static_cast<const float*>(x->data_ptr()), (float)tau,
                          static_cast<int*>(k_active->data_ptr()), static_cast<int*>(appended.data_ptr()),
                          static_cast<float*>(rho.data_ptr()), static_cast<gsi_stream_t>(stream));
  }
  return Py_BuildValue("iNN", status, THPVariable_Wrap(appended), THPVariable_Wrap(rho));
  END_HANDLE_TH_ERRORS
}

// forward_static(Ws (a list), P, p_dtype, W_P, eps, x, y, gate, rho, stream) -> (status, y, gate, rho)
PyObject* py_forward_static(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  HANDLE_TH_ERRORS
  if (!enough(n_args, 10)) return nullptr;
  if (!PyList_Check(args[0])) {
    PyErr_SetString(PyExc_TypeError, "a list of tensors is expected");
    return nullptr;
  }
  const Py_ssize_t maps = PyList_GET_SIZE(args[0]);
  std::vector<const void*> W(maps);
  std::vector<int> d_out(maps);
  int64_t O = 0;
  for (Py_ssize_t j = 0; j < maps; ++j) {
    const at::Tensor* w = tensor_of(PyList_GET_ITEM(args[0], j));
    if (!w) return nullptr;
    W[j] = w->data_ptr();
    d_out[j] = (int)w->size(0);
    O += d_out[j];
  }
  const at::Tensor *P = tensor_of(args[1]), *W_P = P ? tensor_of(args[3]) : nullptr, *x = W_P ? tensor_of(args[5]) : nullptr;
  if (!x) return nullptr;
  const long p_dtype = PyLong_AsLong(args[2]);
  const double eps = PyFloat_AsDouble(args[4]);
  if (PyErr_Occurred()) return nullptr;
  at::Tensor y, gate, rho;
  bool given;
  void* stream;
  if (!output_of(args[6], &y) || !output_of(args[7], &gate) || !output_of(args[8], &rho) ||
      !stream_of(args[9], &given, &stream))
    return nullptr;
  int status;
  {
    NoGil no_gil;
    const int64_t n = x->size(0);
    allocate(*x, n, O, &y, &gate, &rho);
    if (!given) stream = c10::cuda::getCurrentCUDAStream().stream();
    status = forward_static(W.data(), d_out.data(), (int)maps, P->data_ptr(), (gsi_dtype_t)p_dtype, W_P->data_ptr(),
                            (int)P->size(0), (int)P->size(1), (float)eps, static_cast<const float*>(x->data_ptr()), (int)n,
                            static_cast<float*>(y.data_ptr()), static_cast<unsigned char*>(gate.data_ptr()),
                            static_cast<float*>(rho.data_ptr()), static_cast<gsi_stream_t>(stream));
  }
  return Py_BuildValue("iNNN", status, THPVariable_Wrap(y), THPVariable_Wrap(gate), THPVariable_Wrap(rho));
  END_HANDLE_TH_ERRORS
}

// bind(address of gsi_forward_n, of gsi_extend_basis, of gsi_forward_static)
PyObject* py_bind(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  if (!enough(n_args, 3)) return nullptr;
  forward_n = reinterpret_cast<decltype(forward_n)>(PyLong_AsVoidPtr(args[0]));
  extend_basis = reinterpret_cast<decltype(extend_basis)>(PyLong_AsVoidPtr(args[1]));
  forward_static = reinterpret_cast<decltype(forward_static)>(PyLong_AsVoidPtr(args[2]));
  if (PyErr_Occurred()) return nullptr;
  Py_RETURN_NONE;
}

#define METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(forward), METHOD(extend), METHOD(forward_static), METHOD(bind), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_torch_calls", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__torch_calls() { return PyModule_Create(&module); }
