// CPython binding of the library's launching entry points: torch tensors in, status out.
//
// A layer of a few images runs 4 us on the GPU; the Python around its call (a check per tensor, addresses, the stream, a
// foreign call that converts ten arguments by their declared types) took as long again.  Here every argument is converted
// by the type that the C prototype gives it, in one native call:
//   const ssconv_desc_t*   the ctypes structure (any object with a buffer of that size)
//   other pointers         None, or a contiguous CUDA tensor
//   size_t                 the bytes of a tensor (0 for None): scratch is passed twice, as address and size
//   the last void*         the stream: None for the current one, or an object with `cuda_stream`
// The GIL is released around the call.  The entry points and their results are those of include/ssconv.h.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "ssconv.h"

namespace {

struct PythonError {};  // a Python exception is set

[[noreturn]] void raise(PyObject* type, const char* text) {
  PyErr_SetString(type, text);
  throw PythonError{};
}

int64_t as_int(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw PythonError{};
  return v;
}

const at::Tensor& as_tensor(PyObject* o) {
  if (!THPVariable_Check(o)) raise(PyExc_TypeError, "a tensor (or None) is expected");
  return THPVariable_Unpack(o);
}

void* as_address(PyObject* o) {
  if (o == Py_None) return nullptr;
  const at::Tensor& t = as_tensor(o);
  if (!t.is_cuda() || !t.is_contiguous()) raise(PyExc_ValueError, "tensors must be contiguous CUDA tensors");
  return t.mutable_data_ptr();  // (as data_ptr() in Python: a lazily copied tensor becomes one of its own)
}

void* as_stream(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* handle = PyObject_GetAttrString(o, "cuda_stream");
  if (handle == nullptr) throw PythonError{};
  void* s = PyLong_AsVoidPtr(handle);
  Py_DECREF(handle);
  if (s == nullptr && PyErr_Occurred()) throw PythonError{};
  return s;
}

// One argument of type T from a Python object; `held` keeps a descriptor's buffer.
struct Held {
  Py_buffer buffer{};
  ~Held() { PyBuffer_Release(&buffer); }  // (nothing to do if it was never taken)
};
template <class T>
T convert(PyObject* o, Held& held, bool last) {
  if constexpr (std::is_same_v<T, const ssconv_desc_t*>) {
    if (PyObject_GetBuffer(o, &held.buffer, PyBUF_SIMPLE) != 0) throw PythonError{};
    if (held.buffer.len != (Py_ssize_t)sizeof(ssconv_desc_t)) raise(PyExc_TypeError, "a layer descriptor is expected");
    return static_cast<const ssconv_desc_t*>(held.buffer.buf);
  } else if constexpr (std::is_pointer_v<T>) {
    return static_cast<T>(last ? as_stream(o) : as_address(o));
  } else if constexpr (std::is_same_v<T, float>) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PythonError{};
    return (float)v;
  } else if constexpr (std::is_same_v<T, size_t>) {
    return o == Py_None ? 0 : (size_t)as_tensor(o).nbytes();
  } else {
    return (T)as_int(o);
  }
}

template <auto FN>
struct Entry;
template <class... A, int32_t (*FN)(A...)>
struct Entry<FN> {
  template <size_t... I>
  static int32_t run(PyObject* const* args, std::index_sequence<I...>) {
    Held held;
    // (braces: converted from left to right)
    std::tuple<A...> v{convert<A>(args[I], held, I + 1 == sizeof...(A))...};
    int32_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = FN(std::get<I>(v)...);
    Py_END_ALLOW_THREADS
    return rc;
  }
  static PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != (Py_ssize_t)sizeof...(A)) {
      PyErr_Format(PyExc_TypeError, "%zd arguments, %zd expected", n, (Py_ssize_t)sizeof...(A));
      return nullptr;
    }
    int32_t rc;
    try {
      rc = run(args, std::index_sequence_for<A...>{});
    } catch (const PythonError&) {
      return nullptr;
    }
    return PyLong_FromLong(rc);
    END_HANDLE_TH_ERRORS
  }
};

// output(desc, x): an uninitialised bf16 tensor for the layer's output on x's device, or the library's status.
PyObject* output(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  try {
    if (n != 2) raise(PyExc_TypeError, "output(desc, x)");
    Held held;
    const ssconv_desc_t* d = convert<const ssconv_desc_t*>(args[0], held, false);
    const at::Tensor& x = as_tensor(args[1]);
    int32_t ho = 0, wo = 0;
    const int32_t rc = ssconv_out_shape(d, &ho, &wo);
    if (rc != SSCONV_OK) return PyLong_FromLong(rc);
    return THPVariable_Wrap(at::empty({d->N, ho, wo, d->C_out}, at::TensorOptions().dtype(at::kBFloat16).device(x.device())));
  } catch (const PythonError&) {
    return nullptr;
  }
  END_HANDLE_TH_ERRORS
}

// blob(n, x): n uninitialised bytes on x's device.
PyObject* blob(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  try {
    if (n != 2) raise(PyExc_TypeError, "blob(n, x)");
    return THPVariable_Wrap(
        at::empty({as_int(args[0])}, at::TensorOptions().dtype(at::kByte).device(as_tensor(args[1]).device())));
  } catch (const PythonError&) {
    return nullptr;
  }
  END_HANDLE_TH_ERRORS
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))Entry<&name>::call, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    ENTRY(ssconv_select_mask), ENTRY(ssconv_compress), ENTRY(ssconv_maxpool), ENTRY(ssconv_space_to_depth),
    ENTRY(ssconv_forward), ENTRY(ssconv_forward_res), ENTRY(ssconv_forward_dense), ENTRY(ssconv_forward_dense_res),
    ENTRY(ssconv_forward_dense_strided), ENTRY(ssconv_soft_mask), ENTRY(ssconv_mask_grad), ENTRY(ssconv_adamw),
    ENTRY(ssconv_wgrad), ENTRY(ssconv_dgrad), ENTRY(ssconv_forward_grouped), ENTRY(ssconv_forward_dense_grouped),
    ENTRY(ssconv_depthwise), ENTRY(ssconv_layernorm), ENTRY(ssconv_quantize_e4m3), ENTRY(ssconv_forward_fp8),
    ENTRY(ssconv_forward_dense_fp8),
    {"output", (PyCFunction)(void (*)(void))output, METH_FASTCALL, nullptr},
    {"blob", (PyCFunction)(void (*)(void))blob, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() { return PyModule_Create(&module); }
