// The Python binding's way into libnvfp4.so: a call takes tensors, rounding descriptors and numbers as they are and makes the
// C entry point's arguments of them.  A small call is bound by the host, and fetching the arguments one by one in Python and
// passing them through ctypes took 2.7 us of its 6 (three calls on kept weights: 18.4 -> 14.2 us, a 256-token step's two 29.1 -> 22.9).
//
// Argument rules, by what the C parameter is:
//   pointer       a tensor or another object with data_ptr(), or None
//   rounding      a Rounding (the class that bind() was given), or None
//   dtype         an int, or a tensor (its dtype as an nvfp4_dtype): the parameters that NVFP4_CALLS lists
//   size_t        an int, or a tensor (its number of elements): the size of the buffer before it
//   int, int64    an int; a tensor in its place is a misplaced argument and refused
// The last parameter of every entry point is the stream: a torch.cuda.Stream, or None for the current stream.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "nvfp4.h"

namespace {

// Thrown with the Python error set.
struct PythonError {};

[[noreturn]] void type_error(const char* expected, PyObject* got) {
  PyErr_Format(PyExc_TypeError, "expected %s, got %s", expected, Py_TYPE(got)->tp_name);
  throw PythonError{};
}

PyTypeObject* rounding_type = nullptr;             // binding.py's Rounding, a ctypes.Structure laid out as nvfp4_rounding

// The struct is read on the host: nothing but a Rounding will do.
const nvfp4_rounding* convert_rounding(PyObject* o) {
  if (o == Py_None) return nullptr;
  if (!PyObject_TypeCheck(o, rounding_type)) type_error("a Rounding", o);
  Py_buffer view;
  if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw PythonError{};
  void* const p = view.buf;                        // the object outlives the call: the caller holds it
  PyBuffer_Release(&view);
  return static_cast<const nvfp4_rounding*>(p);
}

template <typename T>
T convert_pointer(PyObject* o) {
  if (o == Py_None) return nullptr;
  if (THPVariable_Check(o)) return static_cast<T>(THPVariable_Unpack(o).data_ptr());
  if (!PyObject_HasAttrString(o, "data_ptr")) type_error("a tensor or None", o);
  PyObject* const address = PyObject_CallMethod(o, "data_ptr", nullptr);   // a storage, say
  if (!address) throw PythonError{};
  void* const p = PyLong_AsVoidPtr(address);
  Py_DECREF(address);
  if (!p && PyErr_Occurred()) throw PythonError{};
  return static_cast<T>(p);
}

template <typename T, bool DTYPE>
T convert_number(PyObject* o) {
  if constexpr (DTYPE || std::is_same_v<T, size_t>) {
    if (THPVariable_Check(o)) {
      const at::Tensor& t = THPVariable_Unpack(o);
      if constexpr (!DTYPE) return (T)t.numel();
      if (t.scalar_type() == at::kBFloat16) return (T)NVFP4_BF16;
      if (t.scalar_type() == at::kFloat) return (T)NVFP4_FP32;
      PyErr_Format(PyExc_TypeError, "unsupported dtype %s", c10::toString(t.scalar_type()));
      throw PythonError{};
    }
  }
  if (!PyLong_Check(o)) type_error("an int", o);
  if constexpr (std::is_same_v<T, size_t>) {
    const size_t v = PyLong_AsSize_t(o);
    if (v == (size_t)-1 && PyErr_Occurred()) throw PythonError{};
    return v;
  }
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw PythonError{};
  if constexpr (std::is_same_v<T, int>) {
    if (v != (int)v) {
      PyErr_SetString(PyExc_OverflowError, "argument out of the range of int");
      throw PythonError{};
    }
  }
  return (T)v;
}

void* stream_handle(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* const handle = PyObject_GetAttrString(o, "cuda_stream");
  if (!handle) throw PythonError{};
  void* const p = PyLong_AsVoidPtr(handle);
  Py_DECREF(handle);
  if (!p && PyErr_Occurred()) throw PythonError{};
  return p;
}

template <size_t... S>
constexpr bool one_of(size_t i) { return ((i == S) || ...); }

// DTYPES: the positions of the dtype parameters.
template <size_t... DTYPES, typename... A, size_t... I>
PyObject* call(int (*f)(A...), PyObject* const* args, std::index_sequence<I...>) {
  constexpr size_t kLast = sizeof...(A) - 1;
  std::tuple<A...> a{[&]() -> A {
    if constexpr (I == kLast) return stream_handle(args[I]);
    else if constexpr (std::is_same_v<A, const nvfp4_rounding*>) return convert_rounding(args[I]);
    else if constexpr (std::is_pointer_v<A>) return convert_pointer<A>(args[I]);
    else return convert_number<A, one_of<DTYPES...>(I)>(args[I]);
  }()...};
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = std::apply(f, a);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

template <size_t... DTYPES, typename... A>
PyObject* checked_call(int (*f)(A...), PyObject* const* args, Py_ssize_t n) {
  if (!f) {
    PyErr_SetString(PyExc_RuntimeError, "bind() first");
    return nullptr;
  }
  if (n != (Py_ssize_t)sizeof...(A)) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", (Py_ssize_t)sizeof...(A), n);
    return nullptr;
  }
  try {
    return call<DTYPES...>(f, args, std::index_sequence_for<A...>{});
  } catch (const PythonError&) {
    return nullptr;
  } catch (const std::exception& e) {              // torch's own checks (a tensor without storage, no GPU)
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// The entry points, each with the positions of its dtype parameters.
#define NVFP4_CALLS(X)                                                                                                      \
  X(nvfp4_quantize, 1) X(nvfp4_quantize_dual, 1) X(nvfp4_quantize_mx, 1) X(nvfp4_tensor_amax_scale, 1) X(nvfp4_gemm, 10)    \
  X(nvfp4_gemm_quantized) X(nvfp4_gemm_mx, 10) X(nvfp4_gemm_bf16, 6) X(nvfp4_gemm_bf16_ex, 8) X(nvfp4_linear_fwd, 2, 12)    \
  X(nvfp4_linear_bwd_dx, 2, 12) X(nvfp4_linear_bwd_dw, 2, 12) X(nvfp4_linear_fwd_qout, 2) X(nvfp4_linear_fwd_qin, 4, 12)    \
  X(nvfp4_linear_fwd_save, 2, 14) X(nvfp4_linear_bwd_saved, 1, 12, 14) X(nvfp4_linear_bwd, 3, 16, 18)                       \
  X(nvfp4_linear_bwd_bf16, 7, 9) X(nvfp4_linear_fwd_static, 2, 12)

#define NVFP4_WRAPPER(name, ...)                                                       \
  decltype(&::name) fn_##name = nullptr;                                               \
  PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t n) { return checked_call<__VA_ARGS__>(fn_##name, args, n); }
NVFP4_CALLS(NVFP4_WRAPPER)

// bind(path, Rounding): takes the entry points from the library at `path`, and the class of the rounding descriptors.
PyObject* py_bind(PyObject*, PyObject* args) {
  const char* file;
  PyObject* rounding;
  if (!PyArg_ParseTuple(args, "sO!", &file, &PyType_Type, &rounding)) return nullptr;
  if (reinterpret_cast<PyTypeObject*>(rounding) != rounding_type) {
    Py_XDECREF(rounding_type);
    rounding_type = reinterpret_cast<PyTypeObject*>(Py_NewRef(rounding));
  }
  void* const lib = dlopen(file, RTLD_NOW | RTLD_LOCAL);
  if (!lib) {
    PyErr_SetString(PyExc_OSError, dlerror());
    return nullptr;
  }
  bool all = true;
#define NVFP4_BIND(name, ...) all = (fn_##name = reinterpret_cast<decltype(&::name)>(dlsym(lib, #name))) && all;
  NVFP4_CALLS(NVFP4_BIND)
  if (!all) {
    PyErr_Format(PyExc_OSError, "%s lacks entry points", file);
    return nullptr;
  }
  Py_RETURN_NONE;
}

#define NVFP4_METHOD(name, ...) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr},
PyMethodDef methods[] = {{"bind", py_bind, METH_VARARGS, nullptr}, NVFP4_CALLS(NVFP4_METHOD){nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&module); }
