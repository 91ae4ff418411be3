// Argument marshalling of the Python binding: one native call per entry point of libfasa.so turns a list of
// tensors and integers into its C arguments, checks the tensors and appends the current CUDA stream.
//
// A decode step takes fifteen arguments and the work of a small one on the GPU is about 20 us; checked and
// converted one by one in Python they cost more than the launch itself.  Measured per call of the appending step:
// 11.1 us in Python with ctypes, 4.7 us here.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <utility>

namespace {

constexpr int kMaxArgs = 20;

// All arguments are pointers or 32-bit integers; both travel in 64-bit registers or stack slots of the C calling
// conventions of x86-64 and AArch64, and a callee reads the low half of the latter.
template <size_t... I>
int32_t call_n(void* fn, const int64_t* a, std::index_sequence<I...>) {
  return reinterpret_cast<int32_t (*)(decltype((void)I, int64_t{})...)>(fn)(a[I]...);
}
template <size_t N = 1>
int32_t call(void* fn, const int64_t* a, size_t n) {
  if constexpr (N <= kMaxArgs) {
    if (n == N) return call_n(fn, a, std::make_index_sequence<N>{});
    return call<N + 1>(fn, a, n);
  } else {
    return -1;
  }
}

// The pointer of a tensor argument.  kind 'p': as it is (a cache may be strided, or host memory); 'u': a contiguous
// CUDA tensor; 'b', 'f', 'i', 'l': one of bf16, fp32, int32, int64.  None is a null pointer (not with 'p').
bool tensor_arg(PyObject* o, char kind, int64_t* out) {
  if (o == Py_None && kind != 'p') {
    *out = 0;
    return true;
  }
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a tensor, got %.100s", Py_TYPE(o)->tp_name);
    return false;
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  if (kind != 'p') {
    if (!t.is_cuda()) {
      PyErr_SetString(PyExc_ValueError, "expected a CUDA tensor");
      return false;
    }
    if (!t.is_contiguous()) {
      PyErr_SetString(PyExc_ValueError, "expected a contiguous tensor");
      return false;
    }
    if (kind != 'u') {
      const at::ScalarType want = kind == 'b' ? at::kBFloat16 : kind == 'f' ? at::kFloat : kind == 'i' ? at::kInt : at::kLong;
      if (t.scalar_type() != want) {
        PyErr_Format(PyExc_ValueError, "expected dtype %s, got %s", c10::toString(want), c10::toString(t.scalar_type()));
        return false;
      }
    }
  }
  *out = reinterpret_cast<int64_t>(t.data_ptr());
  return true;
}

// invoke(function address, context address, kinds, *arguments) -> status.  kinds: a letter per argument, 'n' = integer,
// the others as above.  The function is called as f(context, arguments..., current CUDA stream).
PyObject* invoke(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  if (n_args < 3) {
    PyErr_SetString(PyExc_TypeError, "invoke(function, context, kinds, *arguments)");
    return nullptr;
  }
  void* fn = PyLong_AsVoidPtr(args[0]);
  if (!fn) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null function");
    return nullptr;
  }
  int64_t a[kMaxArgs];
  a[0] = args[1] == Py_None ? 0 : reinterpret_cast<int64_t>(PyLong_AsVoidPtr(args[1]));
  if (PyErr_Occurred()) return nullptr;
  Py_ssize_t n_kinds = 0;
  const char* kinds = PyUnicode_AsUTF8AndSize(args[2], &n_kinds);
  if (!kinds) return nullptr;
  if (n_kinds != n_args - 3 || n_kinds + 2 > kMaxArgs) {
    PyErr_SetString(PyExc_TypeError, "one letter per argument");
    return nullptr;
  }
  try {
    for (Py_ssize_t i = 0; i < n_kinds; ++i) {
      if (kinds[i] == 'n') {
        int overflow = 0;
        a[i + 1] = PyLong_AsLongLongAndOverflow(args[i + 3], &overflow);
        if (PyErr_Occurred()) return nullptr;
        if (overflow || a[i + 1] != (int32_t)a[i + 1]) {
          PyErr_SetString(PyExc_OverflowError, "integer argument out of the 32-bit range");
          return nullptr;
        }
      } else if (!tensor_arg(args[i + 3], kinds[i], &a[i + 1])) {
        return nullptr;
      }
    }
    a[n_kinds + 1] = reinterpret_cast<int64_t>(c10::cuda::getCurrentCUDAStream().stream());
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
  int32_t status;
  Py_BEGIN_ALLOW_THREADS
  status = call(fn, a, (size_t)n_kinds + 2);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(status);
}

PyMethodDef kMethods[] = {
    {"invoke", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(invoke)), METH_FASTCALL, "Calls an entry point of libfasa.so."},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// What the build looks for in the file: an extension built for another interpreter or torch is not used.
PyMODINIT_FUNC PyInit__marshal() {
  PyObject* m = PyModule_Create(&kModule);
  if (m && PyModule_AddStringConstant(m, "built_for", FASA_BUILT_FOR) < 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
