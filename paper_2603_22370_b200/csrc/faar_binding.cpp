// Native argument marshalling between Python and libfaar.so (CPython extension module `_faarbind`).
//
// What bounds a small layer is the host: a call through ctypes costs 3-5 us of Python for its dozen tensors and
// structs, as much as the two or three kernel launches behind it.  Here every entry point that enqueues work becomes
// a vectorcall function whose argument conversion is generated from the entry point's own C declaration:
//   pointer            None, an int (address), or a CUDA tensor (its data_ptr(); a host tensor is refused)
//   faar_shape /
//   faar_hparams /
//   faar_model         the binding's ctypes structure, by its buffer
//   int, size_t, float Python numbers
// A function returns the call's status; raising is the Python side's business.  The GIL is released for the call.
// The module holds no device code and does not link libfaar.so: load(path) opens the library the process binds (the
// normal or the bounds-checking build) and resolves the entry points in it.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "faar.h"

namespace {

PyObject* s_data_ptr = nullptr;
PyObject* s_is_cuda = nullptr;

bool to_address(PyObject* o, void** out) {
  if (o == Py_None) { *out = nullptr; return true; }
  if (PyLong_Check(o)) {
    *out = PyLong_AsVoidPtr(o);
    return !(*out == nullptr && PyErr_Occurred());
  }
  PyObject* cuda = PyObject_GetAttr(o, s_is_cuda);
  if (!cuda) return false;
  const bool on_device = cuda == Py_True;
  Py_DECREF(cuda);
  if (!on_device) { PyErr_SetString(PyExc_AssertionError, "device tensors only"); return false; }
  PyObject* args[1] = {o};
  PyObject* p = PyObject_VectorcallMethod(s_data_ptr, args, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, nullptr);
  if (!p) return false;
  *out = PyLong_AsVoidPtr(p);
  Py_DECREF(p);
  return !(*out == nullptr && PyErr_Occurred());
}

// One argument: holds the converted value (and, for the structs, the buffer it was read from).
template <class T, class = void> struct Arg;
template <class T> struct Arg<T, std::enable_if_t<std::is_integral_v<T>>> {
  T v;
  bool set(PyObject* o) {
    if constexpr (std::is_unsigned_v<T>) v = (T)PyLong_AsUnsignedLongLong(o);
    else v = (T)PyLong_AsLongLong(o);
    return !(v == (T)-1 && PyErr_Occurred());
  }
};
template <> struct Arg<float> {
  float v;
  bool set(PyObject* o) {
    v = (float)PyFloat_AsDouble(o);
    return !(v == -1.0f && PyErr_Occurred());
  }
};
template <class T> struct Arg<T, std::enable_if_t<std::is_pointer_v<T>>> {
  using E = std::remove_cv_t<std::remove_pointer_t<T>>;
  static constexpr bool STRUCT = std::is_same_v<E, faar_shape> || std::is_same_v<E, faar_hparams> || std::is_same_v<E, faar_model>;
  T v;
  bool set(PyObject* o) {
    if constexpr (STRUCT) {                        // copied, so nothing is held while the GIL is released
      Py_buffer b;
      if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
      const bool fits = (size_t)b.len == sizeof(E);
      if (fits) copy = *reinterpret_cast<const E*>(b.buf);
      PyBuffer_Release(&b);
      if (!fits) { PyErr_SetString(PyExc_TypeError, "structure of another size"); return false; }
      v = &copy;
      return true;
    } else {
      void* p;
      if (!to_address(o, &p)) return false;
      v = reinterpret_cast<T>(p);
      return true;
    }
  }
  std::conditional_t<STRUCT, E, char> copy;
};

#define ENTRIES(X)                                                                                                        \
  X(faar_workspace_init) X(faar_softquant_init) X(faar_softquant_eval) X(faar_softquant_operand_f32)                      \
  X(faar_transpose_bf16) X(faar_act_fakequant) X(faar_layer_ref) X(faar_layer_fwd) X(faar_layer_dx)                       \
  X(faar_layer_dx_operand) X(faar_silu_mul) X(faar_round_loss) X(faar_round_loss_static) X(faar_layer_bwd)                \
  X(faar_layer_bwd_rowmajor) X(faar_layer_step) X(faar_layer_step_rowmajor) X(faar_layer_step_host) X(faar_nvfp4_expand)                              \
  X(faar_layer_step_host_nvfp4) X(faar_harden_pack) X(faar_align_loss) X(faar_swizzle_scales) X(faar_rmsnorm)             \
  X(faar_rmsnorm_bwd) X(faar_add_rmsnorm) X(faar_rmsnorm_bwd_sum) X(faar_rope) X(faar_silu_mul_bwd) X(faar_embedding)     \
  X(faar_add) X(faar_attention_fwd) X(faar_attention_bwd) X(faar_nvfp4_gemm) X(faar_model_forward) X(faar_model_forward_both) X(faar_model_backward) \
  X(faar_model_forward_stats) X(faar_model_forward_both_stats) X(faar_logit_stats) X(faar_align_loss_stats)

enum {
#define SLOT(name) SLOT_##name,
  ENTRIES(SLOT)
#undef SLOT
  N_SLOTS
};
const char* const entry_names[N_SLOTS] = {
#define NAME(name) #name,
    ENTRIES(NAME)
#undef NAME
};
void* entry_points[N_SLOTS];

template <int SLOT, class F> struct Call;
template <int SLOT, class... A> struct Call<SLOT, int(A...)> {
  template <size_t... I>
  static PyObject* invoke(PyObject* const* args, std::index_sequence<I...>) {
    std::tuple<Arg<A>...> a;
    if (!(std::get<I>(a).set(args[I]) && ...)) return nullptr;
    auto* fn = reinterpret_cast<int (*)(A...)>(entry_points[SLOT]);
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = fn(std::get<I>(a).v...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
  }
  static PyObject* fast(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != (Py_ssize_t)sizeof...(A)) {
      PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, got %zd", entry_names[SLOT], (Py_ssize_t)sizeof...(A), n);
      return nullptr;
    }
    if (!entry_points[SLOT]) {
      PyErr_SetString(PyExc_RuntimeError, "load() has not been called");
      return nullptr;
    }
    return invoke(args, std::index_sequence_for<A...>{});
  }
};

PyObject* load(PyObject*, PyObject* path) {
  const char* p = PyUnicode_AsUTF8(path);
  if (!p) return nullptr;
  void* h = dlopen(p, RTLD_NOW | RTLD_LOCAL);      // the same handle ctypes holds: opened once per process
  if (!h) { PyErr_SetString(PyExc_OSError, dlerror()); return nullptr; }
  void* found[N_SLOTS];
  for (int i = 0; i < N_SLOTS; ++i) {
    found[i] = dlsym(h, entry_names[i]);
    if (!found[i]) { PyErr_Format(PyExc_OSError, "%s: no symbol %s", p, entry_names[i]); return nullptr; }
  }
  for (int i = 0; i < N_SLOTS; ++i) entry_points[i] = found[i];
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"load", load, METH_O, "Resolves the entry points in the library at this path."},
#define METHOD(name)                                                                                                       \
  {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&Call<SLOT_##name, decltype(::name)>::fast)),         \
   METH_FASTCALL, nullptr},
    ENTRIES(METHOD)
#undef METHOD
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_faarbind", "Calls into libfaar.so", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__faarbind(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  if (!s_data_ptr || !s_is_cuda) return nullptr;
  return PyModule_Create(&module);
}
