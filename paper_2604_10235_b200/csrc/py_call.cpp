// Python extension `_cccall`: calls an entry point of libcodecomp with tensors as arguments.
//
// call(fn, spec, *args) turns every argument into one machine word as the characters of spec say and
// calls fn (the address of a C function that takes only pointers and integers) with the GIL
// released; it returns the function's status.  A call marshalled argument by argument through
// ctypes costs about 8 us of host time, as much as a short prompt's kernels take; this costs 1.5 us.
//   i  an integer                         t  a CUDA tensor, or None for NULL
//   p  a CUDA or page-locked host tensor, or None
//   w  a CUDA tensor as two words: address, number of elements
//   L  a sequence of tensors as a host array of addresses, or None
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include <utility>
#include <vector>

namespace {

constexpr int kMaxWords = 20;

PyObject *s_data_ptr, *s_is_cuda, *s_is_pinned, *s_numel;

bool word_of(PyObject* o, uint64_t* out) {
  *out = PyLong_AsUnsignedLongLongMask(o);
  return !(*out == (uint64_t)-1 && PyErr_Occurred());
}

// result of a method without arguments as a word
bool word_from(PyObject* o, PyObject* method, uint64_t* out) {
  PyObject* r = PyObject_CallMethodNoArgs(o, method);
  if (!r) return false;
  const bool ok = word_of(r, out);
  Py_DECREF(r);
  return ok;
}

bool is_true(PyObject* r) {
  const bool yes = r == Py_True;
  Py_XDECREF(r);
  return yes;
}

bool tensor_word(PyObject* o, bool pinned_ok, uint64_t* out) {
  if (o == Py_None) {
    *out = 0;
    return true;
  }
  if (!is_true(PyObject_GetAttr(o, s_is_cuda))) {
    if (PyErr_Occurred()) return false;
    if (!pinned_ok || !is_true(PyObject_CallMethodNoArgs(o, s_is_pinned))) {
      if (!PyErr_Occurred())
        PyErr_SetString(PyExc_ValueError, pinned_ok ? "libcodecomp takes CUDA tensors only (or page-locked host memory here)"
                                                    : "libcodecomp takes CUDA tensors only");
      return false;
    }
  }
  return word_from(o, s_data_ptr, out);
}

template <size_t... I>
int call_n(uint64_t fn, const uint64_t* a, std::index_sequence<I...>) {
  return reinterpret_cast<int (*)(decltype((void)I, uint64_t())...)>(fn)(a[I]...);
}

int dispatch(uint64_t fn, const uint64_t* a, int n) {
  switch (n) {
#define CASE(k) case k: return call_n(fn, a, std::make_index_sequence<k>());
    CASE(5) CASE(6) CASE(7) CASE(8) CASE(9) CASE(10) CASE(11) CASE(12) CASE(13) CASE(14) CASE(15) CASE(16) CASE(17)
#undef CASE
  }
  return 1;
}

PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  uint64_t fn, a[kMaxWords];
  char* spec;
  Py_ssize_t len;
  if (n_args < 2 || !word_of(args[0], &fn) || PyBytes_AsStringAndSize(args[1], &spec, &len) < 0) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "call(fn, spec, *args)");
    return nullptr;
  }
  if (len != n_args - 2) {
    PyErr_SetString(PyExc_TypeError, "one character of spec per argument");
    return nullptr;
  }
  std::vector<std::vector<uint64_t>> lists;      // host arrays of the call (moving the outer one keeps their storage)
  int n = 0;
  for (Py_ssize_t i = 0; i < len; ++i) {
    PyObject* o = args[i + 2];
    bool ok = n + 2 <= kMaxWords;
    switch (ok ? spec[i] : '?') {
      case 'i': ok = word_of(o, &a[n++]); break;
      case 't': ok = tensor_word(o, false, &a[n++]); break;
      case 'p': ok = tensor_word(o, true, &a[n++]); break;
      case 'w': ok = tensor_word(o, false, &a[n]) && word_from(o, s_numel, &a[n + 1]); n += 2; break;
      case 'L': {
        if (o == Py_None) { a[n++] = 0; break; }
        PyObject* seq = PySequence_Fast(o, "a sequence of tensors");
        if (!seq) return nullptr;
        const Py_ssize_t m = PySequence_Fast_GET_SIZE(seq);
        lists.emplace_back((size_t)m + 1);
        for (Py_ssize_t j = 0; j < m && ok; ++j) ok = word_from(PySequence_Fast_GET_ITEM(seq, j), s_data_ptr, &lists.back()[j]);
        Py_DECREF(seq);
        a[n++] = (uint64_t)(uintptr_t)lists.back().data();
        break;
      }
      default: ok = false;
    }
    if (!ok) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "bad spec");
      return nullptr;
    }
  }
  if (n < 5 || n > 17) {
    PyErr_SetString(PyExc_TypeError, "5 to 17 words");
    return nullptr;
  }
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = dispatch(fn, a, n);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

PyMethodDef methods[] = {
    {"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call(fn, spec, *args) -> status"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_cccall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__cccall(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  s_is_pinned = PyUnicode_InternFromString("is_pinned");
  s_numel = PyUnicode_InternFromString("numel");
  return PyModule_Create(&module);
}
