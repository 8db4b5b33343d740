// Python extension `_cccall`: calls an entry point of libcodecomp with tensors as arguments.
//
// bind(name, address, spec) makes a callable of an entry point that takes only pointers and integers: it
// turns every argument into one machine word as the characters of spec say, converts the words to the
// parameter types that codecomp.h declares, calls the function with the GIL released and returns its status.
// A call marshalled argument by argument through ctypes costs about 8 us of host time, as much as a short
// prompt's kernels take; this costs 1.5 us.
//   i  an integer                         t  a CUDA tensor, or None for NULL
//   p  a CUDA or page-locked host tensor, or None
//   w  a CUDA tensor as two words: address, number of elements
//   L  a sequence of tensors as a host array of addresses, or None
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include <new>
#include <type_traits>
#include <utility>
#include <vector>

#include "codecomp.h"

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

template <class T>
T from_word(uint64_t w) {
  if constexpr (std::is_pointer_v<T>) return reinterpret_cast<T>((uintptr_t)w);
  else return static_cast<T>(w);
}

template <class F> struct Caller;
template <class... A>
struct Caller<int (*)(A...)> {
  static constexpr int words = sizeof...(A);
  static_assert(words <= kMaxWords, "words of a call");
  static int call(void* fn, const uint64_t* a) { return spread(fn, a, std::index_sequence_for<A...>()); }
  template <size_t... I>
  static int spread(void* fn, const uint64_t* a, std::index_sequence<I...>) {
    return reinterpret_cast<int (*)(A...)>(fn)(from_word<A>(a[I])...);
  }
};

struct Entry {
  const char* name;
  int words;
  int (*call)(void* fn, const uint64_t* a);
};
#define ENTRY(f) {#f, Caller<decltype(&f)>::words, Caller<decltype(&f)>::call}
const Entry kEntries[] = {ENTRY(cc_score_window), ENTRY(cc_fuse_prior_pool), ENTRY(cc_topk_select),
                          ENTRY(cc_topk_select_static), ENTRY(cc_compact_kv), ENTRY(cc_compress_layer),
                          ENTRY(cc_compress_layers), ENTRY(cc_ppl_chunk_scores), ENTRY(cc_select_chunks)};
#undef ENTRY

struct Bound {                // what a callable holds: an entry point of a loaded library and the spec of its arguments
  const Entry* entry;
  void* fn;
  int n_args;
  char spec[kMaxWords];
};
const char* const kBound = "_cccall.Bound";

PyObject* call_bound(PyObject* self, PyObject* const* args, Py_ssize_t n_args) {
  const Bound* f = static_cast<const Bound*>(PyCapsule_GetPointer(self, kBound));
  if (!f) return nullptr;
  if (n_args != f->n_args) {
    PyErr_Format(PyExc_TypeError, "%s takes %d arguments, %zd were given", f->entry->name, f->n_args, n_args);
    return nullptr;
  }
  uint64_t a[kMaxWords];
  std::vector<std::vector<uint64_t>> lists;      // host arrays of the call (moving the outer one keeps their storage)
  int n = 0;
  for (Py_ssize_t i = 0; i < n_args; ++i) {
    PyObject* o = args[i];
    bool ok = true;
    switch (f->spec[i]) {
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
    }
    if (!ok) return nullptr;
  }
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f->entry->call(f->fn, a);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

PyObject* call(PyObject* self, PyObject* const* args, Py_ssize_t n_args) {
  try {
    return call_bound(self, args, n_args);
  } catch (const std::bad_alloc&) {            // of a host array of addresses
    return PyErr_NoMemory();
  }
}

PyMethodDef bound_call = {"bound", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "an entry point: (*args) -> status"};

PyObject* bind(PyObject*, PyObject* args) {
  const char *name, *spec;
  Py_ssize_t len;
  PyObject* address;
  uint64_t fn;
  if (!PyArg_ParseTuple(args, "sOy#", &name, &address, &spec, &len) || !word_of(address, &fn)) return nullptr;
  const Entry* entry = nullptr;
  for (const Entry& e : kEntries)
    if (strcmp(e.name, name) == 0) entry = &e;
  if (!entry) return PyErr_Format(PyExc_ValueError, "%s cannot be bound", name);
  int words = 0;
  for (Py_ssize_t i = 0; i < len; ++i) {
    if (!spec[i] || !strchr("itpwL", spec[i])) return PyErr_Format(PyExc_ValueError, "unknown kind of argument in the spec of %s", name);
    words += spec[i] == 'w' ? 2 : 1;
  }
  if (words != entry->words) return PyErr_Format(PyExc_ValueError, "%s takes %d words, its spec gives %d", name, entry->words, words);
  Bound* f = new (std::nothrow) Bound{entry, reinterpret_cast<void*>((uintptr_t)fn), (int)len, {}};
  if (!f) return PyErr_NoMemory();
  memcpy(f->spec, spec, (size_t)len);
  PyObject* capsule = PyCapsule_New(f, kBound, [](PyObject* c) { delete static_cast<Bound*>(PyCapsule_GetPointer(c, kBound)); });
  if (!capsule) {
    delete f;
    return nullptr;
  }
  PyObject* callable = PyCFunction_New(&bound_call, capsule);
  Py_DECREF(capsule);
  return callable;
}

PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, "bind(name, address, spec) -> callable"},
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
