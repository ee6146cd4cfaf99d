// The calls of the Python binding.  ptr and stream: the device pointer of a tensor (with the check that it is a contiguous CUDA
// tensor) and the current stream.  bind: callables for entry points of libdet.so that convert their own arguments, tensors, numbers, a
// workspace and the current stream, call with the interpreter's lock released and raise on a status that is not DET_OK.  One call of 19
// arguments took some 7 us of the host through a Python expression per argument and ctypes, and those calls, not the GPU,
// are what a single small linear waits for.  Numbers that are no Python int or float go through ctypes as before.
#include <Python.h>
#include <dlfcn.h>

#include <memory>
#include <string>
#include <type_traits>
#include <utility>

#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/Exceptions.h>
#include <ATen/Context.h>
#include <c10/cuda/CUDAStream.h>

#include "../../include/det.h"

// address of a contiguous CUDA tensor; None is 0 and integers are taken as they are; false with an error set
static bool address_of(PyObject* t, unsigned long long& out) {
  if (THPVariable_Check(t)) {
    const at::Tensor& x = THPVariable_Unpack(t);
    if (!x.is_cuda() || !x.is_contiguous()) {
      PyErr_SetString(PyExc_AssertionError, "tensors must be contiguous CUDA tensors");
      return false;
    }
    out = reinterpret_cast<unsigned long long>(x.data_ptr());
    return true;
  }
  if (t == Py_None) { out = 0; return true; }
  if (PyLong_Check(t)) {
    out = PyLong_AsUnsignedLongLongMask(t);
    return !PyErr_Occurred();
  }
  PyErr_Format(PyExc_TypeError, "expected a CUDA tensor, an address or None, got %s", Py_TYPE(t)->tp_name);
  return false;
}
static unsigned long long current_stream() {
  at::globalContext().lazyInitDevice(c10::DeviceType::CUDA);
  return reinterpret_cast<unsigned long long>(c10::cuda::getCurrentCUDAStream().stream());
}

// None and integers pass through, a tensor becomes its address
static PyObject* ptr(PyObject*, PyObject* t) {
  HANDLE_TH_ERRORS
  if (t == Py_None || PyLong_Check(t)) {
    Py_INCREF(t);
    return t;
  }
  unsigned long long a;
  return address_of(t, a) ? PyLong_FromUnsignedLongLong(a) : nullptr;
  END_HANDLE_TH_ERRORS
}
static PyObject* stream(PyObject*, PyObject*) {
  HANDLE_TH_ERRORS
  return PyLong_FromUnsignedLongLong(current_stream());
  END_HANDLE_TH_ERRORS
}

// ---- entry points ---------------------------------------------------------------------------------------------------
union Slot {                                   // one C argument
  unsigned long long u;
  float f;
};
constexpr int MAX_ARGS = 24;
template <class A>
static A slot_as(const Slot& s) {
  if constexpr (std::is_pointer<A>::value) return reinterpret_cast<A>(s.u);
  else if constexpr (std::is_same<A, float>::value) return s.f;
  else return static_cast<A>(s.u);
}
template <class A>
static constexpr char kind_of() {              // the letters of a signature; v: void*, what a workspace and a stream are declared as
  return std::is_same<A, void*>::value ? 'v' : std::is_pointer<A>::value ? 'p' : std::is_same<A, float>::value ? 'f' : sizeof(A) == 8 ? 'z' : 'i';
}
// whether a pattern gives each C argument what its type takes: a stream and a workspace only where there is a void*
static bool fits(const char* pattern, const std::string& kinds) {
  size_t n = 0;
  for (const char* c = pattern; *c; ++c) {
    const char k = n < kinds.size() ? kinds[n++] : 0;
    if (*c == 'w' ? k != 'v' || kinds[n++] != 'z' : *c == 's' ? k != 'v' : *c == 'p' ? k != 'p' && k != 'v' : k != *c || k == 'v') return false;
  }
  return n == kinds.size();
}
template <class... A, size_t... I>
static int invoke(int (*fn)(A...), const Slot* s, std::index_sequence<I...>) { return fn(slot_as<A>(s[I])...); }
template <class F> struct Typed;
template <class... A>
struct Typed<int(A...)> {
  static_assert(sizeof...(A) <= MAX_ARGS, "more arguments than slots");
  static int call(void* fn, const Slot* s) { return invoke(reinterpret_cast<int (*)(A...)>(fn), s, std::index_sequence_for<A...>()); }
  static std::string kinds() { return std::string{kind_of<A>()...}; }
};

struct Entry {
  const char* name;
  int (*call)(void*, const Slot*);
  std::string (*kinds)();
  PyMethodDef def;
};
static PyObject* entry_call(PyObject* self, PyObject* const* args, Py_ssize_t nargs);
#define DET_ENTRY(f) \
  {#f, &Typed<decltype(f)>::call, &Typed<decltype(f)>::kinds, {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry_call)), METH_FASTCALL, nullptr}}
static Entry entries[] = {
    DET_ENTRY(det_sum), DET_ENTRY(det_sum_static), DET_ENTRY(det_scale_inplace), DET_ENTRY(det_lsq_weight_scale), DET_ENTRY(det_lsq_act_scale_init),
    DET_ENTRY(det_lsq_quantize_weight), DET_ENTRY(det_linear_fwd), DET_ENTRY(det_linear_fwd_q), DET_ENTRY(det_linear_bwd), DET_ENTRY(det_rmsnorm_fwd),
    DET_ENTRY(det_rmsnorm_fwd_q), DET_ENTRY(det_residual_rmsnorm_fwd), DET_ENTRY(det_headnorm_fwd), DET_ENTRY(det_headnorm_bwd), DET_ENTRY(det_rope),
    DET_ENTRY(det_rmsnorm_bwd), DET_ENTRY(det_rmsnorm_bwd_residual), DET_ENTRY(det_xent_fwd), DET_ENTRY(det_xent_bwd), DET_ENTRY(det_attn_fwd),
    DET_ENTRY(det_attn_fwd_q), DET_ENTRY(det_attn_fwd_int8pv), DET_ENTRY(det_attn_bwd), DET_ENTRY(det_attn_bwd_fixq), DET_ENTRY(det_swiglu_fwd),
    DET_ENTRY(det_swiglu_fwd_q), DET_ENTRY(det_swiglu_bwd), DET_ENTRY(det_residual_add), DET_ENTRY(det_embed_fwd), DET_ENTRY(det_embed_bwd),
    DET_ENTRY(det_lmhead_fwd), DET_ENTRY(det_lmhead_fwd_v2), DET_ENTRY(det_lmhead_bwd), DET_ENTRY(det_lmhead_bwd_v2), DET_ENTRY(det_attn_fwd_v2),
    DET_ENTRY(det_tensor_hash_async)};

// One callable that bind returns, owned by the capsule that is its self: nothing is shared between two results of bind.
struct Callable {
  const Entry* entry;
  void* fn;
  std::string pattern;                         // per Python argument: p i z f, or w a workspace (its address and size); s the current stream
  PyObject* general = nullptr;                 // the entry point with its C types declared (ctypes)
  PyObject* raise_status = nullptr;            // raise_status(name, status)
  ~Callable() { Py_XDECREF(general); Py_XDECREF(raise_status); }
};
static void callable_free(PyObject* capsule) { delete static_cast<Callable*>(PyCapsule_GetPointer(capsule, nullptr)); }

// The call with arguments that are not plain Python numbers: addresses, sizes and the stream as they have been found, the numbers as
// they came, so that what is taken for a number, and the error for what is not, are those of the declared types.
static bool call_general(const Callable& e, const Slot* s, PyObject* const* args, int& rc) {
  PyObject* t = PyTuple_New((Py_ssize_t)e.entry->kinds().size());
  if (!t) return false;
  Py_ssize_t n = 0;
  for (const char c : e.pattern) {
    if (c != 's') ++args;
    for (int k = 0; k < (c == 'w' ? 2 : 1); ++k, ++n) {
      PyObject* x = c == 'i' || c == 'z' || c == 'f' ? Py_NewRef(args[-1]) : PyLong_FromUnsignedLongLong(s[n].u);
      if (!x) { Py_DECREF(t); return false; }
      PyTuple_SET_ITEM(t, n, x);
    }
  }
  PyObject* r = PyObject_CallObject(e.general, t);
  Py_DECREF(t);
  if (!r) return false;
  rc = (int)PyLong_AsLong(r);
  Py_DECREF(r);
  return !PyErr_Occurred();
}
static PyObject* entry_call(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
  HANDLE_TH_ERRORS
  const Callable* e = static_cast<const Callable*>(PyCapsule_GetPointer(self, nullptr));
  if (!e) return nullptr;
  const char* name = e->entry->name;
  Slot s[MAX_ARGS];
  int n = 0, rc;
  Py_ssize_t a = 0;
  bool plain = true;                           // every number is a Python int or float
  for (const char c : e->pattern) {
    if (c == 's') { s[n++].u = current_stream(); continue; }
    if (a == nargs) { PyErr_Format(PyExc_TypeError, "%s: too few arguments", name); return nullptr; }
    PyObject* x = args[a++];
    switch (c) {
      case 'p':
        if (!address_of(x, s[n++].u)) return nullptr;
        break;
      case 'w':                                // the size comes from the tensor, so an address alone is no workspace
        if (!address_of(x, s[n].u)) return nullptr;
        if (x == Py_None) s[n + 1].u = 0;
        else if (THPVariable_Check(x)) s[n + 1].u = THPVariable_Unpack(x).nbytes();
        else { PyErr_Format(PyExc_AttributeError, "%s: a workspace is a tensor or None", name); return nullptr; }
        n += 2;
        break;
      case 'f':
        plain = plain && (PyFloat_Check(x) || PyLong_Check(x));
        if (plain) {
          const double d = PyFloat_AsDouble(x);
          s[n].f = static_cast<float>(d);
          if (d == -1.0 && PyErr_Occurred()) { PyErr_Clear(); plain = false; }   // an integer beyond the range
        }
        ++n;
        break;
      default:
        plain = plain && PyLong_Check(x);
        if (plain) s[n].u = PyLong_AsUnsignedLongLongMask(x);
        ++n;
    }
  }
  if (a != nargs) { PyErr_Format(PyExc_TypeError, "%s: too many arguments", name); return nullptr; }
  if (plain) {
    Py_BEGIN_ALLOW_THREADS
    rc = e->entry->call(e->fn, s);
    Py_END_ALLOW_THREADS
  } else if (!call_general(*e, s, args, rc)) {
    return nullptr;
  }
  if (rc != DET_OK) return PyObject_CallFunction(e->raise_status, "si", name, rc);
  Py_RETURN_NONE;
  END_HANDLE_TH_ERRORS
}

// bind(path of libdet.so, {name: pattern}, raise_status, the library with its C types declared) -> {name: callable}
static PyObject* bind(PyObject*, PyObject* args) {
  HANDLE_TH_ERRORS
  const char* path;
  PyObject *patterns, *raise, *declared;
  if (!PyArg_ParseTuple(args, "sO!OO", &path, &PyDict_Type, &patterns, &raise, &declared)) return nullptr;
  void* lib = dlopen(path, RTLD_NOW);
  if (!lib) { PyErr_Format(PyExc_ImportError, "%s", dlerror()); return nullptr; }
  PyObject* out = PyDict_New();
  if (!out) return nullptr;
  for (Entry& e : entries) {
    PyObject* pat = PyDict_GetItemString(patterns, e.name);
    const char* p = pat ? PyUnicode_AsUTF8(pat) : nullptr;
    std::unique_ptr<Callable> own(new Callable);
    own->entry = &e;
    own->fn = dlsym(lib, e.name);
    if (!own->fn || !p || !fits(p, e.kinds())) {
      PyErr_Format(PyExc_ImportError, "%s: %s", e.name, own->fn ? "the pattern does not fit the declaration" : "not in the library");
      Py_DECREF(out);
      return nullptr;
    }
    own->pattern = p;
    own->general = PyObject_GetAttrString(declared, e.name);
    own->raise_status = Py_NewRef(raise);
    PyObject* self = own->general ? PyCapsule_New(own.get(), nullptr, callable_free) : nullptr;
    if (self) own.release();
    PyObject* f = self ? PyCFunction_New(&e.def, self) : nullptr;
    Py_XDECREF(self);
    const int bad = f ? PyDict_SetItemString(out, e.name, f) : -1;
    Py_XDECREF(f);
    if (bad) { Py_DECREF(out); return nullptr; }
  }
  return out;
  END_HANDLE_TH_ERRORS
}
static PyMethodDef methods[] = {{"ptr", ptr, METH_O, "device address of a contiguous CUDA tensor; None and integers as they are"},
                                {"stream", stream, METH_NOARGS, "handle of the current CUDA stream"},
                                {"bind", bind, METH_VARARGS, "callables for the library's entry points"},
                                {nullptr, nullptr, 0, nullptr}};
static PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods};
PyMODINIT_FUNC PyInit__binding() { return PyModule_Create(&module); }
