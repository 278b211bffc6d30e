// The calling side of binding.py: checks of the tensors a call is given, their addresses, the current
// stream, and the call itself, in one step of native code.  (Through ctypes and torch's Python
// attributes the same steps cost 6 us per call, more than the device needs for a small one: a drafted
// token went from 11.0 to 6.2 us.)  The library's functions come as addresses from binding.py,
// which loads it; nothing here computes.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <vector>

#include "ersd.h"

namespace {

decltype(&ersd_race_sample) f_race_sample;
decltype(&ersd_verify) f_verify;
decltype(&ersd_verify_noalloc) f_verify_noalloc;
decltype(&ersd_verify_tokens) f_verify_tokens;
decltype(&ersd_verify_tree) f_verify_tree;
decltype(&ersd_gsd_verify) f_gsd_verify;
decltype(&ersd_gsd_verify_tree) f_gsd_verify_tree;

PyObject* options_type;  // binding.py's ErsdOpts

struct Failed {};  // a Python exception is set

const char* dtype_name(at::ScalarType t) {
  switch (t) {
    case at::kInt: return "torch.int32";
    case at::kLong: return "torch.int64";
    case at::kFloat: return "torch.float32";
    case at::kBFloat16: return "torch.bfloat16";
    case at::kHalf: return "torch.float16";
    case at::kDouble: return "torch.float64";
    default: return c10::toString(t);
  }
}

// A contiguous CUDA tensor (of type `want` unless that is Undefined).
const at::Tensor& tensor(PyObject* o, at::ScalarType want, const char* name) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
    throw Failed();
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_cuda()) {
    PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor", name);
    throw Failed();
  }
  if (want != at::ScalarType::Undefined && t.scalar_type() != want) {
    PyErr_Format(PyExc_TypeError, "%s must be %s", name, dtype_name(want));
    throw Failed();
  }
  if (!t.is_contiguous()) {
    PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
    throw Failed();
  }
  return t;
}
const void* optional_tensor(PyObject* o, at::ScalarType want, const char* name) {
  return o == Py_None ? nullptr : tensor(o, want, name).data_ptr();
}

struct Logits {
  const void* data;
  at::ScalarType type;
  ersd_dtype code;
  int B, rows, V;
};
// Logits [B, rows, ld]; V (None: ld) is the vocabulary's size.
Logits logits(PyObject* o, PyObject* v, const char* name) {
  const at::Tensor& t = tensor(o, at::ScalarType::Undefined, name);
  Logits l;
  l.data = t.data_ptr();
  l.type = t.scalar_type();
  if (t.dim() != 3) {
    PyErr_Format(PyExc_ValueError, "%s must have three dimensions, got %d", name, (int)t.dim());
    throw Failed();
  }
  const int64_t ld = t.size(2);
  int64_t V = ld;
  if (v != Py_None) {
    PyObject* n = PyNumber_Long(v);
    if (!n) throw Failed();
    V = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (V == -1 && PyErr_Occurred()) throw Failed();
    if (V < 1 || V > ld) {
      PyErr_SetString(PyExc_ValueError, "V must be between 1 and the row length of the tensor");
      throw Failed();
    }
  }
  if (t.size(0) > INT32_MAX || t.size(1) > INT32_MAX || V > INT32_MAX) {
    PyErr_Format(PyExc_ValueError, "%s has too many rows or columns", name);
    throw Failed();
  }
  l.B = (int)t.size(0);
  l.rows = (int)t.size(1);
  l.V = (int)V;
  return l;
}
void logits_code(Logits& l) {
  if (l.type == at::kFloat) l.code = ERSD_F32;
  else if (l.type == at::kBFloat16) l.code = ERSD_BF16;
  else {
    PyErr_Format(PyExc_TypeError, "logits must be float32 or bfloat16, got %s", dtype_name(l.type));
    throw Failed();
  }
}

float number(PyObject* o) {
  PyObject* f = PyNumber_Float(o);
  if (!f) throw Failed();
  const double v = PyFloat_AS_DOUBLE(f);
  Py_DECREF(f);
  return (float)v;
}

void* stream_of(PyObject* o) {
  if (o == Py_None) return (void*)c10::cuda::getCurrentCUDAStream().stream();
  PyObject* a = PyObject_GetAttrString(o, "cuda_stream");
  if (!a) throw Failed();
  void* p = PyLong_AsVoidPtr(a);
  Py_DECREF(a);
  if (!p && PyErr_Occurred()) throw Failed();
  return p;
}

// The options structure (an ErsdOpts, which lends its memory), or none.  Nothing else is taken: the
// library copies the whole structure, addresses and all.
struct Options {
  Py_buffer view;
  const ersd_opts* ptr = nullptr;
  explicit Options(PyObject* o) {
    if (o == Py_None) return;
    const int is_options = PyObject_IsInstance(o, options_type);
    if (is_options < 0) throw Failed();
    if (!is_options) {
      PyErr_Format(PyExc_TypeError, "opts must be an ErsdOpts (see make_opts), got %s", Py_TYPE(o)->tp_name);
      throw Failed();
    }
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Failed();
    if (view.len < (Py_ssize_t)sizeof(ersd_opts)) {
      PyBuffer_Release(&view);
      PyErr_Format(PyExc_TypeError, "opts has %d bytes, the library's options %d", (int)view.len, (int)sizeof(ersd_opts));
      throw Failed();
    }
    ptr = (const ersd_opts*)view.buf;
  }
  ~Options() {
    if (ptr) PyBuffer_Release(&view);
  }
  Options(const Options&) = delete;
};

std::vector<int32_t> parents(PyObject* o, int nodes) {
  PyObject* seq = PySequence_Fast(o, "parent must be a sequence of integers");
  if (!seq) throw Failed();
  std::vector<int32_t> p((size_t)PySequence_Fast_GET_SIZE(seq));
  for (size_t i = 0; i < p.size(); ++i) {
    PyObject* n = PyNumber_Long(PySequence_Fast_GET_ITEM(seq, (Py_ssize_t)i));
    const long v = n ? PyLong_AsLong(n) : -1;
    Py_XDECREF(n);
    if (v == -1 && PyErr_Occurred()) {
      Py_DECREF(seq);
      throw Failed();
    }
    p[i] = (int32_t)v;
  }
  Py_DECREF(seq);
  if (p.size() < (size_t)nodes) {
    PyErr_Format(PyExc_ValueError, "parent must have an entry for each of the %d nodes", nodes);
    throw Failed();
  }
  return p;
}

// Runs the call without the interpreter's lock; its status as a Python number.
template <typename F>
PyObject* status_of(F&& call) {
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(status);
}

template <int N, typename F>
PyObject* guarded(Py_ssize_t n, F&& body) {
  if (n != N) {
    PyErr_Format(PyExc_TypeError, "%d arguments wanted, got %d", N, (int)n);
    return nullptr;
  }
  try {
    return body();
  } catch (const Failed&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// race_sample(logits, seeds, T, out_tok, opts, stream, V)
PyObject* race_sample(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded<7>(n, [&]() {
    const Options o(a[4]);
    tensor(a[0], at::ScalarType::Undefined, "logits");
    const void* seeds = tensor(a[1], at::kLong, "seeds").data_ptr();
    int32_t* out = (int32_t*)tensor(a[3], at::kInt, "out_tok").data_ptr();
    Logits l = logits(a[0], a[6], "logits");
    logits_code(l);
    const float T = number(a[2]);
    void* st = stream_of(a[5]);
    return status_of([&] { return f_race_sample(l.data, l.code, (const uint64_t*)seeds, l.B, l.rows, l.V, T, out, o.ptr, st); });
  });
}

// verify(target, draft, seeds, T, out_tokens, out_accept_len, opts, stream, V)
template <typename Fn>
PyObject* verify_with(PyObject* const* a, Py_ssize_t n, Fn fn) {
  return guarded<9>(n, [&]() {
    const Options o(a[6]);
    Logits l = logits(a[0], a[8], "target_logits");
    const void* draft = optional_tensor(a[1], l.type, "draft_logits");
    const void* seeds = tensor(a[2], at::kLong, "seeds").data_ptr();
    int32_t* tok = (int32_t*)tensor(a[4], at::kInt, "out_tokens").data_ptr();
    int32_t* acc = (int32_t*)tensor(a[5], at::kInt, "out_accept_len").data_ptr();
    logits_code(l);
    const float T = number(a[3]);
    void* st = stream_of(a[7]);
    return status_of([&] { return fn(l.data, draft, l.code, (const uint64_t*)seeds, l.B, l.rows - 1, l.V, T, tok, acc, o.ptr, st); });
  });
}
PyObject* verify(PyObject*, PyObject* const* a, Py_ssize_t n) { return verify_with(a, n, f_verify); }
PyObject* verify_noalloc(PyObject*, PyObject* const* a, Py_ssize_t n) { return verify_with(a, n, f_verify_noalloc); }

// verify_tokens(target, draft_tokens, seeds, T, out_tokens, out_accept_len, opts, stream, V)
PyObject* verify_tokens(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded<9>(n, [&]() {
    const Options o(a[6]);
    Logits l = logits(a[0], a[8], "target_logits");
    const void* given = optional_tensor(a[1], at::kInt, "draft_tokens");
    const void* seeds = tensor(a[2], at::kLong, "seeds").data_ptr();
    int32_t* tok = (int32_t*)tensor(a[4], at::kInt, "out_tokens").data_ptr();
    int32_t* acc = (int32_t*)tensor(a[5], at::kInt, "out_accept_len").data_ptr();
    logits_code(l);
    const float T = number(a[3]);
    void* st = stream_of(a[7]);
    return status_of([&] {
      return f_verify_tokens(l.data, (const int32_t*)given, l.code, (const uint64_t*)seeds, l.B, l.rows - 1, l.V, T, tok, acc, o.ptr, st);
    });
  });
}

// verify_tree(target, draft, parent, seeds, T, out_tokens, out_accept_len, opts, stream, V)
PyObject* verify_tree(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded<10>(n, [&]() {
    const Options o(a[7]);
    Logits l = logits(a[0], a[9], "target_logits");
    const void* draft = optional_tensor(a[1], l.type, "draft_logits");
    const void* seeds = tensor(a[3], at::kLong, "seeds").data_ptr();
    int32_t* tok = (int32_t*)tensor(a[5], at::kInt, "out_tokens").data_ptr();
    int32_t* acc = (int32_t*)tensor(a[6], at::kInt, "out_accept_len").data_ptr();
    const std::vector<int32_t> parent = parents(a[2], l.rows);
    logits_code(l);
    const float T = number(a[4]);
    void* st = stream_of(a[8]);
    return status_of([&] {
      return f_verify_tree(l.data, draft, l.code, parent.data(), (const uint64_t*)seeds, l.B, l.rows - 1, l.V, T, tok, acc, o.ptr, st);
    });
  });
}

// gsd_verify(target, draft, draft_tokens, seeds, T, out_tokens, out_accept_len, opts, stream, V)
PyObject* gsd_verify(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded<10>(n, [&]() {
    const Options o(a[7]);
    Logits l = logits(a[0], a[9], "target_logits");
    const void* draft = optional_tensor(a[1], l.type, "draft_logits");
    const void* given = optional_tensor(a[2], at::kInt, "draft_tokens");
    const void* seeds = tensor(a[3], at::kLong, "seeds").data_ptr();
    int32_t* tok = (int32_t*)tensor(a[5], at::kInt, "out_tokens").data_ptr();
    int32_t* acc = (int32_t*)tensor(a[6], at::kInt, "out_accept_len").data_ptr();
    logits_code(l);
    const float T = number(a[4]);
    void* st = stream_of(a[8]);
    return status_of([&] {
      return f_gsd_verify(l.data, draft, (const int32_t*)given, l.code, (const uint64_t*)seeds, l.B, l.rows - 1, l.V, T, tok, acc, o.ptr, st);
    });
  });
}

// gsd_verify_tree(target, draft, draft_tokens, parent, seeds, T, out_tokens, out_accept_len, opts, stream, V)
PyObject* gsd_verify_tree(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded<11>(n, [&]() {
    const Options o(a[8]);
    Logits l = logits(a[0], a[10], "target_logits");
    const void* draft = optional_tensor(a[1], l.type, "draft_logits");
    const void* given = optional_tensor(a[2], at::kInt, "draft_tokens");
    const void* seeds = tensor(a[4], at::kLong, "seeds").data_ptr();
    int32_t* tok = (int32_t*)tensor(a[6], at::kInt, "out_tokens").data_ptr();
    int32_t* acc = (int32_t*)tensor(a[7], at::kInt, "out_accept_len").data_ptr();
    const std::vector<int32_t> parent = parents(a[3], l.rows);
    logits_code(l);
    const float T = number(a[5]);
    void* st = stream_of(a[9]);
    return status_of([&] {
      return f_gsd_verify_tree(l.data, draft, (const int32_t*)given, l.code, parent.data(), (const uint64_t*)seeds, l.B, l.rows - 1, l.V, T,
                               tok, acc, o.ptr, st);
    });
  });
}

// use(race_sample, verify, verify_noalloc, verify_tokens, verify_tree, gsd_verify, gsd_verify_tree, opts): the
// library's functions, as addresses, and the type of the options structure
PyObject* use(PyObject*, PyObject* args) {
  unsigned long long f[7];
  PyObject* type;
  if (!PyArg_ParseTuple(args, "KKKKKKKO", &f[0], &f[1], &f[2], &f[3], &f[4], &f[5], &f[6], &type)) return nullptr;
  if (!PyType_Check(type)) {
    PyErr_SetString(PyExc_TypeError, "the type of the options structure is wanted");
    return nullptr;
  }
  Py_INCREF(type);
  Py_XDECREF(options_type);
  options_type = type;
  f_race_sample = (decltype(f_race_sample))(uintptr_t)f[0];
  f_verify = (decltype(f_verify))(uintptr_t)f[1];
  f_verify_noalloc = (decltype(f_verify_noalloc))(uintptr_t)f[2];
  f_verify_tokens = (decltype(f_verify_tokens))(uintptr_t)f[3];
  f_verify_tree = (decltype(f_verify_tree))(uintptr_t)f[4];
  f_gsd_verify = (decltype(f_gsd_verify))(uintptr_t)f[5];
  f_gsd_verify_tree = (decltype(f_gsd_verify_tree))(uintptr_t)f[6];
  Py_RETURN_NONE;
}

#define FAST(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {{"use", use, METH_VARARGS, nullptr}, FAST(race_sample), FAST(verify), FAST(verify_noalloc), FAST(verify_tokens),
                         FAST(verify_tree), FAST(gsd_verify), FAST(gsd_verify_tree), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_ersd_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (torch_version: the torch this was built against, whose tensors alone it can take apart)
PyMODINIT_FUNC PyInit__ersd_call() {
  PyObject* m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "torch_version", ERSD_TORCH_VERSION) != 0) Py_CLEAR(m);
  return m;
}
