// Python binding of libunitscale (module _binding): argument marshalling in C.  `calls` maps the name of an entry point to a
// function that takes its arguments as torch tensors (for a us_mat, or for a device pointer), ctypes structures and arrays of the
// parameter's type, numbers and None, calls it with the GIL released and returns its status.  prepare() keeps such a call with its arguments
// converted, program() a sequence of them with the descriptions that change from pass to pass, and run() issues one pass.
//
// What a launch costs the host, us: a linear call through ctypes 7.1 (2.5 the launch itself), through this module 3.1; the three launches
// of a 256 x 128 x 512 FFN step 22 -> 12.3, many in a row 21 -> 11.0.
#include <Python.h>

#include <cuda_runtime.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <cstring>
#include <exception>
#include <memory>
#include <tuple>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/unitscale.h"

namespace {

struct Failed {};                                            // a Python exception is set

[[noreturn]] void fail(PyObject* type, const char* what) {
  PyErr_SetString(type, what);
  throw Failed();
}

int dtype_of(const at::Tensor& t) {
  switch (t.scalar_type()) {
    case at::kFloat: return US_F32;
    case at::kBFloat16: return US_BF16;
    case at::kHalf: return US_F16;
    case at::kFloat8_e4m3fn: return US_E4M3;
    case at::kFloat8_e5m2: return US_E5M2;
    default: fail(PyExc_KeyError, "tensor type without a us_dtype");
  }
}

// A 2-D row-major tensor (last stride 1) as a us_mat; a single row has whatever pitch its stride says, but its length at least.
us_mat describe(PyObject* o) {
  const at::Tensor& t = THPVariable_Unpack(o);
  if (t.dim() != 2 || (t.size(1) > 1 && t.stride(1) != 1)) fail(PyExc_ValueError, "expected a 2-D tensor with unit column stride");
  const int64_t rows = t.size(0), cols = t.size(1), ld = t.stride(0);
  return us_mat{t.data_ptr(), dtype_of(t), rows, cols, rows > 1 ? ld : std::max(cols, ld)};
}

// Argument conversion.  `mats` holds descriptions made for one immediate call.
struct Args {
  us_mat mats[16];
  int used = 0;
  bool immediate;                                            // tensors are taken only by calls that are not kept
  explicit Args(bool now) : immediate(now) {}
  us_mat* add(PyObject* tensor) {
    if (!immediate) fail(PyExc_TypeError, "a prepared call takes structures");
    if (used == 16) fail(PyExc_ValueError, "too many tensors");
    mats[used] = describe(tensor);
    return &mats[used++];
  }
};

// ctypes types of the structures (and of host numbers), as register_types() was given them
template <class T>
PyTypeObject* g_type = nullptr;
PyTypeObject* g_ctypes_array = nullptr;

// The memory of a ctypes object of T's type, or of an array of them, that holds `count` at least.
template <class T>
T* structure(PyObject* o, size_t count) {
  bool right = g_type<T> && PyObject_TypeCheck(o, g_type<T>);
  if (!right && PyObject_TypeCheck(o, g_ctypes_array)) {
    PyObject* of = PyObject_GetAttrString(reinterpret_cast<PyObject*>(Py_TYPE(o)), "_type_");
    if (!of) throw Failed();
    right = reinterpret_cast<PyTypeObject*>(of) == g_type<T>;
    Py_DECREF(of);
  }
  if (!right) fail(PyExc_TypeError, "expected a tensor, a ctypes structure or array of the parameter's type, an address or None");
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw Failed();
  void* p = b.buf;
  const bool enough = (size_t)b.len / sizeof(T) >= count;
  PyBuffer_Release(&b);
  if (!enough) fail(PyExc_ValueError, "an array is shorter than the count");
  return static_cast<T*>(p);
}

// Pointers to device memory (and handles) are given as addresses or tensors, those to structures and to arrays on the host are not.
template <class T>
constexpr bool kAddress = std::is_same_v<T, void*> || std::is_same_v<T, float*> || std::is_same_v<T, const float*> || std::is_same_v<T, const int32_t*>;

// ARRAY: a pointer to `count` elements in host memory.
template <class T, bool ARRAY>
T convert(PyObject* o, Args& a, size_t count) {
  if constexpr (std::is_same_v<T, float>) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Failed();
    return (float)v;
  } else if constexpr (std::is_pointer_v<T>) {
    if (o == Py_None) return nullptr;
    if constexpr (std::is_same_v<T, const us_mat*>) {
      if (THPVariable_Check(o) && count <= 1) return a.add(o);
    }
    if constexpr (kAddress<T> && !ARRAY) {
      if (THPVariable_Check(o)) {
        if (!a.immediate) fail(PyExc_TypeError, "a prepared call takes addresses");
        return (T)THPVariable_Unpack(o).data_ptr();
      }
      if (!PyLong_Check(o)) fail(PyExc_TypeError, "expected a tensor, an address or None");
      void* p = PyLong_AsVoidPtr(o);
      if (!p && PyErr_Occurred()) throw Failed();
      return (T)p;
    } else {
      return structure<std::remove_const_t<std::remove_pointer_t<T>>>(o, count);
    }
  } else if constexpr (std::is_same_v<T, size_t>) {
    if (THPVariable_Check(o)) return THPVariable_Unpack(o).nbytes();
    const size_t v = PyLong_AsSize_t(o);
    if (v == (size_t)-1 && PyErr_Occurred()) throw Failed();
    return v;
  } else {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return (T)v;
  }
}

template <class F>
PyObject* guarded(F&& f) {                                    // no C++ exception leaves the module
  try {
    return f();
  } catch (Failed&) {
    return nullptr;
  } catch (std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

struct Prepared {
  virtual ~Prepared() = default;
  virtual int run(void* stream) = 0;
};

// ARRAYS: parameters 1 .. ARRAYS are arrays of as many elements as parameter 0 says.
template <size_t ARRAYS, class... A>
struct Entry {
  using Fn = us_status (*)(A...);
  static constexpr size_t kArgs = sizeof...(A);
  using Tuple = std::tuple<A...>;
  template <size_t... I>
  static Tuple read(PyObject* const* o, Args& a, std::index_sequence<I...>) {
    size_t count = 1;
    if constexpr (ARRAYS > 0) {
      const long n = PyLong_AsLong(o[0]);
      if (n == -1 && PyErr_Occurred()) throw Failed();
      count = n > 0 ? (size_t)n : 0;                          // the library refuses fewer than one
    }
    // a workspace is given twice, for its address and for its size, which one number cannot be
    for (size_t i = 0; a.immediate && i + 1 < kArgs; ++i)
      if (o[i] == o[i + 1] && kSize[i + 1] && !THPVariable_Check(o[i])) fail(PyExc_TypeError, "a workspace is a tensor");
    return Tuple{convert<A, (I >= 1 && I <= ARRAYS)>(o[I], a, I >= 1 && I <= ARRAYS ? count : 1)...};      // braces: left to right
  }
  static constexpr bool kSize[] = {std::is_same_v<A, size_t>...};
  struct Kept : Prepared {
    Fn fn;
    Tuple t;
    int run(void* stream) override {
      std::get<kArgs - 1>(t) = stream;
      return (int)std::apply(fn, t);
    }
  };
  static PyObject* now(Fn fn, PyObject* const* o, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
      if ((size_t)n != kArgs) fail(PyExc_TypeError, "wrong number of arguments");
      Args a(true);
      Tuple t = read(o, a, std::make_index_sequence<kArgs>());
      int status;
      Py_BEGIN_ALLOW_THREADS
      status = (int)std::apply(fn, t);
      Py_END_ALLOW_THREADS
      return PyLong_FromLong(status);
    });
  }
  static Prepared* keep(Fn fn, PyObject* const* o, Py_ssize_t n) {      // every argument but the stream
    if ((size_t)n + 1 != kArgs) fail(PyExc_TypeError, "wrong number of arguments");
    std::vector<PyObject*> all(o, o + n);
    all.push_back(Py_None);
    Args a(false);
    auto k = std::make_unique<Kept>();
    k->fn = fn;
    k->t = read(all.data(), a, std::make_index_sequence<kArgs>());
    return k.release();
  }
};
template <size_t ARRAYS, class... A>
Entry<ARRAYS, A...> entry_of(us_status (*)(A...));

using Keep = Prepared* (*)(PyObject* const*, Py_ssize_t);
struct Known { const char* name; PyCFunction now; Keep keep; };

template <auto F, size_t ARRAYS>
PyObject* now(PyObject*, PyObject* const* o, Py_ssize_t n) { return decltype(entry_of<ARRAYS>(F))::now(F, o, n); }
template <auto F, size_t ARRAYS>
Prepared* keep(PyObject* const* o, Py_ssize_t n) { return decltype(entry_of<ARRAYS>(F))::keep(F, o, n); }
#define US_ARRAYS(f, n) {#f, (PyCFunction)(void (*)(void))now<f, n>, keep<f, n>}
#define US_CALL(f) US_ARRAYS(f, 0)
const Known kKnown[] = {
    US_CALL(us_linear_fwd), US_CALL(us_linear_bwd_x), US_CALL(us_linear_bwd_w), US_CALL(us_linear_fwd_batched), US_CALL(us_linear_bwd_x_batched),
    US_CALL(us_linear_bwd_w_batched), US_ARRAYS(us_linear_group, 1), US_ARRAYS(us_linear_group_any, 1), US_CALL(us_ffn_hidden), US_CALL(us_ffn_hidden_any),
    US_CALL(us_attention_fwd), US_CALL(us_attention_bwd), US_CALL(us_attention_bwd_all), US_CALL(us_cast_fp8), US_ARRAYS(us_cast_fp8_multi, 3),
    US_ARRAYS(us_cast_multi, 3), US_ARRAYS(us_cast_multi_pitched, 3), US_CALL(us_residual_add), US_CALL(us_gelu_fwd), US_CALL(us_gelu_bwd), US_CALL(us_activation_fwd),
    US_CALL(us_activation_bwd), US_ARRAYS(us_weighted_add, 2), US_CALL(us_softmax_fwd), US_CALL(us_softmax_bwd), US_CALL(us_softmax_xent_fwd),
    US_CALL(us_softmax_xent_bwd), US_CALL(us_layer_norm_fwd), US_CALL(us_layer_norm_bwd), US_CALL(us_linear_fwd_cast), US_ARRAYS(us_linear_group_cast, 2),
    US_CALL(us_layer_norm_fwd_cast), US_CALL(us_layer_norm_bwd_cast),
};
constexpr size_t kCount = sizeof(kKnown) / sizeof(kKnown[0]);
PyMethodDef g_calls[kCount];

// ---- kept calls
struct Held {
  std::unique_ptr<Prepared> call;
  PyObject* args = nullptr;                                   // the structures it points into
  ~Held() { Py_XDECREF(args); }
};
void held_free(PyObject* c) { delete static_cast<Held*>(PyCapsule_GetPointer(c, "us.call")); }

PyObject* prepare(PyObject*, PyObject* const* o, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 2 || !PyTuple_Check(o[1])) fail(PyExc_TypeError, "prepare(name, arguments)");
    const char* name = PyUnicode_AsUTF8(o[0]);
    if (!name) throw Failed();
    for (const Known& k : kKnown) {
      if (strcmp(k.name, name)) continue;
      auto h = std::make_unique<Held>();
      std::vector<PyObject*> a;
      for (Py_ssize_t i = 0; i < PyTuple_GET_SIZE(o[1]); ++i) a.push_back(PyTuple_GET_ITEM(o[1], i));
      h->call.reset(k.keep(a.data(), (Py_ssize_t)a.size()));
      h->args = Py_NewRef(o[1]);
      PyObject* c = PyCapsule_New(h.get(), "us.call", held_free);
      if (c) h.release();
      return c;
    }
    fail(PyExc_KeyError, name);
  });
}

// ---- programs
struct Step { int where; Prepared* call; };                   // where: 0 main stream, 1 side stream, 2 join
struct Program {
  std::vector<Step> steps;
  std::vector<std::pair<int, us_mat*>> slots;                 // number of the input, where its description goes
  PyObject* keep = nullptr;
  ~Program() { Py_XDECREF(keep); }
};
void program_free(PyObject* c) { delete static_cast<Program*>(PyCapsule_GetPointer(c, "us.program")); }

// program([(where, prepared call or None)], [(input number, us_mat)])
PyObject* program(PyObject*, PyObject* const* o, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 2 || !PyList_Check(o[0]) || !PyList_Check(o[1])) fail(PyExc_TypeError, "program(steps, slots)");
    auto p = std::make_unique<Program>();
    for (int which = 0; which < 2; ++which) {
      for (Py_ssize_t i = 0; i < PyList_GET_SIZE(o[which]); ++i) {
        PyObject *e = PyList_GET_ITEM(o[which], i), *second;
        if (!PyTuple_Check(e) || PyTuple_GET_SIZE(e) != 2) fail(PyExc_TypeError, "pairs");
        const long first = PyLong_AsLong(PyTuple_GET_ITEM(e, 0));
        if (first == -1 && PyErr_Occurred()) throw Failed();
        second = PyTuple_GET_ITEM(e, 1);
        if (which == 1) {
          p->slots.emplace_back((int)first, structure<us_mat>(second, 1));
        } else if (second == Py_None) {
          p->steps.push_back({(int)first, nullptr});
        } else {
          auto* h = static_cast<Held*>(PyCapsule_GetPointer(second, "us.call"));
          if (!h) throw Failed();
          p->steps.push_back({(int)first, h->call.get()});
        }
      }
    }
    p->keep = PyTuple_Pack(2, o[0], o[1]);
    if (!p->keep) throw Failed();
    PyObject* c = PyCapsule_New(p.get(), "us.program", program_free);
    if (c) p.release();
    return c;
  });
}

// run(program, first step, inputs, main stream, side stream, fork event, join event): one pass from that step on.  -1, or
// (step << 8 | status) of the first call that was refused.  Without a side stream (0) every call goes to the main one.
PyObject* run(PyObject*, PyObject* const* o, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 7 || !PyTuple_Check(o[2])) fail(PyExc_TypeError, "run(program, step, inputs, main, side, fork, join)");
    auto* p = static_cast<Program*>(PyCapsule_GetPointer(o[0], "us.program"));
    if (!p) throw Failed();
    const long first = PyLong_AsLong(o[1]);
    void* h[4];
    for (int i = 0; i < 4; ++i) h[i] = PyLong_AsVoidPtr(o[3 + i]);
    if (PyErr_Occurred()) throw Failed();
    if (first == 0) {
      us_mat m[16];
      const Py_ssize_t count = PyTuple_GET_SIZE(o[2]);
      if (count > 16) fail(PyExc_ValueError, "too many inputs");
      for (Py_ssize_t i = 0; i < count; ++i) {
        PyObject* t = PyTuple_GET_ITEM(o[2], i);
        if (!THPVariable_Check(t)) fail(PyExc_TypeError, "an input is not a tensor");
        m[i] = describe(t);
      }
      for (auto& s : p->slots) {
        if (s.first >= count) fail(PyExc_ValueError, "an input is missing");
        *s.second = m[s.first];
      }
    }
    long bad = -1;
    Py_BEGIN_ALLOW_THREADS
    auto main = static_cast<cudaStream_t>(h[0]), side = static_cast<cudaStream_t>(h[1]);
    auto fork = static_cast<cudaEvent_t>(h[2]), join = static_cast<cudaEvent_t>(h[3]);
    auto after = [&](cudaStream_t from, cudaEvent_t ev, cudaStream_t to) {
      if (cudaEventRecord(ev, from) == cudaSuccess && cudaStreamWaitEvent(to, ev, 0) == cudaSuccess) return (int)US_OK;
      (void)cudaGetLastError();
      return (int)US_ERR_CUDA;
    };
    for (size_t i = (size_t)first; i < p->steps.size() && bad < 0; ++i) {
      const Step& s = p->steps[i];
      int status = US_OK;
      if (s.where == 2) {
        if (side) status = after(side, join, main);
      } else {
        if (s.where == 1 && side) status = after(main, fork, side);
        if (status == US_OK) status = s.call->run(s.where == 1 && side ? side : main);
      }
      if (status != US_OK) bad = (long)i << 8 | status;
    }
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(bad);
  });
}

// unchanged(owned, kept, addresses): whether the tensors of two tuples are the same objects at the addresses they had
PyObject* unchanged(PyObject*, PyObject* const* o, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 3 || !PyTuple_Check(o[0]) || !PyTuple_Check(o[1]) || !PyTuple_Check(o[2])) fail(PyExc_TypeError, "unchanged(owned, kept, addresses)");
    const Py_ssize_t count = PyTuple_GET_SIZE(o[0]);
    if (count != PyTuple_GET_SIZE(o[1]) || count != PyTuple_GET_SIZE(o[2])) Py_RETURN_FALSE;
    for (Py_ssize_t i = 0; i < count; ++i) {
      PyObject* t = PyTuple_GET_ITEM(o[0], i);
      if (t != PyTuple_GET_ITEM(o[1], i) || !THPVariable_Check(t)) Py_RETURN_FALSE;
      if (THPVariable_Unpack(t).data_ptr() != PyLong_AsVoidPtr(PyTuple_GET_ITEM(o[2], i))) Py_RETURN_FALSE;
    }
    Py_RETURN_TRUE;
  });
}

// register_types((us_mat, us_epilogue, us_batch, us_attention_batch, us_attention_bwd_batch, us_attention_bwd_all_batch, us_linear_call,
// c_float)): the ctypes types of the parameters; every argument is checked against its own
template <class... T>
void keep_types(PyObject* types) {
  Py_ssize_t i = 0;
  for (Py_ssize_t k = 0; k < (Py_ssize_t)sizeof...(T); ++k)
    if (!PyType_Check(PyTuple_GET_ITEM(types, k))) fail(PyExc_TypeError, "types");
  (void(g_type<T> = reinterpret_cast<PyTypeObject*>(Py_NewRef(PyTuple_GET_ITEM(types, i++)))), ...);
}
PyObject* register_types(PyObject*, PyObject* const* o, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 1 || !PyTuple_Check(o[0]) || PyTuple_GET_SIZE(o[0]) != 8) fail(PyExc_TypeError, "register_types((eight types))");
    keep_types<us_mat, us_epilogue, us_batch, us_attention_batch, us_attention_bwd_batch, us_attention_bwd_all_batch, us_linear_call, float>(o[0]);
    Py_RETURN_NONE;
  });
}

PyMethodDef g_methods[] = {
    {"register_types", (PyCFunction)(void (*)(void))register_types, METH_FASTCALL, nullptr},
    {"unchanged", (PyCFunction)(void (*)(void))unchanged, METH_FASTCALL, nullptr},
    {"prepare", (PyCFunction)(void (*)(void))prepare, METH_FASTCALL, nullptr},
    {"program", (PyCFunction)(void (*)(void))program, METH_FASTCALL, nullptr},
    {"run", (PyCFunction)(void (*)(void))run, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
const char built_for[] = US_BUILT_FOR;                       // what build.py looks for in the file
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) {
  PyObject* ct = PyImport_ImportModule("ctypes");
  PyObject* array = ct ? PyObject_GetAttrString(ct, "Array") : nullptr;      // kept: lives as long as this module
  Py_XDECREF(ct);
  if (!array) return nullptr;
  g_ctypes_array = reinterpret_cast<PyTypeObject*>(array);
  PyObject* m = PyModule_Create(&g_module);
  PyObject* d = m ? PyDict_New() : nullptr;
  if (!d) { Py_XDECREF(m); return nullptr; }
  for (size_t i = 0; i < kCount; ++i) {
    g_calls[i] = {kKnown[i].name, kKnown[i].now, METH_FASTCALL, nullptr};
    PyObject* f = PyCFunction_New(&g_calls[i], nullptr);
    if (!f || PyDict_SetItemString(d, kKnown[i].name, f) != 0) { Py_XDECREF(f); Py_DECREF(d); Py_DECREF(m); return nullptr; }
    Py_DECREF(f);
  }
  if (PyModule_AddObject(m, "calls", d) != 0) { Py_DECREF(d); Py_DECREF(m); return nullptr; }
  if (PyModule_AddStringConstant(m, "built_for", built_for) != 0) { Py_DECREF(m); return nullptr; }
  return m;
}
