// The calls a decoding program makes over and over, without ctypes: unpacks the arguments, takes the
// tensors' addresses and the current stream, and calls the C entry point with the GIL released.
// A call through ctypes cost 5 to 8 us of host time around a launch of 3, which is more than the
// kernels of a small layer take.
//
// Only the plain cases are handled: a handle, the library's own structures, ints, None, and torch
// tensors that are dense, on a GPU and contiguous. For anything else a function returns
// NotImplemented, and the caller goes through ctypes, which accepts or refuses as it always did.
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/version.h>

#include "blockffn.h"

namespace {

PyObject* g_handle_type = nullptr;    // ctypes.c_void_p
PyObject* g_weights_type = nullptr;   // binding.Weights
PyObject* g_config_type = nullptr;    // binding.Config

struct Args {
  PyObject* const* a;
  bool ok = true;
  // the bytes of a ctypes object of exactly this type
  void* object(PyObject* o, PyObject* type) {
    if (reinterpret_cast<PyObject*>(Py_TYPE(o)) != type) return miss();
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) {
      PyErr_Clear();
      return miss();
    }
    void* p = view.buf;            // (the object owns the bytes: valid while the caller holds it)
    PyBuffer_Release(&view);
    return p;
  }
  blockffn_handle handle(int i) {
    void* p = object(a[i], g_handle_type);
    return p ? *static_cast<blockffn_handle*>(p) : nullptr;
  }
  const blockffn_weights* weights(int i) {
    return static_cast<const blockffn_weights*>(object(a[i], g_weights_type));
  }
  const blockffn_config* config(int i) {
    return static_cast<const blockffn_config*>(object(a[i], g_config_type));
  }
  int32_t number(int i) {
    if (!PyLong_CheckExact(a[i])) {
      miss();
      return 0;
    }
    int over = 0;
    const long v = PyLong_AsLongAndOverflow(a[i], &over);
    if (over || v != static_cast<int32_t>(v)) miss();
    return static_cast<int32_t>(v);
  }
  template <class T>
  T* device(int i) {
    if (a[i] == Py_None) return nullptr;
    if (!THPVariable_CheckExact(a[i])) return static_cast<T*>(miss());
    const at::Tensor& t = THPVariable_Unpack(a[i]);
    if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || !t.has_storage() ||
        !t.unsafeGetTensorImpl()->storage().data() || !t.is_contiguous())
      return static_cast<T*>(miss());
    return static_cast<T*>(t.data_ptr());
  }
  void* stream(int i) {
    if (a[i] != Py_None) return miss();
    return c10::cuda::getCurrentCUDAStream().stream();
  }
  void* miss() {
    ok = false;
    return nullptr;
  }
};

// f(Args&) reads the arguments and returns the call to make
template <class F>
PyObject* run(PyObject* const* a, Py_ssize_t n, Py_ssize_t want, F f) {
  if (n != want) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  int code = 0;
  try {
    Args args{a};
    auto call = f(args);
    if (!args.ok) Py_RETURN_NOTIMPLEMENTED;
    Py_BEGIN_ALLOW_THREADS
    code = call();
    Py_END_ALLOW_THREADS
  } catch (const std::exception&) {
    Py_RETURN_NOTIMPLEMENTED;      // (ctypes then meets the same trouble and says so)
  }
  return PyLong_FromLong(code);
}

PyObject* router(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(a, n, 7, [](Args& g) {
    return [h = g.handle(0), w = g.weights(1), x = g.device<void>(2), L = g.number(3),
            s = g.device<float>(4), m = g.device<uint32_t>(5), st = g.stream(6)] {
      return blockffn_router(h, w, x, L, s, m, st);
    };
  });
}
PyObject* chunk_union(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(a, n, 8, [](Args& g) {
    return [h = g.handle(0), s = g.device<float>(1), L = g.number(2), um = g.device<uint32_t>(3),
            ids = g.device<int32_t>(4), nu = g.device<int32_t>(5), stats = g.device<blockffn_stats>(6),
            st = g.stream(7)] { return blockffn_chunk_union(h, s, L, um, ids, nu, stats, st); };
  });
}
PyObject* expert_ffn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(a, n, 11, [](Args& g) {
    return [h = g.handle(0), w = g.weights(1), x = g.device<void>(2), s = g.device<float>(3),
            L = g.number(4), ids = g.device<int32_t>(5), nu = g.device<int32_t>(6),
            out = g.device<float>(7), xn = g.device<void>(8), fl = g.number(9), st = g.stream(10)] {
      return blockffn_expert_ffn(h, w, x, s, L, ids, nu, out, xn, fl, st);
    };
  });
}
PyObject* expert_ffn_noalloc(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(a, n, 11, [](Args& g) {
    return [c = g.config(0), w = g.weights(1), x = g.device<void>(2), s = g.device<float>(3),
            L = g.number(4), ids = g.device<int32_t>(5), nu = g.device<int32_t>(6),
            out = g.device<float>(7), xn = g.device<void>(8), fl = g.number(9), st = g.stream(10)] {
      return blockffn_expert_ffn_noalloc(c, w, x, s, L, ids, nu, out, xn, fl, st);
    };
  });
}
PyObject* layer_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(a, n, 9, [](Args& g) {
    return [h = g.handle(0), w = g.weights(1), x = g.device<void>(2), L = g.number(3),
            out = g.device<float>(4), xn = g.device<void>(5), stats = g.device<blockffn_stats>(6),
            fl = g.number(7), st = g.stream(8)] {
      return blockffn_layer_forward(h, w, x, L, out, xn, stats, fl, st);
    };
  });
}
PyObject* layer_forward_scores(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(a, n, 10, [](Args& g) {
    return [h = g.handle(0), w = g.weights(1), x = g.device<void>(2), s = g.device<float>(3),
            L = g.number(4), out = g.device<float>(5), xn = g.device<void>(6),
            stats = g.device<blockffn_stats>(7), fl = g.number(8), st = g.stream(9)] {
      return blockffn_layer_forward_scores(h, w, x, s, L, out, xn, stats, fl, st);
    };
  });
}
PyObject* read_routing(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(a, n, 8, [](Args& g) {
    return [h = g.handle(0), L = g.number(1), s = g.device<float>(2), tm = g.device<uint32_t>(3),
            um = g.device<uint32_t>(4), ids = g.device<int32_t>(5), nu = g.device<int32_t>(6),
            st = g.stream(7)] { return blockffn_read_routing(h, L, s, tm, um, ids, nu, st); };
  });
}
PyObject* reuse_ratio(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return run(a, n, 5, [](Args& g) {
    return [h = g.handle(0), s = g.device<float>(1), L = g.number(2), r = g.device<double>(3),
            st = g.stream(4)] { return blockffn_reuse_ratio(h, s, L, r, st); };
  });
}

// scores [L][E] and tok_mask [L][words] (where with_scores), union_mask [words], union_ids [E], n_union [1] on CUDA
// device `index` (-1: the current one)
struct Routing {
  at::Tensor b[5];
  Routing(int64_t L, int64_t E, int64_t words, int with_scores, int index) {
    const auto dev = at::device(at::Device(at::kCUDA, static_cast<c10::DeviceIndex>(index)));
    const auto i32 = dev.dtype(at::kInt);
    if (with_scores) {
      b[0] = at::empty({L, E}, dev.dtype(at::kFloat));
      b[1] = at::empty({L, words}, i32);
    }
    b[2] = at::empty({words}, i32);
    b[3] = at::empty({E}, i32);
    b[4] = at::empty({1}, i32);
  }
};
// t[at ..]: the tensors, None where there is none. False with an error set, and t gone, when that fails.
bool put(PyObject*& t, int at, const at::Tensor* b, int n) {
  for (int k = 0; t && k < n; ++k) {
    PyObject* o = b[k].defined() ? THPVariable_Wrap(b[k]) : Py_NewRef(Py_None);
    if (o) {
      PyTuple_SET_ITEM(t, at + k, o);
    } else {
      Py_CLEAR(t);
    }
  }
  return t != nullptr;
}

// What Layer.forward returns beside out
PyObject* routing_buffers(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 5) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  Args g{a};
  const int64_t L = g.number(0), E = g.number(1), words = g.number(2);
  const int with_scores = g.number(3), index = g.number(4);
  if (!g.ok) Py_RETURN_NOTIMPLEMENTED;
  try {
    const Routing r(L, E, words, with_scores, index);   // (all of them exist before the first becomes a Python object)
    PyObject* t = PyTuple_New(5);
    put(t, 0, r.b, 5);
    return t;
  } catch (const std::exception&) {
    Py_RETURN_NOTIMPLEMENTED;
  }
}

// Layer.forward with nothing given but x: out and the routing buffers, blockffn_layer_forward and
// blockffn_read_routing on the current stream, (status, status, out, the buffers).
// (handle, weights, x, x_next, stats, call_flags, d, E, words, device index)
PyObject* layer_call(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 10) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  bool launched = false;
  try {
    Args g{a};
    const blockffn_handle h = g.handle(0);
    const blockffn_weights* w = g.weights(1);
    const void* x = g.device<void>(2);
    void* xn = g.device<void>(3);
    blockffn_stats* stats = g.device<blockffn_stats>(4);
    const int fl = g.number(5), index = g.number(9);
    const int64_t d = g.number(6), E = g.number(7), words = g.number(8);
    if (!g.ok || !x || THPVariable_Unpack(a[2]).dim() < 1) Py_RETURN_NOTIMPLEMENTED;
    const int64_t L = THPVariable_Unpack(a[2]).size(0);
    if (L > (1 << 20)) Py_RETURN_NOTIMPLEMENTED;       // (refused below; not by running out of memory here)
    const at::Tensor out =
        at::empty({L, d}, at::device(at::Device(at::kCUDA, static_cast<c10::DeviceIndex>(index))).dtype(at::kFloat));
    const Routing r(L, E, words, 1, index);
    void* st = c10::cuda::getCurrentCUDAStream().stream();
    int code[2];
    launched = true;
    Py_BEGIN_ALLOW_THREADS
    code[0] = blockffn_layer_forward(h, w, x, static_cast<int32_t>(L), out.data_ptr<float>(), xn, stats, fl, st);
    code[1] = code[0] != BLOCKFFN_OK
                  ? BLOCKFFN_OK
                  : blockffn_read_routing(h, static_cast<int32_t>(L), r.b[0].data_ptr<float>(),
                                          reinterpret_cast<uint32_t*>(r.b[1].data_ptr<int32_t>()),
                                          reinterpret_cast<uint32_t*>(r.b[2].data_ptr<int32_t>()),
                                          r.b[3].data_ptr<int32_t>(), r.b[4].data_ptr<int32_t>(), st);
    Py_END_ALLOW_THREADS
    PyObject* t = PyTuple_New(8);
    for (int k = 0; t && k < 2; ++k) {
      PyObject* o = PyLong_FromLong(code[k]);
      if (o) {
        PyTuple_SET_ITEM(t, k, o);
      } else {
        Py_CLEAR(t);
      }
    }
    if (t && put(t, 2, &out, 1)) put(t, 3, r.b, 5);
    return t;
  } catch (const std::exception& e) {
    if (!launched) Py_RETURN_NOTIMPLEMENTED;
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyObject* set_types(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 3) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  PyObject** slot[3] = {&g_handle_type, &g_weights_type, &g_config_type};
  for (int i = 0; i < 3; ++i) {
    Py_INCREF(a[i]);
    Py_XDECREF(*slot[i]);
    *slot[i] = a[i];
  }
  Py_RETURN_NONE;
}

template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyMethodDef method(const char* name) {
  return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(F)), METH_FASTCALL, nullptr};
}
PyMethodDef g_methods[] = {
    method<router>("router"),
    method<chunk_union>("chunk_union"),
    method<expert_ffn>("expert_ffn"),
    method<expert_ffn_noalloc>("expert_ffn_noalloc"),
    method<layer_forward>("layer_forward"),
    method<layer_forward_scores>("layer_forward_scores"),
    method<read_routing>("read_routing"),
    method<reuse_ratio>("reuse_ratio"),
    method<routing_buffers>("routing_buffers"),
    method<layer_call>("layer_call"),
    method<set_types>("set_types"),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() {
  PyObject* m = PyModule_Create(&g_module);
  if (m && PyModule_AddStringConstant(m, "TORCH_VERSION", TORCH_VERSION) != 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
