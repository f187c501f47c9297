// The Python binding's calls in native form: host arrays of the entry points as packed bytes (device pointers per layer, donor
// maps), and the calls themselves.
//
// A call passes up to twelve arrays.  Packed in Python one of four tensors takes 0.8 us, most of it in the method call per
// tensor, and small calls are bound by the host: here it takes 0.1 us.  The calls take the arguments of the functions of the same
// name in kvp.py, with the stream behind them, read sizes and pointers off the tensors and call the library.  Measured (us a call
// that launches a small kernel, by ctypes -> so; the launch takes about 2): add 3.5 -> 2.3, rmsnorm 4.3 -> 2.7, rope 4.5 -> 2.6,
// cache_append 4.9 -> 2.8, decode 5.7 -> 2.9, gemm 6.1 -> 3.0.  They take plain tensors, lists, tuples, numbers and the binding's own
// structures; for anything else they return NotImplemented and kvp.py goes through ctypes, which raises what it always has.
#define PY_SSIZE_T_CLEAN
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <new>
#include <optional>
#include <string>

#include "../../include/kvp.h"

namespace {

// An entry point reads an array of L entries (owner layers of some, kvp.h).  What a list does not have is a null pointer to it, and
// refused where it would be read.

// [tensor or None, ...] -> their data pointers (0 for None) as 64-bit integers; at least `entries` of them where that is given, or
// (negative) so many more than the list has
PyObject* pointers(PyObject*, PyObject* args) {
  PyObject* seq;
  Py_ssize_t entries = 0;
  if (!PyArg_ParseTuple(args, "O|n", &seq, &entries)) return nullptr;
  PyObject* fast = PySequence_Fast(seq, "expected a sequence of tensors");
  if (fast == nullptr) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast), all = entries < 0 ? n - entries : std::max(n, entries);
  PyObject* out = PyBytes_FromStringAndSize(nullptr, all * Py_ssize_t(sizeof(uint64_t)));
  uint64_t* dst = out == nullptr ? nullptr : reinterpret_cast<uint64_t*>(PyBytes_AS_STRING(out));
  bool ok = out != nullptr;
  if (ok) std::fill(dst + n, dst + all, uint64_t(0));
  for (Py_ssize_t i = 0; i < n && ok; ++i) {
    PyObject* o = PySequence_Fast_GET_ITEM(fast, i);
    if (o == Py_None) {
      dst[i] = 0;
    } else if (THPVariable_CheckExact(o)) {
      try {
        dst[i] = reinterpret_cast<uint64_t>(THPVariable_Unpack(o).data_ptr());
      } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        ok = false;
      }
    } else {   // subclasses and whatever else has the method
      PyObject* p = PyObject_CallMethod(o, "data_ptr", nullptr);
      dst[i] = p == nullptr ? 0 : PyLong_AsUnsignedLongLong(p);
      Py_XDECREF(p);
      ok = PyErr_Occurred() == nullptr;
    }
  }
  Py_DECREF(fast);
  if (!ok) Py_CLEAR(out);
  return out;
}

// [int, ...] -> 32-bit integers
PyObject* donors(PyObject*, PyObject* seq) {
  PyObject* fast = PySequence_Fast(seq, "expected a sequence of integers");
  if (fast == nullptr) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
  PyObject* out = PyBytes_FromStringAndSize(nullptr, n * Py_ssize_t(sizeof(int32_t)));
  int32_t* dst = out == nullptr ? nullptr : reinterpret_cast<int32_t*>(PyBytes_AS_STRING(out));
  bool ok = out != nullptr;
  for (Py_ssize_t i = 0; i < n && ok; ++i) {
    PyObject* o = PySequence_Fast_GET_ITEM(fast, i);
    PyObject* v = PyLong_CheckExact(o) ? Py_NewRef(o) : PyNumber_Long(o);
    const long long x = v == nullptr ? 0 : PyLong_AsLongLong(v);
    Py_XDECREF(v);
    ok = PyErr_Occurred() == nullptr;
    if (ok && (x < INT32_MIN || x > INT32_MAX)) {
      PyErr_SetString(PyExc_OverflowError, "donor does not fit a 32-bit integer");
      ok = false;
    }
    dst[i] = int32_t(x);
  }
  Py_DECREF(fast);
  if (!ok) Py_CLEAR(out);
  return out;
}

// ---------------------------------------------------------------------------------------------
// the entry points
// ---------------------------------------------------------------------------------------------
struct Library {
  decltype(&kvp_gemm) gemm;
  decltype(&kvp_rmsnorm) rmsnorm;
  decltype(&kvp_rope) rope;
  decltype(&kvp_swiglu) swiglu;
  decltype(&kvp_add) add;
  decltype(&kvp_proj_fwd) proj_fwd;
  decltype(&kvp_proj_bwd) proj_bwd;
  decltype(&kvp_out_proj_fwd) out_proj_fwd;
  decltype(&kvp_out_proj_bwd) out_proj_bwd;
  decltype(&kvp_attn_fwd) attn_fwd;
  decltype(&kvp_attn_bwd) attn_bwd;
  decltype(&kvp_cache_append) cache_append;
  decltype(&kvp_decode) decode;
} lib;
PyTypeObject *shape_type, *desc_type;   // kvp.Shape, kvp.DecodeDesc

// bind(addresses of the entry points in the order above, Shape, DecodeDesc)
PyObject* bind(PyObject*, PyObject* args) {
  PyObject *list, *shape, *desc;
  if (!PyArg_ParseTuple(args, "O!O!O!", &PyList_Type, &list, &PyType_Type, &shape, &PyType_Type, &desc)) return nullptr;
  constexpr Py_ssize_t n = sizeof(Library) / sizeof(void*);
  if (PyList_GET_SIZE(list) != n) return PyErr_Format(PyExc_ValueError, "%zd addresses", n);
  void* at[n];
  for (Py_ssize_t i = 0; i < n; ++i) {
    at[i] = PyLong_AsVoidPtr(PyList_GET_ITEM(list, i));
    if (PyErr_Occurred()) return nullptr;
  }
  memcpy(&lib, at, sizeof(lib));
  shape_type = reinterpret_cast<PyTypeObject*>(Py_NewRef(shape));
  desc_type = reinterpret_cast<PyTypeObject*>(Py_NewRef(desc));
  Py_RETURN_NONE;
}

// The arguments of a call, one after the other; `ok` is false as soon as one is not of the plain kind.
struct Reader {
  PyObject* const* a;
  Py_ssize_t left;
  bool ok;
  int layers = 0;            // L
  Py_ssize_t entries = 0;    // of the arrays, at least
  Reader(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) : a(args), left(n), ok(n == want && lib.add != nullptr) {}
  PyObject* next() { return left-- > 0 ? *a++ : Py_None; }
  const at::Tensor* tensor(int dims) {   // dims < 0: any number
    PyObject* o = next();
    ok = ok && THPVariable_CheckExact(o);
    if (!ok) return nullptr;
    const at::Tensor* t = &THPVariable_Unpack(o);
    ok = dims < 0 || t->dim() == dims;
    return ok ? t : nullptr;
  }
  void* pointer() {
    const at::Tensor* t = tensor(-1);
    return t ? t->data_ptr() : nullptr;
  }
  int flag() {
    PyObject* o = next();
    ok = ok && PyBool_Check(o);
    return o == Py_True;
  }
  long long integer() {   // (of 64 bits: cut to the parameter's size, as ctypes does)
    PyObject* o = next();
    ok = ok && PyLong_CheckExact(o);
    if (!ok) return 0;
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    ok = over == 0;
    return v;
  }
  double real() {
    PyObject* o = next();
    ok = ok && PyFloat_CheckExact(o);
    return ok ? PyFloat_AS_DOUBLE(o) : 0.;
  }
  kvp_stream_t stream() {
    PyObject* o = next();
    ok = ok && PyLong_CheckExact(o);
    if (!ok) return nullptr;
    void* p = PyLong_AsVoidPtr(o);
    ok = PyErr_Occurred() == nullptr;
    if (!ok) PyErr_Clear();
    return static_cast<kvp_stream_t>(p);
  }
  // a structure of the binding (held by the caller for the time of the call)
  template <typename T>
  const T* structure(PyTypeObject* type) {
    PyObject* o = next();
    Py_buffer view;
    ok = ok && Py_TYPE(o) == type;
    if (!ok) return nullptr;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) {
      PyErr_Clear();
      ok = false;
      return nullptr;
    }
    ok = view.len == Py_ssize_t(sizeof(T));
    const T* p = static_cast<const T*>(view.buf);
    PyBuffer_Release(&view);
    if (ok) layers = p->L;
    return p;
  }
  // host arrays
  static constexpr int kRoom = 768;
  void* room[kRoom];
  int32_t numbers[257];
  int used = 0;
  PyObject** items(PyObject* o, Py_ssize_t& n) {
    ok = ok && (PyList_CheckExact(o) || PyTuple_CheckExact(o));
    if (!ok) return nullptr;
    n = PySequence_Fast_GET_SIZE(o);
    return PySequence_Fast_ITEMS(o);
  }
  template <typename T>
  T* pointers(int more = 0) {   // more: entries behind the list (without a donor map, whose length bounds L)
    Py_ssize_t n = 0;
    PyObject** it = items(next(), n);
    const Py_ssize_t all = std::max(n + more, entries);
    ok = ok && used + all <= kRoom;
    if (!ok) return nullptr;
    void** const dst = room + used;
    std::fill(dst + n, dst + all, nullptr);
    for (Py_ssize_t i = 0; i < n && ok; ++i) {
      ok = it[i] == Py_None || THPVariable_CheckExact(it[i]);
      if (ok) dst[i] = it[i] == Py_None ? nullptr : THPVariable_Unpack(it[i]).data_ptr();
    }
    used += int(all);
    return reinterpret_cast<T*>(dst);
  }
  const int32_t* donor_map() {
    Py_ssize_t n = 0;
    PyObject** it = items(next(), n);
    ok = ok && n <= 256;
    for (Py_ssize_t i = 0; i < n && ok; ++i) {
      ok = PyLong_CheckExact(it[i]);
      if (!ok) break;
      int over = 0;
      const long long v = PyLong_AsLongLongAndOverflow(it[i], &over);
      ok = over == 0 && v >= INT32_MIN && v <= INT32_MAX;
      numbers[i] = int32_t(v);
    }
    if (!ok) return nullptr;
    if (n < layers) numbers[n] = -1;   // no donor: the map is refused before anything else is read
    else entries = layers;
    return numbers;
  }
  struct Space {
    void* p;
    size_t n;
  };
  Space workspace() {
    if (left > 0 && *a == Py_None) {
      next();
      return {nullptr, 0};
    }
    const at::Tensor* t = tensor(-1);
    return t ? Space{t->data_ptr(), size_t(t->nbytes())} : Space{nullptr, 0};
  }
};

// Reads the arguments with `read`, which returns the call; what a tensor throws (no storage, symbolic sizes) sends the call to
// kvp.py's own path.  The call itself is made once: what a library function throws becomes an exception of Python's, with the
// interpreter's lock held again.
template <typename F>
PyObject* run(PyObject* const* args, Py_ssize_t n, Py_ssize_t want, F read) {
  Reader r(args, n, want);
  std::optional<decltype(read(r))> call;
  try {
    call.emplace(read(r));
  } catch (const std::exception&) {
    r.ok = false;
  }
  if (!r.ok) {
    if (PyErr_Occurred()) PyErr_Clear();
    Py_RETURN_NOTIMPLEMENTED;
  }
  int status = 0;
  PyObject* thrown = nullptr;   // its kind
  std::string what;
  Py_BEGIN_ALLOW_THREADS
  try {
    status = (*call)();
  } catch (const std::bad_alloc&) {
    thrown = PyExc_MemoryError;
  } catch (const std::exception& e) {
    thrown = PyExc_RuntimeError;
    what = e.what();
  }
  Py_END_ALLOW_THREADS
  if (thrown != nullptr) {
    PyErr_SetString(thrown, what.c_str());
    return nullptr;
  }
  return PyLong_FromLong(status);
}
#define ENTRY(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t n)

ENTRY(gemm) {   // a, b, c, a_mn, b_mn, stream
  return run(args, n, 6, [](Reader& r) {
    const at::Tensor *a = r.tensor(2), *b = r.tensor(2), *c = r.tensor(2);
    const int a_mn = r.flag(), b_mn = r.flag();
    const kvp_stream_t stream = r.stream();
    struct {
      int M, N, K;
      void *a, *b, *c;
      int64_t lda, ldb, ldc;
      int f32;
    } v{};
    if (r.ok)
      v = {int(c->size(0)), int(c->size(1)), int(a->size(a_mn ? 0 : 1)), a->data_ptr(), b->data_ptr(), c->data_ptr(), a->stride(0), b->stride(0),
           c->stride(0), c->scalar_type() == at::kFloat};
    return [=] { return lib.gemm(v.M, v.N, v.K, v.a, v.lda, a_mn, v.b, v.ldb, b_mn, v.c, v.ldc, v.f32, stream); };
  });
}
ENTRY(rmsnorm) {   // x, w, eps, y, stream
  return run(args, n, 5, [](Reader& r) {
    const at::Tensor* x = r.tensor(2);
    void* const w = r.pointer();
    const float eps = float(r.real());
    void* const y = r.pointer();
    const kvp_stream_t stream = r.stream();
    const int T = r.ok ? int(x->size(0)) : 0, D = r.ok ? int(x->size(1)) : 0;
    void* const p = r.ok ? x->data_ptr() : nullptr;
    return [=] { return lib.rmsnorm(T, D, p, w, eps, y, stream); };
  });
}
ENTRY(rope) {   // x, theta, pos0, stream
  return run(args, n, 4, [](Reader& r) {
    const at::Tensor* x = r.tensor(4);
    const float theta = float(r.real());
    const int pos0 = int(r.integer());
    const kvp_stream_t stream = r.stream();
    int d[4] = {};
    for (int i = 0; i < 4 && r.ok; ++i) d[i] = int(x->size(i));
    void* const p = r.ok ? x->data_ptr() : nullptr;
    return [=] { return lib.rope(d[0], d[1], d[2], d[3], theta, pos0, p, stream); };
  });
}
template <bool ADD>
ENTRY(zip) {   // a, b, out, stream
  return run(args, n, 4, [](Reader& r) {
    const at::Tensor* a = r.tensor(-1);
    void *const b = r.pointer(), *const out = r.pointer();
    const kvp_stream_t stream = r.stream();
    const int64_t count = r.ok ? a->numel() : 0;
    void* const p = r.ok ? a->data_ptr() : nullptr;
    return [=] { return ADD ? lib.add(count, p, b, out, stream) : lib.swiglu(count, p, b, out, stream); };
  });
}

typedef const void* const* In;
typedef void* const* Out;
typedef const float* const* InF;
typedef float* const* OutF;
ENTRY(proj_fwd) {   // shape, donor, x, wq, wk, wv, q, k, v, ws, stream
  return run(args, n, 11, [](Reader& r) {
    auto* s = r.structure<kvp_shape>(shape_type);
    auto* donor = r.donor_map();
    In x = r.pointers<const void* const>(), wq = r.pointers<const void* const>(), wk = r.pointers<const void* const>(), wv = r.pointers<const void* const>();
    Out q = r.pointers<void* const>(), k = r.pointers<void* const>(), v = r.pointers<void* const>();
    const Reader::Space ws = r.workspace();
    const kvp_stream_t stream = r.stream();
    return [=] { return lib.proj_fwd(s, donor, x, wq, wk, wv, q, k, v, ws.p, ws.n, stream); };
  });
}
ENTRY(proj_bwd) {   // shape, donor, x, wq, wk, wv, dq, dk_sum, dv_sum, dwq, dwk, dwv, dx, ws, stream
  return run(args, n, 15, [](Reader& r) {
    auto* s = r.structure<kvp_shape>(shape_type);
    auto* donor = r.donor_map();
    In x = r.pointers<const void* const>(), wq = r.pointers<const void* const>(), wk = r.pointers<const void* const>(), wv = r.pointers<const void* const>(),
       dq = r.pointers<const void* const>();
    InF dk = r.pointers<const float* const>(), dv = r.pointers<const float* const>();
    OutF dwq = r.pointers<float* const>(), dwk = r.pointers<float* const>(), dwv = r.pointers<float* const>();
    Out dx = r.pointers<void* const>();
    const Reader::Space ws = r.workspace();
    const kvp_stream_t stream = r.stream();
    return [=] { return lib.proj_bwd(s, donor, x, wq, wk, wv, dq, dk, dv, dwq, dwk, dwv, dx, ws.p, ws.n, stream); };
  });
}
ENTRY(out_proj_fwd) {   // shape, o, wo, y, stream
  return run(args, n, 5, [](Reader& r) {
    auto* s = r.structure<kvp_shape>(shape_type);
    In o = r.pointers<const void* const>(1), wo = r.pointers<const void* const>(1);
    Out y = r.pointers<void* const>(1);
    const kvp_stream_t stream = r.stream();
    return [=] { return lib.out_proj_fwd(s, o, wo, y, stream); };
  });
}
ENTRY(out_proj_bwd) {   // shape, o, wo, dy, d_o, dwo, stream
  return run(args, n, 7, [](Reader& r) {
    auto* s = r.structure<kvp_shape>(shape_type);
    In o = r.pointers<const void* const>(1), wo = r.pointers<const void* const>(1), dy = r.pointers<const void* const>(1);
    Out d_o = r.pointers<void* const>(1);
    OutF dwo = r.pointers<float* const>(1);
    const kvp_stream_t stream = r.stream();
    return [=] { return lib.out_proj_bwd(s, o, wo, dy, d_o, dwo, stream); };
  });
}
ENTRY(attn_fwd) {   // shape, donor, causal, scale, q, k, v, o, lse, ws, stream
  return run(args, n, 11, [](Reader& r) {
    auto* s = r.structure<kvp_shape>(shape_type);
    auto* donor = r.donor_map();
    const int causal = r.flag();
    const float scale = float(r.real());
    In q = r.pointers<const void* const>(), k = r.pointers<const void* const>(), v = r.pointers<const void* const>();
    Out o = r.pointers<void* const>();
    OutF lse = r.pointers<float* const>();
    const Reader::Space ws = r.workspace();
    const kvp_stream_t stream = r.stream();
    return [=] { return lib.attn_fwd(s, donor, causal, scale, q, k, v, o, lse, ws.p, ws.n, stream); };
  });
}
ENTRY(attn_bwd) {   // shape, donor, causal, scale, q, k, v, o, d_o, lse, dq, dk_sum, dv_sum, ws, stream
  return run(args, n, 15, [](Reader& r) {
    auto* s = r.structure<kvp_shape>(shape_type);
    auto* donor = r.donor_map();
    const int causal = r.flag();
    const float scale = float(r.real());
    In q = r.pointers<const void* const>(), k = r.pointers<const void* const>(), v = r.pointers<const void* const>(), o = r.pointers<const void* const>(),
       d_o = r.pointers<const void* const>();
    InF lse = r.pointers<const float* const>();
    Out dq = r.pointers<void* const>();
    OutF dk = r.pointers<float* const>(), dv = r.pointers<float* const>();
    const Reader::Space ws = r.workspace();
    const kvp_stream_t stream = r.stream();
    return [=] { return lib.attn_bwd(s, donor, causal, scale, q, k, v, o, d_o, lse, dq, dk, dv, ws.p, ws.n, stream); };
  });
}
ENTRY(cache_append) {   // desc, donor, k_new, v_new, k_cache, v_cache, block_table, lengths, stream
  return run(args, n, 9, [](Reader& r) {
    auto* d = r.structure<kvp_decode_desc>(desc_type);
    auto* donor = r.donor_map();
    In kn = r.pointers<const void* const>(), vn = r.pointers<const void* const>();
    Out kc = r.pointers<void* const>(), vc = r.pointers<void* const>();
    auto* table = static_cast<const int32_t*>(r.pointer());
    auto* lengths = static_cast<const int32_t*>(r.pointer());
    const kvp_stream_t stream = r.stream();
    return [=] { return lib.cache_append(d, donor, kn, vn, kc, vc, table, lengths, stream); };
  });
}
ENTRY(decode) {   // desc, donor, scale, q, k_cache, v_cache, block_table, lengths, o, lse, layer_begin, layer_end or None, ws, stream
  return run(args, n, 14, [](Reader& r) {
    auto* d = r.structure<kvp_decode_desc>(desc_type);
    auto* donor = r.donor_map();
    const float scale = float(r.real());
    In q = r.pointers<const void* const>(), kc = r.pointers<const void* const>(), vc = r.pointers<const void* const>();
    auto* table = static_cast<const int32_t*>(r.pointer());
    auto* lengths = static_cast<const int32_t*>(r.pointer());
    Out o = r.pointers<void* const>();
    OutF lse = r.pointers<float* const>();
    const int begin = int(r.integer());
    const bool to_end = r.left > 0 && *r.a == Py_None;
    if (to_end) r.next();
    const int end = to_end ? (r.ok ? d->L : 0) : int(r.integer());
    const Reader::Space ws = r.workspace();
    const kvp_stream_t stream = r.stream();
    return [=] { return lib.decode(d, donor, scale, q, kc, vc, table, lengths, o, lse, begin, end, ws.p, ws.n, stream); };
  });
}
#define METHOD(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(fn)), METH_FASTCALL, nullptr}

PyMethodDef methods[] = {{"pointers", pointers, METH_VARARGS, nullptr}, {"donors", donors, METH_O, nullptr}, {"bind", bind, METH_VARARGS, nullptr},
                         METHOD("gemm", gemm), METHOD("rmsnorm", rmsnorm), METHOD("rope", rope), METHOD("swiglu", zip<false>), METHOD("add", zip<true>),
                         METHOD("proj_fwd", proj_fwd), METHOD("proj_bwd", proj_bwd), METHOD("out_proj_fwd", out_proj_fwd), METHOD("out_proj_bwd", out_proj_bwd),
                         METHOD("attn_fwd", attn_fwd), METHOD("attn_bwd", attn_bwd), METHOD("cache_append", cache_append), METHOD("decode", decode),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pack", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pack() { return PyModule_Create(&module); }
