// Python call -> C ABI, the well-formed case: a tensor's checks and address, the shape, the
// positions and the stream are read here instead of through one ctypes conversion each.  A call
// that is anything else (another tensor type, a wrong dtype or size, a CPU tensor, an odd integer)
// returns None before anything is launched, and the Python wrapper takes its general path, which
// raises the errors.
//
// The wrappers' host time bounds the small calls (an append or an attention of a few microseconds
// on the GPU): 8 tensors through ctypes take 8-10 us a call, this takes about 2.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "unstep.h"

namespace {

constexpr int kMaxStreams = 64;   // more streams than this take the general path

decltype(&unstep_rope_table) f_table = nullptr;
decltype(&unstep_rope_kv_append_sink) f_append_sink = nullptr;
decltype(&unstep_rmsnorm_rope_kv_append) f_norm_append = nullptr;
decltype(&unstep_window_attn) f_attn = nullptr;
decltype(&unstep_window_attn) f_attn_noalloc = nullptr;
decltype(&unstep_window_attn_sink) f_attn_sink = nullptr;
PyTypeObject* shape_type = nullptr;

// Reads the arguments of one call; `good` turns false at the first that is not well-formed.
struct Args {
  PyObject* const* a;
  Py_ssize_t n;
  bool good = true;
  Py_ssize_t i = 0;
  unstep_shape_t shape{};
  int64_t tokens = 0, act = 0;   // tokens of a chunk, elements of q

  Args(PyObject* const* args, Py_ssize_t nargs, Py_ssize_t want) : a(args), n(nargs) { good = nargs == want; }

  static bool mul(int64_t x, int64_t y, int64_t* out) { return !__builtin_mul_overflow(x, y, out); }

  const unstep_shape_t* get_shape() {
    if (!good) return nullptr;
    PyObject* o = a[i++];
    Py_buffer view;
    if (Py_TYPE(o) != shape_type || PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) {
      good = false;
      return nullptr;
    }
    good = view.len == static_cast<Py_ssize_t>(sizeof(shape));
    if (good) memcpy(&shape, view.buf, sizeof(shape));
    PyBuffer_Release(&view);
    good = good && shape.batch > 0 && shape.heads > 0 && shape.head_dim > 0 && shape.chunk_frames > 0 &&
           shape.grid_h > 0 && shape.grid_w > 0 && shape.ring_frames > 0 &&
           mul(shape.grid_h, shape.grid_w, &tokens) && mul(tokens, shape.chunk_frames, &tokens) &&
           mul(tokens, shape.batch, &act) && mul(act, shape.heads, &act) && mul(act, shape.head_dim, &act);
    return &shape;
  }
  int64_t cache(int32_t sink) {   // elements of one cache
    int64_t e = static_cast<int64_t>(shape.ring_frames) + sink;
    good = good && mul(e, shape.batch, &e) && mul(e, static_cast<int64_t>(shape.grid_h) * shape.grid_w, &e) &&
           mul(e, static_cast<int64_t>(shape.heads) * shape.head_dim, &e);
    return e;
  }
  int64_t integer(int64_t lo, int64_t hi) {
    if (!good) return 0;
    PyObject* o = a[i++];
    if (!PyLong_CheckExact(o)) {
      good = false;
      return 0;
    }
    int over = 0;
    const int64_t v = PyLong_AsLongLongAndOverflow(o, &over);
    good = over == 0 && v >= lo && v <= hi;
    return v;
  }
  int32_t int32() { return static_cast<int32_t>(integer(INT32_MIN, INT32_MAX)); }
  void starts(int32_t* out) {
    if (!good) return;
    PyObject* o = a[i++];
    if (!(PyList_CheckExact(o) || PyTuple_CheckExact(o)) || shape.batch > kMaxStreams ||
        PySequence_Fast_GET_SIZE(o) != shape.batch) {
      good = false;
      return;
    }
    PyObject** items = PySequence_Fast_ITEMS(o);
    for (int b = 0; b < shape.batch && good; ++b) {
      int over = 0;
      good = PyLong_CheckExact(items[b]);
      if (!good) return;
      const int64_t v = PyLong_AsLongLongAndOverflow(items[b], &over);
      good = over == 0 && v >= INT32_MIN && v <= INT32_MAX;
      out[b] = static_cast<int32_t>(v);
    }
  }
  float real() {
    if (!good) return 0.f;
    PyObject* o = a[i++];
    good = PyFloat_CheckExact(o);
    return good ? static_cast<float>(PyFloat_AS_DOUBLE(o)) : 0.f;
  }
  void* tensor(at::ScalarType type, int64_t numel) {
    if (!good) return nullptr;
    PyObject* o = a[i++];
    if (!THPVariable_CheckExact(o)) {
      good = false;
      return nullptr;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    good = t.is_cuda() && t.scalar_type() == type && t.layout() == at::kStrided && t.is_contiguous() &&
           t.numel() == numel;
    return good ? t.data_ptr() : nullptr;
  }
  void* stream() {
    if (!good) return nullptr;
    PyObject* o = a[i++];
    if (o == Py_None) return static_cast<void*>(c10::cuda::getCurrentCUDAStream().stream());
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (h == nullptr || !PyLong_CheckExact(h)) {
      PyErr_Clear();
      Py_XDECREF(h);
      good = false;
      return nullptr;
    }
    void* p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (PyErr_Occurred()) {
      PyErr_Clear();
      good = false;
    }
    return p;
  }
};

// A tensor wrapper without storage makes its accessors throw: such a call is not well-formed either.
template <typename F>
PyObject* guarded(F&& body) {
  try {
    return body();
  } catch (const std::exception&) {
    PyErr_Clear();
    Py_RETURN_NONE;
  }
}

template <typename F>
PyObject* call(bool good, F&& f) {
  if (!good || PyErr_Occurred()) {
    PyErr_Clear();
    Py_RETURN_NONE;
  }
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

constexpr auto kF32 = at::kFloat;
constexpr auto kBf16 = at::kBFloat16;

// (shape, start_frame, cos, sin, stream)
PyObject* py_table(PyObject*, PyObject* const* args, Py_ssize_t n) {
  return guarded([&] {
    Args a(args, n, 5);
    const unstep_shape_t* s = a.get_shape();
    const int32_t start = a.int32();
    int64_t e = 0;
    a.good = a.good && Args::mul(a.tokens, 64, &e);
    float* cos = static_cast<float*>(a.tensor(kF32, e));
    float* sin = static_cast<float*>(a.tensor(kF32, e));
    void* st = a.stream();
    return call(a.good, [&] { return f_table(s, start, cos, sin, st); });
  });
}

// (shape, sink_frames, start_frame, q, k, v, [gain_q, gain_k, eps,] cos, sin, q_out, cache_k, cache_v,
//  table_stream_stride, stream)
template <bool kNorm>
PyObject* py_append(PyObject*, PyObject* const* args, Py_ssize_t n) {
  return guarded([&] {
    Args a(args, n, kNorm ? 16 : 13);
    int32_t starts[kMaxStreams];
    const unstep_shape_t* s = a.get_shape();
    const int32_t sink = static_cast<int32_t>(a.integer(0, 1 << 20));
    a.starts(starts);
    int64_t stride = 0, table = 0;
    if (a.good) {   // the stride decides the size of the tables
      PyObject* o = args[n - 2];
      int over = 0;
      a.good = PyLong_CheckExact(o);
      if (a.good) stride = PyLong_AsLongLongAndOverflow(o, &over);
      a.good = a.good && over == 0 && stride >= 0 && stride < (int64_t{1} << 40) &&
               Args::mul(a.tokens, 64, &table) && !__builtin_add_overflow(table, (s->batch - 1) * stride, &table);
    }
    const void* q = a.tensor(kBf16, a.act);
    const void* k = a.tensor(kBf16, a.act);
    const void* v = a.tensor(kBf16, a.act);
    const float *gq = nullptr, *gk = nullptr;
    float eps = 0.f;
    if (kNorm) {
      const int64_t wide = static_cast<int64_t>(a.shape.heads) * a.shape.head_dim;
      gq = static_cast<const float*>(a.tensor(kF32, wide));
      gk = static_cast<const float*>(a.tensor(kF32, wide));
      eps = a.real();
    }
    const float* cos = static_cast<const float*>(a.tensor(kF32, table));
    const float* sin = static_cast<const float*>(a.tensor(kF32, table));
    void* q_out = a.tensor(kBf16, a.act);
    const int64_t cache = a.cache(sink);
    void* ck = a.tensor(kBf16, cache);
    void* cv = a.tensor(kBf16, cache);
    ++a.i;   // the stride
    void* st = a.stream();
    return call(a.good, [&] {
      if (kNorm)
        return f_norm_append(s, sink, starts, q, k, v, gq, gk, eps, cos, sin, stride, q_out, ck, cv, st);
      return f_append_sink(s, sink, starts, q, k, v, cos, sin, stride, q_out, ck, cv, st);
    });
  });
}

// (shape, start_frame, window_frames, q, cache_k, cache_v, out, stream), with a sink:
// (shape, sink_frames, start_frame, recent_frames, sink_attend, q, cache_k, cache_v, out, stream)
template <int kKind>   // 0 plain, 1 without allocation, 2 with a sink
PyObject* py_attn(PyObject*, PyObject* const* args, Py_ssize_t n) {
  return guarded([&] {
    Args a(args, n, kKind == 2 ? 10 : 8);
    int32_t starts[kMaxStreams];
    const unstep_shape_t* s = a.get_shape();
    const int32_t sink = kKind == 2 ? static_cast<int32_t>(a.integer(0, 1 << 20)) : 0;
    a.starts(starts);
    const int32_t window = a.int32();
    const int32_t attend = kKind == 2 ? a.int32() : 0;
    const void* q = a.tensor(kBf16, a.act);
    const int64_t cache = a.cache(sink);
    const void* ck = a.tensor(kBf16, cache);
    const void* cv = a.tensor(kBf16, cache);
    void* out = a.tensor(kBf16, a.act);
    void* st = a.stream();
    return call(a.good, [&] {
      if (kKind == 2) return f_attn_sink(s, sink, starts, window, attend, q, ck, cv, out, st);
      return (kKind == 1 ? f_attn_noalloc : f_attn)(s, starts, window, q, ck, cv, out, st);
    });
  });
}

// bind(Shape, table, append_sink, norm_append, attn, attn_noalloc, attn_sink): addresses of the library's functions
PyObject* py_bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != 7 || !PyType_Check(args[0])) {
    PyErr_SetString(PyExc_TypeError, "bind: the Shape type and six addresses");
    return nullptr;
  }
  void* p[6];
  for (int i = 0; i < 6; ++i) {
    p[i] = PyLong_AsVoidPtr(args[i + 1]);
    if (PyErr_Occurred()) return nullptr;
  }
  Py_INCREF(args[0]);
  Py_XDECREF(reinterpret_cast<PyObject*>(shape_type));
  shape_type = reinterpret_cast<PyTypeObject*>(args[0]);
  f_table = reinterpret_cast<decltype(f_table)>(p[0]);
  f_append_sink = reinterpret_cast<decltype(f_append_sink)>(p[1]);
  f_norm_append = reinterpret_cast<decltype(f_norm_append)>(p[2]);
  f_attn = reinterpret_cast<decltype(f_attn)>(p[3]);
  f_attn_noalloc = reinterpret_cast<decltype(f_attn_noalloc)>(p[4]);
  f_attn_sink = reinterpret_cast<decltype(f_attn_sink)>(p[5]);
  Py_RETURN_NONE;
}

template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyCFunction fast() {
  return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(F));
}

PyMethodDef methods[] = {
    {"bind", fast<py_bind>(), METH_FASTCALL, nullptr},
    {"rope_table", fast<py_table>(), METH_FASTCALL, nullptr},
    {"append", fast<py_append<false>>(), METH_FASTCALL, nullptr},
    {"norm_append", fast<py_append<true>>(), METH_FASTCALL, nullptr},
    {"attn", fast<py_attn<0>>(), METH_FASTCALL, nullptr},
    {"attn_noalloc", fast<py_attn<1>>(), METH_FASTCALL, nullptr},
    {"attn_sink", fast<py_attn<2>>(), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void) { return PyModule_Create(&module); }
