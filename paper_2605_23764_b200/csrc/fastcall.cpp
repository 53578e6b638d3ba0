// The calls of a step -- routing, router, layout, forward, backward -- from Python without interpreted marshalling: arguments
// are looked at and outputs allocated in C++, then the C entry point of libmoe_b200 is called with the GIL released.
//
// What bounds the smallest calls is host time: checking six tensors through Python attributes and converting them with
// ctypes took 3-4 us a call, an output allocated from Python 2 us, next to 2-3 us for the launch itself.  Routing + layout of
// 1024 tokens 25 -> 16 us, the router of a few tokens, both directions, 21 -> 14 us.
//
// Every function answers None for arguments it does not take as they are (a wrong type, size, place or layout, an unknown
// context): the caller then goes through the interpreted checks, which say what is wrong.  Otherwise it answers the entry
// point's code, or the outputs it made.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <stdexcept>
#include <unordered_map>

namespace {

struct Shape { int64_t T_max, d, E, k, S, F; };
std::unordered_map<void*, Shape> g_shapes;   // under the GIL

using P = void*;
int (*f_route)(P, const P, int32_t, P, P, P, P);
int (*f_router_fwd)(P, const P, const P, int32_t, P, P, P, P, P);
int (*f_router_bwd)(P, const P, const P, const P, int32_t, P, P);
int (*f_layout_noalloc)(const P, int32_t, int32_t, int32_t, int32_t, P, P, P, P, P, P);
int (*f_ffn_fwd)(P, const P, const P, const P, const P, const P, P, int32_t, P);
int (*f_ffn_bwd)(P, const P, const P, const P, const P, const P, const P, P, P, P, P, int32_t, P);

struct Slow {};   // not for this path

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) throw Slow();
  return THPVariable_Unpack(o);
}
void* check(const at::Tensor& t, at::ScalarType type, int64_t n) {
  if (!t.is_cuda() || t.scalar_type() != type || t.numel() < n || !t.is_contiguous()) throw Slow();
  return t.data_ptr();
}
void* dev(PyObject* o, at::ScalarType type, int64_t n) { return check(tensor(o), type, n); }
void* dev_or_null(PyObject* o, at::ScalarType type, int64_t n) { return o == Py_None ? nullptr : dev(o, type, n); }
int64_t integer(PyObject* o) {
  if (!PyLong_CheckExact(o)) throw Slow();
  int over = 0;
  const long long v = PyLong_AsLongLongAndOverflow(o, &over);
  if (over || v < INT32_MIN || v > INT32_MAX) throw Slow();
  return v;
}
void* handle(PyObject* o) {   // a ctypes.c_void_p
  Py_buffer view;
  if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) {
    PyErr_Clear();
    throw Slow();
  }
  void* h = view.len == (Py_ssize_t)sizeof(void*) ? *static_cast<void**>(view.buf) : nullptr;
  PyBuffer_Release(&view);
  return h;
}
const Shape& shape_of(void* h) {
  const auto it = g_shapes.find(h);
  if (it == g_shapes.end()) throw Slow();
  return it->second;
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

template <class F>
int unlocked(F call) {
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = call();
  Py_END_ALLOW_THREADS
  return rc;
}
at::Tensor empty(at::IntArrayRef size, at::ScalarType type, const at::Tensor& like) {
  return at::empty(size, at::TensorOptions().dtype(type).device(like.device()));
}

constexpr auto BF = at::kBFloat16, I32 = at::kInt, F32 = at::kFloat;

// a function body that may throw Slow (None) or a C++ exception of the allocator (RuntimeError)
template <class F>
PyObject* guarded(F body) {
  try {
    return body();
  } catch (const Slow&) {
    Py_RETURN_NONE;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}
void want(Py_ssize_t n, Py_ssize_t need) { if (n != need) throw Slow(); }

PyObject* setup(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 6) { PyErr_SetString(PyExc_TypeError, "setup: six addresses"); return nullptr; }
  void* p[6];
  for (int i = 0; i < 6; ++i) {
    p[i] = PyLong_AsVoidPtr(a[i]);
    if (!p[i]) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "setup: null address");
      return nullptr;
    }
  }
  f_route = reinterpret_cast<decltype(f_route)>(p[0]);
  f_router_fwd = reinterpret_cast<decltype(f_router_fwd)>(p[1]);
  f_router_bwd = reinterpret_cast<decltype(f_router_bwd)>(p[2]);
  f_layout_noalloc = reinterpret_cast<decltype(f_layout_noalloc)>(p[3]);
  f_ffn_fwd = reinterpret_cast<decltype(f_ffn_fwd)>(p[4]);
  f_ffn_bwd = reinterpret_cast<decltype(f_ffn_bwd)>(p[5]);
  Py_RETURN_NONE;
}
PyObject* add(PyObject*, PyObject* const* a, Py_ssize_t n) {   // handle, T_max, d, E, k, S, F
  return guarded([&]() -> PyObject* {
    want(n, 7);
    Shape s{integer(a[1]), integer(a[2]), integer(a[3]), integer(a[4]), integer(a[5]), integer(a[6])};
    g_shapes[handle(a[0])] = s;
    Py_RETURN_NONE;
  });
}
PyObject* drop(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    want(n, 1);
    g_shapes.erase(handle(a[0]));
    Py_RETURN_NONE;
  });
}

PyObject* route(PyObject*, PyObject* const* a, Py_ssize_t n) {   // ctx, logits, T, ids, w, counts
  return guarded([&]() -> PyObject* {
    want(n, 6);
    void* c = handle(a[0]);
    const Shape& s = shape_of(c);
    const int64_t T = integer(a[2]);
    void *logits = dev(a[1], F32, T * s.E), *ids = dev(a[3], I32, T * s.k), *w = dev(a[4], F32, T * s.k),
         *counts = dev_or_null(a[5], I32, s.E), *st = stream();
    return PyLong_FromLong(unlocked([&] { return f_route(c, logits, (int32_t)T, ids, w, counts, st); }));
  });
}
PyObject* route_new(PyObject*, PyObject* const* a, Py_ssize_t n) {   // ctx, logits -> (code, ids, w)
  return guarded([&]() -> PyObject* {
    want(n, 2);
    void* c = handle(a[0]);
    const Shape& s = shape_of(c);
    const at::Tensor& l = tensor(a[1]);
    if (l.dim() < 1) throw Slow();
    const int64_t T = l.size(0);
    void *logits = check(l, F32, T * s.E), *st = stream();
    at::Tensor ids = empty({T, s.k}, I32, l), w = empty({T, s.k}, F32, l);
    void *pi = ids.data_ptr(), *pw = w.data_ptr();
    const int rc = unlocked([&] { return f_route(c, logits, (int32_t)T, pi, pw, nullptr, st); });
    return Py_BuildValue("(iNN)", rc, THPVariable_Wrap(ids), THPVariable_Wrap(w));
  });
}
PyObject* router_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {   // ctx, x, W_r, T, ids, w, logits, counts
  return guarded([&]() -> PyObject* {
    want(n, 8);
    void* c = handle(a[0]);
    const Shape& s = shape_of(c);
    const int64_t T = integer(a[3]);
    void *x = dev(a[1], BF, T * s.d), *W = dev(a[2], BF, s.E * s.d), *ids = dev(a[4], I32, T * s.k), *w = dev(a[5], F32, T * s.k),
         *logits = dev_or_null(a[6], F32, T * s.E), *counts = dev_or_null(a[7], I32, s.E), *st = stream();
    return PyLong_FromLong(unlocked([&] { return f_router_fwd(c, x, W, (int32_t)T, ids, w, logits, counts, st); }));
  });
}
PyObject* router_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {   // ctx, logits, ids, d_w, T, d_logits
  return guarded([&]() -> PyObject* {
    want(n, 6);
    void* c = handle(a[0]);
    const Shape& s = shape_of(c);
    const int64_t T = integer(a[4]);
    void *logits = dev(a[1], F32, T * s.E), *ids = dev(a[2], I32, T * s.k), *dw = dev(a[3], F32, T * s.k),
         *dl = dev(a[5], F32, T * s.E), *st = stream();
    return PyLong_FromLong(unlocked([&] { return f_router_bwd(c, logits, ids, dw, (int32_t)T, dl, st); }));
  });
}
PyObject* layout_noalloc(PyObject*, PyObject* const* a, Py_ssize_t n) {   // ids, T, E, k, S, counts, offsets, row_of, src_of, status2
  return guarded([&]() -> PyObject* {
    want(n, 10);
    if (!f_layout_noalloc) throw Slow();   // the library is not loaded yet (the other calls have a context)
    const int64_t T = integer(a[1]), E = integer(a[2]), k = integer(a[3]), S = integer(a[4]);
    if (T < 0 || E < 0 || k < 0 || S < 0) throw Slow();
    const int64_t slots = T * (k + S);
    void *ids = dev(a[0], I32, T * k), *counts = dev(a[5], I32, E + S), *offsets = dev(a[6], I32, E + S + 1),
         *row_of = dev(a[7], I32, slots), *src_of = dev(a[8], I32, slots), *status = dev_or_null(a[9], I32, 2), *st = stream();
    return PyLong_FromLong(unlocked([&] {
      return f_layout_noalloc(ids, (int32_t)T, (int32_t)E, (int32_t)k, (int32_t)S, counts, offsets, row_of, src_of, status, st);
    }));
  });
}
PyObject* ffn_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {   // ctx, x, ids, w, W1, W2, out, T
  return guarded([&]() -> PyObject* {
    want(n, 8);
    void* c = handle(a[0]);
    const Shape& s = shape_of(c);
    const int64_t T = integer(a[7]), nw = (s.E + s.S) * s.d * s.F;
    void *x = dev(a[1], BF, T * s.d), *ids = dev(a[2], I32, T * s.k), *w = dev(a[3], F32, T * s.k), *W1 = dev(a[4], BF, 2 * nw),
         *W2 = dev(a[5], BF, nw), *out = dev(a[6], BF, T * s.d), *st = stream();
    return PyLong_FromLong(unlocked([&] { return f_ffn_fwd(c, x, ids, w, W1, W2, out, (int32_t)T, st); }));
  });
}
PyObject* ffn_fwd_new(PyObject*, PyObject* const* a, Py_ssize_t n) {   // ctx, x, ids, w, W1, W2 -> (code, out)
  return guarded([&]() -> PyObject* {
    want(n, 6);
    void* c = handle(a[0]);
    const Shape& s = shape_of(c);
    const at::Tensor& xt = tensor(a[1]);
    if (xt.dim() < 1) throw Slow();
    const int64_t T = xt.size(0), nw = (s.E + s.S) * s.d * s.F;
    void *x = check(xt, BF, T * s.d), *ids = dev(a[2], I32, T * s.k), *w = dev(a[3], F32, T * s.k), *W1 = dev(a[4], BF, 2 * nw),
         *W2 = dev(a[5], BF, nw), *st = stream();
    at::Tensor out = empty({T, s.d}, BF, xt);
    void* po = out.data_ptr();
    const int rc = unlocked([&] { return f_ffn_fwd(c, x, ids, w, W1, W2, po, (int32_t)T, st); });
    return Py_BuildValue("(iN)", rc, THPVariable_Wrap(out));
  });
}
// ctx, dout, x, ids, w, W1, W2, dx, dW1, dW2, d_w, T
PyObject* ffn_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    want(n, 12);
    void* c = handle(a[0]);
    const Shape& s = shape_of(c);
    const int64_t T = integer(a[11]), nw = (s.E + s.S) * s.d * s.F;
    void *dout = dev(a[1], BF, T * s.d), *x = dev(a[2], BF, T * s.d), *ids = dev(a[3], I32, T * s.k), *w = dev(a[4], F32, T * s.k),
         *W1 = dev(a[5], BF, 2 * nw), *W2 = dev(a[6], BF, nw), *dx = dev(a[7], BF, T * s.d), *dW1 = dev(a[8], BF, 2 * nw),
         *dW2 = dev(a[9], BF, nw), *dw = dev_or_null(a[10], F32, T * s.k), *st = stream();
    return PyLong_FromLong(unlocked([&] { return f_ffn_bwd(c, dout, x, ids, w, W1, W2, dx, dW1, dW2, dw, (int32_t)T, st); }));
  });
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(setup), FAST(add), FAST(drop), FAST(route), FAST(route_new), FAST(router_fwd), FAST(router_bwd),
                         FAST(layout_noalloc), FAST(ffn_fwd), FAST(ffn_fwd_new), FAST(ffn_bwd), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() { return PyModule_Create(&module); }
