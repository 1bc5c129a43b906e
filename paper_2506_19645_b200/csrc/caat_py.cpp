// Argument marshalling of the hot calls for the Python binding (caat.py): checks the tensors, takes their addresses and
// the current stream, calls the C ABI.  A few-token step takes about 25 us on the GPU; the same checks written in Python
// and the ctypes conversion cost 14 us of host time per block call, here about one.
//
// An argument that fails a check is handed to the binding's own checking function, which words the exception.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <initializer_list>

#include "caat.h"

namespace {

struct Dims {
  caat_ctx* ctx;
  at::ScalarType td;
  int64_t t, h, ka, km;
};
constexpr const char* kDimsName = "caat.dims";
PyObject* g_explain = nullptr;      // explain(tensor, dtype code, shape, name): raises

void free_dims(PyObject* cap) { delete static_cast<Dims*>(PyCapsule_GetPointer(cap, kDimsName)); }

// dims(ctx address, dtype code, t, h, K_r of attention-out, K_r of MLP-down) -> capsule
PyObject* dims(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 6) { PyErr_SetString(PyExc_TypeError, "dims: six arguments"); return nullptr; }
  const unsigned long long p = PyLong_AsUnsignedLongLong(a[0]);
  long long v[5];
  for (int i = 0; i < 5; ++i) v[i] = PyLong_AsLongLong(a[i + 1]);
  if (PyErr_Occurred()) return nullptr;
  return PyCapsule_New(new Dims{reinterpret_cast<caat_ctx*>(p), v[0] == CAAT_BF16 ? at::kBFloat16 : at::kFloat, v[1], v[2], v[3], v[4]},
                       kDimsName, free_dims);
}

PyObject* set_explain(PyObject*, PyObject* f) {
  Py_XINCREF(f);
  Py_XDECREF(g_explain);
  g_explain = f;
  Py_RETURN_NONE;
}

// The arguments of one call, taken in order.
struct Args {
  PyObject* const* a;
  Py_ssize_t n, i = 0;
  bool ok;
  Dims* d = nullptr;
  int64_t T = 0;

  Args(PyObject* const* args, Py_ssize_t nargs, Py_ssize_t want) : a(args), n(nargs), ok(nargs == want) {
    if (!ok) { PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs); return; }
    d = static_cast<Dims*>(PyCapsule_GetPointer(a[i++], kDimsName));
    ok = d != nullptr;
  }
  int integer() {
    if (!ok) return 0;
    const long v = PyLong_AsLong(a[i++]);
    if (v == -1 && PyErr_Occurred()) ok = false;
    return (int)v;
  }
  int tokens() { T = integer(); return (int)T; }
  void* fail(PyObject* x, at::ScalarType st, std::initializer_list<int64_t> shape, const char* name) {
    ok = false;
    PyObject* sh = PyTuple_New((Py_ssize_t)shape.size());
    Py_ssize_t k = 0;
    for (int64_t v : shape) PyTuple_SET_ITEM(sh, k++, PyLong_FromLongLong(v));
    PyObject* r = PyObject_CallFunction(g_explain, "OiOs", x, st == at::kBFloat16 ? CAAT_BF16 : CAAT_F32, sh, name);
    Py_DECREF(sh);
    if (r) {
      Py_DECREF(r);
      PyErr_Format(PyExc_ValueError, "%s: rejected", name);
    }
    return nullptr;
  }
  void* tensor(at::ScalarType st, std::initializer_list<int64_t> shape, const char* name) {
    if (!ok) return nullptr;
    PyObject* x = a[i++];
    if (x == Py_None) return nullptr;
    if (!THPVariable_Check(x)) return fail(x, st, shape, name);
    const at::Tensor& v = THPVariable_Unpack(x);
    if (!v.is_cuda() || !v.is_contiguous() || v.scalar_type() != st || v.sizes() != at::IntArrayRef(shape)) return fail(x, st, shape, name);
    return v.numel() ? v.data_ptr() : nullptr;
  }
  void* run(std::initializer_list<int64_t> shape, const char* name) { return ok ? tensor(d->td, shape, name) : nullptr; }
  float* f32(std::initializer_list<int64_t> shape, const char* name) { return static_cast<float*>(tensor(at::kFloat, shape, name)); }
  // activations [t, T, h], row statistics [t, T], norm parameters [h]
  void* act(const char* name) { return ok ? run({d->t, T, d->h}, name) : nullptr; }
  float* stat(const char* name) { return ok ? f32({d->t, T}, name) : nullptr; }
  void* vec(const char* name) { return ok ? run({d->h}, name) : nullptr; }
  float* fvec(const char* name) { return ok ? f32({d->h}, name) : nullptr; }
  void* workspace(size_t* bytes) {      // uint8 of any shape
    *bytes = 0;
    if (!ok) return nullptr;
    PyObject* x = a[i++];
    if (x == Py_None) return nullptr;
    if (THPVariable_Check(x)) {
      const at::Tensor& v = THPVariable_Unpack(x);
      if (v.is_cuda() && v.is_contiguous() && v.scalar_type() == at::kByte) {
        *bytes = (size_t)v.numel();
        return v.numel() ? v.data_ptr() : nullptr;
      }
    }
    ok = false;
    PyObject* r = PyObject_CallFunction(g_explain, "OiOs", x, -1, Py_None, "workspace");
    if (r) {
      Py_DECREF(r);
      PyErr_SetString(PyExc_ValueError, "workspace: rejected");
    }
    return nullptr;
  }
};

template <typename F>
PyObject* call(Args& g, F f) {
  if (!g.ok) return nullptr;
  caat_status s;
  void* st = c10::cuda::getCurrentCUDAStream().stream();
  Py_BEGIN_ALLOW_THREADS
  s = f(st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)s);
}

int64_t layer_kr(const Args& g, int layer) { return layer == CAAT_ATTN_OUT ? g.d->ka : g.d->km; }

#define CAAT_FN(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs)

PyObject* forward(PyObject* const* args, Py_ssize_t nargs, bool noalloc) {
  Args g(args, nargs, noalloc ? 12 : 13);
  const int layer = g.integer(), T = g.tokens();
  if (!g.ok) return nullptr;
  const int64_t k = layer_kr(g, layer), t = g.d->t, h = g.d->h;
  void *Y = g.run({t, T, k}, "Y"), *W = g.run({t, h, k}, "W"), *R = g.act("R"), *ga = g.vec("gamma"), *be = g.vec("beta"),
       *Hn = g.act("Hn"), *X = g.act("X");
  float *rs = g.stat("rstd"), *mu = g.stat("mean");
  if (noalloc)
    return call(g, [&](void* st) {
      return caat_rowpar_forward_noalloc(g.d->ctx, (caat_layer)layer, T, Y, W, R, ga, be, Hn, X, rs, mu, st);
    });
  size_t nb;
  void* ws = g.workspace(&nb);
  return call(g, [&](void* st) {
    return caat_rowpar_forward(g.d->ctx, (caat_layer)layer, T, Y, W, R, ga, be, Hn, X, rs, mu, ws, nb, st);
  });
}
CAAT_FN(rowpar_forward) { return forward(args, nargs, false); }
CAAT_FN(rowpar_forward_noalloc) { return forward(args, nargs, true); }

CAAT_FN(rowpar_backward) {
  Args g(args, nargs, 17);
  const int layer = g.integer(), T = g.tokens();
  if (!g.ok) return nullptr;
  const int64_t k = layer_kr(g, layer), t = g.d->t, h = g.d->h;
  void *dX = g.act("dX"), *dHn = g.act("dHn"), *Y = g.run({t, T, k}, "Y"), *W = g.run({t, h, k}, "W"), *Hn = g.act("Hn");
  float *rs = g.stat("rstd"), *mu = g.stat("mean");
  void *ga = g.vec("gamma"), *dY = g.run({t, T, k}, "dY");
  float* dW = g.f32({t, h, k}, "dW");
  void* dR = g.act("dR");
  float *dg = g.fvec("dgamma"), *db = g.fvec("dbeta");
  size_t nb;
  void* ws = g.workspace(&nb);
  return call(g, [&](void* st) {
    return caat_rowpar_backward(g.d->ctx, (caat_layer)layer, T, dX, dHn, Y, W, Hn, rs, mu, ga, dY, dW, dR, dg, db, ws, nb, st);
  });
}

CAAT_FN(block_forward) {
  Args g(args, nargs, 20);
  const int T = g.tokens();
  if (!g.ok) return nullptr;
  const int64_t t = g.d->t, h = g.d->h, ka = g.d->ka, km = g.d->km;
  void *Ya = g.run({t, T, ka}, "Y_attn"), *Wo = g.run({t, h, ka}, "W_o"), *Ym = g.run({t, T, km}, "Y_mlp"),
       *Wd = g.run({t, h, km}, "W_down"), *R0 = g.act("R0"), *g1 = g.vec("gamma1"), *b1 = g.vec("beta1"), *g2 = g.vec("gamma2"),
       *b2 = g.vec("beta2"), *H1 = g.act("Hn1"), *X1 = g.act("X1");
  float *r1 = g.stat("rstd1"), *m1 = g.stat("mean1");
  void *H2 = g.act("Hn2"), *X2 = g.act("X2");
  float *r2 = g.stat("rstd2"), *m2 = g.stat("mean2");
  size_t nb;
  void* ws = g.workspace(&nb);
  return call(g, [&](void* st) {
    return caat_block_forward(g.d->ctx, T, Ya, Wo, Ym, Wd, R0, g1, b1, g2, b2, H1, X1, r1, m1, H2, X2, r2, m2, ws, nb, st);
  });
}

CAAT_FN(block_backward) {
  Args g(args, nargs, 28);
  const int T = g.tokens();
  if (!g.ok) return nullptr;
  const int64_t t = g.d->t, h = g.d->h, ka = g.d->ka, km = g.d->km;
  void *dX1 = g.act("dX1"), *dX2 = g.act("dX2"), *dH2 = g.act("dHn2"), *Ya = g.run({t, T, ka}, "Y_attn"), *Wo = g.run({t, h, ka}, "W_o"),
       *Ym = g.run({t, T, km}, "Y_mlp"), *Wd = g.run({t, h, km}, "W_down"), *H1 = g.act("Hn1");
  float *r1 = g.stat("rstd1"), *m1 = g.stat("mean1");
  void* H2 = g.act("Hn2");
  float *r2 = g.stat("rstd2"), *m2 = g.stat("mean2");
  void *g1 = g.vec("gamma1"), *g2 = g.vec("gamma2"), *dYa = g.run({t, T, ka}, "dY_attn");
  float* dWo = g.f32({t, h, ka}, "dW_o");
  void* dYm = g.run({t, T, km}, "dY_mlp");
  float* dWd = g.f32({t, h, km}, "dW_down");
  void *dR0 = g.act("dR0"), *dH1 = g.act("dHn1");
  float *dg1 = g.fvec("dgamma1"), *db1 = g.fvec("dbeta1"), *dg2 = g.fvec("dgamma2"), *db2 = g.fvec("dbeta2");
  size_t nb;
  void* ws = g.workspace(&nb);
  return call(g, [&](void* st) {
    return caat_block_backward(g.d->ctx, T, dX1, dX2, dH2, Ya, Wo, Ym, Wd, H1, r1, m1, H2, r2, m2, g1, g2, dYa, dWo, dYm, dWd, dR0,
                               dH1, dg1, db1, dg2, db2, ws, nb, st);
  });
}

CAAT_FN(block_forward_compact) {
  Args g(args, nargs, 23);
  const int T = g.tokens();
  if (!g.ok) return nullptr;
  const int64_t t = g.d->t, h = g.d->h, ka = g.d->ka, km = g.d->km, S = caat_shared_channels(g.d->ctx);
  auto sh = [&](const char* n) { return g.run({T, S}, n); };
  auto pr = [&](const char* n) { return g.run({t, T, h - S}, n); };
  void *Ya = g.run({t, T, ka}, "Y_attn"), *Wo = g.run({t, h, ka}, "W_o"), *Ym = g.run({t, T, km}, "Y_mlp"),
       *Wd = g.run({t, h, km}, "W_down"), *R0s = sh("R0s"), *R0p = pr("R0p"), *g1 = g.vec("gamma1"), *b1 = g.vec("beta1"),
       *g2 = g.vec("gamma2"), *b2 = g.vec("beta2"), *H1s = sh("Hn1s"), *H1p = pr("Hn1p"), *X1 = g.act("X1");
  float *r1 = g.stat("rstd1"), *m1 = g.stat("mean1");
  void *H2s = sh("Hn2s"), *H2p = pr("Hn2p"), *X2 = g.act("X2");
  float *r2 = g.stat("rstd2"), *m2 = g.stat("mean2");
  size_t nb;
  void* ws = g.workspace(&nb);
  return call(g, [&](void* st) {
    return caat_block_forward_compact(g.d->ctx, T, Ya, Wo, Ym, Wd, R0s, R0p, g1, b1, g2, b2, H1s, H1p, X1, r1, m1, H2s, H2p, X2, r2,
                                      m2, ws, nb, st);
  });
}

CAAT_FN(block_backward_compact) {
  Args g(args, nargs, 33);
  const int T = g.tokens();
  if (!g.ok) return nullptr;
  const int64_t t = g.d->t, h = g.d->h, ka = g.d->ka, km = g.d->km, S = caat_shared_channels(g.d->ctx);
  auto sh = [&](const char* n) { return g.run({T, S}, n); };
  auto pr = [&](const char* n) { return g.run({t, T, h - S}, n); };
  void *dX1 = g.act("dX1"), *dX2 = g.act("dX2"), *dH2s = sh("dHn2s"), *dH2p = pr("dHn2p"), *Ya = g.run({t, T, ka}, "Y_attn"),
       *Wo = g.run({t, h, ka}, "W_o"), *Ym = g.run({t, T, km}, "Y_mlp"), *Wd = g.run({t, h, km}, "W_down"), *H1s = sh("Hn1s"),
       *H1p = pr("Hn1p");
  float *r1 = g.stat("rstd1"), *m1 = g.stat("mean1");
  void *H2s = sh("Hn2s"), *H2p = pr("Hn2p");
  float *r2 = g.stat("rstd2"), *m2 = g.stat("mean2");
  void *g1 = g.vec("gamma1"), *g2 = g.vec("gamma2"), *dYa = g.run({t, T, ka}, "dY_attn");
  float* dWo = g.f32({t, h, ka}, "dW_o");
  void* dYm = g.run({t, T, km}, "dY_mlp");
  float* dWd = g.f32({t, h, km}, "dW_down");
  void *dR0s = sh("dR0s"), *dR0p = pr("dR0p"), *dH1s = sh("dHn1s"), *dH1p = pr("dHn1p");
  float *dg1 = g.fvec("dgamma1"), *db1 = g.fvec("dbeta1"), *dg2 = g.fvec("dgamma2"), *db2 = g.fvec("dbeta2");
  size_t nb;
  void* ws = g.workspace(&nb);
  return call(g, [&](void* st) {
    return caat_block_backward_compact(g.d->ctx, T, dX1, dX2, dH2s, dH2p, Ya, Wo, Ym, Wd, H1s, H1p, r1, m1, H2s, H2p, r2, m2, g1, g2,
                                       dYa, dWo, dYm, dWd, dR0s, dR0p, dH1s, dH1p, dg1, db1, dg2, db2, ws, nb, st);
  });
}

CAAT_FN(colpar_forward) {
  Args g(args, nargs, 8);
  const int act = g.integer(), n_out = g.integer(), T = g.tokens();
  if (!g.ok) return nullptr;
  const int64_t t = g.d->t, h = g.d->h, wy = act == CAAT_ACT_SWIGLU ? n_out / 2 : n_out;
  void *X = g.act("X"), *A = g.run({t, n_out, h}, "A"), *pre = g.run({t, T, n_out}, "pre"), *Y = g.run({t, T, wy}, "Y");
  return call(g, [&](void* st) { return caat_colpar_forward(g.d->ctx, (caat_activation)act, n_out, T, X, A, pre, Y, st); });
}

CAAT_FN(colpar_backward) {
  Args g(args, nargs, 11);
  const int act = g.integer(), n_out = g.integer(), T = g.tokens();
  if (!g.ok) return nullptr;
  const int64_t t = g.d->t, h = g.d->h, wy = act == CAAT_ACT_SWIGLU ? n_out / 2 : n_out;
  void *dY = g.run({t, T, wy}, "dY"), *X = g.act("X"), *A = g.run({t, n_out, h}, "A"), *pre = g.run({t, T, n_out}, "pre"),
       *dX = g.act("dX");
  float* dA = g.f32({t, n_out, h}, "dA");
  size_t nb;
  void* ws = g.workspace(&nb);
  return call(g, [&](void* st) {
    return caat_colpar_backward(g.d->ctx, (caat_activation)act, n_out, T, dY, X, A, pre, dX, dA, ws, nb, st);
  });
}

// The entry of every call: a tensor's methods throw for a tensor without storage (inside vmap), a sparse one, a machine
// without a device.  C++ exceptions must not leave through Python's C frames; torch's own translation raises what the same
// method raises in Python.
using Fn = PyObject* (*)(PyObject*, PyObject* const*, Py_ssize_t);
template <Fn F>
PyObject* entry(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
  HANDLE_TH_ERRORS
  return F(self, args, nargs);
  END_HANDLE_TH_ERRORS
}

#define CAAT_DEF(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<name>)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    {"set_explain", set_explain, METH_O, nullptr},
    CAAT_DEF(dims), CAAT_DEF(rowpar_forward), CAAT_DEF(rowpar_forward_noalloc), CAAT_DEF(rowpar_backward), CAAT_DEF(block_forward),
    CAAT_DEF(block_backward), CAAT_DEF(block_forward_compact), CAAT_DEF(block_backward_compact), CAAT_DEF(colpar_forward),
    CAAT_DEF(colpar_backward), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_caatpy", "Argument marshalling of the hot calls", -1, kMethods, nullptr, nullptr,
                       nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__caatpy(void) { return PyModule_Create(&kModule); }
