// Native argument marshalling of the four hot-path calls for the Python
// binding: unpack the tensors, make the checks the binding makes, call the
// library.  The same checks in Python and a ctypes call cost 7-8 us a call,
// which for few rows is longer than the kernels: a step of one row x 2048
// kept ids (two calls, 13.7 us of device time) took 25.7 us from Python and
// takes 14.9 us from here; the host's part of any step is 15-20 us shorter.
//
// Every function returns the payload bytes (0 where there is none) when the
// call was made and succeeded, -1 - status when the library refused it, and
// kNotTaken when anything about the arguments is not plain: the binding then
// takes its Python path, which has the last word on what is accepted and
// raises its own errors.  Nothing is remembered between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>

#include <ATen/core/Tensor.h>
#include <torch/csrc/autograd/python_variable.h>

#include "sph.h"

namespace {

constexpr long long kNotTaken = -1000;

decltype(&sph_partial_logits) p_partial = nullptr;
decltype(&sph_fuse_sample) p_fuse = nullptr;
decltype(&sph_split_step) p_split = nullptr;
decltype(&sph_verify_draft) p_verify = nullptr;

// One call's arguments; ok turns false at the first that is not plain.
struct Args {
  PyObject* const* a;
  bool ok = true;
  int dev = -1;              // device of the call's tensors

  const at::Tensor* tensor(int i) {
    PyObject* o = a[i];
    if (!ok || !THPVariable_CheckExact(o)) { ok = false; return nullptr; }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || t.layout() != c10::kStrided || !t.is_cuda()) { ok = false; return nullptr; }
    const int d = (int)t.get_device();
    if (dev < 0) dev = d;
    else if (d != dev) { ok = false; return nullptr; }
    return &t;
  }
  // a 2-D operand with unit inner stride, and its address and row stride
  struct Matrix {
    const at::Tensor* t = nullptr;
    const void* p = nullptr;
    long long ld = 0;
    const at::Tensor* operator->() const { return t; }
  };
  Matrix matrix(int i) {
    const at::Tensor* t = tensor(i);
    if (!t || t->dim() != 2 || t->stride(1) != 1) { ok = false; return {}; }
    return {t, t->const_data_ptr(), (long long)t->stride(0)};
  }
  // a dense buffer of `type` with at least `count` elements (None: nullptr)
  template <class T>
  T* dense(int i, c10::ScalarType type, long long count) {
    if (!ok || a[i] == Py_None) return nullptr;
    const at::Tensor* t = tensor(i);
    if (!t || t->scalar_type() != type || !t->is_contiguous() || t->numel() < count) {
      ok = false;
      return nullptr;
    }
    return static_cast<T*>(t->data_ptr());
  }
  bool none(int i) const { return a[i] == Py_None; }
  long long integer(int i) {
    const long long v = PyLong_CheckExact(a[i]) ? PyLong_AsLongLong(a[i]) : (ok = false, 0);
    if (v == -1 && PyErr_Occurred()) { PyErr_Clear(); ok = false; }
    return v;
  }
  unsigned long long word(int i) {      // modulo 2^64, as the binding masks
    if (!PyLong_CheckExact(a[i])) { ok = false; return 0; }
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(a[i]);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) { PyErr_Clear(); ok = false; }
    return v;
  }
  float real(int i) {
    if (PyFloat_CheckExact(a[i])) return (float)PyFloat_AS_DOUBLE(a[i]);
    if (PyLong_CheckExact(a[i])) {
      const double v = PyLong_AsDouble(a[i]);
      if (!(v == -1.0 && PyErr_Occurred())) return (float)v;
      PyErr_Clear();
    }
    ok = false;
    return 0.f;
  }
  // bf16 or e4m3 weights
  sph_dtype weights(const Matrix& w) {
    if (!w.t) { ok = false; return SPH_DTYPE_BF16; }
    if (w->scalar_type() == c10::kBFloat16) return SPH_DTYPE_BF16;
    if (w->scalar_type() == c10::kFloat8_e4m3fn) return SPH_DTYPE_FP8_E4M3;
    ok = false;
    return SPH_DTYPE_BF16;
  }
};

PyObject* not_taken() { return PyLong_FromLongLong(kNotTaken); }
PyObject* outcome(sph_status st, size_t bytes) {
  return PyLong_FromLongLong(st == SPH_OK ? (long long)bytes : -1 - (long long)st);
}

// The interpreter lock released for the library call (as ctypes makes it),
// and held again however that ends.  Everything a tensor is asked for, which
// may throw, is asked before.
struct Unlocked {
  PyThreadState* saved = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(saved); }
};
template <class F>
sph_status unlocked(F&& f) {
  Unlocked u;
  return f();
}

// No C++ exception crosses into the interpreter: whatever a tensor refuses
// to say (one without storage has no address) is left to the Python path.
template <class F>
PyObject* guarded(F&& f) {
  try {
    return f();
  } catch (...) {
    PyErr_Clear();
    return not_taken();
  }
}

// (ctx, h_cloud, W_h, keep_ids, clip, w_row_scale, bias, act_mode, codes,
//  row_scale, partial_out)
PyObject* partial_logits(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 11) return not_taken();
    Args A{argv};
    auto* ctx = reinterpret_cast<sph_ctx*>((uintptr_t)A.word(0));
    const Args::Matrix h = A.matrix(1);
    const Args::Matrix W = A.matrix(2);
    if (!A.ok || h->scalar_type() != c10::kFloat) return not_taken();
    const sph_dtype wdt = A.weights(W);
    const long long R = h->size(0), dh = h->size(1), V = W->size(0);
    const int32_t* keep = A.dense<int32_t>(3, c10::kInt, 0);
    const long long nk = keep || !A.none(3)
                             ? (A.ok ? (long long)THPVariable_Unpack(argv[3]).numel() : 0) : V;
    const float clip = A.real(4);
    const float* ws = A.dense<float>(5, c10::kFloat, V);
    const float* bias = A.dense<float>(6, c10::kFloat, V);
    const long long act = A.integer(7);
    int8_t* codes = A.dense<int8_t>(8, c10::kChar, R * nk);
    float* scale = A.dense<float>(9, c10::kFloat, R);
    float* part = A.dense<float>(10, c10::kFloat, R * nk);
    if (!A.ok || !ctx) return not_taken();
    size_t pb = 0;
    const sph_status st = unlocked([&] {
      return p_partial(ctx, static_cast<const float*>(h.p), R, h.ld, W.p, wdt, V, dh, W.ld, ws,
                       bias, keep, nk, clip, (sph_act_mode)act, codes, scale, part, &pb);
    });
    return outcome(st, pb);
  });
}

// (ctx, codes, row_scale, h_local, W_l, keep_ids, temperature, seed, offset,
//  tokens, fused_logits_out)
PyObject* fuse_sample(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 11) return not_taken();
    Args A{argv};
    auto* ctx = reinterpret_cast<sph_ctx*>((uintptr_t)A.word(0));
    const Args::Matrix h = A.matrix(3);
    const Args::Matrix W = A.matrix(4);
    if (!A.ok || h->scalar_type() != c10::kFloat || W->scalar_type() != c10::kBFloat16)
      return not_taken();
    const long long R = h->size(0), dl = h->size(1), V = W->size(0);
    const int32_t* keep = A.dense<int32_t>(5, c10::kInt, 0);
    const long long nk = keep || !A.none(5)
                             ? (A.ok ? (long long)THPVariable_Unpack(argv[5]).numel() : 0) : V;
    const int8_t* codes = A.dense<int8_t>(1, c10::kChar, R * nk);
    const float* scale = A.dense<float>(2, c10::kFloat, R);
    const float tau = A.real(6);
    const unsigned long long seed = A.word(7), offset = A.word(8);
    int32_t* tokens = A.dense<int32_t>(9, c10::kInt, R);
    float* z = A.dense<float>(10, c10::kFloat, R * nk);
    if (!A.ok || !ctx) return not_taken();
    return outcome(unlocked([&] {
      return p_fuse(ctx, codes, scale, R, static_cast<const float*>(h.p), h.ld, W.p, V, dl, W.ld,
                    keep, nk, tau, seed, offset, tokens, z);
    }), 0);
  });
}

// (ctx, h, d_l, W_h, W_l, keep_ids, clip, w_row_scale, bias, act_mode,
//  temperature, seed, offset, chunk, endpoint_stream, codes, scales, tokens)
PyObject* split_step(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 18) return not_taken();
    Args A{argv};
    auto* ctx = reinterpret_cast<sph_ctx*>((uintptr_t)A.word(0));
    const Args::Matrix h = A.matrix(1);
    const long long dl = A.integer(2);
    const Args::Matrix Wh = A.matrix(3);
    const Args::Matrix Wl = A.matrix(4);
    if (!A.ok || h->scalar_type() != c10::kFloat || Wl->scalar_type() != c10::kBFloat16)
      return not_taken();
    const sph_dtype wdt = A.weights(Wh);
    const long long R = h->size(0), V = Wh->size(0), dh = Wh->size(1);
    const int32_t* keep = A.dense<int32_t>(5, c10::kInt, 0);
    const long long nk = keep || !A.none(5)
                             ? (A.ok ? (long long)THPVariable_Unpack(argv[5]).numel() : 0) : V;
    const float clip = A.real(6);
    const float* ws = A.dense<float>(7, c10::kFloat, V);
    const float* bias = A.dense<float>(8, c10::kFloat, V);
    const long long act = A.integer(9);
    const float tau = A.real(10);
    const unsigned long long seed = A.word(11), offset = A.word(12);
    const long long chunk = A.integer(13);
    void* es = reinterpret_cast<void*>((uintptr_t)A.word(14));
    if (!A.ok || chunk < 0 || nk < 1) return not_taken();
    const long long L = (chunk == 0 || chunk >= nk) ? nk : chunk;
    int8_t* codes = A.dense<int8_t>(15, c10::kChar, R * nk);
    float* scales = A.dense<float>(16, c10::kFloat, (nk + L - 1) / L * R);
    int32_t* tokens = A.dense<int32_t>(17, c10::kInt, R);
    if (!A.ok || !ctx) return not_taken();
    size_t pb = 0;
    const sph_status st = unlocked([&] {
      return p_split(ctx, static_cast<const float*>(h.p), R, h.ld, dl, dh, Wh.p, wdt, ws, Wh.ld,
                     Wl.p, Wl.ld, V, bias, keep, nk, clip, (sph_act_mode)act, tau, seed, offset,
                     chunk, es, codes, scales, tokens, nullptr, &pb);
    });
    return outcome(st, pb);
  });
}

// (ctx, target_logits, sessions, k, draft_tokens, keep_ids, draft_probs,
//  temperature, seed, offset, n_accepted, next_token)
PyObject* verify_draft(PyObject*, PyObject* const* argv, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 12) return not_taken();
    Args A{argv};
    auto* ctx = reinterpret_cast<sph_ctx*>((uintptr_t)A.word(0));
    const long long S = A.integer(2), k = A.integer(3);
    if (!A.ok || S < 1 || k < 1 || S > (1 << 20) || k > 1024) return not_taken();
    const at::Tensor* t = A.tensor(1);
    if (!t || t->dim() < 1) return not_taken();
    const long long nk = t->size(-1);
    const float* z = A.dense<float>(1, c10::kFloat, S * (k + 1) * nk);
    const int32_t* draft = A.dense<int32_t>(4, c10::kInt, S * k);
    const int32_t* keep = A.dense<int32_t>(5, c10::kInt, nk);
    const float* probs = A.dense<float>(6, c10::kFloat, S * k * nk);
    const float tau = A.real(7);
    const unsigned long long seed = A.word(8), offset = A.word(9);
    int32_t* acc = A.dense<int32_t>(10, c10::kInt, S);
    int32_t* next = A.dense<int32_t>(11, c10::kInt, S);
    if (!A.ok || !ctx) return not_taken();
    return outcome(unlocked([&] {
      return p_verify(ctx, z, S, k, keep, nk, tau, draft, probs, seed, offset, acc, next);
    }), 0);
  });
}

// Find the library's calls in the libsph.so that the binding has loaded.
PyObject* bind(PyObject*, PyObject* path) {
  const char* p = PyUnicode_AsUTF8(path);
  if (!p) return nullptr;
  void* lib = dlopen(p, RTLD_NOW | RTLD_LOCAL);
  auto find = [&](const char* name) { return lib ? dlsym(lib, name) : nullptr; };
  void* const f[4] = {find("sph_partial_logits"), find("sph_fuse_sample"), find("sph_split_step"),
                      find("sph_verify_draft")};
  if (!f[0] || !f[1] || !f[2] || !f[3]) {
    PyErr_Format(PyExc_RuntimeError, "the hot-path calls were not found in %s", p);
    return nullptr;
  }
  p_partial = reinterpret_cast<decltype(p_partial)>(f[0]);
  p_fuse = reinterpret_cast<decltype(p_fuse)>(f[1]);
  p_split = reinterpret_cast<decltype(p_split)>(f[2]);
  p_verify = reinterpret_cast<decltype(p_verify)>(f[3]);
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    {"partial_logits", (PyCFunction)(void (*)(void))partial_logits, METH_FASTCALL, nullptr},
    {"fuse_sample", (PyCFunction)(void (*)(void))fuse_sample, METH_FASTCALL, nullptr},
    {"split_step", (PyCFunction)(void (*)(void))split_step, METH_FASTCALL, nullptr},
    {"verify_draft", (PyCFunction)(void (*)(void))verify_draft, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "py_fast", nullptr, -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_py_fast() { return PyModule_Create(&module); }
