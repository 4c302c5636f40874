// The calls of binding.py without ctypes and without Python's attribute lookups: what a call costs on the host beside its launches is
// 1 to 2 us here and 5 to 8 us there, of shapes that the device is done with in 5 to 15.
//
// A function checks its arguments as binding.py does and makes the call.  It returns the output tensor, or the library's
// status when that is not zero, or None where something is not as the fast path expects (also every error that binding.py
// raises): binding.py then goes the ordinary way, which says what is wrong.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <dlfcn.h>

#include <string>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "gformer.h"

namespace {

struct NotFast {};

// The library beside this module (the one that binding.py has loaded), by path, because several copies of the package
// may be loaded in one process.
struct Api {
  decltype(&gformer_default_h_sparse) default_h_sparse;
  decltype(&gformer_hybrid_attn_w) hybrid_attn;
  decltype(&gformer_hybrid_attn_self_w) hybrid_attn_self;
  decltype(&gformer_window_attn) window_attn, window_attn_self;
  decltype(&gformer_causal_linear_attn_w) causal_linear_attn;
  decltype(&gformer_decode_step_w) decode_step;
  decltype(&gformer_decode_step_ragged_w) decode_step_ragged;
};
Api api;

bool load_api() {
  Dl_info self;
  if (dladdr((const void*)&load_api, &self) == 0 || self.dli_fname == nullptr) return false;
  std::string path(self.dli_fname);
  const size_t slash = path.rfind('/');
  path = (slash == std::string::npos ? std::string() : path.substr(0, slash + 1)) + "libgformer.so";
  void* lib = dlopen(path.c_str(), RTLD_NOW | RTLD_LOCAL);
  if (lib == nullptr) return false;
  auto get = [&](auto& f, const char* name) {
    f = reinterpret_cast<std::remove_reference_t<decltype(f)>>(dlsym(lib, name));
    return f != nullptr;
  };
  return get(api.default_h_sparse, "gformer_default_h_sparse") && get(api.hybrid_attn, "gformer_hybrid_attn_w") &&
         get(api.hybrid_attn_self, "gformer_hybrid_attn_self_w") && get(api.window_attn, "gformer_window_attn") &&
         get(api.window_attn_self, "gformer_window_attn_self") &&
         get(api.causal_linear_attn, "gformer_causal_linear_attn_w") && get(api.decode_step, "gformer_decode_step_w") &&
         get(api.decode_step_ragged, "gformer_decode_step_ragged_w");
}

// A library call with the interpreter's lock released, as ctypes makes it.
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_CheckExact(o)) throw NotFast();
  return THPVariable_Unpack(o);
}
const at::Tensor& cuda_tensor(PyObject* o, int64_t dims) {
  const at::Tensor& t = tensor(o);
  if (!t.is_cuda() || t.dim() != dims || !t.is_contiguous()) throw NotFast();
  return t;
}
long long integer(PyObject* o) {
  if (!PyLong_CheckExact(o)) throw NotFast();
  const long long x = PyLong_AsLongLong(o);
  if (x == -1 && PyErr_Occurred()) throw NotFast();
  return x;
}
int integer32(PyObject* o) {
  const long long x = integer(o);
  if (x != (int)x) throw NotFast();
  return (int)x;
}
float real(PyObject* o) {
  if (PyFloat_CheckExact(o)) return (float)PyFloat_AS_DOUBLE(o);
  return (float)integer(o);
}
void* address(PyObject* o) {  // an int, or None
  if (o == Py_None) return nullptr;
  if (!PyLong_CheckExact(o)) throw NotFast();
  void* p = PyLong_AsVoidPtr(o);
  if (p == nullptr && PyErr_Occurred()) throw NotFast();
  return p;
}
void* stream_of(PyObject* o) {  // binding.py's stream: the handle, or None for the current one
  return o == Py_None ? (void*)c10::cuda::getCurrentCUDAStream().stream() : address(o);
}
int dtype_of(const at::Tensor& t) {
  if (t.scalar_type() == at::kFloat) return GF_F32;
  if (t.scalar_type() == at::kBFloat16) return GF_BF16;
  throw NotFast();
}
const void* projection(PyObject* W, const at::Tensor& q, int64_t heads, int64_t d) {
  if (W == Py_None) return nullptr;
  const at::Tensor& w = cuda_tensor(W, 3);
  if (w.scalar_type() != q.scalar_type() || w.size(0) != heads || w.size(1) != d || w.size(2) != d) throw NotFast();
  return w.data_ptr();
}
float* state_part(PyObject* o, at::IntArrayRef shape) {
  if (o == Py_None) return nullptr;
  const at::Tensor& t = tensor(o);
  if (t.scalar_type() != at::kFloat || !t.is_contiguous() || t.sizes() != shape) throw NotFast();
  return (float*)t.data_ptr();
}

// q, k, v and the output of a call
struct Qkvo {
  const at::Tensor &q, &k, &v;
  at::Tensor o;
  int dtype;
  Qkvo(PyObject* const* a, PyObject* out, int64_t dims)
      : q(cuda_tensor(a[0], dims)), k(cuda_tensor(a[1], dims)), v(cuda_tensor(a[2], dims)), dtype(dtype_of(q)) {
    if (k.sizes() != q.sizes() || v.sizes() != q.sizes() || k.scalar_type() != q.scalar_type() ||
        v.scalar_type() != q.scalar_type())
      throw NotFast();
    o = out == Py_None ? at::empty_like(q) : tensor(out);
  }
};
struct Shape {
  int B, H, N, d;
  Shape(const at::Tensor& q, int layout) {
    const bool bnhd = layout == GF_BNHD;
    for (int64_t i = 0; i < 4; ++i)
      if (q.size(i) != (int)q.size(i)) throw NotFast();
    B = (int)q.size(0);
    H = (int)q.size(bnhd ? 2 : 1);
    N = (int)q.size(bnhd ? 1 : 2);
    d = (int)q.size(3);
  }
};

template <typename F>
PyObject* call(Py_ssize_t have, Py_ssize_t want, PyObject* out, F f) {
  if (have != want) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  try {
    at::Tensor o;
    const int rc = f(o);
    if (rc != GF_OK) return PyLong_FromLong(rc);
    if (out != Py_None) return Py_NewRef(out);
    return THPVariable_Wrap(std::move(o));
  } catch (const NotFast&) {
  } catch (const std::exception&) {
  }
  PyErr_Clear();
  Py_RETURN_NONE;
}

// q k v out W w h_sparse scale chunk layout state ws ws_bytes stream
PyObject* hybrid_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 14, n > 3 ? a[3] : nullptr, [&](at::Tensor& o) {
    Qkvo t(a, a[3], 4);
    const int layout = integer32(a[9]), h_sparse = integer32(a[6]);
    const Shape s(t.q, layout);
    const int h0 = h_sparse < 0 ? api.default_h_sparse(s.H) : h_sparse;
    const void* W = projection(a[4], t.q, s.H - h0, s.d);
    const int w = integer32(a[5]), chunk = integer32(a[8]);
    const float scale = real(a[7]);
    gf_decode_state* st = (gf_decode_state*)address(a[10]);
    void *ws = address(a[11]), *stream = stream_of(a[13]);
    const size_t ws_bytes = (size_t)integer(a[12]);
    o = t.o;
    Unlocked unlocked;
    return api.hybrid_attn(t.q.data_ptr(), t.k.data_ptr(), t.v.data_ptr(), t.o.data_ptr(), s.B, s.H, s.N, s.d, w, h_sparse, scale,
                           W ? GF_PHI_FAVOR_POS : GF_PHI_ELU1, W, chunk, t.dtype, layout, st, ws, ws_bytes, stream);
  });
}
// q k v out W w h_sparse scale layout ws ws_bytes stream
PyObject* hybrid_attn_self(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 12, n > 3 ? a[3] : nullptr, [&](at::Tensor& o) {
    Qkvo t(a, a[3], 4);
    const int layout = integer32(a[8]), h_sparse = integer32(a[6]);
    const Shape s(t.q, layout);
    const int h0 = h_sparse < 0 ? api.default_h_sparse(s.H) : h_sparse;
    const void* W = projection(a[4], t.q, s.H - h0, s.d);
    const int w = integer32(a[5]);
    const float scale = real(a[7]);
    void *ws = address(a[9]), *stream = stream_of(a[11]);
    const size_t ws_bytes = (size_t)integer(a[10]);
    o = t.o;
    Unlocked unlocked;
    return api.hybrid_attn_self(t.q.data_ptr(), t.k.data_ptr(), t.v.data_ptr(), t.o.data_ptr(), s.B, s.H, s.N, s.d, w, h_sparse,
                                scale, W ? GF_PHI_FAVOR_POS : GF_PHI_ELU1, W, t.dtype, layout, ws, ws_bytes, stream);
  });
}
// q k v out w scale layout two_sided ws ws_bytes stream
PyObject* window_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 11, n > 3 ? a[3] : nullptr, [&](at::Tensor& o) {
    Qkvo t(a, a[3], 4);
    const int layout = integer32(a[6]);
    const Shape s(t.q, layout);
    const int w = integer32(a[4]);
    const float scale = real(a[5]);
    void *ws = address(a[8]), *stream = stream_of(a[10]);
    const size_t ws_bytes = (size_t)integer(a[9]);
    o = t.o;
    Unlocked unlocked;
    return (a[7] == Py_True ? api.window_attn_self : api.window_attn)(t.q.data_ptr(), t.k.data_ptr(), t.v.data_ptr(),
                                                                      t.o.data_ptr(), s.B, s.H, s.N, s.d, w, scale, t.dtype,
                                                                      layout, ws, ws_bytes, stream);
  });
}
// q k v out W S z chunk layout ws ws_bytes stream
PyObject* causal_linear_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 12, n > 3 ? a[3] : nullptr, [&](at::Tensor& o) {
    Qkvo t(a, a[3], 4);
    const int layout = integer32(a[8]);
    const Shape s(t.q, layout);
    if ((a[5] == Py_None) != (a[6] == Py_None)) throw NotFast();
    float* S = state_part(a[5], {s.B, s.H, s.d, s.d});
    float* z = state_part(a[6], {s.B, s.H, s.d});
    const void* W = projection(a[4], t.q, s.H, s.d);
    const int chunk = integer32(a[7]);
    void *ws = address(a[9]), *stream = stream_of(a[11]);
    const size_t ws_bytes = (size_t)integer(a[10]);
    o = t.o;
    Unlocked unlocked;
    return api.causal_linear_attn(t.q.data_ptr(), t.k.data_ptr(), t.v.data_ptr(), t.o.data_ptr(), s.B, s.H, s.N, s.d,
                                  W ? GF_PHI_FAVOR_POS : GF_PHI_ELU1, W, chunk, S, z, t.dtype, layout, ws, ws_bytes, stream);
  });
}
// q k v out W state scale t_seq (or None) stream.  As in binding.py, the state says what the tensors hold.
PyObject* decode_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 9, n > 3 ? a[3] : nullptr, [&](at::Tensor& o) {
    const at::Tensor &q = cuda_tensor(a[0], 3), &k = cuda_tensor(a[1], 3), &v = cuda_tensor(a[2], 3);
    gf_decode_state* st = (gf_decode_state*)address(a[5]);
    if (st == nullptr) throw NotFast();
    o = a[3] == Py_None ? at::empty_like(q) : tensor(a[3]);
    const void* W = projection(a[4], q, st->H - st->h_sparse, st->d);
    const int phi = W ? GF_PHI_FAVOR_POS : GF_PHI_ELU1;
    const float scale = real(a[6]);
    void* stream = stream_of(a[8]);
    long long* t_seq = nullptr;
    if (a[7] != Py_None) {
      const at::Tensor& t = tensor(a[7]);
      if (!t.is_cuda() || t.scalar_type() != at::kLong || !t.is_contiguous() || t.numel() != q.size(0)) throw NotFast();
      t_seq = (long long*)t.data_ptr();
    }
    Unlocked unlocked;
    if (a[7] == Py_None)
      return api.decode_step(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), st, scale, phi, W, stream);
    return api.decode_step_ragged(q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), st, t_seq, scale, phi, W, stream);
  });
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(hybrid_attn), FAST(hybrid_attn_self), FAST(window_attn), FAST(causal_linear_attn),
                         FAST(decode_step), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall(void) {
  if (!load_api()) {
    PyErr_SetString(PyExc_ImportError, "libgformer.so beside _fastcall.so cannot be loaded, or is older than it");
    return nullptr;
  }
  PyObject* m = PyModule_Create(&module);
  if (m != nullptr && PyModule_AddStringConstant(m, "built_for", GF_BUILT_FOR) != 0) Py_CLEAR(m);
  return m;
}
