// Python fast path of the binding: argument checks and marshalling of the hot
// entry points in native code.
//
// Every function takes the arguments of the Python function of the same name,
// in order, and either makes the C call and returns its status, or returns
// None without having called anything: whenever an argument is not exactly the
// plain case (a CUDA torch.Tensor of the expected type, shape and device,
// contiguous; a Python int or float; a stream or None).  The Python function
// then goes through its own checks, which raise what is wrong or accept what
// this file does not know (page-locked host outputs, an omitted workspace,
// tensor subclasses).
//
// Measured on the GB300 host (Grace), host time of one call, Python checks against
// this file: decode_append 13.9 -> 2.9 us, append 10.2 -> 2.4, prefill 12.7 -> 3.0,
// backward 20.8 -> 5.0; what remains is the C call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <cstring>
#include <initializer_list>

#include "tk.h"

namespace {

// Entry points of libtk.so, set by bind() from the loaded library.
struct Api {
  decltype(&tk_kv_append) kv_append = nullptr;
  decltype(&tk_attn_decode) decode = nullptr;
  decltype(&tk_attn_decode_append) decode_append = nullptr;
  decltype(&tk_attn_decode_noalloc) decode_noalloc = nullptr;
  decltype(&tk_attn_prefill) prefill = nullptr;
  decltype(&tk_attn_forward) forward = nullptr;
  decltype(&tk_attn_backward) backward = nullptr;
  decltype(&tk_attn_prefill_cached) prefill_cached = nullptr;
} api;

PyObject *s_desc, *s_k, *s_v, *s_k_scale, *s_page_table, *s_cuda_stream;

// The tensor behind o, or nullptr unless o is a plain torch.Tensor (or Parameter).
const at::Tensor* tensor(PyObject* o) {
  return THPVariable_CheckExact(o) ? &THPVariable_Unpack(o) : nullptr;
}

// o as a contiguous CUDA tensor of this type on this device; nullptr if it is not.
const at::Tensor* need(PyObject* o, at::ScalarType type, c10::Device dev) {
  const at::Tensor* t = tensor(o);
  if (!t || !t->defined() || t->scalar_type() != type || t->device() != dev || !t->is_contiguous()) return nullptr;
  return t;
}

bool shape_is(const at::Tensor& t, std::initializer_list<int64_t> s) {
  return t.sizes() == at::IntArrayRef(s);
}

// out: float32 or bfloat16; its tk_dtype in *type
const at::Tensor* need_out(PyObject* o, c10::Device dev, int32_t* type) {
  const at::Tensor* t = tensor(o);
  if (!t || !t->defined()) return nullptr;
  const at::ScalarType s = t->scalar_type();
  if (s != at::kFloat && s != at::kBFloat16) return nullptr;
  *type = s == at::kFloat ? TK_F32 : TK_BF16;
  return need(o, s, dev);
}

bool to_i32(PyObject* o, int32_t* v) {
  if (!PyLong_CheckExact(o)) return false;
  int over = 0;
  const long x = PyLong_AsLongAndOverflow(o, &over);
  if (over || x < INT32_MIN || x > INT32_MAX) return false;
  *v = static_cast<int32_t>(x);
  return true;
}

bool to_scale(PyObject* o, int64_t r, float* v) {
  if (o == Py_None) {
    *v = static_cast<float>(1.0 / std::sqrt(static_cast<double>(r)));
    return r > 0;
  }
  if (!PyFloat_CheckExact(o)) return false;
  *v = static_cast<float>(PyFloat_AS_DOUBLE(o));
  return true;
}

bool to_bool(PyObject* o, int32_t* v) {
  if (o != Py_True && o != Py_False) return false;
  *v = o == Py_True;
  return true;
}

// The stream argument, or the current stream of the current device.
bool to_stream(PyObject* o, void** s) {
  if (o == Py_None) {
    *s = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  PyObject* a = PyObject_GetAttr(o, s_cuda_stream);
  if (!a) {
    PyErr_Clear();
    return false;
  }
  const bool ok = PyLong_CheckExact(a);
  if (ok) *s = PyLong_AsVoidPtr(a);
  Py_DECREF(a);
  if (PyErr_Occurred()) {
    PyErr_Clear();
    return false;
  }
  return ok;
}

// The fields of a ThinKeyCache; holds references to its attributes for the call.
struct Cache {
  tk_cache_desc desc;
  void *k = nullptr, *v = nullptr, *k_scale = nullptr, *page_table = nullptr;
  c10::Device dev{c10::DeviceType::CPU};
  PyObject* ref[4] = {nullptr, nullptr, nullptr, nullptr};
  ~Cache() {
    for (PyObject* r : ref) Py_XDECREF(r);
  }
  bool load(PyObject* o) {
    PyObject* d = PyObject_GetAttr(o, s_desc);
    if (!d) return fail();
    Py_buffer b;
    const bool got = PyObject_GetBuffer(d, &b, PyBUF_SIMPLE) == 0;
    Py_DECREF(d);
    if (!got) return fail();
    const bool fits = b.len == static_cast<Py_ssize_t>(sizeof(desc));
    if (fits) memcpy(&desc, b.buf, sizeof(desc));
    PyBuffer_Release(&b);
    if (!fits) return false;
    PyObject* names[4] = {s_k, s_v, s_k_scale, s_page_table};
    void** ptrs[4] = {&k, &v, &k_scale, &page_table};
    for (int i = 0; i < 4; ++i) {
      ref[i] = PyObject_GetAttr(o, names[i]);
      if (!ref[i]) return fail();
      if (ref[i] == Py_None) continue;
      const at::Tensor* t = tensor(ref[i]);
      if (!t || !t->defined()) return false;
      *ptrs[i] = t->data_ptr();
      if (i == 0) dev = t->device();
    }
    return k && dev.is_cuda();
  }
  bool fail() {
    PyErr_Clear();
    return false;
  }
};

// Holds the GIL released; takes it back however the scope is left.
struct NoGil {
  PyThreadState* state = PyEval_SaveThread();
  ~NoGil() { PyEval_RestoreThread(state); }
};

// Makes the C call without the GIL; its status as a Python int.
template <typename F>
PyObject* call(F&& f) {
  tk_status s;
  {
    NoGil scope;
    s = f();
  }
  return PyLong_FromLong(s);
}

// Runs body(args), which returns nullptr for "not the plain case"; a C++
// exception (a tensor without storage, say) means the same.
template <typename F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F&& body) {
  if (n == want) {
    try {
      PyObject* r = body();
      if (r) return r;
    } catch (...) {
    }
    PyErr_Clear();
  }
  Py_RETURN_NONE;
}

// cache, k_new, v_new, seq_lens, stream
PyObject* kv_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 5, [&]() -> PyObject* {
    Cache c;
    void* s;
    if (!c.load(a[0])) return nullptr;
    const tk_cache_desc& d = c.desc;
    const at::Tensor *kn = need(a[1], at::kBFloat16, c.dev), *vn = need(a[2], at::kBFloat16, c.dev),
                     *sl = need(a[3], at::kInt, c.dev);
    if (!kn || !vn || !sl || kn->dim() != 4 || !to_stream(a[4], &s)) return nullptr;
    const int64_t T = kn->size(2);
    if (T > INT32_MAX || !shape_is(*kn, {d.batch, d.h_kv, T, d.r}) || !shape_is(*vn, {d.batch, d.h_kv, T, d.d_v}))
      return nullptr;
    void *kp = kn->data_ptr(), *vp = vn->data_ptr(), *lp = sl->data_ptr();
    return call([&] {
      return api.kv_append(&d, c.k, c.v, static_cast<float*>(c.k_scale), static_cast<const int32_t*>(c.page_table),
                           static_cast<const int32_t*>(lp), kp, vp, static_cast<int32_t>(T), s);
    });
  });
}

// decode: cache, q, seq_lens, max_seq_len, out, workspace, scale, stream
// (noalloc: the same without the workspace)
template <bool kNoAlloc>
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  constexpr int W = kNoAlloc ? 0 : 1;
  return guarded(n, 7 + W, [&]() -> PyObject* {
    Cache c;
    void* s;
    int32_t bound, type;
    float scale;
    if (!c.load(a[0])) return nullptr;
    const tk_cache_desc& d = c.desc;
    const at::Tensor *q = need(a[1], at::kBFloat16, c.dev), *sl = need(a[2], at::kInt, c.dev),
                     *out = need_out(a[4], c.dev, &type), *ws = kNoAlloc ? nullptr : need(a[5], at::kByte, c.dev);
    if (!q || !sl || !out || (!kNoAlloc && !ws) || !to_i32(a[3], &bound) || !to_scale(a[5 + W], d.r, &scale) ||
        !to_stream(a[6 + W], &s) || !shape_is(*q, {d.batch, d.h_q, d.r}) || !shape_is(*out, {d.batch, d.h_q, d.d_v}))
      return nullptr;
    void *qp = q->data_ptr(), *lp = sl->data_ptr(), *op = out->data_ptr(), *wp = ws ? ws->data_ptr() : nullptr;
    const size_t wn = ws ? static_cast<size_t>(ws->numel()) : 0;
    return call([&] {
      const float* ks = static_cast<const float*>(c.k_scale);
      const int32_t *pt = static_cast<const int32_t*>(c.page_table), *l = static_cast<const int32_t*>(lp);
      return kNoAlloc ? api.decode_noalloc(&d, qp, c.k, c.v, ks, pt, l, bound, op, type, scale, s)
                      : api.decode(&d, qp, c.k, c.v, ks, pt, l, bound, op, type, scale, wp, wn, s);
    });
  });
}

// cache, q, k_new, v_new, seq_lens, max_seq_len, out, workspace, scale, stream
PyObject* decode_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 10, [&]() -> PyObject* {
    Cache c;
    void* s;
    int32_t bound, type;
    float scale;
    if (!c.load(a[0])) return nullptr;
    const tk_cache_desc& d = c.desc;
    const at::Tensor *q = need(a[1], at::kBFloat16, c.dev), *kn = need(a[2], at::kBFloat16, c.dev),
                     *vn = need(a[3], at::kBFloat16, c.dev), *sl = need(a[4], at::kInt, c.dev),
                     *out = need_out(a[6], c.dev, &type), *ws = need(a[7], at::kByte, c.dev);
    if (!q || !kn || !vn || !sl || !out || !ws || !to_i32(a[5], &bound) || !to_scale(a[8], d.r, &scale) ||
        !to_stream(a[9], &s) || !shape_is(*q, {d.batch, d.h_q, d.r}) || !shape_is(*out, {d.batch, d.h_q, d.d_v}) ||
        !shape_is(*kn, {d.batch, d.h_kv, d.r}) || !shape_is(*vn, {d.batch, d.h_kv, d.d_v}))
      return nullptr;
    void *qp = q->data_ptr(), *kp = kn->data_ptr(), *vp = vn->data_ptr(), *lp = sl->data_ptr(), *op = out->data_ptr(),
         *wp = ws->data_ptr();
    const size_t wn = static_cast<size_t>(ws->numel());
    return call([&] {
      return api.decode_append(&d, qp, c.k, c.v, static_cast<float*>(c.k_scale),
                               static_cast<const int32_t*>(c.page_table), static_cast<const int32_t*>(lp), kp, vp,
                               bound, op, type, scale, wp, wn, s);
    });
  });
}

// prefill: q, k, v, out, scale, causal, stream; forward: q, k, v, out, lse, scale, causal, stream
template <bool kLse>
PyObject* prefill(PyObject*, PyObject* const* a, Py_ssize_t n) {
  constexpr int W = kLse ? 1 : 0;
  return guarded(n, 7 + W, [&]() -> PyObject* {
    const at::Tensor* q = tensor(a[0]);
    if (!q || !q->defined() || !q->is_cuda() || q->dim() != 4) return nullptr;
    const c10::Device dev = q->device();
    void* s;
    int32_t type, causal;
    float scale;
    const at::Tensor *k = need(a[1], at::kBFloat16, dev), *v = need(a[2], at::kBFloat16, dev),
                     *out = need_out(a[3], dev, &type), *lse = kLse ? need(a[4], at::kFloat, dev) : nullptr;
    if (!need(a[0], at::kBFloat16, dev) || !k || !v || !out || (kLse && !lse) || k->dim() != 4 || v->dim() != 4)
      return nullptr;
    const int64_t B = q->size(0), hq = q->size(1), S = q->size(2), r = q->size(3), hkv = k->size(1), dv = v->size(3);
    if (B > INT32_MAX || hq > INT32_MAX || S > INT32_MAX || r > INT32_MAX || hkv > INT32_MAX || dv > INT32_MAX ||
        !shape_is(*k, {B, hkv, S, r}) || !shape_is(*v, {B, hkv, S, dv}) || !shape_is(*out, {B, hq, S, dv}) ||
        (kLse && !shape_is(*lse, {B, hq, S})) || !to_scale(a[4 + W], r, &scale) || !to_bool(a[5 + W], &causal) ||
        !to_stream(a[6 + W], &s))
      return nullptr;
    void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr(), *op = out->data_ptr(),
         *lp = lse ? lse->data_ptr() : nullptr;
    const int32_t b = B, x = hq, y = hkv, t = S, w = r, z = dv;
    return call([&] {
      return kLse ? api.forward(qp, kp, vp, op, static_cast<float*>(lp), type, b, x, y, t, w, z, scale, causal, s)
                  : api.prefill(qp, kp, vp, op, type, b, x, y, t, w, z, scale, causal, s);
    });
  });
}

// q, k, v, out, d_out, lse, dq, dk, dv, workspace, scale, causal, stream
PyObject* backward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 13, [&]() -> PyObject* {
    const at::Tensor* q = tensor(a[0]);
    if (!q || !q->defined() || !q->is_cuda() || q->dim() != 4) return nullptr;
    const c10::Device dev = q->device();
    const at::Tensor* t[10];
    for (int i = 0; i < 10; ++i) {
      t[i] = need(a[i], i < 5 ? at::kBFloat16 : (i < 9 ? at::kFloat : at::kByte), dev);
      if (!t[i]) return nullptr;
    }
    if (t[1]->dim() != 4 || t[2]->dim() != 4) return nullptr;
    const int64_t B = q->size(0), hq = q->size(1), S = q->size(2), r = q->size(3), hkv = t[1]->size(1),
                  dv = t[2]->size(3);
    void* s;
    int32_t causal;
    float scale;
    if (B > INT32_MAX || hq > INT32_MAX || S > INT32_MAX || r > INT32_MAX || hkv > INT32_MAX || dv > INT32_MAX ||
        !shape_is(*t[1], {B, hkv, S, r}) || !shape_is(*t[2], {B, hkv, S, dv}) || !shape_is(*t[3], {B, hq, S, dv}) ||
        !shape_is(*t[4], {B, hq, S, dv}) || !shape_is(*t[5], {B, hq, S}) || !shape_is(*t[6], {B, hq, S, r}) ||
        !shape_is(*t[7], {B, hkv, S, r}) || !shape_is(*t[8], {B, hkv, S, dv}) || !to_scale(a[10], r, &scale) ||
        !to_bool(a[11], &causal) || !to_stream(a[12], &s))
      return nullptr;
    void* p[10];
    for (int i = 0; i < 10; ++i) p[i] = t[i]->data_ptr();
    const size_t wn = static_cast<size_t>(t[9]->numel());
    return call([&] {
      return api.backward(p[0], p[1], p[2], p[3], p[4], static_cast<const float*>(p[5]), static_cast<float*>(p[6]),
                          static_cast<float*>(p[7]), static_cast<float*>(p[8]), p[9], wn, static_cast<int32_t>(B),
                          static_cast<int32_t>(hq), static_cast<int32_t>(hkv), static_cast<int32_t>(S),
                          static_cast<int32_t>(r), static_cast<int32_t>(dv), scale, causal, s);
    });
  });
}

// cache, q, k_new, v_new, seq_lens, max_seq_len, out, scale, causal, workspace, stream
PyObject* prefill_cached(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 11, [&]() -> PyObject* {
    Cache c;
    void* s;
    int32_t bound, type, causal;
    float scale;
    if (!c.load(a[0])) return nullptr;
    const tk_cache_desc& d = c.desc;
    const at::Tensor *q = need(a[1], at::kBFloat16, c.dev), *kn = need(a[2], at::kBFloat16, c.dev),
                     *vn = need(a[3], at::kBFloat16, c.dev), *sl = need(a[4], at::kInt, c.dev),
                     *out = need_out(a[6], c.dev, &type);
    const at::Tensor* ws = a[9] == Py_None ? nullptr : need(a[9], at::kByte, c.dev);
    if (!q || !kn || !vn || !sl || !out || q->dim() != 4 || (!ws && (a[9] != Py_None || d.k_dtype != TK_BF16)))
      return nullptr;
    const int64_t S = q->size(2);
    if (S > INT32_MAX || !shape_is(*q, {d.batch, d.h_q, S, d.r}) || !shape_is(*out, {d.batch, d.h_q, S, d.d_v}) ||
        !shape_is(*kn, {d.batch, d.h_kv, S, d.r}) || !shape_is(*vn, {d.batch, d.h_kv, S, d.d_v}) ||
        !to_i32(a[5], &bound) || !to_scale(a[7], d.r, &scale) || !to_bool(a[8], &causal) || !to_stream(a[10], &s))
      return nullptr;
    void *qp = q->data_ptr(), *kp = kn->data_ptr(), *vp = vn->data_ptr(), *lp = sl->data_ptr(), *op = out->data_ptr(),
         *wp = ws ? ws->data_ptr() : nullptr;
    const size_t wn = ws ? static_cast<size_t>(ws->numel()) : 0;
    return call([&] {
      return api.prefill_cached(&d, qp, c.k, c.v, static_cast<float*>(c.k_scale),
                                static_cast<const int32_t*>(c.page_table), static_cast<const int32_t*>(lp), kp, vp,
                                static_cast<int32_t>(S), bound, op, type, scale, causal, wp, wn, s);
    });
  });
}

// Addresses of the library's entry points, in the order of Api.
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void** slots = reinterpret_cast<void**>(&api);
  if (n != static_cast<Py_ssize_t>(sizeof(Api) / sizeof(void*))) {
    PyErr_SetString(PyExc_TypeError, "bind: one address per entry point");
    return nullptr;
  }
  for (Py_ssize_t i = 0; i < n; ++i) {
    void* p = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred()) return nullptr;
    slots[i] = p;
  }
  Py_RETURN_NONE;
}

#define TK_DEF(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(fn)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    TK_DEF("bind", &bind),
    TK_DEF("kv_append", &kv_append),
    TK_DEF("decode", &decode<false>),
    TK_DEF("decode_noalloc", &decode<true>),
    TK_DEF("decode_append", &decode_append),
    TK_DEF("prefill", &prefill<false>),
    TK_DEF("forward", &prefill<true>),
    TK_DEF("backward", &backward),
    TK_DEF("prefill_cached", &prefill_cached),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tkpy", "Native argument checks of the binding's hot calls.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tkpy(void) {
  s_desc = PyUnicode_InternFromString("desc");
  s_k = PyUnicode_InternFromString("k");
  s_v = PyUnicode_InternFromString("v");
  s_k_scale = PyUnicode_InternFromString("k_scale");
  s_page_table = PyUnicode_InternFromString("page_table");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_desc || !s_k || !s_v || !s_k_scale || !s_page_table || !s_cuda_stream) return nullptr;
  return PyModule_Create(&module);
}
