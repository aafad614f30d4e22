// The short way from PyTorch tensors to the C ABI (include/mw_bca.h): checks
// of arguments that need nothing special, output allocation and the call, in
// one native function each.
//
// A call's kernels take from 5 us; the same checks and allocations written in
// Python take 10-40 us of host time a call on the Grace cores (more on the
// autograd thread, whose caches are cold), which is what bounds small windows
// and short streams.  Anything unusual -- another type or layout, buffers the
// caller supplies, a wrapped or fake tensor, sizes that do not fit -- makes a
// function here return None, and the Python binding's full checks then run
// and name what is wrong.  An int is a non-zero mw_status.
//
// The C entry points are handed over as addresses (bind), so that this module
// and the ctypes binding share one loaded library and its options.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <array>
#include <climits>
#include <cmath>
#include <initializer_list>

#include "mw_bca.h"

namespace {

decltype(&mw_bca_fwd) p_fwd = nullptr;
decltype(&mw_bca_bwd) p_bwd = nullptr;
decltype(&mw_bca_bwd_workspace_size) p_bwd_ws = nullptr;
decltype(&mw_bca_cache_workspace_size) p_cache_ws = nullptr;
decltype(&mw_bca_cache_fwd_rope) p_cache = nullptr;
decltype(&mw_bca_cache_step) p_step = nullptr;
decltype(&mw_qkv_rope_split) p_qkv = nullptr;

// A tensor this module may look into: exactly a torch.Tensor or Parameter,
// strided, with storage of its own (no fake, batched or other wrapper).
bool is_real(const at::Tensor& t) {
  return t.unsafeGetTensorImpl()->has_storage() && t.layout() == at::kStrided && t.is_cuda() &&
         !t.unsafeGetTensorImpl()->key_set().has(c10::DispatchKey::Python) && !t.is_neg();
}

// (with a torch function or dispatch mode on, which wants to see every
// allocation, nothing here is taken)
const at::Tensor* tensor(PyObject* o) {
  if (!THPVariable_CheckExact(o) || at::impl::torch_function_mode_enabled() ||
      c10::impl::TorchDispatchModeTLS::any_modes_set())
    return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.defined() && is_real(t) && t.is_contiguous() ? &t : nullptr;
}

// The i-th argument as a bf16 tensor of `dims` dimensions, else null.
const at::Tensor* bf16(PyObject* o, int dims) {
  const at::Tensor* t = tensor(o);
  return t && t->scalar_type() == at::kBFloat16 && t->dim() == dims ? t : nullptr;
}

// The device of all tensors (null pointers skipped), if it is one and current.
bool one_device(std::initializer_list<const at::Tensor*> ts, c10::DeviceIndex* dev) {
  *dev = -1;
  for (const at::Tensor* t : ts) {
    if (!t) continue;
    if (*dev < 0)
      *dev = t->get_device();
    else if (t->get_device() != *dev)
      return false;
  }
  return *dev >= 0 && *dev == c10::cuda::current_device();
}

bool small_int(PyObject* o, int* out) {
  if (!PyLong_CheckExact(o)) return false;
  int over = 0;
  const long v = PyLong_AsLongAndOverflow(o, &over);
  if (over || v < INT_MIN || v > INT_MAX) return false;
  *out = static_cast<int>(v);
  return true;
}

bool real_number(PyObject* o, float* out) {
  if (!PyFloat_CheckExact(o) && !PyLong_CheckExact(o)) return false;
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) {
    PyErr_Clear();
    return false;
  }
  *out = static_cast<float>(v);
  return true;
}

// The softmax scale: None is 1 / sqrt(d).
bool softmax_scale(PyObject* o, int64_t d, float* out) {
  if (o == Py_None) {
    *out = static_cast<float>(1.0 / std::sqrt(static_cast<double>(d)));
    return true;
  }
  return real_number(o, out);
}

bool fits(const at::Tensor& t) {
  for (int64_t s : t.sizes())
    if (s > INT_MAX) return false;
  return true;
}

// Bytes [lo, hi) of a tensor, to see that written buffers stand apart.
struct Span {
  const char* lo;
  const char* hi;
};
Span span(const at::Tensor& t) {
  const char* p = static_cast<const char*>(t.const_data_ptr());
  return {p, p + t.nbytes()};
}

// Sizes of a [B, H, rows, d] tensor, as the outputs are allocated from them.
using Shape = std::array<int64_t, 4>;
Shape shape(const at::Tensor& t) { return {t.size(0), t.size(1), t.size(2), t.size(3)}; }

at::Tensor rows_f32(const Shape& s, const at::TensorOptions& options) {
  return at::empty({s[0], s[1], s[2]}, options.dtype(at::kFloat));
}

at::Tensor scratch(size_t bytes, const at::TensorOptions& options) {
  return at::empty({static_cast<int64_t>(bytes)}, options.dtype(at::kByte));
}

PyObject* none() { Py_RETURN_NONE; }

PyObject* result(std::initializer_list<const at::Tensor*> ts) {
  PyObject* tup = PyTuple_New(static_cast<Py_ssize_t>(ts.size()));
  if (!tup) return nullptr;
  Py_ssize_t i = 0;
  for (const at::Tensor* t : ts) {
    PyObject* o = t->defined() ? THPVariable_Wrap(*t) : Py_NewRef(Py_None);
    if (!o) {
      Py_DECREF(tup);
      return nullptr;
    }
    PyTuple_SET_ITEM(tup, i++, o);
  }
  return tup;
}

// Runs f, which allocates the outputs and launches, without the interpreter lock:
// an allocation can wait for the device, a launch for room in the stream's queue,
// and what they wait for can be a callback that needs the lock.  Sizes and data
// pointers of the arguments are taken before, with the lock.  A guard, since f
// may throw (out of memory).  f returns false for outputs that are not real
// tensors (is_real), and sets the status otherwise.
class WithoutLock {
 public:
  WithoutLock() : state_(PyEval_SaveThread()) {}
  ~WithoutLock() { PyEval_RestoreThread(state_); }
  WithoutLock(const WithoutLock&) = delete;
  WithoutLock& operator=(const WithoutLock&) = delete;

 private:
  PyThreadState* state_;
};

template <class F>
auto call(F&& f) {
  WithoutLock unlocked;
  return f();
}

PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 7) {
    PyErr_SetString(PyExc_TypeError, "bind takes 7 addresses");
    return nullptr;
  }
  void* p[7];
  for (int i = 0; i < 7; ++i) {
    p[i] = PyLong_AsVoidPtr(a[i]);
    if (!p[i]) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null address");
      return nullptr;
    }
  }
  p_fwd = reinterpret_cast<decltype(p_fwd)>(p[0]);
  p_bwd = reinterpret_cast<decltype(p_bwd)>(p[1]);
  p_bwd_ws = reinterpret_cast<decltype(p_bwd_ws)>(p[2]);
  p_cache_ws = reinterpret_cast<decltype(p_cache_ws)>(p[3]);
  p_cache = reinterpret_cast<decltype(p_cache)>(p[4]);
  p_step = reinterpret_cast<decltype(p_step)>(p[5]);
  p_qkv = reinterpret_cast<decltype(p_qkv)>(p[6]);
  Py_RETURN_NONE;
}

// fwd(q, k, v, T_chunk, scale, need_lse) -> (o, lse or None)
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 6 || !p_fwd) return none();
  const at::Tensor *q = bf16(a[0], 4), *k = bf16(a[1], 4), *v = bf16(a[2], 4);
  c10::DeviceIndex dev;
  int T;
  float scale;
  if (!q || !k || !v || k->sizes() != q->sizes() || v->sizes() != q->sizes() || !fits(*q) ||
      !one_device({q, k, v}, &dev) || !small_int(a[3], &T) || T < 1 || q->size(2) % T ||
      !softmax_scale(a[4], q->size(3), &scale) || !PyBool_Check(a[5]))
    return none();
  const Shape sh = shape(*q);
  const at::TensorOptions options = q->options();
  const void *pq = q->const_data_ptr(), *pk = k->const_data_ptr(), *pv = v->const_data_ptr();
  const bool need_lse = a[5] == Py_True;
  at::Tensor o, lse;
  mw_status s = MW_OK;
  const bool real = call([&] {
    o = at::empty(sh, options);
    if (need_lse) lse = rows_f32(sh, options);
    if (!is_real(o) || (need_lse && !is_real(lse))) return false;
    s = p_fwd(pq, pk, pv, o.mutable_data_ptr(),
              need_lse ? static_cast<float*>(lse.mutable_data_ptr()) : nullptr,
              static_cast<int>(sh[0]), static_cast<int>(sh[1]), static_cast<int>(sh[2] / T), T,
              static_cast<int>(sh[3]), scale, c10::cuda::getCurrentCUDAStream(dev).stream());
    return true;
  });
  if (!real) return none();
  if (s != MW_OK) return PyLong_FromLong(s);
  return result({&o, &lse});
  END_HANDLE_TH_ERRORS
}

// bwd(q, k, v, o, lse, dout, T_chunk, scale) -> (dq, dk, dv)
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 8 || !p_bwd) return none();
  const at::Tensor *q = bf16(a[0], 4), *k = bf16(a[1], 4), *v = bf16(a[2], 4), *o = bf16(a[3], 4);
  const at::Tensor *lse = tensor(a[4]), *dout = bf16(a[5], 4);
  c10::DeviceIndex dev;
  int T;
  float scale;
  if (!q || !k || !v || !o || !lse || !dout || k->sizes() != q->sizes() ||
      v->sizes() != q->sizes() || o->sizes() != q->sizes() || dout->sizes() != q->sizes() ||
      !fits(*q) || lse->scalar_type() != at::kFloat || lse->sizes() != q->sizes().slice(0, 3) ||
      !one_device({q, k, v, o, lse, dout}, &dev) || !small_int(a[6], &T) || T < 1 ||
      q->size(2) % T || !softmax_scale(a[7], q->size(3), &scale))
    return none();
  const Shape sh = shape(*q);
  const at::TensorOptions options = q->options();
  const int B = static_cast<int>(sh[0]), H = static_cast<int>(sh[1]);
  const int nc = static_cast<int>(sh[2] / T), d = static_cast<int>(sh[3]);
  const size_t bytes = p_bwd_ws(B, H, nc, T, d);
  const void *pq = q->const_data_ptr(), *pk = k->const_data_ptr(), *pv = v->const_data_ptr();
  const void *po = o->const_data_ptr(), *pdo = dout->const_data_ptr();
  const float* pl = static_cast<const float*>(lse->const_data_ptr());
  at::Tensor ws, dq, dk, dv;
  mw_status s = MW_OK;
  const bool real = call([&] {
    ws = scratch(bytes, options);
    dq = at::empty(sh, options);
    dk = at::empty(sh, options);
    dv = at::empty(sh, options);
    if (!is_real(ws) || !is_real(dq) || !is_real(dk) || !is_real(dv)) return false;
    s = p_bwd(pq, pk, pv, po, pl, pdo, dq.mutable_data_ptr(), dk.mutable_data_ptr(),
              dv.mutable_data_ptr(), bytes ? ws.mutable_data_ptr() : nullptr, bytes, B, H, nc, T, d,
              scale, c10::cuda::getCurrentCUDAStream(dev).stream());
    return true;
  });
  if (!real) return none();
  if (s != MW_OK) return PyLong_FromLong(s);
  return result({&dq, &dk, &dv});
  END_HANDLE_TH_ERRORS
}

// cache(q, k_new, v_new, k_sink, v_sink, k_cache, v_cache, head, len, T_chunk,
//       scale, need_lse, workspace, rope, commit) -> (o, lse or None)
// rope: None or (dims, base, shift); commit: None or (slot, rows)
PyObject* cache(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 15 || !p_cache) return none();
  const at::Tensor *q = bf16(a[0], 4), *kn = bf16(a[1], 4), *vn = bf16(a[2], 4);
  const at::Tensor *kc = bf16(a[5], 4), *vc = bf16(a[6], 4), *ks = nullptr, *vs = nullptr;
  const bool sink = a[3] != Py_None || a[4] != Py_None;
  if (sink) {
    ks = bf16(a[3], 4);
    vs = bf16(a[4], 4);
    if (!ks || !vs || ks->sizes() != vs->sizes() || !fits(*ks)) return none();
  }
  const at::Tensor* given = a[12] == Py_None ? nullptr : tensor(a[12]);
  c10::DeviceIndex dev;
  int head, len, T;
  float scale;
  if (!q || !kn || !vn || !kc || !vc || kn->sizes() != q->sizes() || vn->sizes() != q->sizes() ||
      vc->sizes() != kc->sizes() || !fits(*q) || !fits(*kc) || (a[12] != Py_None && !given) ||
      !one_device({q, kn, vn, kc, vc, ks, vs, given}, &dev) || !small_int(a[7], &head) ||
      !small_int(a[8], &len) || !small_int(a[9], &T) || T < 1 || q->size(2) % T ||
      !softmax_scale(a[10], q->size(3), &scale) || !PyBool_Check(a[11]))
    return none();
  for (const at::Tensor* t : {kc, ks})
    if (t && (t->size(0) != q->size(0) || t->size(1) != q->size(1) || t->size(3) != q->size(3)))
      return none();
  int rope_dims = 0, shift = 0, slot = 0, rows = 0;
  float base = 0.f;
  const bool rope = a[13] != Py_None, commit = a[14] != Py_None;
  if (rope && (!PyTuple_CheckExact(a[13]) || PyTuple_GET_SIZE(a[13]) != 3 ||
               !small_int(PyTuple_GET_ITEM(a[13], 0), &rope_dims) ||
               !real_number(PyTuple_GET_ITEM(a[13], 1), &base) ||
               !small_int(PyTuple_GET_ITEM(a[13], 2), &shift)))
    return none();
  if (commit && (rope || sink || !PyTuple_CheckExact(a[14]) || PyTuple_GET_SIZE(a[14]) != 2 ||
                 !small_int(PyTuple_GET_ITEM(a[14], 0), &slot) ||
                 !small_int(PyTuple_GET_ITEM(a[14], 1), &rows)))
    return none();
  const int sink_len = ks ? static_cast<int>(ks->size(2)) : 0;
  const int64_t keys = static_cast<int64_t>(sink_len) + len;
  if (keys > INT_MAX || keys < 0) return none();
  const Shape sh = shape(*q);
  const at::TensorOptions options = q->options();
  const int B = static_cast<int>(sh[0]), H = static_cast<int>(sh[1]);
  const int W = static_cast<int>(sh[2] / T), d = static_cast<int>(sh[3]);
  const size_t bytes = p_cache_ws(B, H, W, T, d, static_cast<int>(keys));
  // what the call writes shares no byte with anything else of the caller's
  Span spans[8];
  int n_spans = 0, n_written = 0;
  if (given) spans[n_spans++] = span(*given), ++n_written;
  spans[n_spans++] = span(*kc);
  spans[n_spans++] = span(*vc);
  if (commit) n_written += 2;
  for (const at::Tensor* t : {q, kn, vn, ks, vs})
    if (t) spans[n_spans++] = span(*t);
  for (int i = 0; i < n_written; ++i)
    for (int j = i + 1; j < n_spans; ++j)
      if (spans[i].lo < spans[j].hi && spans[j].lo < spans[i].hi) return none();
  const void *pq = q->const_data_ptr(), *pkn = kn->const_data_ptr(), *pvn = vn->const_data_ptr();
  const void *pks = ks ? ks->const_data_ptr() : nullptr, *pvs = vs ? vs->const_data_ptr() : nullptr;
  // (a commit writes the ring; without one it is only read)
  void* const pkc = commit ? kc->mutable_data_ptr() : const_cast<void*>(kc->const_data_ptr());
  void* const pvc = commit ? vc->mutable_data_ptr() : const_cast<void*>(vc->const_data_ptr());
  const int cap = static_cast<int>(kc->size(2));
  const bool need_lse = a[11] == Py_True;
  const bool use_given = bytes > 0 && given && given->nbytes() >= bytes;
  void* const pgiven = use_given ? given->mutable_data_ptr() : nullptr;
  at::Tensor ws, o, lse;
  mw_status s = MW_OK;
  const bool real = call([&] {
    if (bytes > 0 && !use_given) ws = scratch(bytes, options);
    o = at::empty(sh, options);
    if (need_lse) lse = rows_f32(sh, options);
    if (!is_real(o) || (need_lse && !is_real(lse)) || (ws.defined() && !is_real(ws))) return false;
    void* w = ws.defined() ? ws.mutable_data_ptr() : pgiven;
    float* l = need_lse ? static_cast<float*>(lse.mutable_data_ptr()) : nullptr;
    cudaStream_t st = c10::cuda::getCurrentCUDAStream(dev).stream();
    if (commit)
      s = p_step(pq, pkn, pvn, pkc, pvc, cap, head, len, slot, rows, o.mutable_data_ptr(), l, w,
                 bytes, B, H, W, T, d, scale, st);
    else
      s = p_cache(pq, pkn, pvn, pks, pvs, sink_len, pkc, pvc, cap, head, len, rope_dims, base,
                  shift, o.mutable_data_ptr(), l, w, bytes, B, H, W, T, d, scale, st);
    return true;
  });
  if (!real) return none();
  if (s != MW_OK) return PyLong_FromLong(s);
  return result({&o, &lse});
  END_HANDLE_TH_ERRORS
}

// qkv(qkv, rope_dims, rope_base, tokens_per_frame, first_frame) -> (q, k, v)
PyObject* qkv(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 5 || !p_qkv) return none();
  const at::Tensor* x = bf16(a[0], 5);
  c10::DeviceIndex dev;
  int dims, per_frame, first;
  float base;
  if (!x || x->size(2) != 3 || !fits(*x) || !one_device({x}, &dev) || !small_int(a[1], &dims) ||
      !real_number(a[2], &base) || !small_int(a[3], &per_frame) || !small_int(a[4], &first))
    return none();
  const int64_t B = x->size(0), N = x->size(1), H = x->size(3), d = x->size(4);
  const at::TensorOptions options = x->options();
  const void* px = x->const_data_ptr();
  at::Tensor q, k, v;
  mw_status s = MW_OK;
  const bool real = call([&] {
    q = at::empty({B, H, N, d}, options);
    k = at::empty({B, H, N, d}, options);
    v = at::empty({B, H, N, d}, options);
    if (!is_real(q) || !is_real(k) || !is_real(v)) return false;
    s = p_qkv(px, q.mutable_data_ptr(), k.mutable_data_ptr(), v.mutable_data_ptr(),
              static_cast<int>(B), static_cast<int>(N), static_cast<int>(H), static_cast<int>(d),
              dims, base, per_frame, first, c10::cuda::getCurrentCUDAStream(dev).stream());
    return true;
  });
  if (!real) return none();
  if (s != MW_OK) return PyLong_FromLong(s);
  return result({&q, &k, &v});
  END_HANDLE_TH_ERRORS
}

#define MW_FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL
PyMethodDef methods[] = {
    {"bind", MW_FAST(bind), "addresses of the C entry points"},
    {"fwd", MW_FAST(fwd), "mw_bca_fwd"},
    {"bwd", MW_FAST(bwd), "mw_bca_bwd"},
    {"cache", MW_FAST(cache), "mw_bca_cache_fwd in its forms, mw_bca_cache_step"},
    {"qkv", MW_FAST(qkv), "mw_qkv_rope_split"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mw_torch", nullptr, -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

// The PyTorch and Python it was built for: it reads their objects' fields through
// their headers, and another version's symbols may resolve all the same.
PyMODINIT_FUNC PyInit__mw_torch(void) {
  PyObject* m = PyModule_Create(&module);
  if (m && (PyModule_AddStringConstant(m, "torch_version", MW_TORCH_VERSION) < 0 ||
            PyModule_AddIntConstant(m, "python_hexversion", PY_VERSION_HEX) < 0)) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
