// Argument marshalling between torch tensors and the C ABI (libsmartgen.so), as a CPython extension.
//
// The smallest calls of the path take less time on the GPU than a Python layer needs to check and convert their
// arguments (ctypes and tensor attributes: about 9 us per call, 25 us for the three calls of a prefill layer, whose
// kernels take 30).  Here a tensor costs a few dozen nanoseconds.  One function per call, the checks and the messages of
// binding.py's contract, the two sequences a prefill engine issues (all layers, one layer) and a decode call on one layer of
// packed tensors.  Every function returns the
// call's sg_status; a sequence returns status + 256 * (number of the failed call).
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "internal.h"

namespace {

enum Kind { kBf16, kF32, kI32, kI8 };
const char* const kKindName[] = {"(torch.bfloat16, torch.int16, torch.uint16)", "(torch.float32,)", "(torch.int32,)", "(torch.int8,)"};

bool is_kind(at::ScalarType t, Kind k) {
  switch (k) {
    case kBf16: return t == at::kBFloat16 || t == at::kShort || t == at::kUInt16;
    case kF32: return t == at::kFloat;
    case kI32: return t == at::kInt;
    default: return t == at::kChar;
  }
}

// Reads the arguments of one call in order; after the first failure a Python error is set and the rest is skipped.
struct Args {
  PyObject* const* a;
  Py_ssize_t n, i = 0;
  bool ok = true;
  PyObject* held[8];                                    // layers taken out of sequences, kept for the length of the call
  int n_held = 0;
  Args(PyObject* const* a_, Py_ssize_t n_, Py_ssize_t want) : a(a_), n(n_) {
    if (n != want) { PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n); ok = false; }
  }
  Args(const Args&) = delete;
  ~Args() { while (n_held > 0) Py_DECREF(held[--n_held]); }
  const sg_shape* shape() {
    if (!ok) return nullptr;
    Py_buffer view;
    if (PyObject_GetBuffer(a[i++], &view, PyBUF_SIMPLE) != 0) { ok = false; return nullptr; }
    const sg_shape* s = static_cast<const sg_shape*>(view.buf);
    if (view.len < (Py_ssize_t)sizeof(sg_shape)) { PyErr_SetString(PyExc_TypeError, "shape must be a Shape"); ok = false; s = nullptr; }
    PyBuffer_Release(&view);                            // the caller holds the struct for the length of the call
    return s;
  }
  long long integer() {
    if (!ok) return 0;
    const long long v = PyLong_AsLongLong(a[i++]);
    if (v == -1 && PyErr_Occurred()) ok = false;
    return v;
  }
  double number() {
    if (!ok) return 0.0;
    const double v = PyFloat_AsDouble(a[i++]);
    if (v == -1.0 && PyErr_Occurred()) ok = false;
    return v;
  }
  // Checked tensor; undefined when None is given and allowed.  An empty tensor's address is null.
  const at::Tensor* tensor(Kind kind, const char* name, bool allow_none = false, bool whole = true) {
    return ok ? tensor_of(a[i++], kind, name, allow_none, whole) : nullptr;
  }
  const at::Tensor* tensor_of(PyObject* o, Kind kind, const char* name, bool allow_none, bool whole) {
    if (o == Py_None) {
      if (!allow_none) { PyErr_Format(PyExc_TypeError, "%s is required", name); ok = false; }
      return nullptr;
    }
    if (!THPVariable_Check(o) || !THPVariable_Unpack(o).is_cuda()) {
      PyErr_Format(PyExc_TypeError, "%s must be a CUDA tensor", name);
      ok = false;
      return nullptr;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!is_kind(t.scalar_type(), kind)) {
      PyErr_Format(PyExc_TypeError, "%s: expected dtype %s, got torch.%s", name, kKindName[kind], c10::toString(t.scalar_type()));
      ok = false;
      return nullptr;
    }
    if (whole && !t.is_contiguous()) { not_contiguous(name); return nullptr; }
    return &t;
  }
  void not_contiguous(const char* name) {
    PyErr_Format(PyExc_ValueError, "%s must be contiguous (strided caches go through the sg_shape strides)", name);
    ok = false;
  }
  void* ptr(Kind kind, const char* name, bool allow_none = false) {
    const at::Tensor* t = tensor(kind, name, allow_none);
    return t == nullptr || t->numel() == 0 ? nullptr : t->data_ptr();
  }
  // t[layer] of a tensor whose layers are contiguous each, or of a sequence of tensors, one per layer.
  void* layer_ptr(Kind kind, const char* name, long long layer) {
    if (ok && a[i] != Py_None && !THPVariable_Check(a[i])) {
      PyObject* index = PyLong_FromLongLong(layer);
      PyObject* item = index == nullptr ? nullptr : PyObject_GetItem(a[i++], index);
      Py_XDECREF(index);
      if (item == nullptr) { ok = false; return nullptr; }
      held[n_held++] = item;
      const at::Tensor* t = tensor_of(item, kind, name, false, true);
      return t == nullptr || t->numel() == 0 ? nullptr : t->data_ptr();
    }
    const at::Tensor* t = tensor(kind, name, false, false);
    if (t == nullptr) return nullptr;
    if (t->dim() < 1 || layer < -t->size(0) || layer >= t->size(0)) {
      PyErr_Format(PyExc_IndexError, "%s: layer %lld is out of range", name, layer);
      ok = false;
      return nullptr;
    }
    int64_t expect = 1;
    for (int64_t d = t->dim() - 1; d >= 1; --d) {
      if (t->size(d) != 1 && t->stride(d) != expect) { not_contiguous(name); return nullptr; }
      expect *= t->size(d);
    }
    if (layer < 0) layer += t->size(0);
    if (expect == 0) return nullptr;
    return static_cast<char*>(t->data_ptr()) + layer * t->stride(0) * (int64_t)t->element_size();
  }
  // Workspace: any tensor or None.
  void* workspace(size_t* bytes) {
    *bytes = 0;
    if (!ok) return nullptr;
    PyObject* o = a[i++];
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "workspace must be a tensor"); ok = false; return nullptr; }
    const at::Tensor& t = THPVariable_Unpack(o);
    *bytes = t.nbytes();
    return t.data_ptr();
  }
  // None: the current device's current stream; a torch stream; or a raw handle (an integer or a ctypes pointer, 0 or empty
  // for the default stream).
  void* stream() {
    if (!ok) return nullptr;
    PyObject* o = a[i++];
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* raw = Py_NewRef(o);
    for (const char* name : {"cuda_stream", "value"}) {
      if (PyLong_Check(raw) || raw == Py_None) break;
      PyObject* inner = PyObject_GetAttrString(raw, name);
      if (inner == nullptr) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) { Py_DECREF(raw); ok = false; return nullptr; }
        PyErr_Clear();
        continue;
      }
      Py_DECREF(raw);
      raw = inner;
    }
    void* p = nullptr;
    if (raw != Py_None) {
      if (PyLong_Check(raw)) p = PyLong_AsVoidPtr(raw);
      else PyErr_SetString(PyExc_TypeError, "stream must be a stream or a stream handle");
    }
    Py_DECREF(raw);
    if (p == nullptr && PyErr_Occurred()) ok = false;
    return p;
  }
};

template <class F>
PyObject* call(const Args& x, F f) {
  if (!x.ok) return nullptr;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}
// A function of the module.  A tensor's accessors throw C++ exceptions (no storage, no CUDA device); they become Python
// errors here and never leave a C function.
#define SG_FN(name)                                                         \
  PyObject* name##_args(PyObject* const* a, Py_ssize_t n);                  \
  PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n) {             \
    HANDLE_TH_ERRORS                                                        \
    return name##_args(a, n);                                               \
    END_HANDLE_TH_ERRORS                                                    \
  }                                                                         \
  PyObject* name##_args(PyObject* const* a, Py_ssize_t n)

SG_FN(score) {
  Args x(a, n, 7);
  const sg_shape* s = x.shape();
  void *q = x.ptr(kBf16, "q_win"), *k = x.ptr(kBf16, "k_cache"), *imp = x.ptr(kF32, "importance");
  size_t wb;
  void *w = x.workspace(&wb), *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&] { return sg_score(s, q, k, (float*)imp, w, wb, (int32_t*)st, stream); });
}
SG_FN(score_static) {
  Args x(a, n, 6);
  const sg_shape* s = x.shape();
  void *q = x.ptr(kBf16, "q_win"), *k = x.ptr(kBf16, "k_cache"), *imp = x.ptr(kF32, "importance"), *st = x.ptr(kI32, "dev_status", true);
  void* stream = x.stream();
  return call(x, [&] { return sg_score_static(s, q, k, (float*)imp, (int32_t*)st, stream); });
}
SG_FN(select_topk) {
  Args x(a, n, 8);
  const sg_shape* s = x.shape();
  void *imp = x.ptr(kF32, "importance"), *cu_k = x.ptr(kI32, "cu_k");
  const int32_t total = (int32_t)x.integer();
  void *sel = x.ptr(kI32, "sel_idx"), *st, *stream;
  size_t wb;
  void* w = x.workspace(&wb);
  st = x.ptr(kI32, "dev_status", true);
  stream = x.stream();
  return call(x, [&] { return sg_select_topk(s, (float*)imp, (int32_t*)cu_k, total, (int32_t*)sel, w, wb, (int32_t*)st, stream); });
}
SG_FN(pack_kv) {
  Args x(a, n, 10);
  const sg_shape* s = x.shape();
  void *k = x.ptr(kBf16, "k_cache"), *v = x.ptr(kBf16, "v_cache"), *sel = x.ptr(kI32, "sel_idx"), *cu_k = x.ptr(kI32, "cu_k");
  const int32_t total = (int32_t)x.integer();
  void *pk = x.ptr(kBf16, "packed_k"), *pv = x.ptr(kBf16, "packed_v"), *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&] { return sg_pack_kv(s, k, v, (int32_t*)sel, (int32_t*)cu_k, total, pk, pv, (int32_t*)st, stream); });
}
SG_FN(select_pack_kv) {
  Args x(a, n, 11);
  const sg_shape* s = x.shape();
  void *imp = x.ptr(kF32, "importance"), *cu_k = x.ptr(kI32, "cu_k");
  const int32_t total = (int32_t)x.integer();
  void *k = x.ptr(kBf16, "k_cache"), *v = x.ptr(kBf16, "v_cache"), *sel = x.ptr(kI32, "sel_idx", total == 0);
  void *pk = x.ptr(kBf16, "packed_k", total == 0), *pv = x.ptr(kBf16, "packed_v", total == 0), *st = x.ptr(kI32, "dev_status", true);
  void* stream = x.stream();
  return call(x, [&] { return sg_select_pack_kv(s, (float*)imp, (int32_t*)cu_k, total, k, v, (int32_t*)sel, pk, pv, (int32_t*)st, stream); });
}
SG_FN(select_threshold) {
  Args x(a, n, 9);
  const sg_shape* s = x.shape();
  void* scores = x.ptr(kF32, "scores");
  const float alpha = (float)x.number();
  void* cu_cap = x.ptr(kI32, "cu_cap");
  const int32_t total = (int32_t)x.integer();
  void *sel = x.ptr(kI32, "sel_idx", total == 0), *cnt = x.ptr(kI32, "sel_count"), *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&] { return sg_select_threshold(s, (float*)scores, alpha, (int32_t*)cu_cap, total, (int32_t*)sel, (int32_t*)cnt, (int32_t*)st, stream); });
}
SG_FN(pack_kv_counted) {
  Args x(a, n, 11);
  const sg_shape* s = x.shape();
  void *k = x.ptr(kBf16, "k_cache"), *v = x.ptr(kBf16, "v_cache");
  PyObject* const* rest = a + x.i;                      // sel_idx comes before the total that says whether it may be missing
  const bool empty = x.ok && n == 11 && PyLong_Check(rest[2]) && PyLong_AsLongLong(rest[2]) == 0;
  void *sel = x.ptr(kI32, "sel_idx", empty), *cu_cap = x.ptr(kI32, "cu_cap");
  const int32_t total = (int32_t)x.integer();
  void *cnt = x.ptr(kI32, "sel_count"), *pk = x.ptr(kBf16, "packed_k", empty), *pv = x.ptr(kBf16, "packed_v", empty);
  void *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&] { return sg_pack_kv_counted(s, k, v, (int32_t*)sel, (int32_t*)cu_cap, total, (int32_t*)cnt, pk, pv, (int32_t*)st, stream); });
}
SG_FN(sparse_decode_attn) {
  Args x(a, n, 17);
  const sg_shape* s = x.shape();
  void *q = x.ptr(kBf16, "q"), *pk = x.ptr(kBf16, "packed_k", true), *pv = x.ptr(kBf16, "packed_v", true), *cu_k = x.ptr(kI32, "cu_k");
  const int32_t total = (int32_t)x.integer();
  void *lk = x.ptr(kBf16, "local_k", true), *lv = x.ptr(kBf16, "local_v", true), *idx = x.ptr(kI32, "local_idx", true), *cu_n = x.ptr(kI32, "cu_nloc");
  const int32_t nloc = (int32_t)x.integer();
  void *out = x.ptr(kBf16, "out"), *lse = x.ptr(kF32, "lse", true);
  const float scale = (float)x.number();
  size_t wb;
  void *w = x.workspace(&wb), *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&] {
    return sg_sparse_decode_attn(s, q, pk, pv, (int32_t*)cu_k, total, lk, lv, (int32_t*)idx, (int32_t*)cu_n, nloc, scale, out, (float*)lse, w, wb,
                                 (int32_t*)st, stream);
  });
}
// The same with packed tensors of all layers, one of which is meant.
SG_FN(decode_layer) {
  Args x(a, n, 18);
  const sg_shape* s = x.shape();
  const long long layer = x.integer();
  void *q = x.ptr(kBf16, "q"), *pk = x.layer_ptr(kBf16, "packed_k", layer), *pv = x.layer_ptr(kBf16, "packed_v", layer), *cu_k = x.ptr(kI32, "cu_k");
  const int32_t total = (int32_t)x.integer();
  void *lk = x.ptr(kBf16, "local_k", true), *lv = x.ptr(kBf16, "local_v", true), *idx = x.ptr(kI32, "local_idx", true), *cu_n = x.ptr(kI32, "cu_nloc");
  const int32_t nloc = (int32_t)x.integer();
  void *out = x.ptr(kBf16, "out"), *lse = x.ptr(kF32, "lse", true);
  const float scale = (float)x.number();
  size_t wb;
  void *w = x.workspace(&wb), *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&] {
    return sg_sparse_decode_attn(s, q, pk, pv, (int32_t*)cu_k, total, lk, lv, (int32_t*)idx, (int32_t*)cu_n, nloc, scale, out, (float*)lse, w, wb,
                                 (int32_t*)st, stream);
  });
}
SG_FN(sparse_decode_attn_counted) {
  Args x(a, n, 18);
  const sg_shape* s = x.shape();
  void *q = x.ptr(kBf16, "q"), *pk = x.ptr(kBf16, "packed_k", true), *pv = x.ptr(kBf16, "packed_v", true), *cu_k = x.ptr(kI32, "cu_cap");
  const int32_t total = (int32_t)x.integer();
  void* pc = x.ptr(kI32, "packed_count", true);
  void *lk = x.ptr(kBf16, "local_k", true), *lv = x.ptr(kBf16, "local_v", true), *idx = x.ptr(kI32, "local_idx", true), *cu_n = x.ptr(kI32, "cu_nloc");
  const int32_t nloc = (int32_t)x.integer();
  void *out = x.ptr(kBf16, "out"), *lse = x.ptr(kF32, "lse", true);
  const float scale = (float)x.number();
  void *st = x.ptr(kI32, "dev_status", true), *stream = x.stream(), *skip = x.ptr(kI32, "local_skip", true);
  return call(x, [&] {
    return sg_sparse_decode_attn_counted(s, q, pk, pv, (int32_t*)cu_k, total, (int32_t*)pc, lk, lv, (int32_t*)idx, (int32_t*)cu_n, nloc,
                                         (int32_t*)skip, scale, out, (float*)lse, (int32_t*)st, stream);
  });
}
SG_FN(split_index) {
  Args x(a, n, 13);
  const sg_shape* s = x.shape();
  void *idx = x.ptr(kI32, "kv_index"), *cu_k = x.ptr(kI32, "cu_k");
  const int32_t total = (int32_t)x.integer();
  void* mask = x.ptr(kI8, "kv_mask");
  const int32_t reorder = (int32_t)x.integer();
  void *re = x.ptr(kI32, "reordered", true), *lo = x.ptr(kI32, "local_index"), *rem = x.ptr(kI32, "remote_index"), *nl = x.ptr(kI32, "n_local");
  void *nr = x.ptr(kI32, "n_remote"), *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&] {
    return sg_split_index(s, (int32_t*)idx, (int32_t*)cu_k, total, (int8_t*)mask, reorder, (int32_t*)re, (int32_t*)lo, (int32_t*)rem, (int32_t*)nl,
                          (int32_t*)nr, (int32_t*)st, stream);
  });
}
SG_FN(push_blocks) {
  Args x(a, n, 10);
  const sg_shape* s = x.shape();
  const int32_t blocks = (int32_t)x.integer(), layer = (int32_t)x.integer();
  const at::Tensor* sel = x.tensor(kI32, "selected", true);
  void *sk = x.ptr(kBf16, "src_k"), *sv = x.ptr(kBf16, "src_v"), *dk = x.ptr(kBf16, "dst_k"), *dv = x.ptr(kBf16, "dst_v");
  void *mask = x.ptr(kI8, "kv_mask", true), *stream = x.stream();
  const int32_t count = sel ? (int32_t)sel->numel() : 0;
  return call(x, [&] { return sg_push_blocks(s, blocks, layer, count ? (int32_t*)sel->data_ptr() : nullptr, count, sk, sv, dk, dv, (int8_t*)mask, stream); });
}

// ---------------------------------------------------------------- sequences
// sg_score, then sg_select_pack_kv, over all layers of the shape.
SG_FN(prefill) {
  Args x(a, n, 13);
  const sg_shape* s = x.shape();
  void *q = x.ptr(kBf16, "q_win"), *k = x.ptr(kBf16, "k_cache"), *v = x.ptr(kBf16, "v_cache"), *imp = x.ptr(kF32, "importance");
  size_t wb;
  void *w = x.workspace(&wb), *cu_k = x.ptr(kI32, "cu_k");
  const int32_t total = (int32_t)x.integer();
  void *sel = x.ptr(kI32, "sel_idx", total == 0), *pk = x.ptr(kBf16, "packed_k", total == 0), *pv = x.ptr(kBf16, "packed_v", total == 0);
  void *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&]() -> int {
    int rc = sg_internal_score_select_pack(s, q, k, v, (float*)imp, w, wb, (int32_t*)cu_k, total, (int32_t*)sel, pk, pv, (int32_t*)st, stream);
    if (rc != SG_ERR_UNSUPPORTED) return rc;           // one kernel did both
    rc = sg_score(s, q, k, (float*)imp, w, wb, (int32_t*)st, stream);
    if (rc) return rc;
    rc = sg_select_pack_kv(s, (float*)imp, (int32_t*)cu_k, total, k, v, (int32_t*)sel, pk, pv, (int32_t*)st, stream);
    return rc ? rc + 256 : 0;
  });
}
// sg_score, then sg_select_pack_kv, of one layer of tensors that hold all of them (shape: one layer).
SG_FN(prefill_layer) {
  Args x(a, n, 14);
  const sg_shape* s = x.shape();
  const long long layer = x.integer();
  void *q = x.layer_ptr(kBf16, "q_win", layer), *k = x.layer_ptr(kBf16, "k_cache", layer), *v = x.layer_ptr(kBf16, "v_cache", layer);
  void* imp = x.layer_ptr(kF32, "importance", layer);
  size_t wb;
  void *w = x.workspace(&wb), *cu_k = x.ptr(kI32, "cu_k");
  const int32_t total = (int32_t)x.integer();
  void *sel = x.layer_ptr(kI32, "sel_idx", layer), *pk = x.layer_ptr(kBf16, "packed_k", layer), *pv = x.layer_ptr(kBf16, "packed_v", layer);
  void *st = x.ptr(kI32, "dev_status", true), *stream = x.stream();
  return call(x, [&]() -> int {
    int rc = sg_internal_score_select_pack(s, q, k, v, (float*)imp, w, wb, (int32_t*)cu_k, total, (int32_t*)sel, pk, pv, (int32_t*)st, stream);
    if (rc != SG_ERR_UNSUPPORTED) return rc;           // one kernel did both
    rc = sg_score(s, q, k, (float*)imp, w, wb, (int32_t*)st, stream);
    if (rc) return rc;
    rc = sg_select_pack_kv(s, (float*)imp, (int32_t*)cu_k, total, k, v, (int32_t*)sel, pk, pv, (int32_t*)st, stream);
    return rc ? rc + 256 : 0;
  });
}

#define SG_ENTRY(name) {#name, (PyCFunction)(void*)name, METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {SG_ENTRY(score), SG_ENTRY(score_static), SG_ENTRY(select_topk), SG_ENTRY(pack_kv), SG_ENTRY(select_pack_kv),
                          SG_ENTRY(select_threshold), SG_ENTRY(pack_kv_counted), SG_ENTRY(sparse_decode_attn),
                          SG_ENTRY(sparse_decode_attn_counted), SG_ENTRY(split_index), SG_ENTRY(push_blocks), SG_ENTRY(prefill),
                          SG_ENTRY(prefill_layer), SG_ENTRY(decode_layer), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

#ifndef SG_BUILT_FOR
#error "SG_BUILT_FOR: the torch and the interpreter that the module is compiled against (build.py)"
#endif
PyMODINIT_FUNC PyInit__native() {
  PyObject* m = PyModule_Create(&kModule);
  if (m != nullptr && PyModule_AddStringConstant(m, "BUILT_FOR", SG_BUILT_FOR) != 0) Py_CLEAR(m);
  return m;
}
