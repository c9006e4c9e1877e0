// The calls of the Python binding that programs make per layer and step, as one extension call each: arguments taken from the
// tensors, outputs allocated, the C function called on the current stream.  The work of __init__.py's functions and nothing
// else: whatever is not plain (no exact torch.Tensor, not on the GPU, not contiguous, another type or shape, tensors of a
// transform or a mode) is left to them by returning None, so that errors and special cases stay theirs.  What it saves is
// host time per call, which bounds small problems (us, marshalling through ctypes -> here): see __init__.py.
// It reads tensors through inline functions of the torch it is compiled against (LYNX_TORCH_VERSION) and is used with that one alone.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/TensorSubclassLikeUtils.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "lynx.h"

namespace {

constexpr int64_t kD = 128;

// An argument that this file handles itself: the tensor, or nullptr.
const at::Tensor* plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || !t.is_cuda() || at::isTensorSubclassLike(t) || t.is_conj() || t.is_neg() || !t.is_contiguous()) return nullptr;
  return &t;
}
void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
bool is_none(PyObject* o) { return o == Py_None; }

bool int_of(PyObject* o, int32_t* v) {
  if (!PyLong_CheckExact(o) && !PyBool_Check(o)) return false;
  int over = 0;
  const long x = PyLong_AsLongAndOverflow(o, &over);
  if (over || x < INT32_MIN || x > INT32_MAX) return false;
  *v = (int32_t)x;
  return true;
}
bool float_of(PyObject* o, float* v) {
  if (!PyFloat_CheckExact(o)) return false;
  *v = (float)PyFloat_AS_DOUBLE(o);
  return true;
}
PyObject *s_hq, *s_hkv, *s_d, *s_bt, *s_nb, *s_mb, *s_anchor, *s_residual, *s_meta;

bool int_attr(PyObject* o, PyObject* name, int32_t* v) {
  PyObject* a = PyObject_GetAttr(o, name);
  if (!a) { PyErr_Clear(); return false; }
  const bool ok = int_of(a, v);
  Py_DECREF(a);
  return ok;
}
bool shape_of(PyObject* geo, lynx_shape* s) {
  return int_attr(geo, s_hq, &s->num_q_heads) && int_attr(geo, s_hkv, &s->num_kv_heads) && int_attr(geo, s_d, &s->head_dim) &&
         int_attr(geo, s_bt, &s->block_tokens) && int_attr(geo, s_nb, &s->num_blocks) && int_attr(geo, s_mb, &s->max_blocks_per_seq);
}
// (the planes object keeps its tensors alive over the call: the caller holds it)
bool tensor_attr(PyObject* o, PyObject* name, bool optional, void** p) {
  PyObject* a = PyObject_GetAttr(o, name);
  if (!a) { PyErr_Clear(); return false; }
  const at::Tensor* t = plain(a);
  const bool ok = t || (optional && is_none(a));
  *p = ptr(t);
  Py_DECREF(a);
  return ok;
}
bool planes_of(PyObject* o, lynx_plane* pl) {
  return tensor_attr(o, s_anchor, false, (void**)&pl->anchor) && tensor_attr(o, s_residual, true, (void**)&pl->residual) &&
         tensor_attr(o, s_meta, false, (void**)&pl->meta);
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
at::Tensor empty_like_device(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& on) {
  return at::empty(sizes, at::TensorOptions().dtype(type).device(on.device()));
}
// What a call returns: its result, or its status where it is not LYNX_OK (the caller raises).
PyObject* status(lynx_status st) { return PyLong_FromLong((long)st); }

template <class F>
lynx_status unlocked(F f) {
  lynx_status st;
  Py_BEGIN_ALLOW_THREADS
  st = f();
  Py_END_ALLOW_THREADS
  return st;
}
// C++ exceptions (an allocation that fails) become Python ones
template <class F>
PyObject* guarded(F f) {
  try {
    return f();
  } catch (const c10::OutOfMemoryError& e) {
    PyErr_Clear();
    Py_RETURN_NONE;   // the Python path allocates again and raises torch's own error
  } catch (const std::exception& e) {
    PyErr_Clear();
    Py_RETURN_NONE;
  }
}

bool queries(const at::Tensor* q, const lynx_shape& s) {
  return q && q->scalar_type() == at::kBFloat16 && q->dim() == 4 && q->size(3) == kD && q->size(2) == s.num_q_heads &&
         q->size(0) <= INT32_MAX && q->size(1) <= INT32_MAX;
}

// geo, q, K, V, block_table, seq_lens, workspace, causal, softmax_scale, out
PyObject* anchor_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    lynx_shape s;
    lynx_plane K, V;
    int32_t causal;
    float scale;
    if (n != 10 || !shape_of(a[0], &s)) Py_RETURN_NONE;
    const at::Tensor *q = plain(a[1]), *table = plain(a[4]), *lens = plain(a[5]), *ws = plain(a[6]), *given = plain(a[9]);
    if (!queries(q, s) || !table || !lens || !ws || (!given && !is_none(a[9])) || !int_of(a[7], &causal) || !float_of(a[8], &scale) ||
        !planes_of(a[2], &K) || !planes_of(a[3], &V))
      Py_RETURN_NONE;
    at::Tensor out = given ? *given : empty_like_device(q->sizes(), at::kFloat, *q);
    void* st = stream();
    const lynx_status rc = unlocked([&] {
      return lynx_anchor_attention(&s, q->data_ptr(), (int32_t)q->size(0), (int32_t)q->size(1), causal, K, V, (const int32_t*)table->data_ptr(),
                                   (const int32_t*)lens->data_ptr(), scale, (float*)out.data_ptr(), ws->data_ptr(), (size_t)ws->numel(), st);
    });
    if (rc != LYNX_OK) return status(rc);
    return given ? Py_NewRef(a[9]) : THPVariable_Wrap(out);
  });
}

// geo, q, K, V, block_table, seq_lens, workspace, draft_out, atol, rtol, causal, softmax_scale, out_full, first_reject, dev
PyObject* merge_verify_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    lynx_shape s;
    lynx_plane K, V;
    int32_t causal;
    float scale, atol, rtol;
    if (n != 15 || !shape_of(a[0], &s)) Py_RETURN_NONE;
    const at::Tensor *q = plain(a[1]), *table = plain(a[4]), *lens = plain(a[5]), *ws = plain(a[6]), *draft = plain(a[7]);
    const at::Tensor *g_out = plain(a[12]), *g_first = plain(a[13]), *g_dev = plain(a[14]);
    if (!queries(q, s) || !table || !lens || !ws || (!draft && !is_none(a[7])) || (!g_out && !is_none(a[12])) ||
        (!g_first && !is_none(a[13])) || (!g_dev && !is_none(a[14])) || !float_of(a[8], &atol) || !float_of(a[9], &rtol) ||
        !int_of(a[10], &causal) || !float_of(a[11], &scale) || !planes_of(a[2], &K) || !planes_of(a[3], &V))
      Py_RETURN_NONE;
    if (draft && (draft->scalar_type() != at::kFloat || draft->sizes() != q->sizes())) Py_RETURN_NONE;
    at::Tensor out = g_out ? *g_out : empty_like_device(q->sizes(), at::kFloat, *q), first, dev;
    if (g_first) first = *g_first;
    else if (draft) first = empty_like_device({q->size(0)}, at::kInt, *q);
    if (g_dev) dev = *g_dev;
    else if (draft) dev = empty_like_device({q->size(0), q->size(1)}, at::kFloat, *q);
    void* st = stream();
    const lynx_status rc = unlocked([&] {
      return lynx_merge_verify_attention(&s, q->data_ptr(), (int32_t)q->size(0), (int32_t)q->size(1), causal, K, V,
                                         (const int32_t*)table->data_ptr(), (const int32_t*)lens->data_ptr(), scale, (const float*)ptr(draft),
                                         atol, rtol, (float*)out.data_ptr(), first.defined() ? (int32_t*)first.data_ptr() : nullptr,
                                         dev.defined() ? (float*)dev.data_ptr() : nullptr, ws->data_ptr(), (size_t)ws->numel(), st);
    });
    if (rc != LYNX_OK) return status(rc);
    PyObject* r = PyTuple_New(3);
    if (!r) return nullptr;
    PyTuple_SET_ITEM(r, 0, g_out ? Py_NewRef(a[12]) : THPVariable_Wrap(out));
    PyTuple_SET_ITEM(r, 1, g_first || !first.defined() ? Py_NewRef(a[13]) : THPVariable_Wrap(first));
    PyTuple_SET_ITEM(r, 2, g_dev || !dev.defined() ? Py_NewRef(a[14]) : THPVariable_Wrap(dev));
    return r;
  });
}

// geo, q, k_pages, v_pages, block_table, seq_lens, workspace, causal, softmax_scale, out
PyObject* bf16_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    lynx_shape s;
    int32_t causal;
    float scale;
    if (n != 10 || !shape_of(a[0], &s)) Py_RETURN_NONE;
    const at::Tensor *q = plain(a[1]), *k = plain(a[2]), *v = plain(a[3]), *table = plain(a[4]), *lens = plain(a[5]), *ws = plain(a[6]), *given = plain(a[9]);
    if (!queries(q, s) || !k || !v || k->scalar_type() != at::kBFloat16 || v->scalar_type() != at::kBFloat16 || !table || !lens || !ws ||
        (!given && !is_none(a[9])) || !int_of(a[7], &causal) || !float_of(a[8], &scale))
      Py_RETURN_NONE;
    at::Tensor out = given ? *given : empty_like_device(q->sizes(), at::kFloat, *q);
    void* st = stream();
    const lynx_status rc = unlocked([&] {
      return lynx_bf16_attention(&s, q->data_ptr(), (int32_t)q->size(0), (int32_t)q->size(1), causal, k->data_ptr(), v->data_ptr(),
                                 (const int32_t*)table->data_ptr(), (const int32_t*)lens->data_ptr(), scale, (float*)out.data_ptr(), ws->data_ptr(),
                                 (size_t)ws->numel(), st);
    });
    if (rc != LYNX_OK) return status(rc);
    return given ? Py_NewRef(a[9]) : THPVariable_Wrap(out);
  });
}

// src, planes, block_ids, rows_per_block
PyObject* split_quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    lynx_plane pl;
    int32_t rows_per_block;
    if (n != 4) Py_RETURN_NONE;
    const at::Tensor *src = plain(a[0]), *ids = plain(a[2]);
    if (!src || src->scalar_type() != at::kBFloat16 || src->dim() < 1 || src->size(-1) != kD || (!ids && !is_none(a[2])) ||
        !int_of(a[3], &rows_per_block) || !planes_of(a[1], &pl) || (ids && ids->numel() > INT32_MAX))
      Py_RETURN_NONE;
    void* st = stream();
    return status(unlocked([&] {
      return lynx_split_quantize(src->data_ptr(), src->numel() / kD, (const int32_t*)ptr(ids), ids ? (int32_t)ids->numel() : 0, rows_per_block,
                                 const_cast<uint8_t*>(pl.anchor), const_cast<uint8_t*>(pl.residual), const_cast<float*>(pl.meta), st);
    }));
  });
}

// planes, want_codes, want_bf16 -> (codes or None, pages or None)
PyObject* recombine(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    lynx_plane pl;
    if (n != 3 || !PyBool_Check(a[1]) || !PyBool_Check(a[2]) || !planes_of(a[0], &pl) || !pl.residual) Py_RETURN_NONE;
    PyObject* ao = PyObject_GetAttr(a[0], s_anchor);
    if (!ao) { PyErr_Clear(); Py_RETURN_NONE; }
    const at::Tensor anchor = THPVariable_Unpack(ao);
    Py_DECREF(ao);
    if (anchor.dim() < 1) Py_RETURN_NONE;
    c10::SmallVector<int64_t, 6> sizes(anchor.sizes().begin(), anchor.sizes().end());
    sizes.back() = kD;
    at::Tensor codes, pages;
    if (a[1] == Py_True) codes = empty_like_device(sizes, at::kByte, anchor);
    if (a[2] == Py_True) pages = empty_like_device(sizes, at::kBFloat16, anchor);
    void* st = stream();
    const lynx_status rc = unlocked([&] {
      return lynx_recombine(pl.anchor, pl.residual, pl.meta, anchor.numel() / 64, codes.defined() ? (uint8_t*)codes.data_ptr() : nullptr,
                            pages.defined() ? pages.data_ptr() : nullptr, st);
    });
    if (rc != LYNX_OK) return status(rc);
    PyObject* r = PyTuple_New(2);
    if (!r) return nullptr;
    PyTuple_SET_ITEM(r, 0, codes.defined() ? THPVariable_Wrap(codes) : Py_NewRef(Py_None));
    PyTuple_SET_ITEM(r, 1, pages.defined() ? THPVariable_Wrap(pages) : Py_NewRef(Py_None));
    return r;
  });
}

// geo, B, n_q, workspace, bf16 -> the view of the log-sum-exps
PyObject* lse_view(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    lynx_shape s;
    int32_t B, nq;
    if (n != 5 || !shape_of(a[0], &s) || !int_of(a[1], &B) || !int_of(a[2], &nq) || !PyBool_Check(a[4])) Py_RETURN_NONE;
    const at::Tensor* ws = plain(a[3]);
    if (!ws || ws->scalar_type() != at::kByte || ws->dim() != 1) Py_RETURN_NONE;
    const char* base = (const char*)ws->data_ptr();
    const float* p = a[4] == Py_True ? lynx_bf16_workspace_lse(&s, B, nq, base) : lynx_workspace_lse(&s, B, nq, base);
    if (!p) Py_RETURN_NONE;
    const int64_t off = (const char*)p - base, bytes = (int64_t)B * nq * s.num_q_heads * 4;
    if (off < 0 || off + bytes > ws->numel()) Py_RETURN_NONE;
    return THPVariable_Wrap(ws->slice(0, off, off + bytes).view(at::kFloat).view({B, nq, s.num_q_heads}));
  });
}

// out_a, lse_a, out_b, lse_b, out, want_lse -> out or (out, lse)
PyObject* lse_merge(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 6 || !PyBool_Check(a[5])) Py_RETURN_NONE;
    const at::Tensor *oa = plain(a[0]), *la = plain(a[1]), *ob = plain(a[2]), *lb = plain(a[3]), *given = plain(a[4]);
    if (!oa || !la || !ob || !lb || (!given && !is_none(a[4])) || oa->scalar_type() != at::kFloat || ob->scalar_type() != at::kFloat ||
        la->scalar_type() != at::kFloat || lb->scalar_type() != at::kFloat || oa->dim() < 1 || oa->sizes() != ob->sizes() || oa->size(-1) != kD)
      Py_RETURN_NONE;
    const int64_t rows = oa->numel() / kD;
    if (la->numel() != rows || lb->numel() != rows) Py_RETURN_NONE;
    at::Tensor out = given ? *given : at::empty_like(*oa), lse;
    if (a[5] == Py_True) lse = empty_like_device(oa->sizes().slice(0, oa->dim() - 1), at::kFloat, *oa);
    void* st = stream();
    const lynx_status rc = unlocked([&] {
      return lynx_lse_merge((const float*)oa->data_ptr(), (const float*)la->data_ptr(), (const float*)ob->data_ptr(), (const float*)lb->data_ptr(),
                            rows, (float*)out.data_ptr(), lse.defined() ? (float*)lse.data_ptr() : nullptr, st);
    });
    if (rc != LYNX_OK) return status(rc);
    PyObject* o = given ? Py_NewRef(a[4]) : THPVariable_Wrap(out);
    if (!lse.defined()) return o;
    PyObject* r = PyTuple_New(2);
    if (!r) { Py_XDECREF(o); return nullptr; }
    PyTuple_SET_ITEM(r, 0, o);
    PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(lse));
    return r;
  });
}

// src -> the six tensors of HierPlanes
PyObject* hier_quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    const at::Tensor* src = n == 1 ? plain(a[0]) : nullptr;
    if (!src || src->scalar_type() != at::kBFloat16 || src->dim() != 3 || src->size(1) != 256 || src->size(2) != kD) Py_RETURN_NONE;
    const int64_t p = src->size(0);
    at::Tensor t[6] = {empty_like_device({p, 256, 64}, at::kByte, *src), empty_like_device({p, 256, 64}, at::kByte, *src),
                       empty_like_device({p, kD}, at::kFloat, *src),     empty_like_device({p, kD}, at::kFloat, *src),
                       empty_like_device({p, 8, kD}, at::kFloat, *src),  empty_like_device({p, 8, kD}, at::kFloat, *src)};
    void* st = stream();
    const lynx_status rc = unlocked([&] {
      return lynx_hier_quantize(src->data_ptr(), p, (uint8_t*)t[0].data_ptr(), (uint8_t*)t[1].data_ptr(), (float*)t[2].data_ptr(), (float*)t[3].data_ptr(),
                                (float*)t[4].data_ptr(), (float*)t[5].data_ptr(), st);
    });
    if (rc != LYNX_OK) return status(rc);
    PyObject* r = PyTuple_New(6);
    if (!r) return nullptr;
    for (int i = 0; i < 6; ++i) PyTuple_SET_ITEM(r, i, THPVariable_Wrap(t[i]));
    return r;
  });
}

// q_anc, q_res or None, gamma_min, gamma_scale, mu, sigma, out
PyObject* hier_dequantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 7) Py_RETURN_NONE;
    const at::Tensor* t[6];
    for (int i = 0; i < 6; ++i) {
      t[i] = plain(a[i]);
      if (!t[i] && !(i == 1 && is_none(a[1]))) Py_RETURN_NONE;
    }
    const at::Tensor* given = plain(a[6]);
    if ((!given && !is_none(a[6])) || t[0]->dim() < 1) Py_RETURN_NONE;
    const int64_t p = t[0]->size(0);
    at::Tensor out = given ? *given : empty_like_device({p, 256, kD}, at::kBFloat16, *t[0]);
    void* st = stream();
    const lynx_status rc = unlocked([&] {
      return lynx_hier_dequantize((const uint8_t*)t[0]->data_ptr(), (const uint8_t*)ptr(t[1]), p, (const float*)t[2]->data_ptr(), (const float*)t[3]->data_ptr(),
                                  (const float*)t[4]->data_ptr(), (const float*)t[5]->data_ptr(), out.data_ptr(), st);
    });
    if (rc != LYNX_OK) return status(rc);
    return given ? Py_NewRef(a[6]) : THPVariable_Wrap(out);
  });
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(anchor_attention), FAST(merge_verify_attention), FAST(bf16_attention), FAST(split_quantize), FAST(recombine),
                         FAST(lse_view), FAST(lse_merge), FAST(hier_quantize), FAST(hier_dequantize), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  struct { PyObject** s; const char* n; } names[] = {{&s_hq, "num_q_heads"}, {&s_hkv, "num_kv_heads"}, {&s_d, "head_dim"}, {&s_bt, "block_tokens"},
                                                     {&s_nb, "num_blocks"}, {&s_mb, "max_blocks_per_seq"}, {&s_anchor, "anchor"},
                                                     {&s_residual, "residual"}, {&s_meta, "meta"}};
  for (auto& x : names)
    if (!(*x.s = PyUnicode_InternFromString(x.n))) return nullptr;
  PyObject* m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "torch_version", LYNX_TORCH_VERSION)) Py_CLEAR(m);
  return m;
}
