// _pic_native: the tensor-taking entry points of the Python binding, in C++.
// Each function takes what its Python wrapper (same name in __init__.py) is
// given, checks the tensors (device, dtype, contiguity) and calls libpic.
//
// Host work only, and it sets the pace of small requests: the wrappers used to
// check and convert every tensor in Python (0.4 us each, 22 of them for a link,
// and 3 us for the current stream), 20-30 us a call on a Grace core against 8-18
// us of GPU work; here a call's share is about 2 us.
//
// A tensor argument may also be a tuple (tensor, i) or (tensor, i, j): the
// sub-tensor tensor[i] or tensor[i, j], without creating a Python object for it.
// With a list or tuple of tensors in the tensor's place, i picks one of them.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cuda_runtime_api.h>

#include <algorithm>
#include <exception>
#include <vector>

#include "../../include/pic.h"

namespace {

// Thrown with a Python error already set.
struct PyErrorSet : std::exception {};

[[noreturn]] void raise(PyObject *type, const char *fmt, const char *name, const char *more = "") {
  PyErr_Format(type, fmt, name, more);
  throw PyErrorSet();
}

const char *dtype_name(at::ScalarType t) {
  switch (t) {
    case at::kBFloat16: return "torch.bfloat16";
    case at::kInt: return "torch.int32";
    case at::kLong: return "torch.int64";
    case at::kFloat: return "torch.float32";
    case at::kDouble: return "torch.float64";
    case at::kByte: return "torch.uint8";
    default: return c10::toString(t);
  }
}

// Positional arguments, taken one after the other.
struct Args {
  PyObject *const *v;
  Py_ssize_t n, i = 0;
  PyObject *next() {
    if (i >= n) {
      PyErr_SetString(PyExc_TypeError, "too few arguments");
      throw PyErrorSet();
    }
    return v[i++];
  }
  int64_t integer() {
    const unsigned long long x = PyLong_AsUnsignedLongLongMask(next());
    if (PyErr_Occurred()) throw PyErrorSet();
    return (int64_t)x;
  }
  int32_t i32() { return (int32_t)integer(); }
};

// A tensor argument: the sub-tensor `tensor[i]...` at byte offset `offset`,
// its shape the tensor's from dimension `skip` on.
struct View {
  const at::Tensor *t = nullptr;
  int64_t offset = 0, skip = 0;
  explicit operator bool() const { return t != nullptr; }
  int64_t dim() const { return t->dim() - skip; }
  int64_t size(int64_t d) const { return t->size(skip + d); }
  int64_t numel() const {
    int64_t n = 1;
    for (int64_t d = skip; d < t->dim(); ++d) n *= t->size(d);
    return n;
  }
  bool contiguous() const {
    if (skip == 0) return t->is_contiguous();
    if (numel() == 0) return true;
    int64_t stride = 1;
    for (int64_t d = t->dim() - 1; d >= skip; --d) {
      if (t->size(d) != 1 && t->stride(d) != stride) return false;
      stride *= t->size(d);
    }
    return true;
  }
  void *data() const { return static_cast<char *>(t->data_ptr()) + offset; }
};

View view_of(PyObject *o, const char *name) {
  View w;
  if (o == Py_None) return w;
  const bool indexed = PyTuple_CheckExact(o) && PyTuple_GET_SIZE(o) > 0;
  PyObject *base = indexed ? PyTuple_GET_ITEM(o, 0) : o;
  if (base == Py_None) return w;
  const Py_ssize_t n = indexed ? PyTuple_GET_SIZE(o) : 1;
  Py_ssize_t i = 1;
  auto index = [&](int64_t size) {
    long long at = PyLong_AsLongLong(PyTuple_GET_ITEM(o, i++));
    if (PyErr_Occurred()) throw PyErrorSet();
    if (at < 0) at += size;
    if (at < 0 || at >= size) raise(PyExc_IndexError, "%s: index out of range%s", name);
    return (int64_t)at;
  };
  if (n > 1 && (PyList_Check(base) || PyTuple_Check(base)))  // (list, i, ...): the list keeps its item
    base = PySequence_Fast_GET_ITEM(base, index(PySequence_Fast_GET_SIZE(base)));
  if (!THPVariable_Check(base)) raise(PyExc_TypeError, "%s must be a tensor%s", name);
  w.t = &THPVariable_Unpack(base);
  w.skip = n - i;
  if (w.skip > w.t->dim()) raise(PyExc_IndexError, "%s: too many indices%s", name);
  for (int64_t d = 0; d < w.skip; ++d)
    w.offset += index(w.t->size(d)) * w.t->stride(d) * (int64_t)w.t->element_size();
  return w;
}

void *checked(const View &w, at::ScalarType dtype, const char *name, bool optional = false,
              bool pinned_ok = false) {
  if (!w) {
    if (optional) return nullptr;
    raise(PyExc_ValueError, "%s is required%s", name);
  }
  if (!w.t->is_cuda() && !(pinned_ok && w.t->is_pinned()))
    raise(PyExc_ValueError, "%s must be a CUDA tensor%s", name);
  if (w.t->scalar_type() != dtype) {
    PyErr_Format(PyExc_ValueError, "%s must be %s, got %s", name, dtype_name(dtype),
                 dtype_name(w.t->scalar_type()));
    throw PyErrorSet();
  }
  if (!w.contiguous()) raise(PyExc_ValueError, "%s must be contiguous%s", name);
  return w.data();
}

template <typename T = void>
T *ptr(Args &a, at::ScalarType dtype, const char *name, bool optional = false) {
  return static_cast<T *>(checked(view_of(a.next(), name), dtype, name, optional));
}
int32_t *p32(Args &a, const char *name, bool optional = false) {
  return ptr<int32_t>(a, at::kInt, name, optional);
}
int64_t *p64(Args &a, const char *name) { return ptr<int64_t>(a, at::kLong, name); }
void *pbf(Args &a, const char *name, bool optional = false) {
  return ptr(a, at::kBFloat16, name, optional);
}

// The geometry: attributes of the Python dataclass.
struct Geom {
  pic_geom_t g;
  std::vector<double> inv;
  explicit Geom(PyObject *o) {
    static PyObject *names[9] = {};
    if (!names[0]) {
      const char *s[9] = {"num_layers", "num_q_heads", "num_kv_heads", "head_dim", "page_size",
                          "rope_style", "rope_base", "inv_freq", "layer_inv_freq"};
      for (int i = 8; i >= 0; --i) names[i] = PyUnicode_InternFromString(s[i]);
    }
    auto get = [&](int i) {
      PyObject *x = PyObject_GetAttr(o, names[i]);
      if (!x) throw PyErrorSet();
      return x;
    };
    int32_t *ints[6] = {&g.num_layers, &g.num_q_heads, &g.num_kv_heads,
                        &g.head_dim, &g.page_size, &g.rope_style};
    for (int i = 0; i < 6; ++i) {
      PyObject *x = get(i);
      *ints[i] = (int32_t)PyLong_AsUnsignedLongLongMask(x);
      Py_DECREF(x);
      if (PyErr_Occurred()) throw PyErrorSet();
    }
    PyObject *x = get(6);
    g.rope_base = PyFloat_AsDouble(x);
    Py_DECREF(x);
    if (PyErr_Occurred()) throw PyErrorSet();
    g.inv_freq = nullptr;
    g.layer_inv_freq = nullptr;
    x = get(7);
    if (x != Py_None) {
      PyObject *seq = PySequence_Fast(x, "inv_freq must be a sequence");
      if (seq) {
        for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(seq); ++i)
          inv.push_back(PyFloat_AsDouble(PySequence_Fast_GET_ITEM(seq, i)));
        Py_DECREF(seq);
      }
      g.inv_freq = inv.data();
    }
    Py_DECREF(x);
    if (PyErr_Occurred()) throw PyErrorSet();
    x = get(8);
    if (x != Py_None) {
      // the dataclass holds the reference while the call runs
      Py_DECREF(x);
      const View w = view_of(x, "layer_inv_freq");
      if (w.dim() != 2 || w.size(0) != g.num_layers || w.size(1) != g.head_dim / 2)
        raise(PyExc_ValueError, "%s must be [num_layers][head_dim / 2]%s", "layer_inv_freq");
      g.layer_inv_freq = static_cast<const double *>(checked(w, at::kDouble, "layer_inv_freq"));
    } else {
      Py_DECREF(x);
    }
  }
};

pic_stream_t stream_of(PyObject *o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw PyErrorSet();
  const unsigned long long x = PyLong_AsUnsignedLongLongMask(h);
  Py_DECREF(h);
  if (PyErr_Occurred()) throw PyErrorSet();
  return reinterpret_cast<pic_stream_t>((uintptr_t)x);
}

void need_2d(const View &w, const char *name) {
  if (!w) raise(PyExc_ValueError, "%s is required%s", name);
  if (w.dim() != 2) raise(PyExc_ValueError, "%s must have two dimensions%s", name);
}
// The second dimension of a block table or pool.
int64_t second(const View &w, const char *name) {
  if (!w) raise(PyExc_ValueError, "%s is required%s", name);
  if (w.dim() < 2) raise(PyExc_IndexError, "%s must have two dimensions or more%s", name);
  return w.size(1);
}

// Runs one entry point: `body(args)` returns the libpic status.
template <typename F>
PyObject *guarded(PyObject *const *v, Py_ssize_t n, F &&body) {
  try {
    Args a{v, n};
    return PyLong_FromLong(body(a));
  } catch (const PyErrorSet &) {
  } catch (const std::exception &e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
  }
  return nullptr;
}
template <typename F>
int unlocked(F &&call) {
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = call();
  Py_END_ALLOW_THREADS
  return st;
}

struct Layout {  // the request description, as pic_compose and pic_link take it
  View doc_len, ids, bt;
  int32_t *len, *base, *rid, *ndocs, *span, *prefix, *query, *table;
  int64_t *start;
  int32_t B, max_docs;
  explicit Layout(Args &a) {
    doc_len = view_of(a.next(), "doc_len");
    len = static_cast<int32_t *>(checked(doc_len, at::kInt, "doc_len"));
    base = p32(a, "doc_base_pos");
    start = p64(a, "doc_token_start");
    ids = view_of(a.next(), "req_doc_ids");
    need_2d(ids, "req_doc_ids");
    rid = static_cast<int32_t *>(checked(ids, at::kInt, "req_doc_ids"));
    B = (int32_t)ids.size(0), max_docs = (int32_t)ids.size(1);
    ndocs = p32(a, "req_num_docs");
    span = p32(a, "span_len", true);
    prefix = p32(a, "prefix_len");
    query = p32(a, "query_len");
    bt = view_of(a.next(), "block_table");
    table = static_cast<int32_t *>(checked(bt, at::kInt, "block_table"));
    second(bt, "block_table");
  }
};

PyObject *compose(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    Layout l(a);
    const int64_t num_pages = a.integer();
    const int32_t max_ctx = a.i32(), max_inline = a.i32();
    int32_t *off = p32(a, "doc_offset"), *delta = p32(a, "doc_delta");
    int64_t *slots = p64(a, "slot_mapping"), *map = p64(a, "tok_map");
    int32_t *ipos = p32(a, "inline_pos"), *ctx = p32(a, "ctx_len");
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] {
      return pic_compose(&g.g, l.B, l.max_docs, (int32_t)l.doc_len.numel(), l.len, l.base, l.start,
                         l.rid, l.ndocs, l.span, l.prefix, l.query, l.table, (int32_t)l.bt.size(1),
                         num_pages, max_ctx, max_inline, off, delta, slots, map, ipos, ctx, s);
    });
  });
}

PyObject *relocate(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    const View kp = view_of(a.next(), "k_pool");
    const void *k = checked(kp, at::kBFloat16, "k_pool"), *vp = pbf(a, "v_pool");
    const int64_t pool_tokens = second(kp, "k_pool");
    const int64_t *start = p64(a, "doc_token_start");
    const View dl = view_of(a.next(), "doc_len");
    const int32_t *len = static_cast<int32_t *>(checked(dl, at::kInt, "doc_len"));
    const int32_t *base = p32(a, "doc_base_pos");
    const View ids = view_of(a.next(), "req_doc_ids");
    need_2d(ids, "req_doc_ids");
    const int32_t *rid = static_cast<int32_t *>(checked(ids, at::kInt, "req_doc_ids"));
    const int32_t *ndocs = p32(a, "req_num_docs");
    const View tg = view_of(a.next(), "doc_target");
    if (!tg) raise(PyExc_ValueError, "%s is required%s", "doc_target");
    if (tg.dim() != 2 || tg.size(0) != ids.size(0) || tg.size(1) != ids.size(1))
      raise(PyExc_ValueError, "%s must be [batch][max_docs] like req_doc_ids%s", "doc_target");
    const int32_t *target = static_cast<int32_t *>(checked(tg, at::kInt, "doc_target"));
    const View bt = view_of(a.next(), "block_table");
    const int32_t *table = static_cast<int32_t *>(checked(bt, at::kInt, "block_table"));
    const int64_t max_pages = second(bt, "block_table"), num_pages = a.integer();
    void *kc = pbf(a, "k_cache"), *vc = pbf(a, "v_cache");
    const int32_t lb = a.i32(), le = a.i32();
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] {
      return pic_relocate(&g.g, (int32_t)ids.size(0), (int32_t)ids.size(1), (int32_t)dl.numel(), k,
                          vp, pool_tokens, start, len, base, rid, ndocs, target, table,
                          (int32_t)max_pages, num_pages, kc, vc, lb, le, s);
    });
  });
}

PyObject *relocate_mapped(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    const View kp = view_of(a.next(), "k_pool");
    const void *k = checked(kp, at::kBFloat16, "k_pool"), *vp = pbf(a, "v_pool");
    const int64_t pool_tokens = second(kp, "k_pool");
    const int64_t *map = p64(a, "tok_map");
    const View dd = view_of(a.next(), "doc_delta");
    need_2d(dd, "doc_delta");
    const int32_t *delta = static_cast<int32_t *>(checked(dd, at::kInt, "doc_delta"));
    const View sm = view_of(a.next(), "slot_mapping");
    const int64_t *slots = static_cast<int64_t *>(checked(sm, at::kLong, "slot_mapping"));
    const int64_t max_ctx = second(sm, "slot_mapping"), num_pages = a.integer();
    void *kc = pbf(a, "k_cache"), *vc = pbf(a, "v_cache");
    const int32_t lb = a.i32(), le = a.i32();
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] {
      return pic_relocate_mapped(&g.g, (int32_t)dd.size(0), (int32_t)dd.size(1), k, vp, pool_tokens,
                                 map, delta, slots, (int32_t)max_ctx, num_pages, kc, vc, lb, le, s);
    });
  });
}

PyObject *link(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    Layout l(a);
    const int64_t num_pages = a.integer();
    const int32_t max_ctx = a.i32(), max_inline = a.i32();
    const View kp = view_of(a.next(), "k_pool");
    const void *k = checked(kp, at::kBFloat16, "k_pool"), *vp = pbf(a, "v_pool");
    const int64_t pool_tokens = second(kp, "k_pool");
    const int32_t lb = a.i32(), le = a.i32(), app = a.i32();
    const bool opt = app < 0;
    const void *q = pbf(a, "q", opt), *kn = pbf(a, "k_new", opt), *vn = pbf(a, "v_new", opt);
    const int32_t *tin = p32(a, "inline_len", opt);
    void *kc = pbf(a, "k_cache"), *vc = pbf(a, "v_cache");
    int32_t *off = p32(a, "doc_offset"), *delta = p32(a, "doc_delta");
    int64_t *slots = p64(a, "slot_mapping"), *map = p64(a, "tok_map");
    int32_t *ipos = p32(a, "inline_pos"), *ctx = p32(a, "ctx_len");
    const View wv = view_of(a.next(), "workspace");
    void *ws = checked(wv, at::kByte, "workspace", opt);
    const size_t ws_bytes = wv ? (size_t)wv.numel() : 0;
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] {
      return pic_link(&g.g, l.B, l.max_docs, (int32_t)l.doc_len.numel(), l.len, l.base, l.start,
                      l.rid, l.ndocs, l.span, l.prefix, l.query, l.table, (int32_t)l.bt.size(1),
                      num_pages, max_ctx, max_inline, k, vp, pool_tokens, lb, le, app, q, kn, vn,
                      tin, kc, vc, off, delta, slots, map, ipos, ctx, ws, ws_bytes, s);
    });
  });
}

PyObject *append_inline(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    const int32_t layer = a.i32();
    const void *q = pbf(a, "q"), *kn = pbf(a, "k_new"), *vn = pbf(a, "v_new");
    const View ip = view_of(a.next(), "inline_pos");
    need_2d(ip, "inline_pos");
    const int32_t *ipos = static_cast<int32_t *>(checked(ip, at::kInt, "inline_pos"));
    const int32_t *tin = p32(a, "inline_len");
    const View sm = view_of(a.next(), "slot_mapping");
    const int64_t *slots = static_cast<int64_t *>(checked(sm, at::kLong, "slot_mapping"));
    const int64_t max_ctx = second(sm, "slot_mapping"), num_pages = a.integer();
    void *kc = pbf(a, "k_cache"), *vc = pbf(a, "v_cache");
    const View wv = view_of(a.next(), "workspace");
    void *ws = checked(wv, at::kByte, "workspace");
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] {
      return pic_append_inline(&g.g, layer, (int32_t)ip.size(0), (int32_t)ip.size(1), q, kn, vn,
                               ipos, tin, slots, (int32_t)max_ctx, num_pages, kc, vc, ws,
                               (size_t)wv.numel(), s);
    });
  });
}

// Inline projections of a prefill call: all three or none.
struct Projections {
  const void *q, *k, *v;
  explicit Projections(Args &a) {
    const View x[3] = {view_of(a.next(), "q"), view_of(a.next(), "k_new"), view_of(a.next(), "v_new")};
    const int given = (bool)x[0] + (bool)x[1] + (bool)x[2];
    if (given != 0 && given != 3) raise(PyExc_ValueError, "give q, k_new and v_new together, or none%s%s", "");
    q = checked(x[0], at::kBFloat16, "q", true);
    k = checked(x[1], at::kBFloat16, "k_new", true);
    v = checked(x[2], at::kBFloat16, "v_new", true);
  }
};

PyObject *attend_prefill(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    const int32_t layer = a.i32();
    const Projections pr(a);
    const View ip = view_of(a.next(), "inline_pos");
    need_2d(ip, "inline_pos");
    const int32_t *ipos = static_cast<int32_t *>(checked(ip, at::kInt, "inline_pos"));
    const int32_t *tin = p32(a, "inline_len");
    const int32_t max_ctx = a.i32();
    const View bt = view_of(a.next(), "block_table");
    const int32_t *table = static_cast<int32_t *>(checked(bt, at::kInt, "block_table"));
    const int64_t max_pages = second(bt, "block_table"), num_pages = a.integer();
    void *kc = pbf(a, "k_cache"), *vc = pbf(a, "v_cache");
    void *out = checked(view_of(a.next(), "out"), at::kBFloat16, "out", false, true);
    float *lse = ptr<float>(a, at::kFloat, "lse", true);
    const int32_t splits = a.i32();
    const View wv = view_of(a.next(), "workspace");
    void *ws = checked(wv, at::kByte, "workspace");
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] {
      return pic_attend_prefill(&g.g, layer, (int32_t)ip.size(0), (int32_t)ip.size(1), pr.q, pr.k,
                                pr.v, ipos, tin, max_ctx, table, (int32_t)max_pages, num_pages, kc,
                                vc, out, lse, splits, ws, (size_t)wv.numel(), s);
    });
  });
}

PyObject *attend_prefill_fused(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    const int32_t layer = a.i32();
    const Projections pr(a);
    const View ip = view_of(a.next(), "inline_pos");
    need_2d(ip, "inline_pos");
    const int32_t *ipos = static_cast<int32_t *>(checked(ip, at::kInt, "inline_pos"));
    const int32_t *tin = p32(a, "inline_len");
    const int32_t max_ctx = a.i32();
    const View bt = view_of(a.next(), "block_table");
    const int32_t *table = static_cast<int32_t *>(checked(bt, at::kInt, "block_table"));
    const int64_t max_pages = second(bt, "block_table"), num_pages = a.integer();
    void *kc = pbf(a, "k_cache"), *vc = pbf(a, "v_cache");
    const View kp = view_of(a.next(), "k_pool");
    const void *k = checked(kp, at::kBFloat16, "k_pool"), *vp = pbf(a, "v_pool");
    const int64_t pool_tokens = second(kp, "k_pool");
    const View tm = view_of(a.next(), "tok_map");
    if (!tm || tm.dim() != 2 || tm.size(0) != ip.size(0) || tm.size(1) != max_ctx)
      raise(PyExc_ValueError, "%s must be [batch][max_ctx]%s", "tok_map");
    const int64_t *map = static_cast<int64_t *>(checked(tm, at::kLong, "tok_map"));
    const View dd = view_of(a.next(), "doc_delta");
    const int32_t *delta = static_cast<int32_t *>(checked(dd, at::kInt, "doc_delta"));
    const int64_t max_docs = second(dd, "doc_delta");
    void *out = checked(view_of(a.next(), "out"), at::kBFloat16, "out", false, true);
    float *lse = ptr<float>(a, at::kFloat, "lse", true);
    const int32_t splits = a.i32();
    const View wv = view_of(a.next(), "workspace");
    void *ws = checked(wv, at::kByte, "workspace");
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] {
      return pic_attend_prefill_fused(&g.g, layer, (int32_t)ip.size(0), (int32_t)ip.size(1), pr.q,
                                      pr.k, pr.v, ipos, tin, max_ctx, table, (int32_t)max_pages,
                                      num_pages, kc, vc, k, vp, pool_tokens, (int32_t)max_docs, map,
                                      delta, out, lse, splits, ws, (size_t)wv.numel(), s);
    });
  });
}

// One decoding step; the last two arguments of pic_attend_decode's form are
// the workspace and the stream, of the other's the stream alone.
template <bool kWorkspace>
PyObject *attend_decode(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    const int32_t layer = a.i32();
    const void *q = pbf(a, "q"), *kn = pbf(a, "k_new"), *vn = pbf(a, "v_new");
    const View pv = view_of(a.next(), "pos");
    const int32_t *pos = static_cast<int32_t *>(checked(pv, at::kInt, "pos"));
    const int32_t pos_offset = a.i32(), B = (int32_t)pv.numel();
    const View bt = view_of(a.next(), "block_table");
    const int32_t *table = static_cast<int32_t *>(checked(bt, at::kInt, "block_table"));
    const int64_t max_pages = second(bt, "block_table"), num_pages = a.integer();
    void *kc = pbf(a, "k_cache"), *vc = pbf(a, "v_cache"), *out = pbf(a, "out");
    float *lse = ptr<float>(a, at::kFloat, "lse", true);
    const int32_t max_ctx = a.i32(), splits = a.i32();
    if constexpr (kWorkspace) {
      const View wv = view_of(a.next(), "workspace");
      void *ws = checked(wv, at::kByte, "workspace");
      const pic_stream_t s = stream_of(a.next());
      return unlocked([&] {
        return pic_attend_decode(&g.g, layer, B, q, kn, vn, pos, pos_offset, table,
                                 (int32_t)max_pages, num_pages, kc, vc, out, lse, max_ctx, splits,
                                 ws, (size_t)wv.numel(), s);
      });
    } else {
      const pic_stream_t s = stream_of(a.next());
      return unlocked([&] {
        return pic_attend_decode_noalloc(&g.g, layer, B, q, kn, vn, pos, pos_offset, table,
                                         (int32_t)max_pages, num_pages, kc, vc, out, lse, max_ctx,
                                         splits, s);
      });
    }
  });
}

PyObject *copy_async(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    View w[2];
    const char *names[2] = {"dst", "src"};
    for (int i = 0; i < 2; ++i) {
      w[i] = view_of(a.next(), names[i]);
      if (!w[i]) raise(PyExc_ValueError, "%s is required%s", names[i]);
      if (!w[i].contiguous()) raise(PyExc_ValueError, "%s must be contiguous%s", names[i]);
      if (!w[i].t->is_cuda() && !w[i].t->is_pinned())
        raise(PyExc_ValueError, "%s must be a CUDA tensor or pinned host memory%s", names[i]);
    }
    const size_t bytes = (size_t)w[0].numel() * w[0].t->element_size();
    if ((size_t)w[1].numel() * w[1].t->element_size() != bytes)
      raise(PyExc_ValueError, "dst and src differ in size%s%s", "");
    void *d = w[0].data();
    const void *src = w[1].data();
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] { return pic_copy_async(d, src, bytes, s); });
  });
}

// Copies for a served pass: `bytes` bytes at the same byte offset of dst and
// src, or (negative) the whole of two tensors of one shape, by the library's
// copy kernel or (engine) by a copy engine.
PyObject *copy_range(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    View w[2];
    const char *names[2] = {"dst", "src"};
    for (int i = 0; i < 2; ++i) {
      w[i] = view_of(a.next(), names[i]);
      if (!w[i]) raise(PyExc_ValueError, "%s is required%s", names[i]);
      if (!w[i].contiguous()) raise(PyExc_ValueError, "%s must be contiguous%s", names[i]);
      if (!w[i].t->is_cuda() && !w[i].t->is_pinned())
        raise(PyExc_ValueError, "%s must be a CUDA tensor or pinned host memory%s", names[i]);
    }
    if (w[0].t->scalar_type() != w[1].t->scalar_type() || w[0].dim() != w[1].dim())
      raise(PyExc_ValueError, "dst and src differ in dtype or in dimensions%s%s", "");
    const int64_t offset = a.integer();
    int64_t bytes = a.integer();
    const bool engine = a.integer() != 0;
    const int64_t have = std::min(w[0].numel() * (int64_t)w[0].t->element_size(),
                                  w[1].numel() * (int64_t)w[1].t->element_size());
    if (bytes < 0) {
      for (int64_t d = 0; d < w[0].dim(); ++d)
        if (w[0].size(d) != w[1].size(d)) raise(PyExc_ValueError, "dst and src differ in shape%s%s", "");
      bytes = have - offset;
    }
    if (offset < 0 || bytes < 0 || offset + bytes > have)
      raise(PyExc_ValueError, "copy range outside dst or src%s%s", "");
    char *d = static_cast<char *>(w[0].data()) + offset;
    const char *src = static_cast<const char *>(w[1].data()) + offset;
    const pic_stream_t s = stream_of(a.next());
    if (!engine) return unlocked([&]() -> int { return pic_copy_async(d, src, (size_t)bytes, s); });
    const cudaError_t e = (cudaError_t)unlocked(
        [&]() -> int { return cudaMemcpyAsync(d, src, (size_t)bytes, cudaMemcpyDefault, s); });
    if (e != cudaSuccess) raise(PyExc_RuntimeError, "copy failed: %s%s", cudaGetErrorString(e));
    return (int)PIC_OK;
  });
}

PyObject *attention_deviation(PyObject *, PyObject *const *v, Py_ssize_t n) {
  return guarded(v, n, [](Args &a) {
    Geom g(a.next());
    const int32_t layer = a.i32();
    const View ip = view_of(a.next(), "inline_pos");
    need_2d(ip, "inline_pos");
    const int32_t *ipos = static_cast<int32_t *>(checked(ip, at::kInt, "inline_pos"));
    const int32_t *tin = p32(a, "inline_len"), *tq = p32(a, "query_len");
    const int32_t max_query = a.i32();
    const View ids = view_of(a.next(), "req_doc_ids");
    const int32_t *rid = static_cast<int32_t *>(checked(ids, at::kInt, "req_doc_ids"));
    const int64_t max_docs = second(ids, "req_doc_ids");
    const int32_t *len = p32(a, "doc_len"), *off = p32(a, "doc_offset");
    const View sm = view_of(a.next(), "slot_mapping");
    const int64_t *slots = static_cast<int64_t *>(checked(sm, at::kLong, "slot_mapping"));
    const int64_t max_ctx = second(sm, "slot_mapping"), num_pages = a.integer();
    const void *ka = pbf(a, "k_cache_a"), *kb = pbf(a, "k_cache_b");
    const float *la = ptr<float>(a, at::kFloat, "lse_a"), *lb = ptr<float>(a, at::kFloat, "lse_b");
    std::vector<double> edges;
    PyObject *seq = PySequence_Fast(a.next(), "edges must be a sequence");
    if (!seq) throw PyErrorSet();
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(seq); ++i)
      edges.push_back(PyFloat_AsDouble(PySequence_Fast_GET_ITEM(seq, i)));
    Py_DECREF(seq);
    if (PyErr_Occurred()) throw PyErrorSet();
    const View wv = view_of(a.next(), "workspace");
    const void *ws = checked(wv, at::kByte, "workspace");
    double *sums = ptr<double>(a, at::kDouble, "sums");
    int64_t *counts = p64(a, "counts");
    const pic_stream_t s = stream_of(a.next());
    return unlocked([&] {
      return pic_attention_deviation(&g.g, layer, (int32_t)ip.size(0), (int32_t)ip.size(1),
                                     (int32_t)max_docs, (int32_t)max_ctx, num_pages, ipos, tin, tq,
                                     max_query, rid, len, off, slots, ka, kb, la, lb, edges.data(),
                                     (int32_t)edges.size() - 1, ws, (size_t)wv.numel(), sums, counts,
                                     s);
    });
  });
}

#define FAST(name, fn) {name, (PyCFunction)(void (*)(void))(fn), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST("compose", compose),
    FAST("relocate", relocate),
    FAST("relocate_mapped", relocate_mapped),
    FAST("link", link),
    FAST("append_inline", append_inline),
    FAST("attend_prefill", attend_prefill),
    FAST("attend_prefill_fused", attend_prefill_fused),
    FAST("attend_decode", attend_decode<true>),
    FAST("attend_decode_noalloc", attend_decode<false>),
    FAST("copy_async", copy_async),
    FAST("copy_range", copy_range),
    FAST("attention_deviation", attention_deviation),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pic_native", nullptr, -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pic_native() { return PyModule_Create(&module); }
