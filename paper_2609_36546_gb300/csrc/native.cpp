// The Python binding's argument marshalling, against the CPython C API: takes
// tensors (any object with data_ptr(), numel(), element_size() and shape) and
// numbers, and makes the C ABI call declared in include/ipd.h.  No computation
// and no CUDA here.  The calls are a few microseconds of GPU work at small
// sizes, which marshalling through ctypes (about 20 conversions a call, and a
// structure per append or option set) took longer than: 64 requests' K/V append
// 19.7 us a call, of which 4 us are the library's.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>
#include <string.h>

#include "../../include/ipd.h"

namespace {

PyObject *s_data_ptr, *s_numel, *s_element_size, *s_shape, *s_c, *s_k_pages, *s_v_pages;
PyObject *s_out[13];  // names of the score outputs, in the C call's order
const char *const kOutNames[13] = {"logp_s",  "logp_t", "feedback",    "kl_rev", "kl_fwd",
                                   "covered", "margin", "source",      "first_trans",
                                   "n_emit",  "next_driver", "new_len", "done"};

// Every helper returns a value and sets *ok = false with an exception set on
// failure; once *ok is false the later ones do nothing.
long long as_int(PyObject *o, bool *ok) {
  if (!*ok) return 0;
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) *ok = false;
  return v;
}

float as_float(PyObject *o, bool *ok) {
  if (!*ok) return 0.f;
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) *ok = false;
  return (float)v;
}

long long method_int(PyObject *o, PyObject *name, bool *ok) {
  if (!*ok) return 0;
  PyObject *r = PyObject_CallMethodNoArgs(o, name);
  if (!r) {
    *ok = false;
    return 0;
  }
  const unsigned long long v = PyLong_AsUnsignedLongLongMask(r);
  Py_DECREF(r);
  if (v == (unsigned long long)-1 && PyErr_Occurred()) *ok = false;
  return (long long)v;
}

template <typename T = void>
T *ptr(PyObject *o, bool *ok) {  // None is a null pointer
  if (!*ok || o == Py_None) return nullptr;
  return reinterpret_cast<T *>((uintptr_t)method_int(o, s_data_ptr, ok));
}

long long numel(PyObject *o, bool *ok) { return method_int(o, s_numel, ok); }

size_t nbytes(PyObject *o, bool *ok) {
  return (size_t)(numel(o, ok) * method_int(o, s_element_size, ok));
}

// the shape's n sizes; with `exact`, the tensor must have n dimensions
void sizes(PyObject *o, long long *out, Py_ssize_t n, bool exact, bool *ok) {
  if (!*ok) return;
  PyObject *s = PyObject_GetAttr(o, s_shape);
  if (!s) {
    *ok = false;
    return;
  }
  if (!PyTuple_Check(s) || PyTuple_GET_SIZE(s) < n || (exact && PyTuple_GET_SIZE(s) != n)) {
    PyErr_Format(PyExc_ValueError, "expected a tensor of %s%zd dimensions", exact ? "" : "at least ",
                 n);
    *ok = false;
  } else {
    for (Py_ssize_t i = 0; i < n; ++i) out[i] = as_int(PyTuple_GET_ITEM(s, i), ok);
  }
  Py_DECREF(s);
}

ipd_stream_t as_stream(PyObject *o, bool *ok) {
  return reinterpret_cast<ipd_stream_t>((uintptr_t)(o == Py_None ? 0 : as_int(o, ok)));
}

bool n_args(Py_ssize_t n, Py_ssize_t want) {
  if (n != want) PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return n == want;
}

#define IPD_CALL(st, expr)     \
  do {                         \
    Py_BEGIN_ALLOW_THREADS     \
    st = (expr);               \
    Py_END_ALLOW_THREADS       \
  } while (0)

// attn(verify, decode, scale, workspace, stream): sequences of objects whose
// attribute `c` holds an ipd_attn_batch.
Py_ssize_t batches(PyObject *seq, ipd_attn_batch *out, bool *ok) {
  if (!*ok || seq == Py_None) return 0;
  PyObject *f = PySequence_Fast(seq, "batches must be a sequence");
  if (!f) {
    *ok = false;
    return 0;
  }
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(f);
  for (Py_ssize_t i = 0; *ok && i < n && i < IPD_MAX_BATCHES; ++i) {
    PyObject *c = PyObject_GetAttr(PySequence_Fast_GET_ITEM(f, i), s_c);
    Py_buffer b;
    if (!c || PyObject_GetBuffer(c, &b, PyBUF_SIMPLE) != 0) {
      *ok = false;
    } else {
      if (b.len == (Py_ssize_t)sizeof(ipd_attn_batch)) {
        memcpy(&out[i], b.buf, sizeof(ipd_attn_batch));
      } else {
        PyErr_SetString(PyExc_TypeError, "not an attention batch");
        *ok = false;
      }
      PyBuffer_Release(&b);
    }
    Py_XDECREF(c);
  }
  Py_DECREF(f);
  return n;
}

PyObject *attn(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (!n_args(n, 5)) return nullptr;
  bool ok = true;
  ipd_attn_batch ver[IPD_MAX_BATCHES], dec[IPD_MAX_BATCHES];
  const Py_ssize_t nv = batches(a[0], ver, &ok), nd = batches(a[1], dec, &ok);
  const float scale = as_float(a[2], &ok);
  void *ws = ptr(a[3], &ok);
  const size_t wb = nbytes(a[3], &ok);
  const ipd_stream_t st = as_stream(a[4], &ok);
  if (!ok) return nullptr;
  int r = IPD_ERR_INVALID_ARG;  // (more batches than a call takes)
  if (nv + nd <= IPD_MAX_BATCHES)
    IPD_CALL(r, ipd_verify_attn(nv ? ver : nullptr, (int)nv, nd ? dec : nullptr, (int)nd, scale, ws,
                                wb, st));
  return PyLong_FromLong(r);
}

// score(kind, logits_student, logits_teacher, tokens, cu_span, driver,
// prefix_len, K, eos_id, max_span, out, ext, workspace, stream); kind 0:
// ipd_score_span, 1: _needed, 2: _ex (ext a tuple of its fields), 3: _static.
PyObject *score(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (!n_args(n, 14)) return nullptr;
  bool ok = true;
  const int kind = (int)as_int(a[0], &ok);
  const uint16_t *ls = ptr<uint16_t>(a[1], &ok), *lt = ptr<uint16_t>(a[2], &ok);
  const int32_t *tok = ptr<int32_t>(a[3], &ok), *cu = ptr<int32_t>(a[4], &ok);
  const uint8_t *drv = ptr<uint8_t>(a[5], &ok);
  const int32_t *pre = ptr<int32_t>(a[6], &ok);
  const int K = (int)as_int(a[7], &ok), eos = (int)as_int(a[8], &ok);
  const int max_span = (int)as_int(a[9], &ok);
  const int R = (int)numel(a[5], &ok);
  long long tv[2] = {0, 0};
  sizes(a[1], tv, 2, true, &ok);
  const int T = (int)tv[0], V = (int)tv[1];
  if (ok && !PyDict_Check(a[10])) {
    PyErr_SetString(PyExc_TypeError, "out must be a dict of tensors");
    ok = false;
  }
  void *o[13] = {};
  for (int i = 0; ok && i < 13; ++i) {
    PyObject *t = PyDict_GetItemWithError(a[10], s_out[i]);
    if (!t) {
      if (!PyErr_Occurred()) PyErr_SetObject(PyExc_KeyError, s_out[i]);
      ok = false;
    } else {
      o[i] = ptr(t, &ok);
    }
  }
  ipd_score_ext ext;
  memset(&ext, 0, sizeof(ext));
  if (ok && kind == 2) {
    if (!PyTuple_Check(a[11]) || PyTuple_GET_SIZE(a[11]) != 13) {
      PyErr_SetString(PyExc_TypeError, "ext must be a tuple of 13");
      ok = false;
    } else {
      PyObject *const e = a[11];
      auto at = [&](int i) { return PyTuple_GET_ITEM(e, i); };
      ext.takeover_rule = (int)as_int(at(0), &ok);
      ext.handback_rule = (int)as_int(at(1), &ok);
      ext.takeover_tau = as_float(at(2), &ok);
      ext.handback_tau = as_float(at(3), &ok);
      ext.entropy_s = ptr<float>(at(4), &ok);
      ext.entropy_t = ptr<float>(at(5), &ok);
      ext.topk_overlap = ptr<float>(at(6), &ok);
      ext.topk_s = ptr<int32_t>(at(7), &ok);
      ext.topk_t = ptr<int32_t>(at(8), &ok);
      ext.next_token = ptr<int32_t>(at(9), &ok);
      ext.draw_base = ptr<uint64_t>(at(10), &ok);
      if (ok) ext.sample_seed = PyLong_AsUnsignedLongLongMask(at(11));
      if (ok && ext.sample_seed == (uint64_t)-1 && PyErr_Occurred()) ok = false;
      ext.inv_temperature = as_float(at(12), &ok);
    }
  }
  void *ws = kind == 3 ? nullptr : ptr(a[12], &ok);
  const size_t wb = kind == 3 ? 0 : nbytes(a[12], &ok);
  const ipd_stream_t st = as_stream(a[13], &ok);
  if (!ok) return nullptr;
  float *lps = (float *)o[0], *lpt = (float *)o[1], *fb = (float *)o[2], *kr = (float *)o[3],
        *kf = (float *)o[4], *mar = (float *)o[6];
  uint8_t *cov = (uint8_t *)o[5], *src = (uint8_t *)o[7], *nd = (uint8_t *)o[10],
          *dn = (uint8_t *)o[12];
  int32_t *ft = (int32_t *)o[8], *ne = (int32_t *)o[9], *nl = (int32_t *)o[11];
  int r = IPD_ERR_INVALID_ARG;
  if (kind == 0)
    IPD_CALL(r, ipd_score_span(ls, lt, tok, cu, drv, pre, R, T, V, K, eos, lps, lpt, fb, kr, kf, cov,
                               mar, src, ft, ne, nd, nl, dn, ws, wb, st));
  else if (kind == 1)
    IPD_CALL(r, ipd_score_span_needed(ls, lt, tok, cu, drv, pre, R, T, V, K, eos, max_span, lps, lpt,
                                      fb, kr, kf, cov, mar, src, ft, ne, nd, nl, dn, ws, wb, st));
  else if (kind == 2)
    IPD_CALL(r, ipd_score_span_ex(ls, lt, tok, cu, drv, pre, R, T, V, K, eos, lps, lpt, fb, kr, kf,
                                  cov, mar, src, ft, ne, nd, nl, dn, &ext, ws, wb, st));
  else if (kind == 3)
    IPD_CALL(r, ipd_score_span_static(ls, lt, tok, cu, drv, pre, R, T, V, K, eos, lps, lpt, fb, kr,
                                      kf, cov, mar, src, ft, ne, nd, nl, dn, st));
  return PyLong_FromLong(r);
}

// split_loss(kl_rev, kl_fwd, source, cu_span, n_emit, resp_len, agg_mode,
// dir_mode, out8, stream)
PyObject *split_loss(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (!n_args(n, 10)) return nullptr;
  bool ok = true;
  const float *kr = ptr<float>(a[0], &ok), *kf = ptr<float>(a[1], &ok);
  const uint8_t *src = ptr<uint8_t>(a[2], &ok);
  const int32_t *cu = ptr<int32_t>(a[3], &ok), *ne = ptr<int32_t>(a[4], &ok),
                *rl = ptr<int32_t>(a[5], &ok);
  const int agg = (int)as_int(a[6], &ok), dir = (int)as_int(a[7], &ok);
  float *out8 = ptr<float>(a[8], &ok);
  const int R = (int)numel(a[3], &ok) - 1;
  const ipd_stream_t st = as_stream(a[9], &ok);
  if (!ok) return nullptr;
  int r;
  IPD_CALL(r, ipd_split_loss(kr, kf, src, cu, ne, rl, R, agg, dir, out8, nullptr, 0, st));
  return PyLong_FromLong(r);
}

// split_loss_grad(logits_student, logits_teacher, topk_s, topk_t, source,
// cu_span, n_emit, resp_len, loss_out8, K, agg_mode, dir_mode, grad_scale,
// grad_idx, grad_val, grad_dense, dense_dtype, stream)
PyObject *split_loss_grad(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (!n_args(n, 18)) return nullptr;
  bool ok = true;
  const uint16_t *ls = ptr<uint16_t>(a[0], &ok), *lt = ptr<uint16_t>(a[1], &ok);
  const int32_t *ks = ptr<int32_t>(a[2], &ok), *kt = ptr<int32_t>(a[3], &ok);
  const uint8_t *src = ptr<uint8_t>(a[4], &ok);
  const int32_t *cu = ptr<int32_t>(a[5], &ok), *ne = ptr<int32_t>(a[6], &ok),
                *rl = ptr<int32_t>(a[7], &ok);
  const float *out8 = ptr<float>(a[8], &ok);
  const int K = (int)as_int(a[9], &ok), agg = (int)as_int(a[10], &ok),
            dir = (int)as_int(a[11], &ok);
  const float scale = as_float(a[12], &ok);
  int32_t *gi = ptr<int32_t>(a[13], &ok);
  float *gv = ptr<float>(a[14], &ok);
  void *dense = ptr(a[15], &ok);
  const int dtype = (int)as_int(a[16], &ok);
  const int R = (int)numel(a[5], &ok) - 1;
  long long tv[2] = {0, 0};
  sizes(a[0], tv, 2, true, &ok);
  const ipd_stream_t st = as_stream(a[17], &ok);
  if (!ok) return nullptr;
  int r;
  IPD_CALL(r, ipd_split_loss_grad(ls, lt, ks, kt, src, cu, ne, rl, out8, R, (int)tv[0], (int)tv[1],
                                  K, agg, dir, scale, gi, gv, dense, dtype, nullptr, 0, st));
  return PyLong_FromLong(r);
}

// full_kl(logits_student, logits_teacher, kl_rev_full, kl_fwd_full, stream)
PyObject *full_kl(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (!n_args(n, 5)) return nullptr;
  bool ok = true;
  const uint16_t *ls = ptr<uint16_t>(a[0], &ok), *lt = ptr<uint16_t>(a[1], &ok);
  float *rev = ptr<float>(a[2], &ok), *fwd = ptr<float>(a[3], &ok);
  long long tv[2] = {0, 0};
  sizes(a[0], tv, 2, true, &ok);
  const ipd_stream_t st = as_stream(a[4], &ok);
  if (!ok) return nullptr;
  int r;
  IPD_CALL(r, ipd_full_kl(ls, lt, (int)tv[0], (int)tv[1], rev, fwd, st));
  return PyLong_FromLong(r);
}

// sample(logits, seed, draw_id, tokens, workspace, inv_temperature, stream)
PyObject *sample(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (!n_args(n, 7)) return nullptr;
  bool ok = true;
  const uint16_t *l = ptr<uint16_t>(a[0], &ok);
  const unsigned long long seed = PyLong_AsUnsignedLongLongMask(a[1]);
  if (seed == (unsigned long long)-1 && PyErr_Occurred()) return nullptr;
  const uint64_t *draw = ptr<uint64_t>(a[2], &ok);
  int32_t *tok = ptr<int32_t>(a[3], &ok);
  void *ws = ptr(a[4], &ok);
  const size_t wb = nbytes(a[4], &ok);
  const float inv_t = as_float(a[5], &ok);
  long long nv[2] = {0, 0};
  sizes(a[0], nv, 2, true, &ok);
  const ipd_stream_t st = as_stream(a[6], &ok);
  if (!ok) return nullptr;
  int r;
  IPD_CALL(r, ipd_sample(l, (int)nv[0], (int)nv[1], seed, draw, inv_t, tok, ws, wb, st));
  return PyLong_FromLong(r);
}

// kv_append_many(appends, stream): tuples (cache, k_new, v_new, cu_new,
// seq_len, page_table)
PyObject *kv_append_many(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (!n_args(n, 2)) return nullptr;
  bool ok = true;
  PyObject *f = PySequence_Fast(a[0], "appends must be a sequence");
  if (!f) return nullptr;
  ipd_kv_append_desc d[IPD_MAX_BATCHES];
  const Py_ssize_t m = PySequence_Fast_GET_SIZE(f);
  for (Py_ssize_t i = 0; ok && i < m && i < IPD_MAX_BATCHES; ++i) {
    PyObject *t = PySequence_Fast(PySequence_Fast_GET_ITEM(f, i), "an append is a tuple");
    if (!t || PySequence_Fast_GET_SIZE(t) != 6) {
      if (t) PyErr_SetString(PyExc_ValueError, "an append has six members");
      Py_XDECREF(t);
      ok = false;
      break;
    }
    PyObject *const *e = PySequence_Fast_ITEMS(t);
    PyObject *kp = PyObject_GetAttr(e[0], s_k_pages), *vp = PyObject_GetAttr(e[0], s_v_pages);
    if (!kp || !vp) ok = false;
    long long ps[2] = {0, 0}, pt[2] = {0, 0}, kn[1] = {0};
    memset(&d[i], 0, sizeof(d[i]));
    if (ok) {
      d[i].k_pages = ptr<uint16_t>(kp, &ok);
      d[i].v_pages = ptr<uint16_t>(vp, &ok);
      sizes(kp, ps, 2, false, &ok);
      d[i].num_pages = ps[0];
      d[i].num_kv_heads = (int)ps[1];
      d[i].page_size = 16;
      d[i].head_dim = 128;
      d[i].k_new = ptr<uint16_t>(e[1], &ok);
      d[i].v_new = ptr<uint16_t>(e[2], &ok);
      d[i].cu_new = ptr<int32_t>(e[3], &ok);
      d[i].seq_len = ptr<int32_t>(e[4], &ok);
      d[i].page_table = ptr<int32_t>(e[5], &ok);
      sizes(e[5], pt, 2, false, &ok);
      d[i].max_pages = (int)pt[1];
      d[i].num_reqs = (int)numel(e[3], &ok) - 1;
      sizes(e[1], kn, 1, false, &ok);
      d[i].total_new = (int)kn[0];
    }
    Py_XDECREF(kp);
    Py_XDECREF(vp);
    Py_DECREF(t);
  }
  Py_DECREF(f);
  const ipd_stream_t st = as_stream(a[1], &ok);
  if (!ok) return nullptr;
  int r = IPD_ERR_INVALID_ARG;  // (more appends than a call takes)
  if (m <= IPD_MAX_BATCHES) IPD_CALL(r, ipd_kv_append_many(d, (int)m, st));
  return PyLong_FromLong(r);
}

#define IPD_FN(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {IPD_FN(attn),    IPD_FN(score),  IPD_FN(split_loss),
                         IPD_FN(split_loss_grad), IPD_FN(full_kl), IPD_FN(sample),
                         IPD_FN(kv_append_many), {nullptr, nullptr, 0, nullptr}};

PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_ipd_native",
                          "Argument marshalling of libipd.so's calls.", -1, methods,
                          nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__ipd_native() {
  struct {
    PyObject **where;
    const char *name;
  } const names[] = {{&s_data_ptr, "data_ptr"}, {&s_numel, "numel"},
                     {&s_element_size, "element_size"}, {&s_shape, "shape"}, {&s_c, "c"},
                     {&s_k_pages, "k_pages"}, {&s_v_pages, "v_pages"}};
  for (const auto &x : names)
    if (!(*x.where = PyUnicode_InternFromString(x.name))) return nullptr;
  for (int i = 0; i < 13; ++i)
    if (!(s_out[i] = PyUnicode_InternFromString(kOutNames[i]))) return nullptr;
  return PyModule_Create(&module_def);
}
