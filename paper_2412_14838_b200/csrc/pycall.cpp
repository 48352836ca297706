// Native half of binding.py: turns the arguments of the calls a serving loop makes (torch tensors, numpy arrays,
// integer addresses, lists of them, streams) into the C ABI's pointers and makes the call without the GIL.
//
// Why it exists: a decoding step calls the library once per layer and a pass hands over five lists of per-layer
// tensors.  Taking every address through Python attribute look-ups and ctypes arrays costs about 0.3 us a tensor and
// 8 us a call (a 32-layer dkv_decode_attend: 40 us on the host for a kernel of a third of that); here a tensor's
// address is a field read.  Every function returns the library's code; binding.py raises on it.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>

#include "../../include/dkv.h"

namespace {

constexpr Py_ssize_t kMaxList = 4096;       // longest list of per-layer tensors taken

// Address of a torch tensor, an integer, None (NULL), or of anything with data_ptr() (a tensor subclass may have its own)
// or a numpy-like .ctypes.data.
bool address(PyObject* x, void** out) {
  if (x == Py_None) { *out = nullptr; return true; }
  if (THPVariable_CheckExact(x)) { *out = THPVariable_Unpack(x).data_ptr(); return true; }
  PyObject* v = nullptr;
  if (PyLong_Check(x)) {
    v = x;
    Py_INCREF(v);
  } else if (PyObject_HasAttrString(x, "data_ptr")) {
    v = PyObject_CallMethod(x, "data_ptr", nullptr);
  } else if (PyObject_HasAttrString(x, "ctypes")) {
    PyObject* c = PyObject_GetAttrString(x, "ctypes");
    if (c) { v = PyObject_GetAttrString(c, "data"); Py_DECREF(c); }
  } else {
    PyErr_Format(PyExc_TypeError, "cannot take the address of %R", (PyObject*)Py_TYPE(x));
  }
  if (!v) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

// None: torch's current stream; an integer: a cudaStream_t; else an object with .cuda_stream.
bool stream_of(PyObject* x, void** out) {
  if (x == Py_None) { *out = (void*)c10::cuda::getCurrentCUDAStream().stream(); return true; }
  if (PyLong_Check(x)) { *out = PyLong_AsVoidPtr(x); return !PyErr_Occurred(); }
  PyObject* v = PyObject_GetAttrString(x, "cuda_stream");
  if (!v) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

// The addresses of a sequence's items.  The library reads one address a layer, whatever the length of the list: there
// are never fewer than DKV_MAX_LAYERS entries, and a list that is too short ends in NULLs, which the library refuses.
struct Addresses {
  void* few[DKV_MAX_LAYERS] = {};
  void** p = few;
  PyObject* items = nullptr;
  ~Addresses() {
    if (p != few) PyMem_Free(p);
    Py_XDECREF(items);
  }
  bool take(PyObject* seq) {
    items = PySequence_Fast(seq, "a sequence of tensors or addresses is expected");
    if (!items) return false;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(items);
    if (n > kMaxList) { PyErr_SetString(PyExc_ValueError, "too many tensors"); return false; }
    if (n > DKV_MAX_LAYERS) {
      void** more = static_cast<void**>(PyMem_Malloc(sizeof(void*) * n));
      if (!more) { PyErr_NoMemory(); return false; }
      p = more;
    }
    for (Py_ssize_t i = 0; i < n && i < PySequence_Fast_GET_SIZE(items); ++i)      // (an item's own code may shorten its list)
      if (!address(PySequence_Fast_GET_ITEM(items, i), &p[i])) return false;
    return true;
  }
};

// A 32-bit integer; one that does not fit is refused rather than cut to another layer or count.
bool number(PyObject* x, int32_t* out) {
  const long v = PyLong_AsLong(x);
  if (v == -1 && PyErr_Occurred()) return false;
  if (v != (int32_t)v) { PyErr_SetString(PyExc_OverflowError, "an integer does not fit 32 bits"); return false; }
  *out = (int32_t)v;
  return true;
}

// Every function: `n` arguments exactly, conversions by the lines given, then the call without the GIL.
#define DKV_PY(NAME, N, CONVERT, CALL)                                                        \
  PyObject* py_##NAME(PyObject*, PyObject* const* a, Py_ssize_t n) {                          \
    if (n != (N)) { PyErr_SetString(PyExc_TypeError, #NAME ": wrong number of arguments"); return nullptr; } \
    try {                                                                                     \
      CONVERT                                                                                 \
      int rc;                                                                                 \
      Py_BEGIN_ALLOW_THREADS                                                                  \
      rc = CALL;                                                                              \
      Py_END_ALLOW_THREADS                                                                    \
      return PyLong_FromLong(rc);                                                             \
    } catch (const std::exception& e) {                                                       \
      PyErr_SetString(PyExc_RuntimeError, e.what());                                          \
      return nullptr;                                                                         \
    }                                                                                         \
  }
#define CTX(I) void* cp_; if (!address(a[I], &cp_)) return nullptr; dkv_ctx* c = static_cast<dkv_ctx*>(cp_);
#define INT(V, I) int32_t V; if (!number(a[I], &V)) return nullptr;
#define PTR(V, I) void* V; if (!address(a[I], &V)) return nullptr;
#define SIZE(V, I) const uint64_t V = PyLong_AsUnsignedLongLong(a[I]); if (PyErr_Occurred()) return nullptr;
#define STREAM(I) void* st; if (!stream_of(a[I], &st)) return nullptr;
#define LIST(V, I) Addresses V; if (!V.take(a[I])) return nullptr;

DKV_PY(reset, 2, CTX(0) STREAM(1), dkv_reset(c, st))
DKV_PY(score, 6, CTX(0) INT(l, 1) PTR(q, 2) PTR(k, 3) PTR(o, 4) STREAM(5), dkv_score(c, l, q, k, (float*)o, st))
DKV_PY(score_lse, 7, CTX(0) INT(l, 1) PTR(q, 2) PTR(k, 3) PTR(e, 4) PTR(o, 5) STREAM(6),
       dkv_score_lse(c, l, q, k, (const float*)e, (float*)o, st))
DKV_PY(score_static, 5, PTR(cfg, 0) PTR(q, 1) PTR(k, 2) PTR(o, 3) STREAM(4),
       dkv_score_static((const dkv_config*)cfg, q, k, (float*)o, st))
DKV_PY(set_scores, 4, CTX(0) INT(l, 1) PTR(s, 2) STREAM(3), dkv_set_scores(c, l, (const float*)s, st))
DKV_PY(select_topk, 5, CTX(0) INT(l, 1) PTR(i, 2) PTR(r, 3) STREAM(4), dkv_select_topk(c, l, (int32_t*)i, (int32_t*)r, st))
DKV_PY(rebudget, 4, CTX(0) INT(l, 1) PTR(o, 2) STREAM(3), dkv_rebudget(c, l, (int32_t*)o, st))
DKV_PY(compact, 8, CTX(0) INT(l, 1) PTR(ks, 2) PTR(vs, 3) PTR(kb, 4) PTR(vb, 5) PTR(len, 6) STREAM(7),
       dkv_compact(c, l, ks, vs, kb, vb, (int32_t*)len, st))
DKV_PY(compact_all, 5, CTX(0) INT(l, 1) LIST(kb, 2) LIST(vb, 3) STREAM(4), dkv_compact_all(c, l, kb.p, vb.p, st))
DKV_PY(run_prefill_pass, 7, CTX(0) LIST(q, 1) LIST(k, 2) LIST(v, 3) LIST(kb, 4) LIST(vb, 5) STREAM(6),
       dkv_run_prefill_pass(c, q.p, k.p, v.p, kb.p, vb.p, st))
DKV_PY(run_prefill_pass_lse, 8, CTX(0) LIST(q, 1) LIST(k, 2) LIST(v, 3) LIST(e, 4) LIST(kb, 5) LIST(vb, 6) STREAM(7),
       dkv_run_prefill_pass_lse(c, q.p, k.p, v.p, (const float* const*)e.p, kb.p, vb.p, st))
DKV_PY(run_prefill_pass_host, 7, CTX(0) LIST(q, 1) LIST(k, 2) LIST(v, 3) LIST(kb, 4) LIST(vb, 5) PTR(o, 6),
       dkv_run_prefill_pass_host(c, q.p, k.p, v.p, kb.p, vb.p, (int32_t*)o))
DKV_PY(apply_policy, 4, CTX(0) INT(p, 1) PTR(o, 2) STREAM(3), dkv_apply_policy(c, p, (int32_t*)o, st))
DKV_PY(select_positions, 5, CTX(0) INT(l, 1) INT(s, 2) INT(r, 3) STREAM(4), dkv_select_positions(c, l, s, r, st))
DKV_PY(decode_attend, 9, CTX(0) INT(l, 1) INT(nl, 2) INT(nq, 3) LIST(q, 4) LIST(kb, 5) LIST(vb, 6) LIST(o, 7) STREAM(8),
       dkv_decode_attend(c, l, nl, nq, q.p, kb.p, vb.p, (float* const*)o.p, st))
DKV_PY(get_counts, 3, CTX(0) PTR(o, 1) STREAM(2), dkv_get_counts(c, (int32_t*)o, st))
DKV_PY(memcpy_to_host, 5, CTX(0) PTR(dst, 1) PTR(src, 2) SIZE(bytes, 3) STREAM(4), dkv_memcpy_to_host(c, dst, src, bytes, st))
DKV_PY(kept_sorted, 4, CTX(0) INT(l, 1) PTR(o, 2) STREAM(3), dkv_kept_sorted(c, l, (int32_t*)o, st))

#define ENTRY(NAME) {#NAME, (PyCFunction)(void*)py_##NAME, METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    ENTRY(reset), ENTRY(score), ENTRY(score_lse), ENTRY(score_static), ENTRY(set_scores), ENTRY(select_topk),
    ENTRY(rebudget), ENTRY(compact), ENTRY(compact_all), ENTRY(run_prefill_pass), ENTRY(run_prefill_pass_lse),
    ENTRY(run_prefill_pass_host), ENTRY(apply_policy), ENTRY(select_positions), ENTRY(decode_attend),
    ENTRY(get_counts), ENTRY(kept_sorted), ENTRY(memcpy_to_host), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_dkv_pycall", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__dkv_pycall(void) { return PyModule_Create(&kModule); }
