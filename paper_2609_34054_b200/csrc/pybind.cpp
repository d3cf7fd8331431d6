// CPython side of the binding: turns torch tensors into the C-ABI arguments of libprecc.
//
// Host path of one call.  The kernels of a decode step run for 4-10 us, and marshalling through ctypes (a dozen tensor
// attribute look-ups in Python, a dozen argument conversions, the stream look-up) took 7-8 us of a 11 us call: the GPU
// waited for the host.  Here the same work is a few hundred nanoseconds: tensors are unpacked in place, the current
// stream comes from c10, and the descriptor structures are built on the stack.  Nothing is kept from one call to
// the next.  The GIL is released around the library call, as ctypes does.
//
// torch throws C++ exceptions (a tensor without storage, a layout without strides), which must not reach the interpreter's C
// frames: every entry point runs inside `guarded`, dimensions are checked before a size is read, and pointers and sizes
// are taken while the GIL is held.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include "../../include/precc.h"

namespace {

PyObject* g_error = nullptr;   // binding.PreccError
PyObject* g_cache = nullptr;   // binding.Cache
PyObject *s_desc, *s_k_base, *s_v_base, *s_lr_k, *s_lr_v, *s_n_blocks;

// One call's arguments, taken in order; the first problem sets the Python error and makes the rest no-ops.
struct Args {
  PyObject* const* at;
  bool ok;
  Args(PyObject* const* a, Py_ssize_t n, Py_ssize_t want) : at(a), ok(n == want) {
    if (!ok) PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  }
  PyObject* next() { return *at++; }
  void bad(const char* what) { if (ok) { PyErr_SetString(g_error, what); ok = false; } }

  uint64_t u64() {
    PyObject* o = next();
    if (!ok) return 0;
    if (PyLong_CheckExact(o)) return PyLong_AsUnsignedLongLongMask(o);
    PyObject* i = PyNumber_Index(o);
    if (!i) { ok = false; return 0; }
    const uint64_t v = PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    return v;
  }
  int64_t i64() { return static_cast<int64_t>(u64()); }
  int32_t i32() { return static_cast<int32_t>(u64()); }
  precc_ctx* ctx() { return reinterpret_cast<precc_ctx*>(static_cast<uintptr_t>(u64())); }

  // A tensor argument that may be None.
  const at::Tensor* tensor(PyObject* o) {
    if (!ok || o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) { bad("tensor must be a contiguous CUDA tensor"); return nullptr; }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) { bad("tensor must be a contiguous CUDA tensor"); return nullptr; }
    return &t;
  }
  const at::Tensor* tensor() { return tensor(next()); }
  const at::Tensor* required(const char* name) {
    const at::Tensor* t = tensor();
    if (ok && !t) { PyErr_Format(g_error, "%s is None", name); ok = false; }
    return t;
  }
  const at::Tensor* typed(c10::ScalarType type, const char* what) {
    const at::Tensor* t = tensor();
    if (t && t->scalar_type() != type) bad(what);
    return t;
  }
  static void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
  void* tptr() { return ptr(tensor()); }
  // A required tensor of which the library wants the address and the first extent.
  struct Rows { void* p; int32_t n; };
  Rows rows_of(const char* name) {
    const at::Tensor* t = required(name);
    if (t && t->dim() < 1) { PyErr_Format(g_error, "%s has no dimensions", name); ok = false; }
    return ok ? Rows{t->data_ptr(), static_cast<int32_t>(t->size(0))} : Rows{nullptr, 0};
  }
  // Block table or None: [B][stride] for decode (`per_request`), the sequence's own entries for prefill.
  struct Table { const int32_t* p; int32_t n; };
  Table table(bool per_request) {
    const at::Tensor* t = tensor();
    if (t && per_request && t->dim() < 2) bad("block_table must be [B][blocks per request]");
    if (!ok || !t) return {nullptr, 0};
    return {static_cast<const int32_t*>(t->data_ptr()), static_cast<int32_t>(per_request ? t->size(1) : t->numel())};
  }
  // Address and extent of a scratch buffer that may be None.
  struct Buffer { void* p; size_t elements, bytes; };
  Buffer buffer(const at::Tensor* t) {
    if (!ok || !t) return {nullptr, 0, 0};
    const size_t n = static_cast<size_t>(t->numel());
    return {t->data_ptr(), n, n * t->element_size()};
  }

  // LayerDesc (a ctypes structure), copied.
  precc_layer_desc desc() {
    precc_layer_desc d = {};
    copy(next(), &d, sizeof(d), "desc is not a LayerDesc");
    return d;
  }
  void copy(PyObject* o, void* to, size_t n, const char* what) {
    Py_buffer v;
    if (!ok) return;
    if (PyObject_GetBuffer(o, &v, PyBUF_SIMPLE) != 0) { ok = false; return; }
    if (v.len == static_cast<Py_ssize_t>(n)) memcpy(to, v.buf, n);
    else bad(what);
    PyBuffer_Release(&v);
  }
  void* member(PyObject* o, PyObject* name) {
    THPObjectPtr m(ok ? PyObject_GetAttr(o, name) : nullptr);   // (the cache object still holds it afterwards)
    if (!m) { ok = false; return nullptr; }
    return ptr(tensor(m));
  }
  // A Cache is read member by member; any other object (a subclass, a view with a layout of its own) is asked for its desc().
  precc_cache cache() {
    precc_cache c = {};
    PyObject* o = next();
    if (!ok) return c;
    if (reinterpret_cast<PyObject*>(Py_TYPE(o)) != g_cache) {
      THPObjectPtr d(PyObject_CallMethodNoArgs(o, s_desc));
      if (!d) { ok = false; return c; }
      copy(d, &c, sizeof(c), "cache.desc() is not a CacheDesc");
      return c;
    }
    c.k_base = member(o, s_k_base);
    c.v_base = member(o, s_v_base);
    c.lr_k = member(o, s_lr_k);
    c.lr_v = member(o, s_lr_v);
    THPObjectPtr n(ok ? PyObject_GetAttr(o, s_n_blocks) : nullptr);
    if (!n) { ok = false; return c; }
    c.n_blocks = PyLong_AsLongLong(n);
    if (c.n_blocks == -1 && PyErr_Occurred()) ok = false;
    return c;
  }
  // Rotary table fp32 [max_pos][hd/2][2], optionally followed by (positions, start_pos).
  precc_rope rope(bool with_positions) {
    precc_rope r = {};
    const at::Tensor* t = required("rope table");
    if (ok && (t->scalar_type() != at::kFloat || t->dim() != 3 || t->size(2) != 2)) bad("rope table must be fp32 [max_pos][hd/2][2]");
    if (ok) { r.table = static_cast<const float*>(t->data_ptr()); r.max_pos = static_cast<int32_t>(t->size(0)); }
    if (with_positions) {
      r.positions = static_cast<const int32_t*>(tptr());
      r.start_pos = i64();
    }
    return r;
  }
};

const int32_t* i32p(const at::Tensor* t) { return static_cast<const int32_t*>(Args::ptr(t)); }

struct GilRelease {        // (an object, so that an exception on the way leaves with the GIL held)
  PyThreadState* state = PyEval_SaveThread();
  ~GilRelease() { PyEval_RestoreThread(state); }
};

template <typename F>
PyObject* finish(precc_ctx* ctx, const char* what, F&& call) {
  void* stream = c10::cuda::getCurrentCUDAStream().stream();
  int32_t rc;
  {
    GilRelease unlocked;
    rc = call(stream);
  }
  if (rc == PRECC_OK) Py_RETURN_NONE;
  PyErr_Format(g_error, "%s: %s: %s", what, precc_error_name(rc), precc_last_error(ctx));
  return nullptr;
}

#define NATIVE(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs)

// ------------------------------------------------------------------------------------------------ projections
NATIVE(lr_precompute) {
  Args a(args, nargs, 8);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows H = a.rows_of("H");
  void* A = a.tptr();
  const precc_cache c = a.cache();
  const int64_t start = a.i64();
  const int32_t* slots = i32p(a.tensor());
  const uint64_t mask = a.u64();
  if (!a.ok) return nullptr;
  return finish(ctx, "precc_lr_precompute", [&](void* st) {
    return precc_lr_precompute(ctx, &d, H.p, H.n, A, slots, start, mask, &c, st); });
}

NATIVE(turn_project) {
  Args a(args, nargs, 8);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows H = a.rows_of("H");
  void* WA = a.tptr();
  const precc_cache c = a.cache();
  const int64_t start = a.i64();
  const int32_t* slots = i32p(a.tensor());
  const uint64_t mask = a.u64();
  if (!a.ok) return nullptr;
  return finish(ctx, "precc_turn_project", [&](void* st) {
    return precc_turn_project(ctx, &d, H.p, H.n, WA, slots, start, mask, &c, st); });
}

NATIVE(turn_project_rows) {
  Args a(args, nargs, 8);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows H = a.rows_of("H");
  void* WA = a.tptr();
  const precc_cache c = a.cache();
  const int32_t* slots = i32p(a.tensor());
  const uint64_t* masks = static_cast<const uint64_t*>(Args::ptr(a.typed(at::kLong, "row_masks must be int64 (bit patterns of uint64 masks)")));
  const int32_t* copies = i32p(a.typed(at::kInt, "lr_copy_slots must be int32"));
  if (!a.ok) return nullptr;
  return finish(ctx, "precc_turn_project_rows", [&](void* st) {
    return precc_turn_project_rows(ctx, &d, H.p, H.n, WA, slots, masks, copies, &c, st); });
}

NATIVE(rebase_project) {
  Args a(args, nargs, 7);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows H = a.rows_of("H");
  void* W = a.tptr();
  const precc_cache c = a.cache();
  const int64_t start = a.i64();
  const int32_t* slots = i32p(a.tensor());
  if (!a.ok) return nullptr;
  return finish(ctx, "precc_rebase_project", [&](void* st) {
    return precc_rebase_project(ctx, &d, H.p, H.n, W, slots, start, &c, st); });
}

NATIVE(rebase_project_rope) {
  Args a(args, nargs, 10);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows H = a.rows_of("H");
  void* W = a.tptr();
  const precc_cache c = a.cache();
  const precc_rope r = a.rope(true);
  const int64_t start = a.i64();
  const int32_t* slots = i32p(a.tensor());
  if (!a.ok) return nullptr;
  return finish(ctx, "precc_rebase_project_rope", [&](void* st) {
    return precc_rebase_project_rope(ctx, &d, H.p, H.n, W, slots, start, &r, &c, st); });
}

NATIVE(turn_project_rope) {
  Args a(args, nargs, 11);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows H = a.rows_of("H");
  void* WA = a.tptr();
  const precc_cache c = a.cache();
  const precc_rope r = a.rope(true);
  const int64_t start = a.i64();
  const int32_t* slots = i32p(a.tensor());
  const uint64_t mask = a.u64();
  if (!a.ok) return nullptr;
  return finish(ctx, "precc_turn_project_rope", [&](void* st) {
    return precc_turn_project_rope(ctx, &d, H.p, H.n, WA, slots, start, mask, &r, &c, st); });
}

// ------------------------------------------------------------------------------------------------ decode
// (ctx, desc, q, agent_id, ctx_len, max_ctx, B_k, B_v, [rope,] cache, out, [workspace,] block_table, first_block)
enum DecodeForm { PLAIN, ROPE, STATIC };
template <DecodeForm FORM>
NATIVE(decode) {
  Args a(args, nargs, FORM == ROPE ? 14 : FORM == PLAIN ? 13 : 12);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows q = a.rows_of("q");
  const int32_t* agent = i32p(a.tensor());
  const int32_t* len = i32p(a.tensor());
  const int32_t max_ctx = a.i32();
  void* Bk = a.tptr();
  void* Bv = a.tptr();
  precc_rope r = {};
  if (FORM == ROPE) r = a.rope(false);
  const precc_cache c = a.cache();
  void* out = a.tptr();
  const Args::Buffer ws = a.buffer(FORM == STATIC ? nullptr : a.required("workspace"));
  const Args::Table table = a.table(true);
  const int32_t* first = i32p(a.tensor());
  if (!a.ok) return nullptr;
  const char* what = FORM == ROPE ? "precc_lr_attend_decode_rope" : FORM == PLAIN ? "precc_lr_attend_decode" : "precc_lr_attend_decode_static";
  return finish(ctx, what, [&](void* st) {
    if (FORM == STATIC)
      return precc_lr_attend_decode_static(ctx, &d, q.p, q.n, agent, len, table.p, table.n, first, max_ctx,
                                           Bk, Bv, &c, out, st);
    if (FORM == ROPE)
      return precc_lr_attend_decode_rope(ctx, &d, q.p, q.n, agent, len, table.p, table.n, first, max_ctx,
                                         Bk, Bv, &r, &c, out, ws.p, ws.elements, st);
    return precc_lr_attend_decode(ctx, &d, q.p, q.n, agent, len, table.p, table.n, first, max_ctx, Bk, Bv,
                                  &c, out, ws.p, ws.elements, st); });
}

NATIVE(decode_partial) {
  Args a(args, nargs, 12);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows q = a.rows_of("q");
  const int32_t* agent = i32p(a.tensor());
  const int32_t* len = i32p(a.tensor());
  const int32_t max_ctx = a.i32();
  void* Bk = a.tptr();
  const precc_cache c = a.cache();
  float* records = static_cast<float*>(Args::ptr(a.typed(at::kFloat, "records must be fp32")));
  const Args::Buffer ws = a.buffer(a.required("workspace"));
  const Args::Table table = a.table(true);
  const int32_t* first = i32p(a.tensor());
  if (!a.ok) return nullptr;
  return finish(ctx, "precc_lr_attend_decode_partial", [&](void* st) {
    return precc_lr_attend_decode_partial(ctx, &d, q.p, q.n, agent, len, table.p, table.n, first, max_ctx,
                                          Bk, &c, records, ws.p, ws.elements, st); });
}

NATIVE(combine_partials) {
  Args a(args, nargs, 6);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows records = a.rows_of("records");
  const int32_t* agent = i32p(a.tensor());
  void* Bv = a.tptr();
  const Args::Rows out = a.rows_of("out");
  if (!a.ok) return nullptr;
  return finish(ctx, "precc_combine_partials", [&](void* st) {
    return precc_combine_partials(ctx, &d, static_cast<const float*>(records.p), records.n, out.n, agent, Bv, out.p, st); });
}

// ------------------------------------------------------------------------------------------------ prefill
// (ctx, desc, q, agent, ctx_len, B_k, B_v, [rope,] cache, out, [workspace or key scratch,] block_table, first_block)
enum PrefillForm { PF_PLAIN, PF_WS, PF_ROPE, PF_SCRATCH };
template <PrefillForm FORM>
NATIVE(prefill) {
  Args a(args, nargs, FORM == PF_PLAIN ? 11 : FORM == PF_SCRATCH ? 13 : 12);
  if (!a.ok) return nullptr;
  precc_ctx* ctx = a.ctx();
  const precc_layer_desc d = a.desc();
  const Args::Rows q = a.rows_of("q");
  const int32_t agent = a.i32(), T = a.i32();
  void* Bk = a.tptr();
  void* Bv = a.tptr();
  precc_rope r = {};
  if (FORM == PF_ROPE || FORM == PF_SCRATCH) r = a.rope(false);
  const precc_cache c = a.cache();
  void* out = a.tptr();
  const Args::Buffer extra = a.buffer(FORM == PF_WS ? a.tensor() : FORM == PF_SCRATCH ? a.required("key_scratch") : nullptr);
  const Args::Table table = a.table(false);
  const int32_t first = a.i32();
  if (!a.ok) return nullptr;
  const char* what = FORM == PF_PLAIN ? "precc_lr_attend_prefill" : FORM == PF_WS ? "precc_lr_attend_prefill_ws" :
                     FORM == PF_ROPE ? "precc_lr_attend_prefill_rope" : "precc_lr_attend_prefill_rope_scratch";
  return finish(ctx, what, [&](void* st) {
    switch (FORM) {
      case PF_WS:
        return precc_lr_attend_prefill_ws(ctx, &d, q.p, q.n, agent, T, table.p, table.n, first, Bk, Bv, &c, out,
                                          extra.p, extra.bytes, st);
      case PF_ROPE:
        return precc_lr_attend_prefill_rope(ctx, &d, q.p, q.n, agent, T, table.p, table.n, first, Bk, Bv, &r, &c, out, st);
      case PF_SCRATCH:
        return precc_lr_attend_prefill_rope_scratch(ctx, &d, q.p, q.n, agent, T, table.p, table.n, first, Bk, Bv, &r,
                                                    &c, out, extra.p, extra.bytes, st);
      default:
        return precc_lr_attend_prefill(ctx, &d, q.p, q.n, agent, T, table.p, table.n, first, Bk, Bv, &c, out, st);
    }
  });
}

// (error class, cache class) of binding.py
PyObject* set_types(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != 2) { PyErr_SetString(PyExc_TypeError, "set_types(error, cache)"); return nullptr; }
  Py_XSETREF(g_error, Py_NewRef(args[0]));
  Py_XSETREF(g_cache, Py_NewRef(args[1]));
  Py_RETURN_NONE;
}

// Entry point as the interpreter sees it: C++ exceptions become Python errors (the GIL is held wherever they arrive here).
using Entry = PyObject* (*)(PyObject*, PyObject* const*, Py_ssize_t);
template <Entry FN>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
  try {
    return FN(self, args, nargs);
  } catch (python_error& e) {
    e.restore();
  } catch (const c10::Error& e) {
    PyErr_SetString(g_error, e.what_without_backtrace());
  } catch (const std::exception& e) {
    PyErr_SetString(g_error, e.what());
  } catch (...) {
    PyErr_SetString(g_error, "unknown C++ exception");
  }
  return nullptr;
}

#define FAST(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(&guarded<fn>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST("set_types", set_types),
    FAST("lr_precompute", lr_precompute), FAST("rebase_project", rebase_project), FAST("turn_project", turn_project),
    FAST("turn_project_rows", turn_project_rows), FAST("rebase_project_rope", rebase_project_rope),
    FAST("turn_project_rope", turn_project_rope),
    FAST("lr_attend_decode", decode<PLAIN>), FAST("lr_attend_decode_rope", decode<ROPE>), FAST("lr_attend_decode_static", decode<STATIC>),
    FAST("lr_attend_decode_partial", decode_partial), FAST("combine_partials", combine_partials),
    FAST("lr_attend_prefill", prefill<PF_PLAIN>), FAST("lr_attend_prefill_ws", prefill<PF_WS>),
    FAST("lr_attend_prefill_rope", prefill<PF_ROPE>), FAST("lr_attend_prefill_rope_scratch", prefill<PF_SCRATCH>),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling of the precc calls.", -1, methods,
                          nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  s_desc = PyUnicode_InternFromString("desc");
  s_k_base = PyUnicode_InternFromString("k_base");
  s_v_base = PyUnicode_InternFromString("v_base");
  s_lr_k = PyUnicode_InternFromString("lr_k");
  s_lr_v = PyUnicode_InternFromString("lr_v");
  s_n_blocks = PyUnicode_InternFromString("n_blocks");
  Py_INCREF(PyExc_RuntimeError);
  g_error = PyExc_RuntimeError;
  return PyModule_Create(&module_def);
}
