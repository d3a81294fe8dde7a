// CPython extension behind binding.py: the enqueueing calls of one context as C methods.
//
// A decode step of a short session is shorter on the GPU than a handful of foreign calls made through ctypes are on the
// host (4 to 6 us each: argument objects, type conversions, a stream object per call; 50 us per step of a 4096-token
// session against 20 us here), so the marshalling is native: positional or keyword arguments as in binding.py's
// documentation, tensors read through their data_ptr() method, the layout through the buffer protocol, the current stream through
// torch's raw-stream getter.  Nothing is computed here and nothing is cached but interned names and torch's two dtype
// objects.  The GIL is released around every library call: a launch may wait for room in the stream's queue.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <climits>
#include <cstring>
#include <memory>

#include "fathom.h"

namespace {

struct ContextObject {
  PyObject_HEAD
  fathom_ctx* ctx;
};

PyObject *s_data_ptr, *s_dtype, *s_cuda_stream;              // interned attribute names
PyObject *t_f32, *t_bf16;                                    // torch.float32, torch.bfloat16
PyObject *f_device, *f_raw_stream, *f_first_stream;          // torch._C getters; torch.cuda.current_stream (initialises CUDA)
PyObject* f_raise;                                           // binding._raise(status, context address)
bool stream_ready = false;                                   // torch.cuda.current_stream() has succeeded once

// ---- arguments: `names` lists all parameters; the first `required` have no default.  got[i] is borrowed, nullptr if absent.
bool take(const char* fn, const char* const* names, int total, int required, PyObject* const* args, Py_ssize_t nargs, PyObject* kw,
          PyObject** got) {
  if (nargs > total) {
    PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", fn, total, nargs);
    return false;
  }
  for (int i = 0; i < total; ++i) got[i] = i < nargs ? args[i] : nullptr;
  const Py_ssize_t nkw = kw ? PyTuple_GET_SIZE(kw) : 0;
  for (Py_ssize_t j = 0; j < nkw; ++j) {
    PyObject* key = PyTuple_GET_ITEM(kw, j);
    int at = -1;
    for (int i = 0; i < total && at < 0; ++i)
      if (PyUnicode_CompareWithASCIIString(key, names[i]) == 0) at = i;
    if (at < 0) {
      PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", fn, key);
      return false;
    }
    if (got[at]) {
      PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%s'", fn, names[at]);
      return false;
    }
    got[at] = args[nargs + j];
  }
  for (int i = 0; i < required; ++i)
    if (!got[i]) {
      PyErr_Format(PyExc_TypeError, "%s() missing argument '%s'", fn, names[i]);
      return false;
    }
  return true;
}

// None -> null, an int as it is, anything else through data_ptr()
bool pointer(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = nullptr;
    return true;
  }
  PyObject* v = o;
  if (PyLong_Check(o)) Py_INCREF(v);
  else if (!(v = PyObject_CallMethodNoArgs(o, s_data_ptr))) return false;
  const unsigned long long p = PyLong_AsUnsignedLongLongMask(v);
  Py_DECREF(v);
  if (p == (unsigned long long)-1 && PyErr_Occurred()) return false;
  *out = reinterpret_cast<void*>((uintptr_t)p);
  return true;
}

bool integer(PyObject* o, int* out) {
  const unsigned long v = PyLong_AsUnsignedLongMask(o);      // wraps like a C int does
  if (v == (unsigned long)-1 && PyErr_Occurred()) return false;
  *out = (int)v;
  return true;
}

bool layout_of(PyObject* o, fathom_layout* out) {
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
  const bool ok = b.len == (Py_ssize_t)sizeof(fathom_layout);
  if (ok) memcpy(out, b.buf, sizeof(fathom_layout));
  PyBuffer_Release(&b);
  if (!ok) PyErr_SetString(PyExc_TypeError, "layout must be a Layout");
  return ok;
}

// an explicit dtype code, or that of a tensor
bool dtype_code(PyObject* code, PyObject* tensor, int* out) {
  if (code && code != Py_None) return integer(code, out);
  PyObject* d = PyObject_GetAttr(tensor, s_dtype);
  if (!d) return false;
  const bool f32 = d == t_f32, bf16 = d == t_bf16;
  if (!f32 && !bf16) PyErr_Format(PyExc_TypeError, "unsupported dtype %S", d);
  Py_DECREF(d);
  *out = f32 ? FATHOM_F32 : FATHOM_BF16;
  return f32 || bf16;
}

// None: torch's current stream on its current device; an int as it is; else the object's cuda_stream
bool stream_of(PyObject* o, void** out) {
  PyObject* v = nullptr;
  if (!o || o == Py_None) {
    if (stream_ready) {
      PyObject* dev = PyObject_CallNoArgs(f_device);
      if (!dev) return false;
      v = PyObject_CallOneArg(f_raw_stream, dev);
      Py_DECREF(dev);
    } else {
      PyObject* s = PyObject_CallNoArgs(f_first_stream);
      if (!s) return false;
      v = PyObject_GetAttr(s, s_cuda_stream);
      Py_DECREF(s);
      stream_ready = v != nullptr;
    }
  } else if (PyLong_Check(o)) {
    v = Py_NewRef(o);
  } else {
    v = PyObject_GetAttr(o, s_cuda_stream);
  }
  if (!v) return false;
  const unsigned long long p = PyLong_AsUnsignedLongLongMask(v);
  Py_DECREF(v);
  if (p == (unsigned long long)-1 && PyErr_Occurred()) return false;
  *out = reinterpret_cast<void*>((uintptr_t)p);
  return true;
}

PyObject* finish(int rc, const fathom_ctx* ctx) {
  if (rc == FATHOM_OK) Py_RETURN_NONE;
  PyObject* r = PyObject_CallFunction(f_raise, "iK", rc, (unsigned long long)(uintptr_t)ctx);
  if (r) {                                                    // it always raises
    Py_DECREF(r);
    PyErr_SetString(PyExc_RuntimeError, "fathom error handler returned");
  }
  return nullptr;
}

// ---- a method: parameter names, its arguments' kinds, and the library call.  Kinds: L layout, P pointer, I int, F float,
//      S stream (optional), T pointer whose tensor gives the dtype code unless the trailing D argument does.
union Value {
  void* p;
  int i;
  float f;
};
struct Parsed {
  fathom_layout layout;
  Value v[16];
  int dtype;
};

bool parse(const char* fn, const char* const* names, const char* kinds, PyObject* const* args, Py_ssize_t nargs, PyObject* kw, Parsed* out) {
  const int total = (int)strlen(kinds);
  int required = total;
  while (required > 0 && (kinds[required - 1] == 'S' || kinds[required - 1] == 'D')) --required;
  PyObject* got[16];
  if (!take(fn, names, total, required, args, nargs, kw, got)) return false;
  PyObject *typed = nullptr, *code = nullptr;
  for (int i = 0; i < total; ++i) {
    bool ok = true;
    switch (kinds[i]) {
      case 'L': ok = layout_of(got[i], &out->layout); break;
      case 'T': typed = got[i];                               // (fall through)
      case 'P': ok = pointer(got[i], &out->v[i].p); break;
      case 'I': ok = integer(got[i], &out->v[i].i); break;
      case 'F': {
        const double d = PyFloat_AsDouble(got[i]);
        ok = !(d == -1.0 && PyErr_Occurred());
        out->v[i].f = (float)d;
        break;
      }
      case 'S': ok = stream_of(got[i], &out->v[i].p); break;
      case 'D': code = got[i]; break;
    }
    if (!ok) return false;
  }
  return !typed || dtype_code(code, typed, &out->dtype);
}

#define METHOD(NAME, KINDS, CALL, ...)                                                                             \
  PyObject* m_##NAME(PyObject* self, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {                      \
    static const char* const names[] = {__VA_ARGS__};                                                              \
    static_assert(sizeof(names) / sizeof(names[0]) == sizeof(KINDS) - 1, "one name per kind");                     \
    Parsed a;                                                                                                      \
    if (!parse(#NAME, names, KINDS, args, nargs, kw, &a)) return nullptr;                                          \
    fathom_ctx* ctx = reinterpret_cast<ContextObject*>(self)->ctx;                                                 \
    const fathom_layout* L = &a.layout;                                                                            \
    const Value* v = a.v;                                                                                          \
    int rc;                                                                                                        \
    Py_BEGIN_ALLOW_THREADS rc = CALL;                                                                              \
    Py_END_ALLOW_THREADS (void)L;                                                                                  \
    return finish(rc, ctx);                                                                                        \
  }
#define F32P(i) static_cast<float*>(v[i].p)
#define U64P(i) static_cast<uint64_t*>(v[i].p)
#define U16P(i) static_cast<uint16_t*>(v[i].p)
#define U8P(i) static_cast<uint8_t*>(v[i].p)
#define I32P(i) static_cast<int32_t*>(v[i].p)

METHOD(fathom_build_planes, "LTPPSD", fathom_build_planes(ctx, L, v[1].p, a.dtype, U64P(2), U16P(3), v[4].p),
       "layout", "K", "planes", "scales", "stream", "k_dtype")
METHOD(fathom_alloc_depth, "LPPIIIPS", fathom_alloc_depth(ctx, L, F32P(1), F32P(2), v[3].i, v[4].i, v[5].i, U8P(6), v[7].p),
       "layout", "q", "var", "mode", "budget", "heads_per_plan", "depth", "stream")
METHOD(fathom_scan, "LPPPPIPS", fathom_scan(ctx, L, U64P(1), U16P(2), F32P(3), U8P(4), v[5].i, F32P(6), v[7].p),
       "layout", "planes", "scales", "q", "depth", "heads_per_plan", "scores", "stream")
METHOD(fathom_topk, "LPIIIPS", fathom_topk(ctx, L, F32P(1), v[2].i, v[3].i, v[4].i, I32P(5), v[6].p),
       "layout", "scores", "k", "n_sink", "n_local", "idx", "stream")
METHOD(fathom_sparse_attend, "LPTPPIFPSD",
       fathom_sparse_attend(ctx, L, F32P(1), v[2].p, v[3].p, a.dtype, I32P(4), v[5].i, v[6].f, F32P(7), v[8].p),
       "layout", "q", "Krows", "Vrows", "idx", "k", "softmax_scale", "out", "stream", "row_dtype")
METHOD(fathom_calibrate, "LTPPS", fathom_calibrate(ctx, L, v[1].p, a.dtype, F32P(2), F32P(3), v[4].p), "layout", "K", "mean", "cov",
       "stream")
METHOD(fathom_channel_variance, "LTPPS", fathom_channel_variance(ctx, L, v[1].p, a.dtype, F32P(2), F32P(3), v[4].p), "layout", "K",
       "mean", "var", "stream")
METHOD(fathom_klt_basis, "LPPPS", fathom_klt_basis(ctx, L, F32P(1), F32P(2), F32P(3), v[4].p), "layout", "cov", "basis",
       "eigenvalues", "stream")
METHOD(fathom_rotate_keys, "LTPPPS", fathom_rotate_keys(ctx, L, v[1].p, a.dtype, F32P(2), F32P(3), F32P(4), v[5].p), "layout", "K",
       "mean", "basis", "K_rot", "stream")
METHOD(fathom_build_planes_rotated, "LTPPPPS",
       fathom_build_planes_rotated(ctx, L, v[1].p, a.dtype, F32P(2), F32P(3), U64P(4), U16P(5), v[6].p), "layout", "K", "mean", "basis",
       "planes", "scales", "stream")
METHOD(fathom_rotate_query, "LPPPS", fathom_rotate_query(ctx, L, F32P(1), F32P(2), F32P(3), v[4].p), "layout", "q", "basis", "q_rot",
       "stream")
METHOD(fathom_scan_topk, "LPPPPIIIIPS",
       fathom_scan_topk(ctx, L, U64P(1), U16P(2), F32P(3), U8P(4), v[5].i, v[6].i, v[7].i, v[8].i, I32P(9), v[10].p), "layout", "planes",
       "scales", "q", "depth", "heads_per_plan", "k", "n_sink", "n_local", "idx", "stream")
METHOD(fathom_gather_union, "LPITPPPPPSD",
       fathom_gather_union(ctx, L, I32P(1), v[2].i, v[3].p, v[4].p, a.dtype, v[5].p, v[6].p, I32P(7), I32P(8), v[9].p), "layout", "idx",
       "k", "Krows", "Vrows", "K_stage", "V_stage", "idx_local", "union_count", "stream", "row_dtype")

// items: a sequence of (layout, planes, scales, q, depth, scores)
PyObject* m_fathom_scan_batch(PyObject* self, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {
  static const char* const names[] = {"items", "heads_per_plan", "stream"};
  PyObject* got[3];
  if (!take("fathom_scan_batch", names, 3, 2, args, nargs, kw, got)) return nullptr;
  PyObject* seq = PySequence_Fast(got[0], "items must be a sequence");
  if (!seq) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
  if (n > INT_MAX) {
    Py_DECREF(seq);
    PyErr_SetString(PyExc_OverflowError, "too many items");
    return nullptr;
  }
  struct Free { void operator()(void* p) const { PyMem_Free(p); } };
  std::unique_ptr<fathom_scan_item[], Free> items(static_cast<fathom_scan_item*>(PyMem_Malloc((size_t)n * sizeof(fathom_scan_item))));
  if (!items) {
    Py_DECREF(seq);
    return PyErr_NoMemory();
  }
  bool ok = true;
  for (Py_ssize_t i = 0; i < n && ok; ++i) {
    PyObject* t = PySequence_Fast(PySequence_Fast_GET_ITEM(seq, i), "an item is (layout, planes, scales, q, depth, scores)");
    if (!t) { ok = false; break; }
    if (PySequence_Fast_GET_SIZE(t) != 6) {
      PyErr_SetString(PyExc_ValueError, "an item is (layout, planes, scales, q, depth, scores)");
      ok = false;
    } else {
      void* p[6];
      ok = layout_of(PySequence_Fast_GET_ITEM(t, 0), &items[i].layout);
      for (int x = 1; x < 6 && ok; ++x) ok = pointer(PySequence_Fast_GET_ITEM(t, x), &p[x]);
      if (ok) {
        items[i].planes = static_cast<uint64_t*>(p[1]);
        items[i].scales = static_cast<uint16_t*>(p[2]);
        items[i].q = static_cast<float*>(p[3]);
        items[i].depth = static_cast<uint8_t*>(p[4]);
        items[i].scores = static_cast<float*>(p[5]);
      }
    }
    Py_DECREF(t);
  }
  Py_DECREF(seq);
  int hpp = 0;
  void* st = nullptr;
  if (!ok || !integer(got[1], &hpp) || !stream_of(got[2], &st)) return nullptr;
  fathom_ctx* ctx = reinterpret_cast<ContextObject*>(self)->ctx;
  int rc;
  Py_BEGIN_ALLOW_THREADS rc = fathom_scan_batch(ctx, items.get(), (int)n, hpp, st);
  Py_END_ALLOW_THREADS
  return finish(rc, ctx);
}

// the context's address as an int; 0 detaches (every later call is then refused by the library)
PyObject* m_attach(PyObject* self, PyObject* address) {
  void* p = nullptr;
  if (!pointer(address, &p)) return nullptr;
  reinterpret_cast<ContextObject*>(self)->ctx = static_cast<fathom_ctx*>(p);
  Py_RETURN_NONE;
}

#define ENTRY(NAME) {#NAME, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(m_##NAME)), METH_FASTCALL | METH_KEYWORDS, nullptr}
PyMethodDef context_methods[] = {ENTRY(fathom_build_planes), ENTRY(fathom_alloc_depth), ENTRY(fathom_scan), ENTRY(fathom_scan_batch),
                                 ENTRY(fathom_topk), ENTRY(fathom_sparse_attend), ENTRY(fathom_calibrate), ENTRY(fathom_channel_variance),
                                 ENTRY(fathom_klt_basis), ENTRY(fathom_rotate_keys), ENTRY(fathom_build_planes_rotated),
                                 ENTRY(fathom_rotate_query), ENTRY(fathom_scan_topk), ENTRY(fathom_gather_union),
                                 {"_attach", m_attach, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};

PyType_Slot context_slots[] = {{Py_tp_methods, context_methods}, {Py_tp_new, reinterpret_cast<void*>(PyType_GenericNew)}, {0, nullptr}};
PyType_Spec context_spec = {"paper_2609_17652_b200._native.ContextCalls", sizeof(ContextObject), 0,
                            Py_TPFLAGS_DEFAULT | Py_TPFLAGS_BASETYPE, context_slots};

// _setup(float32, bfloat16, get_device, raw_stream, current_stream, raise)
PyObject* setup(PyObject*, PyObject* args) {
  PyObject** slot[6] = {&t_f32, &t_bf16, &f_device, &f_raw_stream, &f_first_stream, &f_raise};
  if (PyTuple_GET_SIZE(args) != 6) {
    PyErr_SetString(PyExc_TypeError, "_setup takes six objects");
    return nullptr;
  }
  for (int i = 0; i < 6; ++i) Py_XSETREF(*slot[i], Py_NewRef(PyTuple_GET_ITEM(args, i)));
  Py_RETURN_NONE;
}

PyMethodDef module_methods[] = {{"_setup", setup, METH_VARARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, module_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_dtype = PyUnicode_InternFromString("dtype");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_data_ptr || !s_dtype || !s_cuda_stream) return nullptr;
  PyObject* m = PyModule_Create(&module_def);
  if (!m) return nullptr;
  PyObject* t = PyType_FromSpec(&context_spec);
  if (!t || PyModule_AddObjectRef(m, "ContextCalls", t) != 0) {
    Py_XDECREF(t);
    Py_DECREF(m);
    return nullptr;
  }
  Py_DECREF(t);
  return m;
}
