// Argument marshalling of the Python binding in native code: tensors to device pointers, the current
// CUDA stream, the call.  Every function takes the address of the context (0 after destroy) and
// returns the library's status; a tensor that the library cannot take raises ValueError.
//
// The entry points of the path are called once per layer or per layer and token: through ctypes a
// decode step cost 11 us on the host, of which 8 us were attribute look-ups and argument conversion.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <dlfcn.h>

#include <exception>
#include <vector>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "cake.h"

namespace {

struct Lib {
  decltype(&cake_begin) begin;
  decltype(&cake_score_layer) score_layer;
  decltype(&cake_allocate) allocate;
  decltype(&cake_evict) evict;
  decltype(&cake_compact) compact;
  decltype(&cake_compact_int4) compact_int4;
  decltype(&cake_clear_unused) clear_unused;
  decltype(&cake_decode_step) decode_step;
  decltype(&cake_decode_get_state) decode_get_state;
  decltype(&cake_select_positions_static) select_positions_static;
} lib;

// The current CUDA stream; false with a Python error set if there is none (no usable device).
bool stream(void** st) {
  try {
    *st = (void*)c10::cuda::getCurrentCUDAStream().stream();
    return true;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return false;
  }
}

cake_ctx* ctx_of(PyObject* h) { return (cake_ctx*)PyLong_AsVoidPtr(h); }

constexpr at::ScalarType kAny = at::ScalarType::Undefined;
at::ScalarType element(PyObject* is_fp32) {
  return PyObject_IsTrue(is_fp32) ? at::ScalarType::Float : at::ScalarType::BFloat16;
}

// Device pointer of a tensor (null for None); false with a Python error set if the library cannot
// take it.
bool ptr(PyObject* o, at::ScalarType want, void** out, bool pinned_ok = false) {
  *out = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) {
    PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor or None");
    return false;
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  try {
    if (!t.is_cuda() && !(pinned_ok && t.is_pinned())) {
      PyErr_SetString(PyExc_ValueError, pinned_ok ? "libcake takes CUDA tensors only (or pinned host tensors here)"
                                                  : "libcake takes CUDA tensors only");
      return false;
    }
    if (!t.is_contiguous()) {
      PyErr_SetString(PyExc_ValueError, "tensor must be contiguous");
      return false;
    }
    if (want != kAny && t.scalar_type() != want) {
      PyErr_Format(PyExc_ValueError, "expected torch.%s, got torch.%s",
                   want == at::ScalarType::Float ? "float32" : want == at::ScalarType::BFloat16 ? "bfloat16"
                   : want == at::ScalarType::Long ? "int64" : "int32",
                   c10::toString(t.scalar_type()));
      return false;
    }
    *out = t.data_ptr();
    return true;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return false;
  }
}

// The pointers of a sequence of tensors.
bool ptrs(PyObject* seq, at::ScalarType want, bool pinned_ok, std::vector<const void*>& out) {
  PyObject* fast = PySequence_Fast(seq, "expected a sequence of tensors");
  if (!fast) return false;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
  out.resize((size_t)n);
  bool ok = true;
  for (Py_ssize_t i = 0; ok && i < n; ++i) {
    void* p;
    ok = ptr(PySequence_Fast_GET_ITEM(fast, i), want, &p, pinned_ok);
    out[(size_t)i] = p;
  }
  Py_DECREF(fast);
  return ok;
}

// One pointer per layer in both arrays; missing ones are null.
bool per_layer(std::vector<const void*>& k, std::vector<const void*>& v, long layers) {
  if (PyErr_Occurred()) return false;               // `layers` was not a number
  if (layers < 0 || layers > CAKE_MAX_LAYERS) {
    PyErr_SetString(PyExc_ValueError, "no such number of layers");
    return false;
  }
  if (k.size() > (size_t)layers || v.size() > (size_t)layers) {
    PyErr_SetString(PyExc_IndexError, "more tensors than layers");
    return false;
  }
  k.resize((size_t)layers, nullptr);
  v.resize((size_t)layers, nullptr);
  return true;
}

bool integers(PyObject* seq, std::vector<int64_t>& out) {
  PyObject* fast = PySequence_Fast(seq, "expected a sequence of integers");
  if (!fast) return false;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
  out.resize((size_t)n);
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* v = PyNumber_Long(PySequence_Fast_GET_ITEM(fast, i));
    out[(size_t)i] = v ? PyLong_AsLongLong(v) : -1;
    Py_XDECREF(v);
    if (PyErr_Occurred()) break;
  }
  Py_DECREF(fast);
  return !PyErr_Occurred();
}

bool arity(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return false;
}

#define INT(i) ((int32_t)PyLong_AsLong(a[i]))
// Makes the call on the current stream, `st` in its arguments, without the interpreter lock (it may
// wait for room in the launch queue).
#define DONE(call)                            \
  do {                                        \
    if (PyErr_Occurred()) return nullptr;     \
    int32_t rc_;                              \
    void* st;                                 \
    if (!stream(&st)) return nullptr;         \
    Py_BEGIN_ALLOW_THREADS                    \
    rc_ = (call);                             \
    Py_END_ALLOW_THREADS                      \
    return PyLong_FromLong((long)rc_);        \
  } while (0)

// init(path of libcake.so)
PyObject* init(PyObject*, PyObject* path) {
  const char* p = PyUnicode_AsUTF8(path);
  if (!p) return nullptr;
  void* h = dlopen(p, RTLD_NOW | RTLD_LOCAL);
  if (!h) {
    PyErr_SetString(PyExc_ImportError, dlerror());
    return nullptr;
  }
#define SYM(name)                                                  \
  lib.name = (decltype(lib.name))dlsym(h, "cake_" #name);          \
  if (!lib.name) {                                                 \
    PyErr_SetString(PyExc_ImportError, "libcake lacks cake_" #name); \
    return nullptr;                                                \
  }
  SYM(begin) SYM(score_layer) SYM(allocate) SYM(evict) SYM(compact) SYM(compact_int4) SYM(clear_unused)
  SYM(decode_step) SYM(decode_get_state) SYM(select_positions_static)
#undef SYM
  Py_RETURN_NONE;
}

// begin(ctx, cu_seqlens)
PyObject* begin(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 2)) return nullptr;
  std::vector<int64_t> cu;
  if (!integers(a[1], cu)) return nullptr;
  cake_ctx* c = ctx_of(a[0]);
  DONE(lib.begin(c, (int32_t)cu.size() - 1, cu.data(), st));
}

// score_layer(ctx, layer, is_fp32, q_win, k, lse)
PyObject* score_layer(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *q, *k, *lse;
  if (!arity(n, 6)) return nullptr;
  const at::ScalarType e = element(a[2]);
  if (!ptr(a[3], e, &q) || !ptr(a[4], e, &k) || !ptr(a[5], at::ScalarType::Float, &lse)) return nullptr;
  cake_ctx* c = ctx_of(a[0]);
  const int32_t layer = INT(1);
  DONE(lib.score_layer(c, layer, q, k, (const float*)lse, st));
}

PyObject* allocate(PyObject*, PyObject* const* a, Py_ssize_t n) {      // (ctx, stage)
  if (!arity(n, 2)) return nullptr;
  cake_ctx* c = ctx_of(a[0]);
  const int32_t stage = INT(1);
  DONE(lib.allocate(c, stage, st));
}

PyObject* evict(PyObject*, PyObject* const* a, Py_ssize_t n) {         // (ctx, stage)
  if (!arity(n, 2)) return nullptr;
  cake_ctx* c = ctx_of(a[0]);
  const int32_t stage = INT(1);
  DONE(lib.evict(c, stage, st));
}

// prefill(ctx, n_layers, is_fp32, q_layers, k_layers): score, allocate and evict of every layer
PyObject* prefill(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 5)) return nullptr;
  const at::ScalarType e = element(a[2]);
  const int32_t layers = INT(1);
  std::vector<const void*> q, k;
  if (!ptrs(a[3], e, false, q) || !ptrs(a[4], e, false, k) || PyErr_Occurred()) return nullptr;
  if ((int64_t)q.size() < layers || (int64_t)k.size() < layers) {
    PyErr_SetString(PyExc_IndexError, "fewer tensors than layers");
    return nullptr;
  }
  cake_ctx* c = ctx_of(a[0]);
  auto all = [&](void* st) {
    int32_t rc = CAKE_OK;
    for (int32_t l = 0; l < layers && rc == CAKE_OK; ++l) {
      rc = lib.score_layer(c, l, q[l], k[l], nullptr, st);
      if (rc == CAKE_OK) rc = lib.allocate(c, l, st);
      if (rc == CAKE_OK) rc = lib.evict(c, l, st);
    }
    return rc;
  };
  DONE(all(st));
}

// compact(ctx, n_layers, is_fp32, lo, hi, k_layers, v_layers, k_out, v_out, row_offsets, positions)
PyObject* compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 11)) return nullptr;
  const at::ScalarType e = element(a[2]);
  std::vector<const void*> k, v;
  void *ko, *vo, *off, *pos;
  // K/V of a layer may also live in pinned host memory: the gather then fetches only the retained
  // rows over the bus
  if (!ptrs(a[5], e, true, k) || !ptrs(a[6], e, true, v) || !ptr(a[7], kAny, &ko) || !ptr(a[8], kAny, &vo) ||
      !ptr(a[9], at::ScalarType::Long, &off) || !ptr(a[10], at::ScalarType::Int, &pos)) return nullptr;
  if (!per_layer(k, v, PyLong_AsLong(a[1]))) return nullptr;
  cake_ctx* c = ctx_of(a[0]);
  const int32_t lo = INT(3), hi = INT(4);
  DONE(lib.compact(c, lo, hi, k.data(), v.data(), ko, vo, (int64_t*)off, (int32_t*)pos, st));
}

// compact_int4(ctx, n_layers, is_fp32, group, k_layers, v_layers, k_codes, k_scale, k_zero, v_codes,
//              v_scale, v_zero, row_offsets, kgroup_offsets, positions)
PyObject* compact_int4(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 15)) return nullptr;
  const at::ScalarType e = element(a[2]);
  std::vector<const void*> k, v;
  void* o[9];
  if (!ptrs(a[4], e, false, k) || !ptrs(a[5], e, false, v)) return nullptr;
  for (int i = 0; i < 9; ++i)
    if (!ptr(a[6 + i], kAny, &o[i])) return nullptr;
  if (!per_layer(k, v, PyLong_AsLong(a[1]))) return nullptr;
  cake_ctx* c = ctx_of(a[0]);
  const int32_t layers = INT(1), group = INT(3);
  DONE(lib.compact_int4(c, 0, layers, k.data(), v.data(), group, (uint8_t*)o[0], (float*)o[1], (float*)o[2], (uint8_t*)o[3],
                        (float*)o[4], (float*)o[5], (int64_t*)o[6], (int64_t*)o[7], (int32_t*)o[8], st));
}

// clear_unused(tensors, offsets): zeroes the rows of every tensor beyond the last entry of its offsets
PyObject* clear_unused(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 2)) return nullptr;
  void* bufs[CAKE_CLEAR_MAX];
  const int64_t* used[CAKE_CLEAR_MAX];
  int64_t bytes[CAKE_CLEAR_MAX], rows[CAKE_CLEAR_MAX];
  int32_t m = 0;
  auto fill = [&](PyObject* tensors, PyObject* offsets) {
    const Py_ssize_t count = PySequence_Fast_GET_SIZE(tensors);
    if (count > CAKE_CLEAR_MAX || PySequence_Fast_GET_SIZE(offsets) != count) {
      PyErr_SetString(PyExc_ValueError, "clear_unused: too many tensors, or not an offsets tensor for each");
      return false;
    }
    for (; m < (int32_t)count; ++m) {
      PyObject *x = PySequence_Fast_GET_ITEM(tensors, m), *o = PySequence_Fast_GET_ITEM(offsets, m);
      void* off;
      if (!THPVariable_Check(x) || !THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor");
        return false;
      }
      if (!ptr(x, kAny, &bufs[m]) || !ptr(o, at::ScalarType::Long, &off)) return false;
      const at::Tensor &t = THPVariable_Unpack(x), &u = THPVariable_Unpack(o);
      if (t.dim() < 1 || u.numel() < 1) {
        PyErr_SetString(PyExc_ValueError, "clear_unused: a tensor without rows, or empty offsets");
        return false;
      }
      rows[m] = t.size(0);
      bytes[m] = rows[m] > 0 ? (int64_t)t.nbytes() / rows[m] : 0;
      used[m] = (const int64_t*)off + (u.numel() - 1);
    }
    return true;
  };
  PyObject* tensors = PySequence_Fast(a[0], "expected a sequence of tensors");
  PyObject* offsets = tensors ? PySequence_Fast(a[1], "expected a sequence of tensors") : nullptr;
  const bool ok = offsets && fill(tensors, offsets);
  Py_XDECREF(tensors);
  Py_XDECREF(offsets);
  if (!ok) return nullptr;
  DONE(lib.clear_unused(m, bufs, bytes, rows, used, st));
}

// decode_step(ctx, layer, is_fp32, q_new, k_new, v_new, k_cache, v_cache)
PyObject* decode_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *q, *k, *v, *kc, *vc;
  if (!arity(n, 8)) return nullptr;
  const at::ScalarType e = element(a[2]);
  if (!ptr(a[3], e, &q) || !ptr(a[4], e, &k) || !ptr(a[5], e, &v) || !ptr(a[6], kAny, &kc) || !ptr(a[7], kAny, &vc))
    return nullptr;
  cake_ctx* c = ctx_of(a[0]);
  const int32_t layer = INT(1);
  DONE(lib.decode_step(c, layer, q, k, v, kc, vc, st));
}

// decode_get_state(ctx, req, layer, positions, scores, slots)
PyObject* decode_get_state(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *p, *s, *sl;
  if (!arity(n, 6)) return nullptr;
  if (!ptr(a[3], kAny, &p) || !ptr(a[4], kAny, &s) || !ptr(a[5], kAny, &sl)) return nullptr;
  cake_ctx* c = ctx_of(a[0]);
  const int32_t req = INT(1), layer = INT(2);
  DONE(lib.decode_get_state(c, req, layer, (int32_t*)p, (float*)s, (int32_t*)sl, st));
}

// select(values, n_heads, n, keep, out)
PyObject* select(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *v, *o;
  if (!arity(n, 5)) return nullptr;
  if (!ptr(a[0], at::ScalarType::Float, &v) || !ptr(a[4], at::ScalarType::Int, &o)) return nullptr;
  const int32_t heads = INT(1), len = INT(2), keep = INT(3);
  DONE(lib.select_positions_static((const float*)v, heads, len, keep, (int32_t*)o, st));
}

#define FAST(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {{"init", init, METH_O, nullptr},
                         FAST(begin), FAST(score_layer), FAST(allocate), FAST(evict), FAST(prefill), FAST(compact),
                         FAST(compact_int4), FAST(clear_unused), FAST(decode_step), FAST(decode_get_state), FAST(select),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_cake_py", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__cake_py() { return PyModule_Create(&module); }
