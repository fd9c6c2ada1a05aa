// CPython extension of the binding: the calls of a training step on the current stream, for arguments that are plain
// tensors of the right shapes.  It checks what binding.py checks and calls the same entry points of the library, whose
// addresses binding.py hands over; for anything else it returns None, and binding.py takes the call and says what is
// wrong with it.  A call through ctypes costs 4 to 9 us of the host, a small launch less on the GPU.
#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "psa.h"

namespace {

struct Entry {   // in the order of binding.py's _NATIVE_ENTRIES
  decltype(&::psa_fwd) fwd;
  decltype(&::psa_bwd) bwd;
  decltype(&::psa_bwd_f32) bwd_f32;
  decltype(&::dpo_logp_f64sum) logp;
  decltype(&::dpo_logp_bwd) logp_bwd;
  decltype(&::dpo_loss) dpo;
  decltype(&::simpo_loss) simpo;
  decltype(&::orpo_loss) orpo;
  decltype(&::psa_rope) rope;
  decltype(&::psa_plan) plan;
  decltype(&::psa_plan_stats) stats;
  decltype(&::psa_plan_destroy) destroy;
} g_lib;
bool g_ready = false;

// A tensor that is nothing but one: no subclass, wrapper or mode that would see the calls of binding.py.
const at::Tensor* plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.defined() && t.has_storage() && t.is_cuda() && !t.is_conj() && !t.is_neg() ? &t : nullptr;
}
bool modes_off() { return g_ready && !at::impl::torch_function_mode_enabled(); }

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Takes `o` as a contiguous tensor of this type and shape.
bool take3(PyObject* o, at::ScalarType type, int64_t a, int64_t b, int64_t c, void** p) {
  const at::Tensor* t = plain(o);
  if (!t || t->scalar_type() != type || t->dim() != 3 || t->size(0) != a || t->size(1) != b || t->size(2) != c ||
      !t->is_contiguous())
    return false;
  *p = t->data_ptr();
  return true;
}
bool take2(PyObject* o, at::ScalarType type, int64_t a, int64_t b, void** p) {
  const at::Tensor* t = plain(o);
  if (!t || t->scalar_type() != type || t->dim() != 2 || t->size(0) != a || t->size(1) != b || !t->is_contiguous()) return false;
  *p = t->data_ptr();
  return true;
}
bool take_n(PyObject* o, at::ScalarType type, int64_t n, void** p) {
  const at::Tensor* t = plain(o);
  if (!t || t->scalar_type() != type || t->numel() != n || !t->is_contiguous()) return false;
  *p = t->data_ptr();
  return true;
}
bool take_status(PyObject* o, void** p) {
  *p = nullptr;
  if (o == Py_None) return true;
  const at::Tensor* t = plain(o);
  if (!t || (t->numel() > 0 && t->nbytes() < 4)) return false;
  *p = t->data_ptr();
  return reinterpret_cast<uintptr_t>(*p) % 4 == 0;
}
bool take_int(PyObject* o, int64_t* v) {
  if (!PyLong_CheckExact(o)) return false;
  int over = 0;
  *v = PyLong_AsLongLongAndOverflow(o, &over);
  return over == 0;
}
bool take_float(PyObject* o, float* v) {
  if (PyFloat_CheckExact(o)) *v = float(PyFloat_AS_DOUBLE(o));
  else return false;
  return true;
}

// What binding.Plan keeps for these calls: (handle, tokens, query heads, kv heads, head size, workspace bytes).
struct PlanKey {
  psa_plan_t* plan;
  int64_t T, Hq, Hkv, d, ws;
};
bool take_plan(PyObject* o, PlanKey* k) {
  if (!PyTuple_CheckExact(o) || PyTuple_GET_SIZE(o) != 6) return false;
  k->plan = static_cast<psa_plan_t*>(PyLong_AsVoidPtr(PyTuple_GET_ITEM(o, 0)));
  int64_t* v[] = {&k->T, &k->Hq, &k->Hkv, &k->d, &k->ws};
  for (int i = 0; i < 5; ++i)
    if (!take_int(PyTuple_GET_ITEM(o, i + 1), v[i])) return false;
  return k->plan != nullptr;
}

PyObject* none() { Py_RETURN_NONE; }
// The library's calls run without the interpreter's lock, as those of ctypes do: a full launch queue must not hold it.
template <typename F>
psa_status_t unlocked(F f) {
  struct Unlock {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlock() { PyEval_RestoreThread(state); }
  } unlock;
  return f();
}
// An exception on the C++ side becomes binding.py's turn.
template <typename F>
PyObject* guarded(F f) {
  try {
    return f();
  } catch (const std::exception&) {
    PyErr_Clear();
    Py_RETURN_NONE;
  }
}

PyObject* init(PyObject*, PyObject* addresses) {
  constexpr Py_ssize_t n = sizeof(Entry) / sizeof(void*);
  if (!PyTuple_CheckExact(addresses) || PyTuple_GET_SIZE(addresses) != n) Py_RETURN_FALSE;
  void** to = reinterpret_cast<void**>(&g_lib);
  for (Py_ssize_t i = 0; i < n; ++i) to[i] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(addresses, i));
  if (PyErr_Occurred()) return nullptr;
  g_ready = true;
  Py_RETURN_TRUE;
}

// fwd(key, q, k, v, o, lse, status) -> status code, or None
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    PlanKey p;
    void *q, *k, *v, *o, *lse, *st;
    const auto b = at::kBFloat16;
    if (n != 7 || !modes_off() || !take_plan(a[0], &p) || !take3(a[1], b, p.T, p.Hq, p.d, &q) ||
        !take3(a[2], b, p.T, p.Hkv, p.d, &k) || !take3(a[3], b, p.T, p.Hkv, p.d, &v) || !take3(a[4], b, p.T, p.Hq, p.d, &o) ||
        !take2(a[5], at::kFloat, p.Hq, p.T, &lse) || !take_status(a[6], &st))
      return none();
    void* const on = stream();
    return PyLong_FromLong(unlocked([&] {
      return g_lib.fwd(p.plan, q, k, v, o, static_cast<float*>(lse), static_cast<int32_t*>(st), on);
    }));
  });
}

// bwd(f32, key, d_o, q, k, v, o, lse, dq, dk, dv, workspace, status) -> status code, or None
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    PlanKey p;
    void *d_o, *q, *k, *v, *o, *lse, *dq, *dk, *dv, *st;
    const auto b = at::kBFloat16;
    if (n != 13 || !modes_off()) return none();
    const bool f32 = a[0] == Py_True;
    const auto g = f32 ? at::kFloat : b;
    if (!take_plan(a[1], &p) || !take3(a[2], b, p.T, p.Hq, p.d, &d_o) || !take3(a[3], b, p.T, p.Hq, p.d, &q) ||
        !take3(a[4], b, p.T, p.Hkv, p.d, &k) || !take3(a[5], b, p.T, p.Hkv, p.d, &v) || !take3(a[6], b, p.T, p.Hq, p.d, &o) ||
        !take2(a[7], at::kFloat, p.Hq, p.T, &lse) || !take3(a[8], g, p.T, p.Hq, p.d, &dq) ||
        !take3(a[9], g, p.T, p.Hkv, p.d, &dk) || !take3(a[10], g, p.T, p.Hkv, p.d, &dv) || !take_status(a[12], &st))
      return none();
    const at::Tensor* ws = plain(a[11]);
    if (!ws || int64_t(ws->nbytes()) < p.ws ||
        int64_t(ws->storage().nbytes()) - ws->storage_offset() * int64_t(ws->itemsize()) < p.ws)
      return none();
    const float* l = static_cast<const float*>(lse);
    int32_t* s = static_cast<int32_t*>(st);
    void *const w = ws->data_ptr(), *const on = stream();
    return PyLong_FromLong(unlocked([&] {
      return f32 ? g_lib.bwd_f32(p.plan, d_o, q, k, v, o, l, static_cast<float*>(dq), static_cast<float*>(dk),
                                 static_cast<float*>(dv), w, s, on)
                 : g_lib.bwd(p.plan, d_o, q, k, v, o, l, dq, dk, dv, w, s, on);
    }));
  });
}

// Logits [n_rows, vocab] with unit column stride and the labels of dpo_logp.
struct Labelled {
  const at::Tensor* x;
  int32_t dtype;
  int64_t rows, vocab, stride, n_forks;
  void *targets, *segments, *fork[3];
};
bool take_labelled(PyObject* logits, PyObject* targets, PyObject* segments, PyObject* const* forks, Labelled* l) {
  l->x = plain(logits);
  if (!l->x || l->x->dim() != 2 || l->x->stride(1) != 1) return false;
  if (l->x->scalar_type() == at::kFloat) l->dtype = PSA_DTYPE_F32;
  else if (l->x->scalar_type() == at::kBFloat16) l->dtype = PSA_DTYPE_BF16;
  else return false;
  l->rows = l->x->size(0);
  l->vocab = l->x->size(1);
  l->stride = l->rows > 1 ? l->x->stride(0) : l->vocab;
  if (!take_n(targets, at::kInt, l->rows, &l->targets) || !take_n(segments, at::kInt, l->rows, &l->segments)) return false;
  l->n_forks = 0;
  l->fork[0] = l->fork[1] = l->fork[2] = nullptr;
  if (forks[0] == Py_None) return true;
  const at::Tensor* f = plain(forks[0]);
  if (!f) return false;
  if (f->numel() == 0) return true;
  l->n_forks = f->numel();
  for (int i = 0; i < 3; ++i)
    if (!take_n(forks[i], at::kInt, l->n_forks, &l->fork[i])) return false;
  return l->n_forks <= INT32_MAX;
}

at::Tensor device_tensor(int64_t n, at::ScalarType type, const at::Tensor& like) {
  return at::empty({n}, at::TensorOptions().dtype(type).device(like.device()));
}

// logp(logits, targets, segments, n_segments, fork_rows, fork_targets, fork_segments, status) -> out, a status code (not
// 0), or None
PyObject* logp(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    Labelled l;
    int64_t groups;
    void* st;
    if (n != 8 || !modes_off() || !take_labelled(a[0], a[1], a[2], a + 4, &l) || !take_int(a[3], &groups) || groups < 0 ||
        groups > INT32_MAX || !take_status(a[7], &st) || l.x->device().index() != c10::cuda::current_device())
      return none();
    at::Tensor out = device_tensor(groups, at::kFloat, *l.x), sums = device_tensor(groups + 1, at::kDouble, *l.x);
    void *const x = l.x->data_ptr(), *const scratch = sums.data_ptr(), *const on = stream();
    float* const to = out.data_ptr<float>();
    const psa_status_t rc = unlocked([&] {
      return g_lib.logp(x, l.dtype, l.rows, l.vocab, l.stride, static_cast<int32_t*>(l.targets),
                        static_cast<int32_t*>(l.segments), static_cast<int32_t*>(l.fork[0]), static_cast<int32_t*>(l.fork[1]),
                        static_cast<int32_t*>(l.fork[2]), int32_t(l.n_forks), int32_t(groups), to, scratch,
                        static_cast<int32_t*>(st), on);
    });
    return rc == PSA_OK ? THPVariable_Wrap(out) : PyLong_FromLong(rc);
  });
}

// logp_bwd(logits, targets, segments, coef, fork_rows, fork_targets, fork_segments, dlogits, status) -> status code, or None
PyObject* logp_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    Labelled l;
    void* st;
    if (n != 9 || !modes_off() || !take_labelled(a[0], a[1], a[2], a + 4, &l) || !take_status(a[8], &st)) return none();
    const at::Tensor *coef = plain(a[3]), *d = plain(a[7]);
    if (!coef || coef->scalar_type() != at::kFloat || !coef->is_contiguous() || coef->numel() > INT32_MAX || !d ||
        d->scalar_type() != l.x->scalar_type() || d->sizes() != l.x->sizes() || d->strides() != l.x->strides())
      return none();
    void *const x = l.x->data_ptr(), *const to = d->data_ptr(), *const on = stream();
    const float* const c = static_cast<const float*>(coef->data_ptr());
    const int32_t groups = int32_t(coef->numel());
    return PyLong_FromLong(unlocked([&] {
      return g_lib.logp_bwd(x, l.dtype, l.rows, l.vocab, l.stride, static_cast<int32_t*>(l.targets),
                            static_cast<int32_t*>(l.segments), static_cast<int32_t*>(l.fork[0]),
                            static_cast<int32_t*>(l.fork[1]), static_cast<int32_t*>(l.fork[2]), int32_t(l.n_forks), groups, c,
                            to, static_cast<int32_t*>(st), on);
    }));
  });
}

// loss(kind, policy, other, x, y, status) -> (loss, coef), a status code (not 0), or None; kind 0 dpo (other: reference
// log-probs, x beta), 1 simpo (lengths, beta, gamma), 2 orpo (lengths, lambda)
PyObject* loss(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    int64_t kind;
    float x, y;
    void* st;
    if (n != 6 || !modes_off() || !take_int(a[0], &kind) || !take_float(a[3], &x) || !take_float(a[4], &y) ||
        !take_status(a[5], &st))
      return none();
    const at::Tensor *pol = plain(a[1]), *other = plain(a[2]);
    if (!pol || pol->scalar_type() != at::kFloat || !pol->is_contiguous() || !other || other->sizes() != pol->sizes() ||
        !other->is_contiguous() || other->scalar_type() != (kind == 0 ? at::kFloat : at::kInt) || pol->numel() > INT32_MAX)
      return none();
    const int32_t half = int32_t(pol->numel() / 2);
    at::Tensor out = device_tensor(1, at::kFloat, *pol), coef = device_tensor(2 * int64_t(half), at::kFloat, *pol);
    const float* p = static_cast<const float*>(pol->data_ptr());
    float *lo = out.data_ptr<float>(), *co = coef.data_ptr<float>();
    int32_t* s = static_cast<int32_t*>(st);
    void *const r = other->data_ptr(), *const on = stream();
    const psa_status_t rc = unlocked([&] {
      return kind == 0   ? g_lib.dpo(p, static_cast<const float*>(r), half, x, lo, co, on)
             : kind == 1 ? g_lib.simpo(p, static_cast<const int32_t*>(r), half, x, y, lo, co, s, on)
                         : g_lib.orpo(p, static_cast<const int32_t*>(r), half, x, lo, co, s, on);
    });
    if (rc != PSA_OK) return PyLong_FromLong(rc);
    return Py_BuildValue("(NN)", THPVariable_Wrap(out), THPVariable_Wrap(coef));
  });
}

// rope(x, position_ids, theta, out) -> status code, or None
PyObject* rope(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    float theta;
    void *pos, *out;
    if (n != 4 || !modes_off() || !take_float(a[2], &theta)) return none();
    const at::Tensor* x = plain(a[0]);
    if (!x || x->scalar_type() != at::kBFloat16 || x->dim() != 3 || !x->is_contiguous() ||
        !take3(a[3], at::kBFloat16, x->size(0), x->size(1), x->size(2), &out) || !take_n(a[1], at::kInt, x->size(0), &pos) ||
        x->size(1) > INT32_MAX || x->size(2) > INT32_MAX)
      return none();
    void *const from = x->data_ptr(), *const on = stream();
    const int64_t T = x->size(0), H = x->size(1), d = x->size(2);
    return PyLong_FromLong(unlocked([&] {
      return g_lib.rope(from, out, static_cast<int32_t*>(pos), T, int32_t(H), int32_t(d), theta, on);
    }));
  });
}

// plan(cu, prefix, chosen, rejected, n_q_heads, n_kv_heads, head_dim, scale) -> (handle, tokens, pairs, live tiles, partial
// tiles, workspace bytes), a status code (not 0), or None.  The arrays are int32 buffers, contiguous and one-dimensional.
PyObject* plan(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    int64_t v[3];
    float scale;
    if (n != 8 || !g_ready || !take_float(a[7], &scale)) return none();
    for (int i = 0; i < 3; ++i)
      if (!take_int(a[4 + i], &v[i]) || v[i] < INT32_MIN || v[i] > INT32_MAX) return none();
    struct Buffers {
      Py_buffer b[4];
      int held = 0;
      ~Buffers() {
        while (held > 0) PyBuffer_Release(&b[--held]);
      }
    } buffers;
    const Py_buffer* b = buffers.b;
    for (int i = 0; i < 4; ++i) {
      if (PyObject_GetBuffer(a[i], &buffers.b[i], PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) {
        PyErr_Clear();
        return none();
      }
      buffers.held = i + 1;
      if (b[i].ndim != 1 || b[i].itemsize != 4 || !b[i].format || b[i].format[0] != 'i' || b[i].format[1]) return none();
    }
    if (b[1].shape[0] >= INT32_MAX || b[0].shape[0] != b[1].shape[0] + 1 || b[2].shape[0] != b[1].shape[0] ||
        b[3].shape[0] != b[1].shape[0])
      return none();
    psa_plan_t* p = nullptr;
    int64_t T = 0, pairs = 0, live = 0, partial = 0;
    size_t ws = 0;
    void* const st = stream();
    const psa_status_t rc = unlocked([&] {
      const psa_status_t made = g_lib.plan(static_cast<int32_t*>(b[0].buf), static_cast<int32_t*>(b[1].buf),
                                           static_cast<int32_t*>(b[2].buf), static_cast<int32_t*>(b[3].buf),
                                           int32_t(b[1].shape[0]), int32_t(v[0]), int32_t(v[1]), int32_t(v[2]), scale, 0, st, &p);
      return made == PSA_OK ? g_lib.stats(p, &T, &pairs, &live, &partial, &ws) : made;
    });
    return rc == PSA_OK ? Py_BuildValue("(NLLLLn)", PyLong_FromVoidPtr(p), (long long)T, (long long)pairs, (long long)live,
                                        (long long)partial, Py_ssize_t(ws))
                        : PyLong_FromLong(rc);
  });
}

// destroy(handle)
PyObject* destroy(PyObject*, PyObject* handle) {
  psa_plan_t* const p = static_cast<psa_plan_t*>(PyLong_AsVoidPtr(handle));
  if (PyErr_Occurred()) return nullptr;
  unlocked([&] { return g_lib.destroy(p); });
  Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {{"init", init, METH_O, nullptr}, FAST(fwd),  FAST(bwd),  FAST(logp), FAST(logp_bwd),
                           FAST(loss),                      FAST(rope), FAST(plan), {"destroy", destroy, METH_O, nullptr},
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "psa_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_psa_native() { return PyModule_Create(&g_module); }
