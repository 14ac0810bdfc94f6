// binding.cpp - the Python calls' argument marshalling in native code: checks a call's tensors,
// allocates its outputs and calls the C entry point on the current stream.
//
// A call marshalled in Python (attribute lookups, torch.empty, ctypes) kept the host busy for 22 us
// (attention) to 28 us (scoring), longer than a small call's kernel runs; marshalled here it takes 5
// and 10 us, launch included. Every function returns None, with nothing launched, for a call that
// is not made of plain, contiguous CUDA tensors (a tensor subclass, an active dispatch or function
// mode, a Stream object, caller-made output dicts, anything that a check would refuse), and the
// caller (api.py) then goes through its own checks, which raise the errors. Otherwise it returns the
// call's results, or the entry point's status code (an int) when that is not zero.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/Context.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>

#include "cover.h"

namespace {

using at::Tensor;

// The C entry points, as found in the loaded library by the caller (bind).
decltype(&cover_attn_fwd) f_attn;
decltype(&cover_attn_fwd_f32) f_attn_f32;
decltype(&cover_attn_fwd_prefix) f_prefix;
decltype(&cover_attn_fwd_prefix_f32) f_prefix_f32;
decltype(&cover_score_fwd) f_score;
decltype(&cover_score_decide_fwd) f_decide;
decltype(&cover_attn_mass_fwd) f_mass;
decltype(&cover_seed_kv_gather) f_gather;
decltype(&cover_seed_kv_override) f_override;

bool none(PyObject* o) { return o == Py_None; }

int dim(const Tensor& t, int i) { return static_cast<int>(t.size(i)); }

template <typename T>
T* ptr(const Tensor& t) {
  return static_cast<T*>(t.data_ptr());
}

// Reads a call's arguments. The first one that is not of the plain form ends it: ok is false from then on,
// what is returned is without meaning, and the call goes to the caller's own path. (No exception
// says so: throwing and catching one took 6 to 10 us of a call that is then marshalled in Python.)
struct Args {
  bool ok = !c10::impl::TorchDispatchModeTLS::any_modes_set() && at::impl::PythonTorchFunctionTLS::stack_len() == 0 &&
            !at::globalContext().deterministicAlgorithms();

  void need(bool cond) { ok = ok && cond; }

  const Tensor& any_tensor(PyObject* o) {
    static const Tensor nothing;
    need(THPVariable_CheckExact(o));
    return ok ? THPVariable_Unpack(o) : nothing;
  }

  const Tensor& tensor(PyObject* o, at::ScalarType dtype, int dims) {
    const Tensor& t = any_tensor(o);
    if (!ok) return t;
    need(t.scalar_type() == dtype && t.is_cuda() && t.dim() == dims && t.is_contiguous());
    for (const int64_t n : t.sizes()) need(n <= INT_MAX);
    return t;
  }

  template <typename T>
  T* pointer(PyObject* o, at::ScalarType dtype, int dims) {
    const Tensor& t = tensor(o, dtype, dims);
    return ok ? ptr<T>(t) : nullptr;
  }
  template <typename T>
  T* pointer_or_null(PyObject* o, at::ScalarType dtype, int dims) {
    return none(o) ? nullptr : pointer<T>(o, dtype, dims);
  }

  int integer(PyObject* o) {
    need(PyLong_CheckExact(o));
    if (!ok) return 0;
    int over = 0;
    const long v = PyLong_AsLongAndOverflow(o, &over);
    need(over == 0 && v >= INT_MIN && v <= INT_MAX);
    return static_cast<int>(v);
  }

  double real(PyObject* o) {
    need(PyFloat_CheckExact(o));
    return ok ? PyFloat_AS_DOUBLE(o) : 0.0;
  }

  // An object whose truth value raises goes to the caller's own path, which raises it before anything is launched.
  bool truth(PyObject* o) {
    if (!ok) return false;
    const int t = PyObject_IsTrue(o);
    need(t >= 0);
    return t > 0;
  }

  void* stream(PyObject* o) {
    need(none(o));
    return ok ? c10::cuda::getCurrentCUDAStream().stream() : nullptr;
  }
};

Tensor empty(at::IntArrayRef sizes, at::ScalarType dtype, const Tensor& like) {
  return at::detail::empty_cuda(sizes, dtype, like.device(), std::nullopt);
}

PyObject* wrap(Tensor t) { return THPVariable_Wrap(std::move(t)); }

// Calls an entry point without the interpreter's lock, as ctypes does.
struct NoGil {
  PyThreadState* state = PyEval_SaveThread();
  ~NoGil() { PyEval_RestoreThread(state); }
};
template <typename F>
int call(bool& launched, F&& f) {
  NoGil unlocked;
  launched = true;
  return f();
}

// (a, b) with each the given object or, where that is None, the new tensor (None if undefined).
PyObject* pair(PyObject* a, Tensor ta, PyObject* b, Tensor tb) {
  PyObject* x = none(a) && ta.defined() ? wrap(std::move(ta)) : Py_NewRef(a);
  PyObject* y = none(b) && tb.defined() ? wrap(std::move(tb)) : Py_NewRef(b);
  PyObject* r = x != nullptr && y != nullptr ? PyTuple_Pack(2, x, y) : nullptr;
  Py_XDECREF(x);
  Py_XDECREF(y);
  return r;
}

struct Item {
  const char* key;
  Tensor value;
};
template <size_t N>
PyObject* dict_of(Item (&items)[N]) {
  PyObject* d = PyDict_New();
  for (size_t i = 0; d != nullptr && i < N; ++i) {
    PyObject* v = wrap(std::move(items[i].value));
    if (v == nullptr || PyDict_SetItemString(d, items[i].key, v) != 0) Py_CLEAR(d);
    Py_XDECREF(v);
  }
  return d;
}

// Runs f(args, launched), which returns null for a call of another form; such a call, or one that an
// exception ended before its entry point was called, is None.
template <typename F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F&& f) {
  if (n != want) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  bool launched = false;
  Args args;
  try {
    PyObject* r = args.ok ? f(args, launched) : nullptr;
    if (r != nullptr || launched) return r;
  } catch (const std::exception& e) {
    if (launched) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
      return nullptr;
    }
  }
  PyErr_Clear();
  Py_RETURN_NONE;
}

// attn(kind, q, k, v, km, vm, seed_idx, q0, out, lse, want_lse, stream); kind: 0 bf16, 1 f32 (whole
// sequence), 2 bf16, 3 f32 (window at q0)
PyObject* attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 12, [&](Args& in, bool& launched) -> PyObject* {
    const int kind = in.integer(a[0]);
    const bool window = kind >= 2;
    const at::ScalarType dt = (kind & 1) != 0 ? at::kFloat : at::kBFloat16;
    const Tensor &q = in.tensor(a[1], dt, 4), &k = in.tensor(a[2], dt, 4), &v = in.tensor(a[3], dt, 4);
    if (!in.ok) return nullptr;
    const int B = dim(q, 0), Hq = dim(q, 1), Lq = dim(q, 2), D = dim(q, 3), Hkv = dim(k, 1), L = dim(k, 2);
    in.need(dim(k, 0) == B && dim(k, 3) == D && (window || L == Lq) && v.sizes() == k.sizes());
    int S = 0;
    const void *km = nullptr, *vm = nullptr;
    const int32_t* idx = nullptr;
    if (!none(a[6])) {
      const Tensor& seeds = in.any_tensor(a[6]);
      if (!in.ok || seeds.dim() != 2) return nullptr;
      if (seeds.size(1) > 0) {
        const Tensor &si = in.tensor(a[6], at::kInt, 2), &tk = in.tensor(a[4], dt, 4), &tv = in.tensor(a[5], dt, 4);
        if (!in.ok) return nullptr;
        S = dim(si, 1);
        in.need(dim(si, 0) == B && dim(tk, 0) == B && dim(tk, 1) == Hkv && dim(tk, 2) == S && dim(tk, 3) == D &&
             tv.sizes() == tk.sizes());
        km = ptr<void>(tk), vm = ptr<void>(tv), idx = ptr<int32_t>(si);
      }
    }
    const int q0 = window ? in.integer(a[7]) : 0;
    void* stream = in.stream(a[11]);
    void* out = in.pointer_or_null<void>(a[8], dt, 4);
    float* lse = in.pointer_or_null<float>(a[9], at::kFloat, 3);
    const bool make_lse = none(a[9]) && in.truth(a[10]);
    if (!in.ok) return nullptr;
    Tensor new_out, new_lse;
    if (none(a[8])) out = ptr<void>(new_out = empty(q.sizes(), dt, q));
    if (make_lse) lse = ptr<float>(new_lse = empty(q.sizes().slice(0, 3), at::kFloat, q));
    const void *pq = ptr<void>(q), *pk = ptr<void>(k), *pv = ptr<void>(v);
    const auto f = [](const void* p) { return static_cast<const float*>(p); };
    const int rc = call(launched, [&] {
      switch (kind) {
        case 0: return f_attn(pq, pk, pv, km, vm, idx, S, B, Hq, Hkv, L, D, out, lse, stream);
        case 1:
          return f_attn_f32(f(pq), f(pk), f(pv), f(km), f(vm), idx, S, B, Hq, Hkv, L, D, static_cast<float*>(out), lse,
                            stream);
        case 2: return f_prefix(pq, pk, pv, km, vm, idx, S, B, Hq, Hkv, Lq, L, q0, D, out, lse, stream);
        default:
          return f_prefix_f32(f(pq), f(pk), f(pv), f(km), f(vm), idx, S, B, Hq, Hkv, Lq, L, q0, D,
                              static_cast<float*>(out), lse, stream);
      }
    });
    if (rc != 0) return PyLong_FromLong(rc);
    return pair(a[8], std::move(new_out), a[9], std::move(new_lse));
  });
}

// score(logits, n_seq, topk, cur_tok, d_in, d_out, eligible, workspace, out, stream)
PyObject* score(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 10, [&](Args& in, bool& launched) -> PyObject* {
    const Tensor& x = in.tensor(a[0], at::kBFloat16, 2);
    if (!in.ok) return nullptr;
    const int N = dim(x, 0), V = dim(x, 1), n_seq = in.integer(a[1]), topk = in.integer(a[2]);
    in.need(n_seq >= 1 && topk >= 0 && none(a[8]));
    const int32_t* cur = in.pointer_or_null<int32_t>(a[3], at::kInt, 1);
    const float *d_in = in.pointer_or_null<float>(a[4], at::kFloat, 1), *d_out = in.pointer_or_null<float>(a[5], at::kFloat, 1);
    const uint8_t* eligible = in.pointer_or_null<uint8_t>(a[6], at::kByte, 1);
    in.need(topk == 0 || !none(a[7]));   // the caller allocates a missing workspace
    void* stream = in.stream(a[9]);
    const Tensor& work = none(a[7]) ? x : in.any_tensor(a[7]);
    if (!in.ok) return nullptr;
    void* ws = none(a[7]) ? nullptr : ptr<void>(work);
    Item r[] = {{"maxprob", empty({N}, at::kFloat, x)},
                {"entropy", empty({N}, at::kFloat, x)},
                {"argmax", empty({N}, at::kInt, x)},
                {"score", empty({N}, at::kFloat, x)},
                {"topk_idx", empty({n_seq, topk}, at::kInt, x)},
                {"topk_score", empty({n_seq, topk}, at::kFloat, x)}};
    const void* logits = ptr<void>(x);
    const int rc = call(launched, [&] {
      return f_score(logits, N, V, n_seq, cur, d_in, d_out, eligible, topk, ptr<float>(r[0].value),
                     ptr<float>(r[1].value), ptr<int32_t>(r[2].value), ptr<float>(r[3].value),
                     topk > 0 ? ptr<int32_t>(r[4].value) : nullptr, topk > 0 ? ptr<float>(r[5].value) : nullptr, ws,
                     stream);
    });
    return rc != 0 ? PyLong_FromLong(rc) : dict_of(r);
  });
}

// decide(logits, n_seq, tok, flags, remask_cnt, tau_draft, draft_budget, remask_budget, mask_id,
// min_one, pos0, max_seeds, phase, d_in, d_out, draft_ok, workspace, out, stream)
PyObject* decide(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 19, [&](Args& in, bool& launched) -> PyObject* {
    const Tensor& x = in.tensor(a[0], at::kBFloat16, 2);
    if (!in.ok) return nullptr;
    const int N = dim(x, 0), V = dim(x, 1), n_seq = in.integer(a[1]);
    int32_t* tok = in.pointer<int32_t>(a[2], at::kInt, 1);
    uint8_t *flags = in.pointer<uint8_t>(a[3], at::kByte, 1), *cnt = in.pointer<uint8_t>(a[4], at::kByte, 1);
    const float tau = static_cast<float>(in.real(a[5]));
    const int budget = in.integer(a[6]), remask = in.integer(a[7]), mask_id = in.integer(a[8]);
    const int min_one = in.truth(a[9]) ? 1 : 0;
    const int pos0 = in.integer(a[10]), max_seeds = in.integer(a[11]), phase = in.integer(a[12]);
    const float *d_in = in.pointer_or_null<float>(a[13], at::kFloat, 1), *d_out = in.pointer_or_null<float>(a[14], at::kFloat, 1);
    const uint8_t* draft_ok = in.pointer_or_null<uint8_t>(a[15], at::kByte, 1);
    in.need(n_seq >= 1 && max_seeds >= 0 && none(a[17]));
    void* stream = in.stream(a[18]);
    const Tensor& work = in.any_tensor(a[16]);
    if (!in.ok) return nullptr;
    void* ws = ptr<void>(work);
    Item r[] = {{"maxprob", empty({N}, at::kFloat, x)},
                {"entropy", empty({N}, at::kFloat, x)},
                {"argmax", empty({N}, at::kInt, x)},
                {"score", empty({N}, at::kFloat, x)},
                {"seed_idx", empty({n_seq, max_seeds}, at::kInt, x)},
                {"n_seeds", empty({n_seq}, at::kInt, x)},
                {"stats", empty({n_seq, 6}, at::kInt, x)}};
    const void* logits = ptr<void>(x);
    const int rc = call(launched, [&] {
      return f_decide(logits, N, V, n_seq, d_in, d_out, draft_ok, tau, budget, remask, mask_id, min_one, pos0, max_seeds,
                      phase, tok, flags, cnt, ptr<float>(r[0].value), ptr<float>(r[1].value), ptr<int32_t>(r[2].value),
                      ptr<float>(r[3].value), max_seeds > 0 ? ptr<int32_t>(r[4].value) : nullptr,
                      ptr<int32_t>(r[5].value), ptr<int32_t>(r[6].value), ws, stream);
    });
    return rc != 0 ? PyLong_FromLong(rc) : dict_of(r);
  });
}

// mass(q, k, lse, tok, flags, mask_id, pos0, per, k_seedmask, seed_idx, workspace, d_in, d_out, stream)
PyObject* mass(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 14, [&](Args& in, bool& launched) -> PyObject* {
    const Tensor &q = in.tensor(a[0], at::kBFloat16, 4), &k = in.tensor(a[1], at::kBFloat16, 4);
    const Tensor &lse = in.tensor(a[2], at::kFloat, 3), &tok = in.tensor(a[3], at::kInt, 1), &flags = in.tensor(a[4], at::kByte, 1);
    if (!in.ok) return nullptr;
    const int B = dim(q, 0), Hq = dim(q, 1), L = dim(q, 2), D = dim(q, 3), Hkv = dim(k, 1);
    const int mask_id = in.integer(a[5]), pos0 = in.integer(a[6]), per = in.integer(a[7]);
    const int64_t rows = static_cast<int64_t>(B) * per;
    in.need(per >= 1 && tok.size(0) == rows && flags.size(0) == rows);
    int S = 0;
    const void* km = nullptr;
    const int32_t* idx = nullptr;
    if (!none(a[9])) {
      const Tensor& seeds = in.any_tensor(a[9]);
      if (!in.ok || seeds.dim() != 2) return nullptr;
      if (seeds.size(1) > 0) {
        idx = in.pointer<int32_t>(a[9], at::kInt, 2);
        km = in.pointer<void>(a[8], at::kBFloat16, 4);
        S = dim(seeds, 1);
      }
    }
    void* stream = in.stream(a[13]);
    const Tensor &work = in.any_tensor(a[10]), &given_in = none(a[11]) ? q : in.any_tensor(a[11]),
                 &given_out = none(a[12]) ? q : in.any_tensor(a[12]);
    if (!in.ok) return nullptr;
    void* ws = ptr<void>(work);
    Tensor new_in, new_out;
    float* d_in = ptr<float>(none(a[11]) ? (new_in = empty({rows}, at::kFloat, q)) : given_in);
    float* d_out = ptr<float>(none(a[12]) ? (new_out = empty({rows}, at::kFloat, q)) : given_out);
    const void *pq = ptr<void>(q), *pk = ptr<void>(k);
    const float* pl = ptr<float>(lse);
    const int32_t* pt = ptr<int32_t>(tok);
    const uint8_t* pf = ptr<uint8_t>(flags);
    const int rc = call(launched, [&] {
      return f_mass(pq, pk, km, idx, S, pl, B, Hq, Hkv, L, D, pt, pf, mask_id, pos0, per, ws, d_in, d_out, stream);
    });
    if (rc != 0) return PyLong_FromLong(rc);
    return pair(a[11], std::move(new_in), a[12], std::move(new_out));
  });
}

// kv(swap, k, v, seed_idx, k_cache, v_cache, stream)
PyObject* kv(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 7, [&](Args& in, bool& launched) -> PyObject* {
    const bool swap = in.integer(a[0]) != 0;
    const Tensor& any_k = in.any_tensor(a[1]);
    if (!in.ok) return nullptr;
    const at::ScalarType dt = any_k.scalar_type();
    in.need(dt == at::kBFloat16 || dt == at::kFloat);
    const Tensor &k = in.tensor(a[1], dt, 4), &v = in.tensor(a[2], dt, 4), &seeds = in.tensor(a[3], at::kInt, 2);
    if (!in.ok) return nullptr;
    const int B = dim(k, 0), Hkv = dim(k, 1), L = dim(k, 2), D = dim(k, 3), S = dim(seeds, 1);
    in.need(v.sizes() == k.sizes() && S > 0 && dim(seeds, 0) == B && none(a[4]) == none(a[5]) && (!swap || !none(a[4])));
    void* stream = in.stream(a[6]);
    if (!in.ok) return nullptr;
    Tensor new_k, new_v;
    const Tensor& kc = none(a[4]) ? (new_k = empty({B, Hkv, S, D}, dt, k)) : in.tensor(a[4], dt, 4);
    const Tensor& vc = none(a[5]) ? (new_v = empty({B, Hkv, S, D}, dt, k)) : in.tensor(a[5], dt, 4);
    if (!in.ok || dim(kc, 0) != B || dim(kc, 1) != Hkv || dim(kc, 2) != S || dim(kc, 3) != D || vc.sizes() != kc.sizes())
      return nullptr;
    void *pk = ptr<void>(k), *pv = ptr<void>(v), *pkc = ptr<void>(kc), *pvc = ptr<void>(vc);
    const int32_t* idx = ptr<int32_t>(seeds);
    const int elem = static_cast<int>(k.element_size());
    const int rc = call(launched, [&] {
      return swap ? f_override(pk, pv, idx, S, B, Hkv, L, D, elem, pkc, pvc, stream)
                  : f_gather(pk, pv, idx, S, B, Hkv, L, D, elem, pkc, pvc, stream);
    });
    if (rc != 0) return PyLong_FromLong(rc);
    return pair(a[4], std::move(new_k), a[5], std::move(new_v));
  });
}

// bind(addresses): the entry points' addresses, in the order below
PyObject* bind(PyObject*, PyObject* list) {
  unsigned long long p[9];
  PyObject* t = PySequence_Tuple(list);
  if (t == nullptr) return nullptr;
  if (PyTuple_GET_SIZE(t) != 9) {
    Py_DECREF(t);
    PyErr_SetString(PyExc_ValueError, "nine addresses are expected");
    return nullptr;
  }
  for (int i = 0; i < 9; ++i) p[i] = PyLong_AsUnsignedLongLong(PyTuple_GET_ITEM(t, i));
  Py_DECREF(t);
  if (PyErr_Occurred()) return nullptr;
  const auto at = [&](int i) { return reinterpret_cast<void*>(static_cast<uintptr_t>(p[i])); };
  f_attn = reinterpret_cast<decltype(f_attn)>(at(0));
  f_attn_f32 = reinterpret_cast<decltype(f_attn_f32)>(at(1));
  f_prefix = reinterpret_cast<decltype(f_prefix)>(at(2));
  f_prefix_f32 = reinterpret_cast<decltype(f_prefix_f32)>(at(3));
  f_score = reinterpret_cast<decltype(f_score)>(at(4));
  f_decide = reinterpret_cast<decltype(f_decide)>(at(5));
  f_mass = reinterpret_cast<decltype(f_mass)>(at(6));
  f_gather = reinterpret_cast<decltype(f_gather)>(at(7));
  f_override = reinterpret_cast<decltype(f_override)>(at(8));
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"attn", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(attn)), METH_FASTCALL, nullptr},
    {"score", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(score)), METH_FASTCALL, nullptr},
    {"decide", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(decide)), METH_FASTCALL, nullptr},
    {"mass", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(mass)), METH_FASTCALL, nullptr},
    {"kv", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(kv)), METH_FASTCALL, nullptr},
    {"bind", bind, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", "Native argument marshalling of the calls in api.py.", -1,
                      methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() { return PyModule_Create(&module); }
