// The host side of the calls that are short on the GPU (per-token values, small batches): unpacks torch tensors, allocates the
// outputs and calls the C ABI, without the interpreter in between.  Every function returns NotImplemented when an argument is
// anything but what the call documents (another type or dtype, a tensor without memory, too small a workspace, an option that
// is not handled here); the caller then takes the general path, which accepts or refuses it as ever.  Host time of advantages and
// loss forward and backward 41 -> 26 us, of advantages, KL-shaped returns and per-token loss 36.5 -> 20.3 (which was what a
// batch of 300 thousand tokens took: 35.4 -> 24.3), of scoring 19 -> 11.
#include <Python.h>
#include <ATen/ops/empty.h>
#include <torch/csrc/autograd/python_variable.h>

#include "rlhead.h"

namespace {

struct Abi {
  decltype(&rl_workspace_bytes) workspace_bytes;
  decltype(&rl_workspace_bytes_logprobs) workspace_bytes_logprobs;
  decltype(&rl_set_workspace) set_workspace;
  decltype(&rl_grpo_advantages_ex) grpo_advantages_ex;
  decltype(&rl_kl_shaped_returns) kl_shaped_returns;
  decltype(&rl_token_loss) token_loss;
  decltype(&rl_token_logprobs) token_logprobs;
  decltype(&rl_policy_loss_fwd_bwd_ex) policy_loss_fwd_bwd_ex;
} abi;

// Thrown where the general path has to take over.
struct General {};

// Positional arguments; each reader throws General when the argument is not what it reads.
struct Args {
  PyObject* const* a;
  Py_ssize_t n, i = 0;
  Args(PyObject* const* args, Py_ssize_t nargs, Py_ssize_t expect) : a(args), n(nargs) {
    if (n != expect) throw General();
  }
  int64_t integer() {
    PyObject* o = a[i++];
    if (PyBool_Check(o)) return o == Py_True;
    if (!PyLong_CheckExact(o)) throw General();
    int overflow = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
    if (overflow) throw General();
    return v;
  }
  int small() {   // an int of the ABI
    const int64_t v = integer();
    if (v != (int)v) throw General();
    return (int)v;
  }
  float real() {
    PyObject* o = a[i++];
    if (PyFloat_CheckExact(o)) return (float)PyFloat_AS_DOUBLE(o);
    if (!PyLong_CheckExact(o)) throw General();
    const double v = PyLong_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) { PyErr_Clear(); throw General(); }
    return (float)v;
  }
  rl_ctx* context() { return reinterpret_cast<rl_ctx*>(integer()); }
  // nullptr for None where that is allowed
  const at::Tensor* tensor(bool none_ok) {
    PyObject* o = a[i++];
    if (o == Py_None) {
      if (!none_ok) throw General();
      return nullptr;
    }
    if (!THPVariable_CheckExact(o)) throw General();
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || !t.has_storage()) throw General();
    return &t;
  }
  const at::Tensor* of(at::ScalarType type, bool none_ok) {
    const at::Tensor* t = tensor(none_ok);
    if (t && t->scalar_type() != type) throw General();
    return t;
  }
  // [n] contiguous entries of a type
  const at::Tensor* array(at::ScalarType type, int64_t n, bool none_ok) {
    const at::Tensor* t = of(type, none_ok);
    if (t && (t->numel() != n || !t->is_contiguous())) throw General();
    return t;
  }
  const at::Tensor* values(int64_t n, bool none_ok) { return array(at::kFloat, n, none_ok); }
  // [n] one-byte entries or None
  const at::Tensor* mask(int64_t n) {
    const at::Tensor* t = tensor(true);
    if (t && (t->element_size() != 1 || t->numel() != n || !t->is_contiguous())) throw General();
    return t;
  }
  // rows of bf16, contiguous within a row
  const at::Tensor* rows() {
    const at::Tensor* t = of(at::kBFloat16, false);
    if (t->dim() != 2 || t->stride(1) != 1) throw General();
    return t;
  }
};

template <class T>
T* data(const at::Tensor* t) { return t ? static_cast<T*>(t->data_ptr()) : nullptr; }

// The interpreter's lock is given up for as long as this lives, as ctypes and torch give it up: an allocation may wait for the GPU,
// the call may lead back into Python (a hook), and other threads launch what the GPU waits for.
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};

// What a call returns.
struct Outputs {
  at::Tensor t[4];
  int n = 0;
  void* add(at::Tensor x) {
    t[n] = std::move(x);
    return t[n++].data_ptr();
  }
  // [n] fp32 on the device of `like`
  float* values(int64_t n_values, const at::Tensor& like) {
    return static_cast<float*>(add(at::empty({n_values}, like.options().dtype(at::kFloat).requires_grad(false))));
  }
};

// f reads the arguments, allocates the outputs and makes the call, last; a status other than RL_OK is returned as an int for the
// caller to raise.  Only what is thrown before the call sends its caller to the general path, which makes the call again.
template <class F>
PyObject* guarded(F f) {
  Outputs out;
  rl_status s;
  try {
    s = f(out);
  } catch (...) {   // General, or e.g. a tensor whose memory cannot be taken: the general path says why
    PyErr_Clear();
    return Py_NewRef(Py_NotImplemented);
  }
  if (s != RL_OK) return PyLong_FromLong((long)s);
  PyObject* result = PyTuple_New(out.n);
  for (int i = 0; result && i < out.n; ++i) {
    PyObject* o = nullptr;
    try {
      o = THPVariable_Wrap(std::move(out.t[i]));
    } catch (...) {
      if (!PyErr_Occurred()) PyErr_NoMemory();
    }
    if (o) PyTuple_SET_ITEM(result, i, o);
    else   Py_CLEAR(result);
  }
  return result;
}

// (context, rewards, group_size, ddof, eps_std, seq_offsets, T) -> (adv_seq, adv_tok)
PyObject* grpo_advantages(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  return guarded([&](Outputs& out) {
    Args a(args, nargs, 7);
    rl_ctx* c = a.context();
    const at::Tensor* rewards = a.of(at::kFloat, false);
    if (!rewards->is_contiguous()) throw General();
    const int group = a.small(), ddof = a.small();
    const float eps = a.real();
    const at::Tensor* offsets = a.of(at::kInt, false);
    const int64_t T = a.integer();
    if (T < 0) throw General();
    const float* r = data<float>(rewards);
    const int32_t* o = data<int32_t>(offsets);
    const int64_t n = rewards->numel();
    Unlocked u;
    float* seq = static_cast<float*>(out.add(at::empty(rewards->sizes(), rewards->options().requires_grad(false))));
    float* tok = out.values(T, *rewards);
    return abi.grpo_advantages_ex(c, r, n, group, ddof, eps, o, T, seq, tok);
  });
}

// (context, seq_value, logp, ref_logp, mask, seq_offsets, T, beta, gamma, kind, kl_tok) -> (shaped, returns)
PyObject* kl_shaped_returns(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  return guarded([&](Outputs& out) {
    Args a(args, nargs, 11);
    rl_ctx* c = a.context();
    const at::Tensor* value = a.of(at::kFloat, false);
    if (!value->is_contiguous()) throw General();
    Args peek = a;
    peek.i += 4;
    const int64_t T = peek.integer();
    if (T < 0) throw General();
    const at::Tensor *logp = a.values(T, true), *ref = a.values(T, true), *mask = a.mask(T), *offsets = a.of(at::kInt, false);
    ++a.i;
    const float beta = a.real(), gamma = a.real();
    const int kind = a.small();
    const at::Tensor* kl = a.values(T, true);
    const float *pv = data<float>(value), *pl = data<float>(logp), *pr = data<float>(ref), *pk = data<float>(kl);
    const uint8_t* pm = static_cast<const uint8_t*>(data<void>(mask));
    const int32_t* po = data<int32_t>(offsets);
    const int64_t n = offsets->numel() - 1;
    if (value->numel() != n) throw General();
    Unlocked u;
    float *shaped = out.values(T, *value), *returns = out.values(T, *value);
    return abi.kl_shaped_returns(c, pv, pl, pr, pk, pm, po, n, T, beta, gamma, kind, shaped, returns);
  });
}

// (context, logp, entropy, old_logp, ref_logp, adv, mask, eps_low, eps_high, beta, ent_coef, token_weight, token_count)
// -> (loss, dlogp, dentropy, metrics)
PyObject* token_loss(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  return guarded([&](Outputs& out) {
    Args a(args, nargs, 13);
    rl_ctx* c = a.context();
    const at::Tensor* logp = a.of(at::kFloat, false);
    const int64_t T = logp->numel();
    if (!logp->is_contiguous()) throw General();
    const at::Tensor *ent = a.values(T, true), *old = a.values(T, true), *ref = a.values(T, true), *adv = a.values(T, true);
    const at::Tensor* mask = a.array(at::kByte, T, true);
    const float lo = a.real(), hi = a.real(), beta = a.real(), ec = a.real();
    const at::Tensor *weight = a.values(T, true), *count = a.of(at::kLong, true);
    const float *pl = data<float>(logp), *pe = data<float>(ent), *po = data<float>(old), *pr = data<float>(ref), *pa = data<float>(adv),
                *pw = data<float>(weight);
    const uint8_t* pm = data<uint8_t>(mask);
    const void* pc = data<void>(count);
    Unlocked u;
    float *loss = out.values(1, *logp), *dlogp = out.values(T, *logp), *dent = out.values(T, *logp), *metrics = out.values(8, *logp);
    return abi.token_loss(c, pl, pe, po, pr, pa, pm, T, lo, hi, beta, ec, pw, pc, loss, dlogp, dent, metrics);
  });
}

void bind_workspace(rl_ctx* c, const at::Tensor* ws, decltype(&rl_workspace_bytes) bytes, int64_t T, int64_t d, int64_t V) {
  size_t need = 0;
  if (bytes(c, T, d, V, &need) != RL_OK || !ws || (size_t)ws->numel() < need) throw General();
  if (abi.set_workspace(c, ws->data_ptr(), (size_t)ws->numel()) != RL_OK) throw General();
}

// (context, workspace, H, W, tokens, mask) -> (logp, entropy, lse)
PyObject* token_logprobs(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  return guarded([&](Outputs& out) {
    Args a(args, nargs, 6);
    rl_ctx* c = a.context();
    const at::Tensor *ws = a.tensor(true), *H = a.rows(), *W = a.rows();
    const int64_t T = H->size(0), d = H->size(1), V = W->size(0);
    if (T == 0) throw General();
    const at::Tensor *tokens = a.array(at::kInt, T, false), *mask = a.mask(T);
    bind_workspace(c, ws, abi.workspace_bytes_logprobs, T, d, V);
    const void *ph = H->data_ptr(), *pw = W->data_ptr();
    const int64_t ldH = H->stride(0), ldW = W->stride(0);
    const int32_t* pt = data<int32_t>(tokens);
    const uint8_t* pm = static_cast<const uint8_t*>(data<void>(mask));
    Unlocked u;
    float *logp = out.values(T, *H), *ent = out.values(T, *H), *lse = out.values(T, *H);
    return abi.token_logprobs(c, ph, ldH, pw, ldW, pt, pm, T, d, V, logp, ent, lse);
  });
}

// (context, workspace, H, W, tokens, old_logp, ref_logp, adv, mask, eps_low, eps_high, beta, ent_coef, token_weight, accumulate_dW,
//  dW, dH, loss, agg_mode, sequence_level, seq_offsets, dH_fp32, token_count) -> (logp, entropy, metrics); loss, dH and dW are the
// caller's
PyObject* policy_loss(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  return guarded([&](Outputs& out) {
    Args a(args, nargs, 23);
    rl_ctx* c = a.context();
    const at::Tensor *ws = a.tensor(true), *H = a.rows(), *W = a.rows();
    const int64_t T = H->size(0), d = H->size(1), V = W->size(0);
    if (T == 0) throw General();
    const at::Tensor *tokens = a.array(at::kInt, T, false), *old = a.values(T, false), *ref = a.values(T, true), *adv = a.values(T, false),
                     *mask = a.mask(T);
    const float lo = a.real(), hi = a.real(), beta = a.real();
    rl_loss_opts o;
    memset(&o, 0, sizeof(o));
    o.struct_size = sizeof(o);
    o.ent_coef = a.real();
    o.token_weight = data<float>(a.values(T, true));
    o.accumulate_dW = a.integer() != 0;
    const at::Tensor *dW = a.values(V * d, false), *dH = a.tensor(false), *loss = a.values(1, false);
    o.agg_mode = a.small();
    o.sequence_level = a.integer() != 0;
    const at::Tensor* offsets = a.of(at::kInt, true);
    if (offsets) {
      o.seq_offsets = data<int32_t>(offsets);
      o.n_seq = offsets->numel() - 1;
    }
    o.dH_dtype = a.small();   // (the library says which values it knows)
    if (dH->scalar_type() != (o.dH_dtype ? at::kFloat : at::kBFloat16) || dH->numel() != T * d || !dH->is_contiguous()) throw General();
    const at::Tensor* count = a.of(at::kLong, true);
    if (count && count->numel() != 1) throw General();
    o.token_count = data<int64_t>(count);
    bind_workspace(c, ws, abi.workspace_bytes, T, d, V);
    const void *ph = H->data_ptr(), *pw = W->data_ptr();
    const int64_t ldH = H->stride(0), ldW = W->stride(0);
    const int32_t* pt = data<int32_t>(tokens);
    const float *po = data<float>(old), *pr = data<float>(ref), *pa = data<float>(adv);
    const uint8_t* pm = static_cast<const uint8_t*>(data<void>(mask));
    float *pl = data<float>(loss), *pd = data<float>(dW);
    void* ph_out = data<void>(dH);
    Unlocked u;
    o.logp_out = out.values(T, *W);
    o.entropy_out = out.values(T, *W);
    o.metrics_out = out.values(8, *W);
    return abi.policy_loss_fwd_bwd_ex(c, ph, ldH, pw, ldW, pt, po, pr, pa, pm, T, d, V, lo, hi, beta, pl, ph_out, pd, &o);
  });
}

// (addresses of the ABI's functions, in the order of Abi)
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  void** slot = reinterpret_cast<void**>(&abi);
  if (nargs != (Py_ssize_t)(sizeof(abi) / sizeof(void*))) {
    PyErr_SetString(PyExc_TypeError, "bind: number of addresses");
    return nullptr;
  }
  for (Py_ssize_t i = 0; i < nargs; ++i) {
    slot[i] = PyLong_AsVoidPtr(args[i]);
    if (!slot[i]) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "bind: null address");
      return nullptr;
    }
  }
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(bind), METH_FASTCALL, nullptr},
    {"grpo_advantages", reinterpret_cast<PyCFunction>(grpo_advantages), METH_FASTCALL, nullptr},
    {"kl_shaped_returns", reinterpret_cast<PyCFunction>(kl_shaped_returns), METH_FASTCALL, nullptr},
    {"token_loss", reinterpret_cast<PyCFunction>(token_loss), METH_FASTCALL, nullptr},
    {"token_logprobs", reinterpret_cast<PyCFunction>(token_logprobs), METH_FASTCALL, nullptr},
    {"policy_loss", reinterpret_cast<PyCFunction>(policy_loss), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_calls() { return PyModule_Create(&module); }
