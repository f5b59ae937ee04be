// The host side of one attention call, compiled: checks of the tensors, allocation of the results, the current
// stream, and the call into libsigattn.so's C ABI.  The Python wrappers of binding.py hand their arguments over as
// they are.  The smallest calls take the device 6-10 us; the same steps in Python took 16 us (forward) and 25 us
// (backward) of host time a call, here 4 and 10, most of it the launches themselves.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <memory>
#include <stdexcept>
#include <string>

#include "../../include/sigattn.h"

namespace {

PyObject* g_error = nullptr;   // binding.SigattnError

// A Python exception has been set.
struct PyError {};

struct Release {
  void operator()(PyObject* o) const { Py_DECREF(o); }
};

[[noreturn]] void fail(PyObject* type, const std::string& text) {
  PyErr_SetString(type, text.c_str());
  throw PyError();
}
[[noreturn]] void bad(const std::string& text) { fail(PyExc_ValueError, text); }

const at::Tensor* tensor_or_null(PyObject* o) { return THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr; }

double number(PyObject* o) {
  const double x = PyFloat_AsDouble(o);
  if (x == -1.0 && PyErr_Occurred()) throw PyError();
  return x;
}

bool truth(PyObject* o) {
  const int x = PyObject_IsTrue(o);
  if (x < 0) throw PyError();
  return x != 0;
}

// One [B, H, N, D] operand: a contiguous CUDA tensor.
const at::Tensor& operand(PyObject* o, const char* name) {
  const at::Tensor* t = tensor_or_null(o);
  if (!t || !t->is_cuda()) bad(std::string(name) + " must be a CUDA tensor");
  if (t->dim() != 4) bad("tensors must be [B, H, N, D]");
  if (!t->is_contiguous()) bad(std::string(name) + " must be contiguous [B, H, N, D]");
  return *t;
}

// ... of the same shape, dtype and device as `ref`.
const at::Tensor& like(PyObject* o, const at::Tensor& ref, const char* name, const char* ref_name) {
  const at::Tensor* t = tensor_or_null(o);
  if (!t || !t->is_cuda()) bad(std::string(name) + " must be a CUDA tensor");
  if (!t->sizes().equals(ref.sizes()) || t->scalar_type() != ref.scalar_type() || t->device() != ref.device())
    bad(std::string(name) + " must match " + ref_name + " in shape, dtype and device");
  if (!t->is_contiguous()) bad(std::string(name) + " must be contiguous [B, H, N, D]");
  return *t;
}

// A small contiguous CUDA vector or matrix on q's device.
bool side_ok(const at::Tensor* t, const at::Tensor& q, at::ScalarType type) {
  return t && t->is_cuda() && t->device() == q.device() && t->scalar_type() == type && t->is_contiguous();
}

// Which entry points: how k, v relate to q, and what else a call carries.
enum Mode : long { kPlain = 0, kBiasVec, kGqa, kNk, kShard, kVarlen, kRagged, kRowscale, kDecode, kDtemp };

struct Call {
  Mode mode;
  const at::Tensor *q, *k, *v;
  int B, H, H_kv, N_q, N_k, D, dtype;
  float scale, bias = 0.0f;
  const float* bias_vec = nullptr;
  int causal;
  const float* slopes = nullptr;
  const int *seqlens = nullptr, *cu = nullptr;
  const float* row_scale = nullptr;
  int n_seqs = 0, pos0 = 0;
  void* stream = nullptr;
};

void* stream_of(PyObject* o, const at::Tensor& q) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream(q.device().index()).stream();
  PyObject* h = PyLong_Check(o) ? Py_NewRef(o) : PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw PyError();
  void* p = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (!p && PyErr_Occurred()) throw PyError();
  return p;
}

Call parse(PyObject* mode, PyObject* q_, PyObject* k_, PyObject* v_, PyObject* scale, PyObject* bias, PyObject* causal,
           PyObject* slopes, PyObject* aux, PyObject* stream) {
  Call c;
  c.mode = static_cast<Mode>(PyLong_AsLong(mode));
  const at::Tensor& q = operand(q_, "q");
  c.q = &q;
  if (c.mode == kPlain || c.mode == kBiasVec || c.mode == kDtemp) {
    c.k = &like(k_, q, "k", "q");
    c.v = &like(v_, q, "v", "q");
  } else {
    const bool any_len = c.mode == kNk || c.mode == kShard || c.mode == kRowscale || c.mode == kDecode;
    const at::Tensor &k = operand(k_, "k"), &v = operand(v_, "v");
    if (!k.sizes().equals(v.sizes()) || k.size(0) != q.size(0) || (!any_len && k.size(2) != q.size(2)) ||
        k.size(3) != q.size(3) || k.scalar_type() != q.scalar_type() || v.scalar_type() != q.scalar_type() ||
        k.device() != q.device() || v.device() != q.device())
      bad(any_len ? "k, v must be [B, H_kv, N_k, D] with q's B, D, dtype and device"
                  : "k, v must be [B, H_kv, N, D] with q's B, N, D, dtype and device");
    c.k = &k;
    c.v = &v;
  }
  auto size = [](int64_t n) {   // sizes past int's range: the library would see another shape
    if (n > INT32_MAX) bad("tensor extents must be below 2^31");
    return static_cast<int>(n);
  };
  c.B = size(q.size(0));
  c.H = size(q.size(1));
  c.N_q = size(q.size(2));
  c.D = size(q.size(3));
  c.H_kv = size(c.k->size(1));
  c.N_k = size(c.k->size(2));
  if (q.scalar_type() == at::kBFloat16) c.dtype = SIGATTN_DTYPE_BF16;
  else if (q.scalar_type() == at::kFloat) c.dtype = SIGATTN_DTYPE_FP32;
  else fail(PyExc_TypeError, std::string("sigattn supports bfloat16 and float32 tensors, got ") + c10::toString(q.scalar_type()));

  if (c.mode == kRagged) {
    if (c.B != 1) bad("a batch without padding has B = 1: q [1, H, T, D], k, v [1, H_kv, T, D]");
    const at::Tensor* cu = tensor_or_null(aux);
    if (!side_ok(cu, q, at::kInt) || cu->dim() != 1 || cu->numel() < 2)
      bad("cu_seqlens must be a contiguous int32 CUDA tensor of n_seqs + 1 row offsets on q's device");
    c.cu = cu->const_data_ptr<int>();
    c.n_seqs = size(cu->numel() - 1);
  } else if (c.mode == kVarlen) {
    const at::Tensor* s = tensor_or_null(aux);
    if (!side_ok(s, q, at::kInt) || s->dim() != 1 || s->numel() != c.B)
      bad("seqlens must be a contiguous int32 CUDA tensor of shape [B] on q's device");
    c.seqlens = s->const_data_ptr<int>();
  } else if (c.mode == kRowscale) {
    const at::Tensor* r = tensor_or_null(aux);
    if (!side_ok(r, q, at::kFloat) || r->dim() != 1 || r->numel() != c.N_q)
      bad("row_scale must be a contiguous float32 CUDA tensor of shape [N_q] on q's device");
    c.row_scale = r->const_data_ptr<float>();
  } else if (c.mode == kShard) {
    PyObject* n = PyNumber_Long(aux);
    if (!n) throw PyError();
    const long long x = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (x == -1 && PyErr_Occurred()) throw PyError();
    if (x > INT32_MAX || x < INT32_MIN) bad("pos0 must fit 32 bits");
    c.pos0 = static_cast<int>(x);
  }

  const at::Tensor* bv = tensor_or_null(bias);
  if (bv || c.mode == kBiasVec) {
    if (c.mode == kPlain) {
      c.bias = static_cast<float>(number(bias));   // a one-element tensor converts like any number
    } else {
      if (!side_ok(bv, q, at::kFloat) || bv->dim() != 2 || bv->size(0) != (c.cu ? c.n_seqs : c.B) || bv->size(1) != c.H)
        bad(c.cu ? "bias must be a float or a contiguous float32 CUDA tensor [n_seqs, H] on q's device"
                 : "bias_bh must be a contiguous float32 CUDA tensor of shape [B, H] on q's device");
      c.bias_vec = bv->const_data_ptr<float>();
    }
  } else {
    c.bias = static_cast<float>(number(bias));
  }
  c.scale = static_cast<float>(number(scale));
  c.causal = truth(causal) ? 1 : 0;
  if (slopes != Py_None) {
    const at::Tensor* s = tensor_or_null(slopes);
    if (!side_ok(s, q, at::kFloat) || s->numel() != c.H)
      bad("alibi_slopes must be a contiguous float32 CUDA tensor of " + std::to_string(c.H) +
          " slopes (one per query head) on q's device");
    c.slopes = s->const_data_ptr<float>();
  }
  c.stream = stream_of(stream, q);
  return c;
}

// The caller's scratch tensor, or one allocated here (kept alive in `hold`) when the call needs any.
void* workspace_of(PyObject* o, const at::Tensor& q, size_t need, at::Tensor* hold, size_t* bytes) {
  *bytes = 0;
  if (o == Py_None) {
    if (need == 0) return nullptr;
    *hold = at::empty({static_cast<int64_t>(need)}, q.options().dtype(at::kByte));
    *bytes = need;
    return hold->data_ptr();
  }
  const at::Tensor* w = tensor_or_null(o);
  if (!side_ok(w, q, at::kByte)) bad("workspace must be a contiguous uint8 CUDA tensor on q's device");
  *bytes = static_cast<size_t>(w->numel());
  return w->data_ptr();
}

void check_rc(int rc) {
  if (rc == SIGATTN_OK) return;
  PyObject* e = PyObject_CallFunction(g_error, "i", rc);
  if (e) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  throw PyError();
}

template <class F>
PyObject* guarded(F f) {
  HANDLE_TH_ERRORS
  try {
    return f();
  } catch (const PyError&) {
    return nullptr;
  }
  END_HANDLE_TH_ERRORS
}

// fwd(mode, q, k, v, scale, bias, causal, slopes, aux, workspace, out, stream) -> O
PyObject* host_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 12) fail(PyExc_TypeError, "fwd takes 12 arguments");
    const Call c = parse(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[11]);
    const at::Tensor& q = *c.q;
    const c10::cuda::OptionalCUDAGuard guard(q.device());
    at::Tensor made, hold;
    if (a[10] == Py_None) made = at::empty_like(q);
    else like(a[10], q, "out", "q");
    const at::Tensor& out = a[10] == Py_None ? made : THPVariable_Unpack(a[10]);
    const void *qp = q.const_data_ptr(), *kp = c.k->const_data_ptr(), *vp = c.v->const_data_ptr();
    void* op = out.data_ptr();
    int rc = SIGATTN_ERR_FLAG;
    switch (c.mode) {
      case kPlain:
        rc = sigattn_fwd(qp, kp, vp, op, c.B, c.H, c.N_q, c.D, c.scale, c.bias, c.causal, c.slopes, c.dtype, c.stream);
        break;
      case kBiasVec:
        rc = sigattn_fwd_bias_vec(qp, kp, vp, op, c.B, c.H, c.N_q, c.D, c.scale, c.bias_vec, c.causal, c.slopes, c.dtype,
                                  c.stream);
        break;
      case kGqa:
        rc = sigattn_fwd_gqa(qp, kp, vp, op, c.B, c.H, c.H_kv, c.N_q, c.D, c.scale, c.bias, c.bias_vec, c.causal, c.slopes,
                             c.dtype, c.stream);
        break;
      case kNk:
        rc = sigattn_fwd_nk(qp, kp, vp, op, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                            c.slopes, c.dtype, c.stream);
        break;
      case kShard:
        rc = sigattn_fwd_shard(qp, kp, vp, op, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                               c.pos0, c.slopes, c.dtype, c.stream);
        break;
      case kVarlen:
        rc = sigattn_fwd_varlen(qp, kp, vp, op, c.B, c.H, c.H_kv, c.N_q, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                                c.seqlens, c.slopes, c.dtype, c.stream);
        break;
      case kRagged:
        rc = sigattn_fwd_ragged(qp, kp, vp, op, c.H, c.H_kv, c.N_q, c.D, c.cu, c.n_seqs, c.scale, c.bias, c.bias_vec,
                                c.causal, c.slopes, c.dtype, c.stream);
        break;
      case kRowscale:
        rc = sigattn_fwd_rowscale(qp, kp, vp, op, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec,
                                  c.causal, c.row_scale, c.slopes, c.dtype, c.stream);
        break;
      case kDecode: {
        size_t bytes = 0;
        void* ws = workspace_of(a[9], q, sigattn_fwd_decode_workspace_bytes(c.B, c.H, c.N_q, c.D, c.dtype), &hold, &bytes);
        rc = sigattn_fwd_decode(qp, kp, vp, op, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                                c.slopes, c.dtype, ws, bytes, c.stream);
        break;
      }
      default:
        break;
    }
    check_rc(rc);
    return a[10] == Py_None ? THPVariable_Wrap(std::move(made)) : Py_NewRef(a[10]);
  });
}

// bwd(mode, q, k, v, d_o, scale, bias, causal, slopes, aux, want_dbias, workspace, out, stream) ->
// (dQ, dK, dV), with dbias or None as a fourth (not for the plain call); the temperature's gradient comes before it
PyObject* host_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 14) fail(PyExc_TypeError, "bwd takes 14 arguments");
    const Call c = parse(a[0], a[1], a[2], a[3], a[5], a[6], a[7], a[8], a[9], a[13]);
    const at::Tensor& q = *c.q;
    const at::Tensor& d_o = like(a[4], q, "d_o", "q");
    const c10::cuda::OptionalCUDAGuard guard(q.device());
    at::Tensor g[3];
    std::unique_ptr<PyObject, Release> given[3];   // (an iterable other than a list or a tuple may hold no reference itself)
    if (a[12] == Py_None) {
      g[0] = at::empty_like(q);
      g[1] = at::empty_like(*c.k);
      g[2] = at::empty_like(*c.v);
    } else {
      static const char* names[3] = {"dq", "dk", "dv"};
      const std::unique_ptr<PyObject, Release> seq(PySequence_Fast(a[12], "out must be (dq, dk, dv)"));
      if (!seq) throw PyError();
      if (PySequence_Fast_GET_SIZE(seq.get()) != 3) bad("out must be (dq, dk, dv)");
      for (int i = 0; i < 3; ++i) {
        given[i].reset(Py_NewRef(PySequence_Fast_GET_ITEM(seq.get(), i)));
        g[i] = like(given[i].get(), i == 0 ? q : *c.k, names[i], i == 0 ? "q" : "k");
      }
    }
    const auto f32 = q.options().dtype(at::kFloat);
    at::Tensor dbias, dtemp, hold;
    if (truth(a[10])) dbias = at::empty({c.cu ? c.n_seqs : c.B, c.H}, f32);
    if (c.mode == kDtemp) dtemp = at::empty({c.B, c.H}, f32);
    float* db = dbias.defined() ? dbias.data_ptr<float>() : nullptr;
    size_t bytes = 0;
    void* ws = workspace_of(a[11], q, sigattn_bwd_workspace_bytes(c.B, c.H, c.N_q, c.D, c.dtype), &hold, &bytes);
    const void *qp = q.const_data_ptr(), *kp = c.k->const_data_ptr(), *vp = c.v->const_data_ptr(), *dop = d_o.const_data_ptr();
    void *dq = g[0].data_ptr(), *dk = g[1].data_ptr(), *dv = g[2].data_ptr();
    int rc = SIGATTN_ERR_FLAG;
    switch (c.mode) {
      case kPlain:
        rc = sigattn_bwd(qp, kp, vp, dop, dq, dk, dv, c.B, c.H, c.N_q, c.D, c.scale, c.bias, c.causal, c.slopes, c.dtype, ws,
                         bytes, c.stream);
        break;
      case kBiasVec:
        rc = sigattn_bwd_bias_vec(qp, kp, vp, dop, dq, dk, dv, c.B, c.H, c.N_q, c.D, c.scale, c.bias_vec, c.causal, c.slopes,
                                  c.dtype, db, ws, bytes, c.stream);
        break;
      case kGqa:
        rc = sigattn_bwd_gqa(qp, kp, vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                             c.slopes, c.dtype, db, ws, bytes, c.stream);
        break;
      case kNk:
        rc = sigattn_bwd_nk(qp, kp, vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec,
                            c.causal, c.slopes, c.dtype, db, ws, bytes, c.stream);
        break;
      case kShard:
        rc = sigattn_bwd_shard(qp, kp, vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec,
                               c.causal, c.pos0, c.slopes, c.dtype, db, ws, bytes, c.stream);
        break;
      case kVarlen:
        rc = sigattn_bwd_varlen(qp, kp, vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.D, c.scale, c.bias, c.bias_vec,
                                c.causal, c.seqlens, c.slopes, c.dtype, db, ws, bytes, c.stream);
        break;
      case kRagged:
        rc = sigattn_bwd_ragged(qp, kp, vp, dop, dq, dk, dv, c.H, c.H_kv, c.N_q, c.D, c.cu, c.n_seqs, c.scale, c.bias,
                                c.bias_vec, c.causal, c.slopes, c.dtype, db, ws, bytes, c.stream);
        break;
      case kRowscale:
        rc = sigattn_bwd_rowscale(qp, kp, vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias,
                                  c.bias_vec, c.causal, c.row_scale, c.slopes, c.dtype, db, ws, bytes, c.stream);
        break;
      case kDtemp:
        rc = sigattn_bwd_dtemp(qp, kp, vp, dop, dq, dk, dv, c.B, c.H, c.N_q, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                               c.slopes, c.dtype, db, dtemp.data_ptr<float>(), ws, bytes, c.stream);
        break;
      default:
        break;
    }
    check_rc(rc);
    const int extra = c.mode == kPlain ? 0 : c.mode == kDtemp ? 2 : 1;
    PyObject* out = PyTuple_New(3 + extra);
    if (!out) throw PyError();
    for (int i = 0; i < 3; ++i) PyTuple_SET_ITEM(out, i, given[i] ? given[i].release() : THPVariable_Wrap(std::move(g[i])));
    if (extra == 2) PyTuple_SET_ITEM(out, 3, THPVariable_Wrap(std::move(dtemp)));
    if (extra) PyTuple_SET_ITEM(out, 2 + extra, db ? THPVariable_Wrap(std::move(dbias)) : Py_NewRef(Py_None));
    return out;
  });
}

PyObject* host_set_error(PyObject*, PyObject* type) {
  Py_XSETREF(g_error, Py_NewRef(type));
  Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(host_fwd)), METH_FASTCALL, nullptr},
    {"bwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(host_bwd)), METH_FASTCALL, nullptr},
    {"set_error", host_set_error, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_sigattn_host", "Host side of the attention calls.", -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sigattn_host(void) {
  PyObject* m = PyModule_Create(&g_module);
  if (!m) return nullptr;
  for (const auto& e : {std::pair<const char*, long>{"PLAIN", kPlain}, {"BIAS_VEC", kBiasVec}, {"GQA", kGqa}, {"NK", kNk},
                        {"SHARD", kShard}, {"VARLEN", kVarlen}, {"RAGGED", kRagged}, {"ROWSCALE", kRowscale},
                        {"DECODE", kDecode}, {"DTEMP", kDtemp}})
    if (PyModule_AddIntConstant(m, e.first, e.second) < 0) return nullptr;
  return m;
}
