// The host side of one attention call, compiled: checks of the tensors, allocation of the results, the current
// stream, and the call into libsigattn.so's C ABI.  The Python wrappers of binding.py hand their arguments over as
// they are.  The smallest calls take the device 6-10 us; the same steps in Python took 16 us (forward) and 25 us
// (backward) of host time a call, here 4 and 10, most of it the launches themselves.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDACachingAllocator.h>
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
  const void *qp, *kp, *vp;   // their data
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
  c.qp = q.const_data_ptr();
  c.kp = c.k->const_data_ptr();
  c.vp = c.v->const_data_ptr();
  return c;
}

// The caller's scratch tensor, if one was given.
struct Scratch {
  void* ptr = nullptr;
  size_t bytes = 0;
};
Scratch given_scratch(PyObject* o, const at::Tensor& q) {
  if (o == Py_None) return {};
  const at::Tensor* w = tensor_or_null(o);
  if (!side_ok(w, q, at::kByte)) bad("workspace must be a contiguous uint8 CUDA tensor on q's device");
  return {w->data_ptr(), static_cast<size_t>(w->numel())};
}

// ... or one allocated here when the call needs any.
at::Tensor own_scratch(const at::Tensor& q, size_t need, Scratch* s) {
  if (need == 0) return {};
  at::Tensor t = at::empty({static_cast<int64_t>(need)}, q.options().dtype(at::kByte));
  *s = {t.data_ptr(), need};
  return t;
}

// Allocations and launches run without the interpreter lock: a launch waits when the stream's queue is full, and the
// other threads of the process (one of them may be what the queue waits for) have to run meanwhile.
class Unlocked {
 public:
  Unlocked() : state_(PyEval_SaveThread()) {}
  ~Unlocked() { PyEval_RestoreThread(state_); }
  Unlocked(const Unlocked&) = delete;
  Unlocked& operator=(const Unlocked&) = delete;

 private:
  PyThreadState* state_;
};

// Memory that a call allocates is used on the call's stream.  Where that is not the current one, it is made the
// current one for the allocations: the allocator then hands out memory that is free in that stream's order, and takes
// scratch back in that order.  Results are used on the caller's current stream as well, which the allocator is told.
class OnStream {
 public:
  OnStream(const at::Tensor& q, void* stream) : device_(q.device()), current_(c10::cuda::getCurrentCUDAStream(device_.index())) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (s == cudaStreamPerThread) return;   // (the allocator knows no such stream)
    if (s == cudaStreamLegacy) s = nullptr;
    if (s != current_.stream()) other_.reset_stream(c10::cuda::getStreamFromExternal(s, device_.index()));
  }
  at::Tensor result(at::Tensor t) const {
    if (other_.current_stream()) c10::cuda::CUDACachingAllocator::recordStream(t.storage().data_ptr(), current_);
    return t;
  }

 private:
  c10::Device device_;
  c10::cuda::CUDAStream current_;
  c10::cuda::CUDAGuard on_device_{device_};
  c10::cuda::OptionalCUDAStreamGuard other_;
};

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

int launch_fwd(const Call& c, void* op, const Scratch& ws) {
  switch (c.mode) {
    case kPlain:
      return sigattn_fwd(c.qp, c.kp, c.vp, op, c.B, c.H, c.N_q, c.D, c.scale, c.bias, c.causal, c.slopes, c.dtype, c.stream);
    case kBiasVec:
      return sigattn_fwd_bias_vec(c.qp, c.kp, c.vp, op, c.B, c.H, c.N_q, c.D, c.scale, c.bias_vec, c.causal, c.slopes, c.dtype,
                                  c.stream);
    case kGqa:
      return sigattn_fwd_gqa(c.qp, c.kp, c.vp, op, c.B, c.H, c.H_kv, c.N_q, c.D, c.scale, c.bias, c.bias_vec, c.causal, c.slopes,
                             c.dtype, c.stream);
    case kNk:
      return sigattn_fwd_nk(c.qp, c.kp, c.vp, op, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                            c.slopes, c.dtype, c.stream);
    case kShard:
      return sigattn_fwd_shard(c.qp, c.kp, c.vp, op, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                               c.pos0, c.slopes, c.dtype, c.stream);
    case kVarlen:
      return sigattn_fwd_varlen(c.qp, c.kp, c.vp, op, c.B, c.H, c.H_kv, c.N_q, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                                c.seqlens, c.slopes, c.dtype, c.stream);
    case kRagged:
      return sigattn_fwd_ragged(c.qp, c.kp, c.vp, op, c.H, c.H_kv, c.N_q, c.D, c.cu, c.n_seqs, c.scale, c.bias, c.bias_vec,
                                c.causal, c.slopes, c.dtype, c.stream);
    case kRowscale:
      return sigattn_fwd_rowscale(c.qp, c.kp, c.vp, op, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec,
                                  c.causal, c.row_scale, c.slopes, c.dtype, c.stream);
    case kDecode:
      return sigattn_fwd_decode(c.qp, c.kp, c.vp, op, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                                c.slopes, c.dtype, ws.ptr, ws.bytes, c.stream);
    default:
      return SIGATTN_ERR_FLAG;
  }
}

int launch_bwd(const Call& c, const void* dop, void* dq, void* dk, void* dv, float* db, float* dtemp, const Scratch& ws) {
  switch (c.mode) {
    case kPlain:
      return sigattn_bwd(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.B, c.H, c.N_q, c.D, c.scale, c.bias, c.causal, c.slopes, c.dtype, ws.ptr,
                         ws.bytes, c.stream);
    case kBiasVec:
      return sigattn_bwd_bias_vec(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.B, c.H, c.N_q, c.D, c.scale, c.bias_vec, c.causal, c.slopes,
                                  c.dtype, db, ws.ptr, ws.bytes, c.stream);
    case kGqa:
      return sigattn_bwd_gqa(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                             c.slopes, c.dtype, db, ws.ptr, ws.bytes, c.stream);
    case kNk:
      return sigattn_bwd_nk(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec,
                            c.causal, c.slopes, c.dtype, db, ws.ptr, ws.bytes, c.stream);
    case kShard:
      return sigattn_bwd_shard(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias, c.bias_vec,
                               c.causal, c.pos0, c.slopes, c.dtype, db, ws.ptr, ws.bytes, c.stream);
    case kVarlen:
      return sigattn_bwd_varlen(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.D, c.scale, c.bias, c.bias_vec,
                                c.causal, c.seqlens, c.slopes, c.dtype, db, ws.ptr, ws.bytes, c.stream);
    case kRagged:
      return sigattn_bwd_ragged(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.H, c.H_kv, c.N_q, c.D, c.cu, c.n_seqs, c.scale, c.bias,
                                c.bias_vec, c.causal, c.slopes, c.dtype, db, ws.ptr, ws.bytes, c.stream);
    case kRowscale:
      return sigattn_bwd_rowscale(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.B, c.H, c.H_kv, c.N_q, c.N_k, c.D, c.scale, c.bias,
                                  c.bias_vec, c.causal, c.row_scale, c.slopes, c.dtype, db, ws.ptr, ws.bytes, c.stream);
    case kDtemp:
      return sigattn_bwd_dtemp(c.qp, c.kp, c.vp, dop, dq, dk, dv, c.B, c.H, c.N_q, c.D, c.scale, c.bias, c.bias_vec, c.causal,
                               c.slopes, c.dtype, db, dtemp, ws.ptr, ws.bytes, c.stream);
    default:
      return SIGATTN_ERR_FLAG;
  }
}

// fwd(mode, q, k, v, scale, bias, causal, slopes, aux, workspace, out, stream) -> O
PyObject* host_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 12) fail(PyExc_TypeError, "fwd takes 12 arguments");
    const Call c = parse(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[11]);
    const bool given = a[10] != Py_None, decode = c.mode == kDecode;
    at::Tensor out;
    if (given) out = like(a[10], *c.q, "out", "q");
    Scratch ws = given_scratch(decode ? a[9] : Py_None, *c.q);
    int rc;
    {
      const Unlocked unlocked;
      const OnStream on(*c.q, c.stream);
      if (!given) out = on.result(at::empty_like(*c.q));
      at::Tensor hold;
      if (decode && a[9] == Py_None)
        hold = own_scratch(*c.q, sigattn_fwd_decode_workspace_bytes(c.B, c.H, c.N_q, c.D, c.dtype), &ws);
      rc = launch_fwd(c, out.data_ptr(), ws);
    }
    check_rc(rc);
    return given ? Py_NewRef(a[10]) : THPVariable_Wrap(std::move(out));
  });
}

// bwd(mode, q, k, v, d_o, scale, bias, causal, slopes, aux, want_dbias, workspace, out, stream) ->
// (dQ, dK, dV), with dbias or None as a fourth (not for the plain call); the temperature's gradient comes before it
PyObject* host_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    if (n != 14) fail(PyExc_TypeError, "bwd takes 14 arguments");
    const Call c = parse(a[0], a[1], a[2], a[3], a[5], a[6], a[7], a[8], a[9], a[13]);
    const at::Tensor& q = *c.q;
    const void* dop = like(a[4], q, "d_o", "q").const_data_ptr();
    at::Tensor g[3];
    std::unique_ptr<PyObject, Release> given[3];   // (an iterable other than a list or a tuple may hold no reference itself)
    if (a[12] != Py_None) {
      static const char* names[3] = {"dq", "dk", "dv"};
      const std::unique_ptr<PyObject, Release> seq(PySequence_Fast(a[12], "out must be (dq, dk, dv)"));
      if (!seq) throw PyError();
      if (PySequence_Fast_GET_SIZE(seq.get()) != 3) bad("out must be (dq, dk, dv)");
      for (int i = 0; i < 3; ++i) {
        given[i].reset(Py_NewRef(PySequence_Fast_GET_ITEM(seq.get(), i)));
        g[i] = like(given[i].get(), i == 0 ? q : *c.k, names[i], i == 0 ? "q" : "k");
      }
    }
    const bool want_dbias = truth(a[10]), want_dtemp = c.mode == kDtemp;
    Scratch ws = given_scratch(a[11], q);
    at::Tensor dbias, dtemp;
    int rc;
    {
      const Unlocked unlocked;
      const OnStream on(q, c.stream);
      for (int i = 0; i < 3; ++i)
        if (!given[i]) g[i] = on.result(at::empty_like(i == 0 ? q : *c.k));
      const auto f32 = q.options().dtype(at::kFloat);
      if (want_dbias) dbias = on.result(at::empty({c.cu ? c.n_seqs : c.B, c.H}, f32));
      if (want_dtemp) dtemp = on.result(at::empty({c.B, c.H}, f32));
      at::Tensor hold;
      if (a[11] == Py_None) hold = own_scratch(q, sigattn_bwd_workspace_bytes(c.B, c.H, c.N_q, c.D, c.dtype), &ws);
      rc = launch_bwd(c, dop, g[0].data_ptr(), g[1].data_ptr(), g[2].data_ptr(), want_dbias ? dbias.data_ptr<float>() : nullptr,
                      want_dtemp ? dtemp.data_ptr<float>() : nullptr, ws);
    }
    check_rc(rc);
    const int extra = c.mode == kPlain ? 0 : want_dtemp ? 2 : 1;
    PyObject* out = PyTuple_New(3 + extra);
    if (!out) throw PyError();
    for (int i = 0; i < 3; ++i) PyTuple_SET_ITEM(out, i, given[i] ? given[i].release() : THPVariable_Wrap(std::move(g[i])));
    if (extra == 2) PyTuple_SET_ITEM(out, 3, THPVariable_Wrap(std::move(dtemp)));
    if (extra) PyTuple_SET_ITEM(out, 2 + extra, want_dbias ? THPVariable_Wrap(std::move(dbias)) : Py_NewRef(Py_None));
    return out;
  });
}

// workspace_ptr(workspace, q) -> the address of a scratch tensor that passes the calls' check, None for None
PyObject* host_workspace_ptr(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    const at::Tensor* q = n == 2 ? tensor_or_null(a[1]) : nullptr;
    if (!q) fail(PyExc_TypeError, "workspace_ptr takes (workspace, q)");
    if (a[0] == Py_None) return Py_NewRef(Py_None);
    return PyLong_FromVoidPtr(given_scratch(a[0], *q).ptr);
  });
}

PyObject* host_set_error(PyObject*, PyObject* type) {
  Py_XSETREF(g_error, Py_NewRef(type));
  Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(host_fwd)), METH_FASTCALL, nullptr},
    {"bwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(host_bwd)), METH_FASTCALL, nullptr},
    {"workspace_ptr", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(host_workspace_ptr)), METH_FASTCALL, nullptr},
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
