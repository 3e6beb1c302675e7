// The binding's per-call host work in native code (CPython module `_native`): argument checks, output and workspace
// allocation, marshalling into the C ABI of include/mdn.h.
//
// Why: the smallest calls are bound by the host.  A decode step of one sequence takes 5 us on the GPU; the Python
// marshalling around it (attribute checks of nine tensors, ctypes conversion of twelve arguments, the stream query)
// took 23 us per call and set the call rate.
//
// Contract with binding.py: a function here either does exactly what the Python code of the same name does, or returns
// None without side effects whenever anything about the arguments is not the plain valid case; the Python code then
// runs and raises its own error (or handles the unusual case).  A failed C call returns its status as an int.
#include <Python.h>

#include <cmath>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>

#include "mdn.h"

namespace {

using at::Tensor;

// Releases the GIL for the C call (it can block when the launch queue is full); allocations need no GIL either.
struct NoGil {
  PyThreadState* state;
  NoGil() : state(PyEval_SaveThread()) {}
  ~NoGil() { PyEval_RestoreThread(state); }
};

bool io_dtype_code(at::ScalarType t, int32_t* code) {
  if (t == at::kFloat) { *code = MDN_F32; return true; }
  if (t == at::kBFloat16) { *code = MDN_BF16; return true; }
  return false;
}

// The tensor behind a Python object if it is a contiguous CUDA tensor of `dtype` on `dev`, else nullptr.
const Tensor* cuda_tensor(PyObject* obj, at::ScalarType dtype, c10::DeviceIndex dev) {
  if (!THPVariable_Check(obj)) return nullptr;
  const Tensor& t = THPVariable_Unpack(obj);
  if (!t.defined() || !t.is_cuda() || t.scalar_type() != dtype || t.get_device() != dev || !t.is_contiguous()) return nullptr;
  return &t;
}

bool has_shape(const Tensor& t, std::initializer_list<int64_t> shape) { return t.sizes() == at::IntArrayRef(shape); }

// q, k, v and the four gates of a call (eta may be None), as _check_inputs of binding.py wants them.
struct Inputs {
  const Tensor *q, *k, *v;
  const float *beta, *log_alpha, *log_mu, *eta;
  int64_t B, T, H, dk, dv;
  c10::DeviceIndex dev;
  at::ScalarType dtype;
  int32_t code;
};

bool parse_inputs(PyObject* const* a, Inputs* in) {   // a[0..6]
  if (!THPVariable_Check(a[0])) return false;
  const Tensor& q = THPVariable_Unpack(a[0]);
  if (!q.defined() || !q.is_cuda() || q.dim() != 4 || !q.is_contiguous()) return false;
  in->q = &q;
  in->dev = q.get_device();
  in->dtype = q.scalar_type();
  if (!io_dtype_code(in->dtype, &in->code) || in->dev != c10::cuda::current_device()) return false;
  in->k = cuda_tensor(a[1], in->dtype, in->dev);
  in->v = cuda_tensor(a[2], in->dtype, in->dev);
  if (!in->k || !in->v || in->v->dim() != 4 || in->k->sizes() != q.sizes()) return false;
  in->B = q.size(0); in->T = q.size(1); in->H = q.size(2); in->dk = q.size(3); in->dv = in->v->size(3);
  constexpr int64_t kMax = INT32_MAX;
  if (in->B > kMax || in->T > kMax || in->H > kMax || in->dk > kMax || in->dv > kMax) return false;
  if (!has_shape(*in->v, {in->B, in->T, in->H, in->dv})) return false;
  const float** dst[4] = {&in->beta, &in->log_alpha, &in->log_mu, &in->eta};
  for (int i = 0; i < 4; ++i) {
    *dst[i] = nullptr;
    if (a[3 + i] == Py_None) {
      if (i < 3) return false;
      continue;
    }
    const Tensor* g = cuda_tensor(a[3 + i], at::kFloat, in->dev);
    if (!g || !has_shape(*g, {in->B, in->T, in->H})) return false;
    *dst[i] = static_cast<const float*>(g->const_data_ptr());
  }
  return true;
}

// A state [n, H, dk, dv] fp32 or None.
bool parse_state(PyObject* obj, const Inputs& in, int64_t n, float** out) {
  *out = nullptr;
  if (obj == Py_None) return true;
  const Tensor* t = cuda_tensor(obj, at::kFloat, in.dev);
  if (!t || !has_shape(*t, {n, in.H, in.dk, in.dv})) return false;
  *out = static_cast<float*>(t->data_ptr());
  return true;
}

bool parse_scale(PyObject* obj, int64_t dk, float* out) {
  if (obj == Py_None) { *out = static_cast<float>(1.0 / std::sqrt(static_cast<double>(dk))); return true; }
  if (!PyFloat_Check(obj)) return false;
  *out = static_cast<float>(PyFloat_AS_DOUBLE(obj));
  return true;
}

bool parse_o_dtype(PyObject* obj, const Inputs& in, at::ScalarType* dt, int32_t* code) {
  *dt = in.dtype;
  if (obj != Py_None) {
    if (!THPDtype_Check(obj)) return false;
    *dt = reinterpret_cast<THPDtype*>(obj)->scalar_type;
  }
  return io_dtype_code(*dt, code);
}

bool parse_cu(PyObject* obj, c10::DeviceIndex dev, const int32_t** cu, int64_t* n) {
  *cu = nullptr; *n = 0;
  if (obj == Py_None) return true;
  const Tensor* t = cuda_tensor(obj, at::kInt, dev);
  if (!t || t->numel() < 2) return false;
  *cu = static_cast<const int32_t*>(t->const_data_ptr());
  *n = t->numel() - 1;
  return *n <= INT32_MAX;
}

Tensor empty(at::IntArrayRef shape, at::ScalarType dt, c10::DeviceIndex dev) {
  return at::detail::empty_cuda(shape, dt, c10::Device(c10::kCUDA, dev), std::nullopt);
}

// A buffer that starts on a 1024-byte boundary (chunk states and the backward's workspaces): the allocator's blocks start on
// 512-byte ones, most of them on coarser.
Tensor empty_1024(int64_t bytes, c10::DeviceIndex dev) {
  Tensor t = empty({bytes}, at::kByte, dev);
  if (reinterpret_cast<uintptr_t>(t.data_ptr()) % 1024 == 0) return t;
  t = empty({bytes + 1024}, at::kByte, dev);
  return t.narrow(0, (int64_t)((1024 - reinterpret_cast<uintptr_t>(t.data_ptr()) % 1024) % 1024), bytes);
}

void* stream_of(c10::DeviceIndex dev) { return c10::cuda::getCurrentCUDAStream(dev).stream(); }

mdn_params params_of(const Inputs& in, int64_t num_seqs, int32_t o_code, int32_t path, float scale, int32_t segments) {
  return mdn_params{(int32_t)in.B, (int32_t)in.T, (int32_t)in.H, (int32_t)in.dk, (int32_t)in.dv, 64, (int32_t)num_seqs,
                    in.code, o_code, path, scale, segments};
}

// layer_ops: the address of an mdn_layer_ops, 0 for none
bool parse_ops(PyObject* obj, const mdn_layer_ops** ops) {
  if (!PyLong_Check(obj)) return false;
  *ops = static_cast<const mdn_layer_ops*>(PyLong_AsVoidPtr(obj));
  return !PyErr_Occurred();
}

// C++ exceptions as torch's own functions hand them on: out of memory, ValueError and so on as those types, and what Python code
// raised underneath (saved-tensor hooks, which activation checkpointing leaves by an exception) as itself.
#define NATIVE_TRY try {
#define NATIVE_CATCH                                                 \
  } catch (const std::exception&) {                                  \
    torch::translate_exception_to_python(std::current_exception());  \
    return nullptr;                                                  \
  }

// decode_step(q, k, v, beta, log_alpha, log_mu, eta, S, M, scale, o_dtype, out, ops) -> o
PyObject* decode_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  NATIVE_TRY
  Inputs in;
  float *S, *M, scale;
  at::ScalarType odt;
  int32_t ocode;
  const mdn_layer_ops* ops;
  if (n != 13 || !parse_inputs(a, &in) || in.T != 1 || !parse_state(a[7], in, in.B, &S) || !S ||
      !parse_state(a[8], in, in.B, &M) || !M || !parse_scale(a[9], in.dk, &scale) || !parse_o_dtype(a[10], in, &odt, &ocode) ||
      !parse_ops(a[12], &ops))
    return Py_NewRef(Py_None);
  Tensor o;
  if (a[11] != Py_None) {
    const Tensor* t = cuda_tensor(a[11], odt, in.dev);
    if (!t || !has_shape(*t, {in.B, 1, in.H, in.dv})) return Py_NewRef(Py_None);
    o = *t;
  }
  const mdn_params p = params_of(in, 0, ocode, MDN_PATH_AUTO, scale, 0);
  mdn_status st;
  {
    NoGil g;
    if (!o.defined()) o = empty({in.B, 1, in.H, in.dv}, odt, in.dev);
    st = mdn_decode_step_fused(&p, ops, in.q->const_data_ptr(), in.k->const_data_ptr(), in.v->const_data_ptr(), in.beta,
                               in.log_alpha, in.log_mu, in.eta, S, M, o.data_ptr(), stream_of(in.dev));
  }
  if (st != MDN_OK) return PyLong_FromLong(st);
  return THPVariable_Wrap(o);
  NATIVE_CATCH
}

// chunk_fwd(q, k, v, beta, log_alpha, log_mu, eta, initial_S, initial_M, cu_seqlens, scale, o_dtype, path,
//           output_final_state, workspace, out, segments, ops, keep) -> (o, S, M) or (o, S, M, chunk_states, workspace)
PyObject* chunk_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  NATIVE_TRY
  Inputs in;
  float *S0, *M0, scale;
  const int32_t* cu;
  int64_t N;
  at::ScalarType odt;
  int32_t ocode;
  const mdn_layer_ops* ops;
  if (n != 19 || !parse_inputs(a, &in) || !parse_cu(a[9], in.dev, &cu, &N)) return Py_NewRef(Py_None);
  const int64_t nst = N > 0 ? N : in.B;
  if (!parse_state(a[7], in, nst, &S0) || !parse_state(a[8], in, nst, &M0) || !parse_scale(a[10], in.dk, &scale) ||
      !parse_o_dtype(a[11], in, &odt, &ocode) || !parse_ops(a[17], &ops) || !PyLong_Check(a[12]) || !PyLong_Check(a[16]))
    return Py_NewRef(Py_None);
  const int32_t path = (int32_t)PyLong_AsLong(a[12]), segments = (int32_t)PyLong_AsLong(a[16]);
  const bool finals = a[13] == Py_True, keep = a[18] == Py_True;
  if (PyErr_Occurred() || (keep && ops)) { PyErr_Clear(); return Py_NewRef(Py_None); }
  const mdn_params p = params_of(in, N, ocode, path, scale, segments);
  const size_t need = ops ? mdn_chunk_fwd_fused_workspace_bytes(&p, ops) : mdn_chunk_fwd_workspace_bytes(&p);
  const size_t state_bytes = keep ? mdn_chunk_states_bytes(&p) : 0;
  if (need == 0 || (keep && state_bytes == 0)) return Py_NewRef(Py_None);
  Tensor ws, o, Sf, Mf, states;
  if (a[14] != Py_None) {
    const Tensor* t = cuda_tensor(a[14], at::kByte, in.dev);
    if (!t) return Py_NewRef(Py_None);
    ws = *t;
  }
  if (a[15] != Py_None) {
    const Tensor* t = cuda_tensor(a[15], odt, in.dev);
    if (!t || !has_shape(*t, {in.B, in.T, in.H, in.dv})) return Py_NewRef(Py_None);
    o = *t;
  }
  mdn_status st;
  {
    NoGil g;
    if (!ws.defined()) ws = empty({(int64_t)need}, at::kByte, in.dev);
    if (!o.defined()) o = empty({in.B, in.T, in.H, in.dv}, odt, in.dev);
    if (finals) {
      Sf = empty({nst, in.H, in.dk, in.dv}, at::kFloat, in.dev);
      Mf = empty({nst, in.H, in.dk, in.dv}, at::kFloat, in.dev);
    }
    float* sf = finals ? static_cast<float*>(Sf.data_ptr()) : nullptr;
    float* mf = finals ? static_cast<float*>(Mf.data_ptr()) : nullptr;
    const void *q = in.q->const_data_ptr(), *k = in.k->const_data_ptr(), *v = in.v->const_data_ptr();
    void* stream = stream_of(in.dev);
    if (keep) {
      states = empty_1024((int64_t)state_bytes, in.dev);
      st = mdn_chunk_fwd_keep_states(&p, q, k, v, in.beta, in.log_alpha, in.log_mu, in.eta, S0, M0, cu, o.data_ptr(), sf, mf,
                                     states.data_ptr(), ws.data_ptr(), (size_t)ws.numel(), stream);
    } else {
      st = mdn_chunk_fwd_fused(&p, ops, q, k, v, in.beta, in.log_alpha, in.log_mu, in.eta, S0, M0, cu, o.data_ptr(), sf, mf,
                               ws.data_ptr(), (size_t)ws.numel(), stream);
    }
  }
  if (st != MDN_OK) return PyLong_FromLong(st);
  PyObject* r = PyTuple_New(keep ? 5 : 3);
  if (!r) return nullptr;
  PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(o));
  PyTuple_SET_ITEM(r, 1, finals ? THPVariable_Wrap(Sf) : Py_NewRef(Py_None));
  PyTuple_SET_ITEM(r, 2, finals ? THPVariable_Wrap(Mf) : Py_NewRef(Py_None));
  if (keep) {
    PyTuple_SET_ITEM(r, 3, THPVariable_Wrap(states));
    PyTuple_SET_ITEM(r, 4, THPVariable_Wrap(ws));
  }
  return r;
  NATIVE_CATCH
}

// chunk_bwd(q, k, v, beta, log_alpha, log_mu, eta, d_o, initial_S, initial_M, cu_seqlens, d_final_S, d_final_M, scale,
//           workspace, method, fwd_workspace, chunk_states) -> (dq, dk, dv, dbeta, dlog_alpha, dlog_mu, deta, dS0, dM0)
// method: 0 stepwise, 1 chunked, 2 chunked on saved states, 3 the same with dq, dk, dv in the i/o dtype
PyObject* chunk_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  NATIVE_TRY
  Inputs in;
  float *S0, *M0, *dSf, *dMf, scale;
  const int32_t* cu;
  int64_t N;
  if (n != 18 || !parse_inputs(a, &in) || !parse_cu(a[10], in.dev, &cu, &N) || !THPVariable_Check(a[7])) return Py_NewRef(Py_None);
  const int64_t nst = N > 0 ? N : in.B;
  const at::ScalarType odt = THPVariable_Unpack(a[7]).scalar_type();
  int32_t ocode;
  const Tensor* d_o = cuda_tensor(a[7], odt, in.dev);
  if (!d_o || !io_dtype_code(odt, &ocode) || !has_shape(*d_o, {in.B, in.T, in.H, in.dv}) || !parse_state(a[8], in, nst, &S0) ||
      !parse_state(a[9], in, nst, &M0) || !parse_state(a[11], in, nst, &dSf) || !parse_state(a[12], in, nst, &dMf) ||
      !parse_scale(a[13], in.dk, &scale) || !PyLong_Check(a[15]))
    return Py_NewRef(Py_None);
  const long method = PyLong_AsLong(a[15]);
  const mdn_params p = params_of(in, N, ocode, method == 0 ? MDN_PATH_AUTO : MDN_PATH_TENSOR, scale, 0);
  const size_t need = method == 0 ? mdn_chunk_bwd_workspace_bytes(&p)
                                  : method == 1 ? mdn_chunk_bwd_chunked_workspace_bytes(&p) : mdn_chunk_bwd_saved_workspace_bytes(&p);
  if (need == 0) return Py_NewRef(Py_None);
  Tensor ws;
  if (a[14] != Py_None) {
    const Tensor* t = cuda_tensor(a[14], at::kByte, in.dev);
    if (!t) return Py_NewRef(Py_None);
    ws = *t;
  }
  const Tensor *fws = nullptr, *states = nullptr;
  if (method >= 2 && (!(fws = cuda_tensor(a[16], at::kByte, in.dev)) || !(states = cuda_tensor(a[17], at::kByte, in.dev))))
    return Py_NewRef(Py_None);
  Tensor g[9];
  mdn_status st;
  {
    NoGil gil;
    if (!ws.defined()) ws = empty_1024((int64_t)need, in.dev);
    const at::ScalarType gdt = method == 3 ? in.dtype : at::kFloat;
    g[0] = empty({in.B, in.T, in.H, in.dk}, gdt, in.dev);
    g[1] = empty({in.B, in.T, in.H, in.dk}, gdt, in.dev);
    g[2] = empty({in.B, in.T, in.H, in.dv}, gdt, in.dev);
    for (int i = 3; i < (in.eta ? 7 : 6); ++i) g[i] = empty({in.B, in.T, in.H}, at::kFloat, in.dev);
    g[7] = empty({nst, in.H, in.dk, in.dv}, at::kFloat, in.dev);
    g[8] = empty({nst, in.H, in.dk, in.dv}, at::kFloat, in.dev);
    float* gp[9];
    for (int i = 0; i < 9; ++i) gp[i] = g[i].defined() ? static_cast<float*>(g[i].data_ptr()) : nullptr;   // (0..2: the i/o dtype for method 3)
    const void *q = in.q->const_data_ptr(), *k = in.k->const_data_ptr(), *v = in.v->const_data_ptr();
    void* stream = stream_of(in.dev);
    if (method == 2)
      st = mdn_chunk_bwd_saved(&p, q, k, v, in.beta, in.log_alpha, in.log_mu, in.eta, cu, fws->data_ptr(), (size_t)fws->numel(),
                               states->const_data_ptr(), d_o->const_data_ptr(), dSf, dMf, gp[0], gp[1], gp[2], gp[3], gp[4],
                               gp[5], gp[6], gp[7], gp[8], ws.data_ptr(), (size_t)ws.numel(), stream);
    else if (method == 3)
      st = mdn_chunk_bwd_saved_io(&p, q, k, v, in.beta, in.log_alpha, in.log_mu, in.eta, cu, fws->data_ptr(), (size_t)fws->numel(),
                                  states->const_data_ptr(), d_o->const_data_ptr(), dSf, dMf, gp[0], gp[1], gp[2], gp[3], gp[4],
                                  gp[5], gp[6], gp[7], gp[8], ws.data_ptr(), (size_t)ws.numel(), stream);
    else
      st = (method == 1 ? mdn_chunk_bwd_chunked : mdn_chunk_bwd)(
          &p, q, k, v, in.beta, in.log_alpha, in.log_mu, in.eta, S0, M0, cu, d_o->const_data_ptr(), dSf, dMf, gp[0], gp[1],
          gp[2], gp[3], gp[4], gp[5], gp[6], gp[7], gp[8], ws.data_ptr(), (size_t)ws.numel(), stream);
  }
  if (st != MDN_OK) return PyLong_FromLong(st);
  PyObject* r = PyTuple_New(9);
  if (!r) return nullptr;
  for (int i = 0; i < 9; ++i) PyTuple_SET_ITEM(r, i, g[i].defined() ? THPVariable_Wrap(g[i]) : Py_NewRef(Py_None));
  return r;
  NATIVE_CATCH
}

PyObject* mdn_error = nullptr;   // binding.py's MdnError, set when it loads this module

// set_error_class(MdnError)
PyObject* set_error_class(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 1) { PyErr_SetString(PyExc_TypeError, "set_error_class(class)"); return nullptr; }
  Py_XDECREF(mdn_error);
  mdn_error = Py_NewRef(a[0]);
  return Py_NewRef(Py_None);
}

// Throws MdnError(status, where) for a failed call: it arrives as that in Python, from autograd's threads too.  The GIL need not
// be held.
void check(mdn_status st, const char* where) {
  if (st == MDN_OK) return;
  const PyGILState_STATE gil = PyGILState_Ensure();
  PyObject* e = PyObject_CallFunction(mdn_error, "is", (int)st, where);
  if (e) {
    PyErr_SetObject(mdn_error, e);
    Py_DECREF(e);
  }
  python_error err;
  err.persist();
  PyGILState_Release(gil);
  throw err;
}

// ---- chunk_attention: the differentiable forward.  The same two calls as _ChunkAttention of binding.py, as a C++ autograd
// node: a training step of a few hundred tokens takes 55 us on the GPU, and the Python node (apply, saved tensors, the
// engine's way back into Python) made it 138 us.
struct AttnPtrs {   // device pointers of defined tensors, NULL otherwise
  static const float* f(const Tensor& t) { return t.defined() ? static_cast<const float*>(t.const_data_ptr()) : nullptr; }
};

class ChunkAttention : public torch::autograd::Function<ChunkAttention> {
  static mdn_params params(const Tensor& q, const Tensor& v, const Tensor& cu, double scale) {
    const int64_t N = cu.defined() ? cu.numel() - 1 : 0;
    return mdn_params{(int32_t)q.size(0), (int32_t)q.size(1), (int32_t)q.size(2), (int32_t)q.size(3), (int32_t)v.size(3), 64, (int32_t)N,
                      MDN_BF16, MDN_BF16, MDN_PATH_TENSOR, (float)scale, 0};
  }
  // A saved tensor as it was handed to save_for_backward: hooks may have brought back something else.
  static const Tensor& same(const Tensor& t, at::ScalarType dtype, c10::DeviceIndex dev, at::IntArrayRef shape) {
    TORCH_CHECK_VALUE(!t.defined() || (t.is_cuda() && t.get_device() == dev && t.scalar_type() == dtype && t.is_contiguous() && t.sizes() == shape),
                      "a tensor saved for chunk_attention's backward came back with another device, type, shape or stride");
    return t;
  }
  // A byte buffer of the forward on the boundary that it needs (copied there where hooks have moved it).
  static Tensor buffer(const Tensor& t, int64_t bytes, c10::DeviceIndex dev) {
    same(t, at::kByte, dev, {bytes});
    if (reinterpret_cast<uintptr_t>(t.const_data_ptr()) % 1024 == 0) return t;
    return empty_1024(bytes, dev).copy_(t);
  }

 public:
  static torch::autograd::variable_list forward(torch::autograd::AutogradContext* ctx, const Tensor& q, const Tensor& k, const Tensor& v,
                                                const Tensor& beta, const Tensor& log_alpha, const Tensor& log_mu,
                                                const std::optional<Tensor>& eta_, const std::optional<Tensor>& S0_,
                                                const std::optional<Tensor>& M0_, const std::optional<Tensor>& cu_, double scale) {
    auto get = [](const std::optional<Tensor>& t) { return t.has_value() ? *t : Tensor(); };
    const Tensor eta = get(eta_), S0 = get(S0_), M0 = get(M0_), cu = get(cu_);
    const mdn_params p = params(q, v, cu, scale);
    const c10::DeviceIndex dev = q.get_device();
    const int64_t n = p.num_seqs > 0 ? p.num_seqs : p.B;
    const size_t state_bytes = mdn_chunk_states_bytes(&p);
    mdn_ws_layout lay;
    check(state_bytes != 0 ? mdn_workspace_layout(&p, &lay) : MDN_ERR_UNSUPPORTED, "mdn_chunk_fwd_workspace_bytes");
    // the scan's scratch is given back here: what is kept for the backward lives until then, in every layer
    const int64_t need = (int64_t)lay.off_seg, scan = (int64_t)(lay.total_bytes - lay.off_seg);
    Tensor ws = empty({need}, at::kByte, dev), states = empty_1024((int64_t)state_bytes, dev), scratch;
    if (scan > 0) scratch = empty({scan}, at::kByte, dev);
    Tensor o = empty(v.sizes(), q.scalar_type(), dev);
    Tensor Sf = empty({n, p.H, p.dk, p.dv}, at::kFloat, dev), Mf = empty({n, p.H, p.dk, p.dv}, at::kFloat, dev);
    check(mdn_chunk_fwd_keep_states_scratch(
              &p, q.const_data_ptr(), k.const_data_ptr(), v.const_data_ptr(), AttnPtrs::f(beta), AttnPtrs::f(log_alpha),
              AttnPtrs::f(log_mu), AttnPtrs::f(eta), AttnPtrs::f(S0), AttnPtrs::f(M0),
              cu.defined() ? static_cast<const int32_t*>(cu.const_data_ptr()) : nullptr, o.data_ptr(), static_cast<float*>(Sf.data_ptr()),
              static_cast<float*>(Mf.data_ptr()), states.data_ptr(), ws.data_ptr(), (size_t)need, scan > 0 ? scratch.data_ptr() : nullptr,
              (size_t)scan, stream_of(dev)),
          "mdn_chunk_fwd_keep_states");
    ctx->set_materialize_grads(false);
    ctx->save_for_backward({q, k, v, beta, log_alpha, log_mu, eta, S0, M0, cu, states, ws});
    ctx->saved_data["scale"] = scale;
    ctx->saved_data["device"] = (int64_t)dev;
    ctx->saved_data["qk"] = q.sizes().vec();
    ctx->saved_data["v"] = v.sizes().vec();
    ctx->saved_data["seqs"] = (int64_t)p.num_seqs;
    return {o, Sf, Mf};
  }

  static torch::autograd::variable_list backward(torch::autograd::AutogradContext* ctx, torch::autograd::variable_list grads) {
    const auto s = ctx->get_saved_variables();
    const c10::DeviceIndex dev = (c10::DeviceIndex)ctx->saved_data["device"].toInt();
    const auto qk_shape = ctx->saved_data["qk"].toIntVector(), v_shape = ctx->saved_data["v"].toIntVector();
    const Tensor &q = same(s[0], at::kBFloat16, dev, qk_shape), &k = same(s[1], at::kBFloat16, dev, qk_shape);
    const Tensor &v = same(s[2], at::kBFloat16, dev, v_shape), &cu = same(s[9], at::kInt, dev, {ctx->saved_data["seqs"].toInt() + 1});
    for (int i = 3; i < 7; ++i) same(s[i], at::kFloat, dev, {qk_shape[0], qk_shape[1], qk_shape[2]});
    const Tensor &eta = s[6], &S0 = s[7], &M0 = s[8];
    const mdn_params p = params(q, v, cu, ctx->saved_data["scale"].toDouble());
    const int64_t n = p.num_seqs > 0 ? p.num_seqs : p.B;
    mdn_ws_layout lay;
    check(mdn_workspace_layout(&p, &lay), "mdn_workspace_layout");
    const Tensor states = buffer(s[10], (int64_t)mdn_chunk_states_bytes(&p), dev), ws = buffer(s[11], (int64_t)lay.off_seg, dev);
    const Tensor d_o = grads[0].defined() ? grads[0].to(q.scalar_type()).contiguous() : at::zeros_like(v);
    const Tensor dSf = grads[1].defined() ? grads[1].to(at::kFloat).contiguous() : Tensor();
    const Tensor dMf = grads[2].defined() ? grads[2].to(at::kFloat).contiguous() : Tensor();
    const size_t need = mdn_chunk_bwd_saved_workspace_bytes(&p);
    Tensor work = empty_1024((int64_t)need, dev);
    Tensor dq = empty(q.sizes(), q.scalar_type(), dev), dk = empty(q.sizes(), q.scalar_type(), dev), dv = empty(v.sizes(), q.scalar_type(), dev);
    Tensor g[4], dS0, dM0;   // d beta, d log_alpha, d log_mu, d eta
    float* gp[4] = {nullptr, nullptr, nullptr, nullptr};
    for (int i = 0; i < (eta.defined() ? 4 : 3); ++i) {
      g[i] = empty({p.B, p.T, p.H}, at::kFloat, dev);
      gp[i] = static_cast<float*>(g[i].data_ptr());
    }
    if (S0.defined()) dS0 = empty({n, p.H, p.dk, p.dv}, at::kFloat, dev);
    if (M0.defined()) dM0 = empty({n, p.H, p.dk, p.dv}, at::kFloat, dev);
    check(mdn_chunk_bwd_saved_io(&p, q.const_data_ptr(), k.const_data_ptr(), v.const_data_ptr(), AttnPtrs::f(s[3]), AttnPtrs::f(s[4]),
                                 AttnPtrs::f(s[5]), AttnPtrs::f(eta), cu.defined() ? static_cast<const int32_t*>(cu.const_data_ptr()) : nullptr,
                                 ws.data_ptr(), (size_t)ws.numel(), states.const_data_ptr(), d_o.const_data_ptr(), AttnPtrs::f(dSf),
                                 AttnPtrs::f(dMf), dq.data_ptr(), dk.data_ptr(), dv.data_ptr(), gp[0], gp[1], gp[2], gp[3],
                                 dS0.defined() ? static_cast<float*>(dS0.data_ptr()) : nullptr,
                                 dM0.defined() ? static_cast<float*>(dM0.data_ptr()) : nullptr, work.data_ptr(), need, stream_of(dev)),
          "mdn_chunk_bwd_saved_io");
    return {dq, dk, dv, g[0], g[1], g[2], g[3], dS0, dM0, Tensor(), Tensor()};
  }
};

// chunk_attention(q, k, v, beta, log_alpha, log_mu, eta, initial_S, initial_M, cu_seqlens, scale) -> (o, S, M)
PyObject* chunk_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  NATIVE_TRY
  Inputs in;
  float *S0, *M0, scale;
  const int32_t* cu;
  int64_t N;
  if (n != 11 || !parse_inputs(a, &in) || in.dtype != at::kBFloat16 || in.dk != 128 || in.dv != 128 || !parse_cu(a[9], in.dev, &cu, &N) ||
      (N > 0 && in.B != 1) || in.B == 0 || in.T == 0 || in.H == 0)
    return Py_NewRef(Py_None);
  const int64_t nst = N > 0 ? N : in.B;
  if (!parse_state(a[7], in, nst, &S0) || !parse_state(a[8], in, nst, &M0) || !parse_scale(a[10], in.dk, &scale)) return Py_NewRef(Py_None);
  auto maybe = [&](int i) { return a[i] == Py_None ? std::optional<Tensor>() : std::optional<Tensor>(THPVariable_Unpack(a[i])); };
  torch::autograd::variable_list r;
  {
    const Tensor t[6] = {THPVariable_Unpack(a[0]), THPVariable_Unpack(a[1]), THPVariable_Unpack(a[2]),
                         THPVariable_Unpack(a[3]), THPVariable_Unpack(a[4]), THPVariable_Unpack(a[5])};
    const std::optional<Tensor> o[4] = {maybe(6), maybe(7), maybe(8), maybe(9)};
    NoGil g;
    r = ChunkAttention::apply(t[0], t[1], t[2], t[3], t[4], t[5], o[0], o[1], o[2], o[3], (double)scale);
  }
  PyObject* out = PyTuple_New(3);
  if (!out) return nullptr;
  for (int i = 0; i < 3; ++i) PyTuple_SET_ITEM(out, i, THPVariable_Wrap(r[i]));
  return out;
  NATIVE_CATCH
}

// ---- make_layer_ops: fills the mdn_layer_ops at an address from the binding's dicts
bool dict_float(PyObject* d, const char* key, float* out, bool required = true) {
  PyObject* v = PyDict_GetItemString(d, key);
  if (!v) return !required;
  if (PyFloat_Check(v)) *out = static_cast<float>(PyFloat_AS_DOUBLE(v));
  else if (PyLong_Check(v)) *out = static_cast<float>(PyLong_AsDouble(v));
  else return false;
  return true;
}
bool dict_vec(PyObject* d, const char* key, int64_t len, bool optional, c10::DeviceIndex dev, const float** out) {
  *out = nullptr;
  PyObject* v = PyDict_GetItemString(d, key);
  if (!v || v == Py_None) return optional;
  const Tensor* t = cuda_tensor(v, at::kFloat, dev);
  if (!t || t->numel() != len) return false;
  *out = static_cast<const float*>(t->const_data_ptr());
  return true;
}

// fill_layer_ops(address, q, v, gate_param, qk_norm, out_norm_gate, placement) -> True
PyObject* fill_layer_ops(PyObject*, PyObject* const* a, Py_ssize_t n) {
  NATIVE_TRY
  if (n != 7 || !THPVariable_Check(a[1]) || !THPVariable_Check(a[2])) return Py_NewRef(Py_None);
  const Tensor &q = THPVariable_Unpack(a[1]), &v = THPVariable_Unpack(a[2]);
  if (!q.is_cuda() || q.dim() != 4 || v.dim() != 4) return Py_NewRef(Py_None);
  const int64_t H = q.size(2), dv = v.size(3);
  const c10::DeviceIndex dev = q.get_device();
  mdn_layer_ops ops{};
  if (a[3] != Py_None) {
    ops.raw_gates = 1;
    ops.log_mu_min = -1.0f;
    if (!PyDict_Check(a[3]) || !dict_vec(a[3], "a_alpha", H, false, dev, &ops.decay_a_alpha) ||
        !dict_vec(a[3], "b_alpha", H, false, dev, &ops.decay_b_alpha) || !dict_vec(a[3], "a_mu", H, false, dev, &ops.decay_a_mu) ||
        !dict_vec(a[3], "b_mu", H, false, dev, &ops.decay_b_mu) || !dict_float(a[3], "s", &ops.s) ||
        !dict_float(a[3], "tau", &ops.tau) || !dict_float(a[3], "log_mu_min", &ops.log_mu_min, false))
      return Py_NewRef(Py_None);
  }
  if (a[4] != Py_None) {
    ops.qk_norm = 1;
    if (!PyDict_Check(a[4]) || !dict_vec(a[4], "d", H, true, dev, &ops.d) || !dict_float(a[4], "eps", &ops.qk_eps))
      return Py_NewRef(Py_None);
  }
  if (a[5] != Py_None) {
    if (!PyDict_Check(a[5])) return Py_NewRef(Py_None);
    PyObject* gobj = PyDict_GetItemString(a[5], "g");
    const Tensor* g = gobj ? cuda_tensor(gobj, q.scalar_type(), dev) : nullptr;
    if (!g || g->sizes() != v.sizes() || !dict_vec(a[5], "w", dv, true, dev, &ops.w) || !dict_float(a[5], "eps", &ops.rms_eps))
      return Py_NewRef(Py_None);
    ops.out_norm_gate = 1;
    ops.g = g->const_data_ptr();
  }
  if (!PyUnicode_Check(a[6])) return Py_NewRef(Py_None);
  if (PyUnicode_CompareWithASCIIString(a[6], "fused") == 0) ops.placement = 0;
  else if (PyUnicode_CompareWithASCIIString(a[6], "separate") == 0) ops.placement = 1;
  else return Py_NewRef(Py_None);
  mdn_layer_ops* dst = static_cast<mdn_layer_ops*>(PyLong_AsVoidPtr(a[0]));
  if (!dst) return nullptr;
  *dst = ops;
  return Py_NewRef(Py_True);
  NATIVE_CATCH
}

PyMethodDef methods[] = {
    {"decode_step", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(decode_step)), METH_FASTCALL, nullptr},
    {"chunk_fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(chunk_fwd)), METH_FASTCALL, nullptr},
    {"chunk_bwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(chunk_bwd)), METH_FASTCALL, nullptr},
    {"chunk_attention", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(chunk_attention)), METH_FASTCALL, nullptr},
    {"set_error_class", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(set_error_class)), METH_FASTCALL, nullptr},
    {"fill_layer_ops", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fill_layer_ops)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Per-call host work of the binding.", -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
