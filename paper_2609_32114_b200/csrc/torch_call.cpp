// The two torch entry points of binding.py (ha_la_prefill, ha_la_decode) as one native call each: tensors are unpacked,
// checked, missing outputs allocated and the C struct filled here instead of in Python (one decoding step cost its caller
// 12 us of interpreter and ctypes time around a 3 us kernel).  Nothing is computed here.  A call that is not entirely
// ordinary -- a tensor of another type, layout, size or device, the batch dimension left out -- returns None, and binding.py
// takes it through its own marshalling, which also words the errors.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <optional>

#include "ha_la.h"

namespace {

int (*g_prefill)(const ha_la_prefill_args*, void*) = nullptr;
int (*g_prefill_bytes)(const ha_la_prefill_args*, size_t*) = nullptr;
int (*g_decode)(const ha_la_decode_args*, void*) = nullptr;

// a tensor, or nullptr for None; anything else is not ordinary
bool unpack(PyObject* o, const at::Tensor** t) {
  *t = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) return false;
  *t = &THPVariable_Unpack(o);
  return true;
}
bool plain(const at::Tensor* t, at::ScalarType type, int64_t dim) {
  return t && t->is_cuda() && t->scalar_type() == type && t->dim() == dim && t->is_contiguous();
}
// q [rows.., HK, dk] sets the sizes of k, v [rows.., HV, dv], g [rows.., HV] (KDA: and dk) and beta [rows.., HV].  The others may
// have more rows than q where they lie one behind the other.
bool inputs(const at::Tensor* q, const at::Tensor* k, const at::Tensor* v, const at::Tensor* g, const at::Tensor* beta,
            int64_t dim, bool kda) {
  if (!q || !(q->scalar_type() == at::kBFloat16 || q->scalar_type() == at::kFloat)) return false;
  if (!plain(q, q->scalar_type(), dim) || !plain(k, q->scalar_type(), dim) || !plain(v, q->scalar_type(), dim) ||
      !plain(g, at::kFloat, kda ? dim : dim - 1) || !plain(beta, at::kFloat, dim - 1))
    return false;
  // (as arrays: a tensor's size(i) is a call and a range check each)
  const int64_t *qs = q->sizes().data(), *ks = k->sizes().data(), *vs = v->sizes().data(), *gs = g->sizes().data(), *bs = beta->sizes().data();
  const int h = (int)dim - 2;                            // (dimension of the heads)
  const auto device = q->device();
  for (const at::Tensor* t : {k, v, g, beta})
    if (t->device() != device) return false;
  for (const int64_t* ts : {ks, vs, gs, bs}) {
    if (ts[0] < qs[0]) return false;
    if (h == 2 && !(ts[1] == qs[1] || (qs[0] == 1 && ts[1] > qs[1]))) return false;
  }
  return ks[h] == qs[h] && ks[h + 1] == qs[h + 1] && gs[h] == vs[h] && bs[h] == vs[h] && (!kda || gs[h + 1] == qs[h + 1]);
}
// an optional tensor with room for n elements that the kernels can take by its address
bool room(const at::Tensor* t, const at::Tensor& q, at::ScalarType type, int64_t n) {
  return !t || (t->device() == q.device() && t->scalar_type() == type && t->is_contiguous() && t->numel() >= n);
}
void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }

// The stream of a call.  Where the caller names another than torch's current one, that is the current one while this lives:
// tensors that the call allocates and fills come from that stream's pool and are filled in its order, and nothing that is
// queued on the current stream can still be using (or clear, in the status word's case) what the kernels write.  The caller
// reads them on the current stream once it has waited, so they are recorded there too and not reused before that is over.
struct CallStream {
  void* handle = nullptr;
  std::optional<c10::cuda::CUDAStream> current;          // (set: another stream's call)
  std::optional<c10::cuda::CUDAStreamGuard> guard;
  bool set(PyObject* stream, const at::Tensor& q) {      // false: Python error
    if (stream == Py_None) {
      handle = at::cuda::getCurrentCUDAStream(q.get_device()).stream();
      return true;
    }
    handle = PyLong_AsVoidPtr(stream);
    return !PyErr_Occurred();
  }
  void will_allocate(PyObject* stream, const at::Tensor& q) {
    if (stream == Py_None || current) return;
    const c10::cuda::CUDAStream c = c10::cuda::getCurrentCUDAStream(q.get_device());
    if (c.stream() == handle) return;
    current = c;
    guard.emplace(c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(handle), q.get_device()));
  }
  void allocated(const at::Tensor& t) const {
    if (current) t.record_stream(current->unwrap());
  }
};

// (prefill, workspace bytes, decode): the library's entry points, as addresses
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 3) { PyErr_SetString(PyExc_TypeError, "three addresses"); return nullptr; }
  g_prefill = reinterpret_cast<decltype(g_prefill)>(PyLong_AsVoidPtr(a[0]));
  g_prefill_bytes = reinterpret_cast<decltype(g_prefill_bytes)>(PyLong_AsVoidPtr(a[1]));
  g_decode = reinterpret_cast<decltype(g_decode)>(PyLong_AsVoidPtr(a[2]));
  if (PyErr_Occurred()) return nullptr;
  Py_RETURN_NONE;
}

// decode(q, k, v, g, beta, state, stream, kda, scale, o, state_out) -> (o, state_out) | status | None
PyObject* decode_call(PyObject* const* a, Py_ssize_t n) {
  if (n != 11 || !g_decode) { PyErr_SetString(PyExc_TypeError, "eleven arguments"); return nullptr; }
  const at::Tensor *q, *k, *v, *g, *beta, *st, *o, *so;
  const bool kda = a[7] == Py_True;
  if (!unpack(a[0], &q) || !unpack(a[1], &k) || !unpack(a[2], &v) || !unpack(a[3], &g) || !unpack(a[4], &beta) ||
      !unpack(a[5], &st) || !unpack(a[9], &o) || !unpack(a[10], &so) || !inputs(q, k, v, g, beta, 3, kda))
    Py_RETURN_NONE;
  const int64_t state = q->size(0) * v->size(1) * q->size(2) * v->size(2);
  if (!room(st, *q, at::kFloat, state) || !room(so, *q, at::kFloat, state) ||
      !room(o, *q, q->scalar_type(), q->size(0) * v->size(1) * v->size(2)))
    Py_RETURN_NONE;
  ha_la_decode_args d{};
  d.variant = kda;
  d.dtype = q->scalar_type() == at::kFloat;
  d.num_seqs = (int32_t)q->size(0);
  d.num_qk_heads = (int32_t)q->size(1);
  d.num_v_heads = (int32_t)v->size(1);
  d.d_k = (int32_t)q->size(2);
  d.d_v = (int32_t)v->size(2);
  d.scale = (float)PyFloat_AsDouble(a[8]);
  if (PyErr_Occurred()) return nullptr;
  CallStream on;
  if (!on.set(a[6], *q)) return nullptr;
  at::Tensor o_new, s_new;
  if (!o || (!so && !st)) on.will_allocate(a[6], *q);
  if (!o) { o_new = at::empty(v->sizes(), v->options()); o = &o_new; on.allocated(o_new); }
  if (!so) {
    if (st) so = st;
    else { s_new = at::empty({d.num_seqs, d.num_v_heads, d.d_k, d.d_k}, g->options()); so = &s_new; on.allocated(s_new); }
  }
  d.q = ptr(q); d.k = ptr(k); d.v = ptr(v);
  d.g = (const float*)ptr(g); d.beta = (const float*)ptr(beta);
  d.h_in = (const float*)ptr(st); d.h_out = (float*)ptr(so); d.o = ptr(o);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = g_decode(&d, on.handle);
  Py_END_ALLOW_THREADS
  if (rc != HA_LA_OK) return PyLong_FromLong(rc);
  PyObject* po = o == &o_new ? THPVariable_Wrap(o_new) : Py_NewRef(a[9]);
  PyObject* ps = so == &s_new ? THPVariable_Wrap(s_new) : Py_NewRef(so == st ? a[5] : a[10]);
  PyObject* r = PyTuple_Pack(2, po, ps);
  Py_XDECREF(po);
  Py_XDECREF(ps);
  return r;
}

// prefill(q, k, v, g, beta, h0, cu_seqlens, max_seqlen, stream, kda, scale, o, hT, want_hT, workspace, status_word)
//   -> (o, hT | None, status_word, workspace) | status | None
PyObject* prefill_call(PyObject* const* a, Py_ssize_t n) {
  if (n != 16 || !g_prefill) { PyErr_SetString(PyExc_TypeError, "sixteen arguments"); return nullptr; }
  const at::Tensor *q, *k, *v, *g, *beta, *h0, *cu, *o, *hT, *ws, *sw;
  if (a[9] != Py_True && a[9] != Py_False) Py_RETURN_NONE;
  const bool kda = a[9] == Py_True;
  if (!unpack(a[0], &q) || !unpack(a[1], &k) || !unpack(a[2], &v) || !unpack(a[3], &g) || !unpack(a[4], &beta) ||
      !unpack(a[5], &h0) || !unpack(a[6], &cu) || !unpack(a[11], &o) || !unpack(a[12], &hT) || !unpack(a[14], &ws) ||
      !unpack(a[15], &sw) || !inputs(q, k, v, g, beta, 4, kda))
    Py_RETURN_NONE;
  if (cu && (!plain(cu, at::kInt, 1) || cu->device() != q->device() || q->size(0) != 1)) Py_RETURN_NONE;
  if (ws && (!plain(ws, at::kByte, 1) || ws->device() != q->device())) Py_RETURN_NONE;
  const int64_t N = cu ? cu->numel() - 1 : q->size(0), state = N * v->size(2) * q->size(3) * v->size(3);
  if (!room(h0, *q, at::kFloat, state) || !room(hT, *q, at::kFloat, state) ||
      !room(o, *q, q->scalar_type(), q->size(0) * q->size(1) * v->size(2) * v->size(3)) || !room(sw, *q, at::kInt, 1))
    Py_RETURN_NONE;
  ha_la_prefill_args d{};
  d.variant = kda;
  d.dtype = q->scalar_type() == at::kFloat;
  d.batch = (int32_t)q->size(0);
  d.seqlen = (int32_t)q->size(1);
  d.num_qk_heads = (int32_t)q->size(2);
  d.num_v_heads = (int32_t)v->size(2);
  d.d_k = (int32_t)q->size(3);
  d.d_v = (int32_t)v->size(3);
  d.chunk = 64;
  d.scale = (float)PyFloat_AsDouble(a[10]);
  d.num_seqs = cu ? (int32_t)N : 0;
  d.max_seqlen = (int32_t)PyLong_AsLong(a[7]);
  if (PyErr_Occurred()) return nullptr;
  d.q = ptr(q); d.k = ptr(k); d.v = ptr(v);
  d.g = (const float*)ptr(g); d.beta = (const float*)ptr(beta);
  d.h0 = (const float*)ptr(h0); d.cu_seqlens = (const int32_t*)ptr(cu);
  size_t need = 0;
  int rc = g_prefill_bytes(&d, &need);
  if (rc != HA_LA_OK) Py_RETURN_NONE;                     // (binding.py words the error)
  at::Tensor o_new, h_new, w_new, s_new;
  // (asked for its truth value only where the call has to know: when it brings no hT)
  const int want_hT = hT ? 0 : PyObject_IsTrue(a[13]);
  if (want_hT < 0) return nullptr;
  CallStream on;
  if (!on.set(a[8], *q)) return nullptr;
  if (!o || (!hT && want_hT) || !ws || !sw) on.will_allocate(a[8], *q);
  if (!o) { o_new = at::empty(v->sizes(), v->options()); o = &o_new; on.allocated(o_new); }
  if (!hT && want_hT) { h_new = at::empty({N, v->size(2), q->size(3), v->size(3)}, g->options()); hT = &h_new; on.allocated(h_new); }
  if (!ws) { w_new = at::empty({(int64_t)need + 256}, g->options().dtype(at::kByte)); ws = &w_new; on.allocated(w_new); }
  if (!sw) { s_new = at::zeros({1}, g->options().dtype(at::kInt)); sw = &s_new; on.allocated(s_new); }
  d.o = ptr(o); d.hT = (float*)ptr(hT); d.status_word = (int32_t*)ptr(sw);
  const uintptr_t base = (uintptr_t)ws->data_ptr(), al = (base + 255) / 256 * 256;
  d.workspace = (void*)al;
  const int64_t pad = (int64_t)(al - base);
  d.workspace_bytes = ws->numel() > pad ? (size_t)(ws->numel() - pad) : 0;   // (a buffer may end before its first aligned byte)
  Py_BEGIN_ALLOW_THREADS
  rc = g_prefill(&d, on.handle);
  Py_END_ALLOW_THREADS
  if (rc != HA_LA_OK) return PyLong_FromLong(rc);
  PyObject* r = PyTuple_New(4);
  if (!r) return nullptr;
  PyTuple_SET_ITEM(r, 0, o == &o_new ? THPVariable_Wrap(o_new) : Py_NewRef(a[11]));
  PyTuple_SET_ITEM(r, 1, hT == &h_new && hT ? THPVariable_Wrap(h_new) : Py_NewRef(a[12]));
  PyTuple_SET_ITEM(r, 2, sw == &s_new ? THPVariable_Wrap(s_new) : Py_NewRef(a[15]));
  PyTuple_SET_ITEM(r, 3, ws == &w_new ? THPVariable_Wrap(w_new) : Py_NewRef(a[14]));
  return r;
}

// torch's C++ calls throw (no memory, no driver, a tensor without storage).  An exception that left these functions would go
// through the interpreter's C frames and end the process; torch's own translation gives the caller the type that the same
// call raises in Python.
template <PyObject* (*call)(PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  return call(a, n);
  END_HANDLE_TH_ERRORS
}

PyMethodDef kMethods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&bind)), METH_FASTCALL, nullptr},
    {"decode", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&guarded<decode_call>)), METH_FASTCALL, nullptr},
    {"prefill", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&guarded<prefill_call>)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "ha_la_torch_call", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_ha_la_torch_call(void) { return PyModule_Create(&kModule); }
