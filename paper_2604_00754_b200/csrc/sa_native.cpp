// Python entry of the calls a model makes per layer: takes torch tensors, allocates what the call
// returns and enqueues the C ABI call on the current stream.  A pass over a small problem is bound
// by host work, and through ctypes that work (struct and pointer objects, one Python call per
// allocation, the stream look-up) was several times the launches themselves: make_perm 36 us and
// the forward 18 us of host time, of which 12 and 3 us were launches.  The functions take their
// arguments by position; defaults and names live in the Python wrappers.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/EmptyTensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "sa.h"

namespace {

PyObject* g_error_class = nullptr;   // binding.SaError

struct Raised {};                    // a Python exception is set

[[noreturn]] void raise(PyObject* type, const char* text) {
  PyErr_SetString(type, text);
  throw Raised{};
}

void check(int status, const char* where) {
  if (status == SA_OK) return;
  PyObject* e = PyObject_CallFunction(g_error_class, "is", status, where);
  if (e) {
    PyErr_SetObject(g_error_class, e);
    Py_DECREF(e);
  }
  throw Raised{};
}

// The C call, with its arguments in hand, without the interpreter's lock: a launch waits for room
// where the device's queue is full, and other threads go on meanwhile.
template <typename... P, typename... A>
int unlocked(sa_status (*call)(P...), A... args) {
  PyThreadState* state = PyEval_SaveThread();
  const int status = call(static_cast<P>(args)...);
  PyEval_RestoreThread(state);
  return status;
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a tensor");
  return THPVariable_Unpack(o);
}
const at::Tensor* tensor_or_null(PyObject* o) { return o == Py_None ? nullptr : &tensor(o); }
void* ptr(const at::Tensor& t) { return t.data_ptr(); }
void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }

unsigned long long integer_mask(PyObject* o) {        // as int(o), modulo 2^64
  PyObject* i = PyLong_CheckExact(o) ? o : PyNumber_Long(o);
  if (!i) throw Raised{};
  const unsigned long long v = PyLong_AsUnsignedLongLongMask(i);
  if (i != o) Py_DECREF(i);
  return v;
}
long long integer(PyObject* o) { return (long long)integer_mask(o); }
int64_t size(PyObject* o) {                           // a tensor's extent: whole numbers only
  const Py_ssize_t v = PyNumber_AsSsize_t(o, PyExc_OverflowError);
  if (v == -1 && PyErr_Occurred()) throw Raised{};
  return v;
}
double real(PyObject* o) {                            // as float(o)
  PyObject* f = PyFloat_CheckExact(o) ? o : PyNumber_Float(o);
  if (!f) throw Raised{};
  const double v = PyFloat_AS_DOUBLE(f);
  if (f != o) Py_DECREF(f);
  return v;
}
bool truth(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw Raised{};
  return v != 0;
}

sa_stream_t stream() { return (sa_stream_t)c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor fresh(at::IntArrayRef sizes, at::ScalarType type, c10::Device dev) {
  if (!dev.is_cuda()) return at::empty(sizes, at::TensorOptions().dtype(type).device(dev));
  return at::detail::empty_cuda(sizes, type, dev, std::nullopt);
}
void same_layout(const at::Tensor& ref, const at::Tensor* t) {
  if (t && (t->sizes() != ref.sizes() || t->strides() != ref.strides() ||
            t->scalar_type() != ref.scalar_type()))
    raise(PyExc_ValueError, "tensor does not share the layout of its reference tensor");
}

// A tensor with the shape, strides and type of `t`.  A slice of a larger tensor or an expanded one
// has strides that a fresh tensor cannot have: the kernels, which are told one set of strides for
// both, would write outside it.
at::Tensor fresh_like(const at::Tensor& t) {
  if (t.is_cuda() && t.is_non_overlapping_and_dense())
    return at::detail::empty_strided_cuda(t.sizes(), t.strides(), t.scalar_type(), t.device());
  const at::Tensor r = at::empty_like(t);
  same_layout(t, &r);
  return r;
}

sa_problem problem(const at::Tensor& q, const at::Tensor& k, PyObject* w, uint32_t flags,
                   PyObject* scale) {
  sa_problem p{};
  if (q.scalar_type() == at::kFloat) p.dtype = SA_F32;
  else if (q.scalar_type() == at::kBFloat16) p.dtype = SA_BF16;
  else raise(PyExc_TypeError, "q/k/v must be float32 or bfloat16");
  if (q.dim() != 4 || k.dim() != 4) raise(PyExc_ValueError, "q, k, v must be [B,H,n,d]");
  p.B = (int32_t)q.size(0);
  p.Hq = (int32_t)q.size(1);
  p.Hkv = (int32_t)k.size(1);
  p.n = (int32_t)q.size(2);
  p.d = (int32_t)q.size(3);
  p.w = (int32_t)integer(w);
  p.flags = flags;
  p.softmax_scale = (float)real(scale);
  if (q.stride(3) != 1 || k.stride(3) != 1)
    raise(PyExc_ValueError, "the head dimension must be contiguous");
  for (int i = 0; i < 3; ++i) {
    p.q_stride[i] = q.stride(i);
    p.kv_stride[i] = k.stride(i);
  }
  return p;
}

size_t ws_bytes(const sa_problem& p, int op) {
  const size_t n = sa_workspace_bytes(&p, op);
  if (n == (size_t)-1) check(SA_ERR_INVALID_ARG, "sa_workspace_bytes");
  return n;
}

// Scratch for the SA branch's key lists, from the allocator's pool of the current stream; undefined
// where the problem has no use for any, and, with a warning (the sums run in another order then), where there
// is no memory for it.
at::Tensor key_lists(const sa_problem& p, c10::Device dev) {
  const size_t n = sa_workspace_bytes(&p, SA_OP_KEY_LISTS);
  if (n == 0 || n == (size_t)-1) return at::Tensor();
  try {
    return fresh({(int64_t)n}, at::kByte, dev);
  } catch (const c10::OutOfMemoryError&) {
    if (PyErr_WarnEx(PyExc_RuntimeWarning, "no memory for the key lists: the call goes without them", 1) < 0)
      throw Raised{};
    return at::Tensor();
  }
}
void* ptr_or_null(const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }
size_t bytes_of(const at::Tensor& t) { return t.defined() ? (size_t)t.numel() : 0; }

PyObject* wrap(at::Tensor t) { return THPVariable_Wrap(std::move(t)); }
PyObject* pass(PyObject* o) {
  Py_INCREF(o);
  return o;
}

PyObject* tuple(std::initializer_list<PyObject*> items) {
  PyObject* r = PyTuple_New((Py_ssize_t)items.size());
  Py_ssize_t i = 0;
  for (PyObject* o : items) PyTuple_SET_ITEM(r, i++, o);
  return r;
}

// An output: the caller's tensor, or a fresh one (kept alive by `own`).
struct Out {
  at::Tensor own;
  PyObject* given = nullptr;
  const at::Tensor* t = nullptr;
  PyObject* result() { return given ? pass(given) : wrap(own); }
};
template <typename F>
Out output(PyObject* o, F&& make) {
  Out r;
  if (o != Py_None) {
    r.given = o;
    r.t = &tensor(o);
  } else {
    r.own = make();
  }
  return r;
}
void* ptr(const Out& o) { return o.t ? o.t->data_ptr() : o.own.data_ptr(); }

at::Tensor rows_f32(const at::Tensor& q) {
  return fresh({q.size(0), q.size(1), q.size(2)}, at::kFloat, q.device());
}

// make_perm(seed, layer, B, n, perm, inv, ws): perm or inv None: made on the current device
PyObject* make_perm(PyObject* const* a) {
  const int64_t B = size(a[2]), n = size(a[3]);
  const c10::Device dev = a[4] != Py_None ? tensor(a[4]).device()
                                          : c10::Device(c10::kCUDA, c10::cuda::current_device());
  auto make = [&] { return fresh({B, n}, at::kInt, dev); };
  sa_problem p{};
  p.B = (int32_t)B;
  p.n = (int32_t)n;
  const size_t need = ws_bytes(p, SA_OP_MAKE_PERM);
  Out perm = output(a[4], make), inv = output(a[5], make);
  at::Tensor own;
  const at::Tensor* ws = tensor_or_null(a[6]);
  if (!ws) ws = &(own = fresh({(int64_t)need}, at::kByte, dev));
  check(unlocked(sa_make_perm, integer_mask(a[0]), (uint32_t)integer(a[1]), p.B, p.n, (int32_t*)ptr(perm),
                     (int32_t*)ptr(inv), ptr(*ws), (size_t)ws->numel(), stream()),
        "sa_make_perm");
  return tuple({perm.result(), inv.result()});
}

// forward(q, k, v, perm, inv, w, flags, scale, y, want_lse, lse)
PyObject* forward(PyObject* const* a) {
  const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]);
  same_layout(k, &v);
  const sa_problem p = problem(q, k, a[5], (uint32_t)integer(a[6]), a[7]);
  Out y = output(a[8], [&] { return fresh_like(q); });
  same_layout(q, y.t);
  const bool has_lse = a[10] != Py_None || truth(a[9]);
  Out lse;
  if (has_lse) lse = output(a[10], [&] { return rows_f32(q); });
  at::Tensor lists = key_lists(p, q.device());
  check(unlocked(sa_forward_lists, &p, ptr(q), ptr(k), ptr(v), (const int32_t*)ptr(tensor(a[3])),
                   (const int32_t*)ptr(tensor(a[4])), ptr(y), has_lse ? (float*)ptr(lse) : nullptr,
                   ptr_or_null(lists), bytes_of(lists), stream()),
        "sa_forward");
  return has_lse ? tuple({y.result(), lse.result()}) : y.result();
}

// gated_forward(q, k, v, perm, inv, gate_logits, w, flags, scale, save_for_bwd,
//               y, y_sa, y_swa, lse_sa, lse_swa, ws)
PyObject* gated_forward(PyObject* const* a) {
  const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]);
  same_layout(k, &v);
  const bool save = truth(a[9]);
  const uint32_t flags = (uint32_t)integer(a[7]) | (save ? SA_SAVE_FOR_BWD : 0u);
  auto like_q = [&] { return fresh_like(q); };
  auto rows = [&] { return rows_f32(q); };
  Out y = output(a[10], like_q), branch[2], lse[2];
  same_layout(q, y.t);
  for (int x = 0; x < 2; ++x) {
    if (save || a[11 + x] != Py_None) branch[x] = output(a[11 + x], like_q);
    same_layout(q, branch[x].t);
    if (save || a[13 + x] != Py_None) lse[x] = output(a[13 + x], rows);
  }
  auto at_or_null = [](const Out& o) { return o.t || o.own.defined() ? ptr(o) : nullptr; };
  const sa_problem p = problem(q, k, a[6], flags, a[8]);
  const at::Tensor* ws = tensor_or_null(a[15]);
  if (ws && ((uintptr_t)ptr(ws) & 15u)) check(SA_ERR_INVALID_ARG, "sa_swa_gated_forward");
  at::Tensor lists = key_lists(p, q.device());
  check(unlocked(sa_swa_gated_forward_lists, &p, ptr(q), ptr(k), ptr(v), (const int32_t*)ptr(tensor(a[3])),
                             (const int32_t*)ptr(tensor(a[4])), (const float*)ptr(tensor(a[5])),
                             ptr(y), at_or_null(branch[0]), at_or_null(branch[1]),
                             (float*)at_or_null(lse[0]), (float*)at_or_null(lse[1]), ptr_or_null(lists),
                             bytes_of(lists), stream()),
        "sa_swa_gated_forward");
  if (!save) return y.result();
  return tuple({y.result(), branch[0].result(), branch[1].result(), lse[0].result(),
                lse[1].result()});
}

// backward(q, k, v, perm, inv, gate_logits, y_sa, y_swa, lse_sa, lse_swa, dy, w, flags, scale, ws,
//          dq, dk, dv, dgate)
PyObject* backward(PyObject* const* a) {
  const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]);
  same_layout(k, &v);
  const at::Tensor *gate = tensor_or_null(a[5]), *y_swa = tensor_or_null(a[7]),
                   *lse_swa = tensor_or_null(a[9]);
  const at::Tensor &y_sa = tensor(a[6]), &dy = tensor(a[10]);
  same_layout(q, &dy);
  same_layout(q, &y_sa);
  same_layout(q, y_swa);
  Out dq = output(a[15], [&] { return fresh_like(q); });
  Out dk = output(a[16], [&] { return fresh_like(k); });
  Out dv = output(a[17], [&] { return fresh_like(v); });
  same_layout(q, dq.t);
  same_layout(k, dk.t);
  same_layout(k, dv.t);
  Out dgate;
  if (gate) dgate = output(a[18], [&] { return fresh({2, q.size(1)}, at::kFloat, q.device()); });
  const sa_problem p = problem(q, k, a[11], (uint32_t)integer(a[12]), a[13]);
  at::Tensor own;
  const at::Tensor* ws = tensor_or_null(a[14]);
  if (!ws) ws = &(own = fresh({(int64_t)ws_bytes(p, SA_OP_BACKWARD)}, at::kByte, q.device()));
  check(unlocked(sa_backward, &p, ptr(q), ptr(k), ptr(v), (const int32_t*)ptr(tensor(a[3])),
                    (const int32_t*)ptr(tensor(a[4])), (const float*)ptr(gate), ptr(y_sa),
                    ptr(y_swa), (const float*)ptr(tensor(a[8])), (const float*)ptr(lse_swa),
                    ptr(dy), ptr(dq), ptr(dk), ptr(dv), gate ? (float*)ptr(dgate) : nullptr,
                    ptr(*ws), (size_t)ws->numel(), stream()),
        "sa_backward");
  return tuple({dq.result(), dk.result(), dv.result(), gate ? dgate.result() : pass(Py_None)});
}

template <PyObject* (*F)(PyObject* const*), int kArgs>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs != kArgs) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  try {
    return F(args);
  } catch (const Raised&) {
  } catch (const c10::OutOfMemoryError& e) {
    PyObject* torch_module = PyImport_ImportModule("torch");
    PyObject* type = torch_module ? PyObject_GetAttrString(torch_module, "OutOfMemoryError") : nullptr;
    if (type) PyErr_SetString(type, e.what_without_backtrace());
    Py_XDECREF(type);
    Py_XDECREF(torch_module);
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
  }
  return nullptr;
}

PyObject* set_error_class(PyObject*, PyObject* cls) {
  Py_INCREF(cls);
  Py_XDECREF(g_error_class);
  g_error_class = cls;
  Py_RETURN_NONE;
}

#define SA_FAST(name, n) \
  {#name, (PyCFunction)(void (*)(void))entry<name, n>, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    SA_FAST(make_perm, 7),
    SA_FAST(forward, 11),
    SA_FAST(gated_forward, 16),
    SA_FAST(backward, 19),
    {"set_error_class", set_error_class, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&g_module); }
