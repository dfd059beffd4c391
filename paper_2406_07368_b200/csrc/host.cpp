// Native side of the Python binding: takes torch tensors, checks them, allocates the outputs the caller did not bring
// and calls the C entry points of include/la.h.
//
// What bounds a small call (one decode step, a round on one draft tree) is the host: with the checks and the argument
// marshalling in Python (ctypes) a decode step of one sequence took 16 us and a verify + accept + commit round 64 us
// whatever the kernels' own time.  Here the same work is a few hundred nanoseconds beside the launch itself.
#include <Python.h>

#include <ATen/EmptyTensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <initializer_list>

#include "la.h"
#include "la_internal.h"

namespace {

// One per Context: the C handle and what the checks need to know about it.
struct Plan {
  PyObject_HEAD
  la_ctx* ctx;
  int64_t H, d, W, max_depth;
  at::ScalarType io;
};

PyObject *s_S, *s_z, *s_win, *s_pos, *s_cuda_stream, *g_error;   // interned names; the binding's exception class

// A Python exception is set; unwinds to the method's edge.
struct Raised {};

[[noreturn]] void fail(const char* fn, la_status code) {
  PyObject* e = PyObject_CallFunction(g_error, "si", fn, (int)code);
  if (e) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  throw Raised();
}
inline void check(const char* fn, la_status code) {
  if (code != LA_OK) fail(fn, code);
}

const at::Tensor& tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor", name);
    throw Raised();
  }
  return THPVariable_Unpack(o);
}
const char* dtype_name(at::ScalarType t) {
  return t == at::kFloat ? "torch.float32" : t == at::kBFloat16 ? "torch.bfloat16" : t == at::kInt ? "torch.int32" : "torch.int64";
}
using Shape = std::initializer_list<int64_t>;

// Device pointer of a tensor with exactly this type and shape; null for None (the C side says where that is an error).
void* ptr(PyObject* o, at::ScalarType dtype, Shape shape, const char* name) {
  if (o == Py_None) return nullptr;
  const at::Tensor& t = tensor(o, name);
  if (!t.is_cuda() || !t.is_contiguous()) {
    PyErr_Format(PyExc_ValueError, "%s must be a contiguous CUDA tensor", name);
    throw Raised();
  }
  if (t.scalar_type() != dtype) {
    PyErr_Format(PyExc_ValueError, "%s must have dtype %s", name, dtype_name(dtype));
    throw Raised();
  }
  if (t.sizes() != at::IntArrayRef(shape)) {
    PyObject* want = PyTuple_New((Py_ssize_t)shape.size());
    Py_ssize_t i = 0;
    for (int64_t x : shape) PyTuple_SET_ITEM(want, i++, PyLong_FromLongLong(x));
    PyErr_Format(PyExc_ValueError, "%s must have shape %R", name, want);
    Py_DECREF(want);
    throw Raised();
  }
  return t.data_ptr();
}

// Small int32 outputs of one call that the caller did not bring share one allocation (a trip through the allocator costs a
// fifth of a launch); each starts on a 64-byte boundary of it.
struct Pool {
  at::Tensor base;
  int64_t used = 0;
  at::Tensor take(const at::Tensor& like, Shape shape, int64_t room) {
    if (!base.defined()) base = at::detail::empty_cuda({room}, at::kInt, like.device(), std::nullopt);
    at::Tensor t = at::detail::make_tensor<at::TensorImpl>(c10::Storage(base.storage()), base.key_set(), base.dtype());
    t.unsafeGetTensorImpl()->set_storage_offset(used);
    t.unsafeGetTensorImpl()->set_sizes_contiguous(at::IntArrayRef(shape));
    used += padded(t.numel());
    return t;
  }
  static int64_t padded(int64_t n) { return (n + 15) & ~int64_t(15); }
};

// The given tensor, or a new one on the device of `like`.  Holds the reference that is returned to Python.
struct Out {
  PyObject* obj = nullptr;
  void* p = nullptr;
  Out(PyObject* given, const at::Tensor& like, at::ScalarType dtype, Shape shape, const char* name) {
    if (given != Py_None) {
      p = ptr(given, dtype, shape, name);
      Py_INCREF(given);
      obj = given;
    } else {
      at::Tensor t = at::detail::empty_cuda(at::IntArrayRef(shape), dtype, like.device(), std::nullopt);
      p = t.data_ptr();
      obj = THPVariable_Wrap(std::move(t));
      if (!obj) throw Raised();
    }
  }
  Out(PyObject* given, const at::Tensor& like, Shape shape, const char* name, Pool& pool, int64_t room) {
    if (given != Py_None) {
      p = ptr(given, at::kInt, shape, name);
      Py_INCREF(given);
      obj = given;
    } else {
      at::Tensor t = pool.take(like, shape, room);
      p = t.data_ptr();
      obj = THPVariable_Wrap(std::move(t));
      if (!obj) throw Raised();
    }
  }
  Out(const Out&) = delete;
  ~Out() { Py_XDECREF(obj); }
  PyObject* release() {
    PyObject* o = obj;
    obj = nullptr;
    return o;
  }
};

// First argument of a call: a CUDA tensor with this many dimensions (its sizes give B and T or N).
const at::Tensor& lead(PyObject* o, int64_t dims, const char* name) {
  const at::Tensor& t = tensor(o, name);
  if (t.dim() != dims) {
    PyErr_Format(PyExc_ValueError, "%s must have %d dimensions", name, (int)dims);
    throw Raised();
  }
  if (!t.is_cuda()) {
    PyErr_Format(PyExc_ValueError, "%s must be a contiguous CUDA tensor", name);
    throw Raised();
  }
  return t;
}

// The state's four tensors.  They are held until the call is over: an attribute may be a property that makes a view anew.
struct StateArg {
  la_state st;
  PyObject* held[4] = {nullptr, nullptr, nullptr, nullptr};
  StateArg(const Plan* p, PyObject* state, int64_t B) {
    try {
      st.S = (float*)field(0, state, s_S, at::kFloat, {B, p->H, p->d, p->d}, "state.S");
      st.z = (float*)field(1, state, s_z, at::kFloat, {B, p->H, p->d}, "state.z");
      st.win = field(2, state, s_win, p->io, {B, p->H, p->W - 1, p->d}, "state.win");
      st.pos = (int64_t*)field(3, state, s_pos, at::kLong, {B}, "state.pos");
    } catch (...) {
      release();
      throw;
    }
    if (p->W == 1) st.win = nullptr;
  }
  StateArg(const StateArg&) = delete;
  ~StateArg() { release(); }
  void release() {
    for (PyObject*& o : held) Py_CLEAR(o);
  }
  void* field(int i, PyObject* state, PyObject* attr, at::ScalarType dtype, Shape shape, const char* name) {
    held[i] = PyObject_GetAttr(state, attr);
    if (!held[i]) throw Raised();
    return ptr(held[i], dtype, shape, name);
  }
};

void* stream_of(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* v = PyObject_GetAttr(o, s_cuda_stream);
  if (!v) throw Raised();
  void* s = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  if (PyErr_Occurred()) throw Raised();
  return s;
}
// int(o) and float(o): whatever those take (a group size computed as 64.0, a one-element tensor).
long integer(PyObject* o) {
  PyObject* n = PyNumber_Long(o);
  if (!n) throw Raised();
  const long v = PyLong_AsLong(n);
  Py_DECREF(n);
  if (v == -1 && PyErr_Occurred()) throw Raised();
  return v;
}
float real(PyObject* o) {
  PyObject* n = PyNumber_Float(o);
  if (!n) throw Raised();
  const double v = PyFloat_AS_DOUBLE(n);
  Py_DECREF(n);
  return (float)v;
}
bool truth(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw Raised();
  return v != 0;
}

// Runs a C entry point with the interpreter lock released (a launch blocks while the stream's queue is full).
template <typename F> la_status unlocked(F&& f) {
  la_status r;
  Py_BEGIN_ALLOW_THREADS
  r = f();
  Py_END_ALLOW_THREADS
  return r;
}
// Method edge: arity check, C++ exceptions to Python ones.
template <typename F> PyObject* method(Py_ssize_t got, Py_ssize_t want, F&& f) {
  if (got != want) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
    return nullptr;
  }
  try {
    return f();
  } catch (const Raised&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}
PyObject* pair(Out& a, Out& b) {
  PyObject* t = PyTuple_New(2);
  if (!t) throw Raised();
  PyTuple_SET_ITEM(t, 0, a.release());
  PyTuple_SET_ITEM(t, 1, b.release());
  return t;
}

// (q, k, v, conv_w, state, init_state, out, stream)
PyObject* prefill(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Plan* p = (Plan*)self;
  return method(n, 8, [&] {
    const at::Tensor& q = lead(a[0], 4, "q");
    const int64_t B = q.size(0), T = q.size(2);
    const Shape shp = {B, p->H, T, p->d};
    StateArg st(p, a[4], B);
    const void *qp = ptr(a[0], p->io, shp, "q"), *kp = ptr(a[1], p->io, shp, "k"), *vp = ptr(a[2], p->io, shp, "v");
    const float* w = (const float*)ptr(a[3], at::kFloat, {p->H, p->d, p->W}, "conv_w");
    const int init = truth(a[5]);
    Out o(a[6], q, p->io, shp, "o");
    void* s = stream_of(a[7]);
    check("la_prefill", unlocked([&] { return la_prefill(p->ctx, (int32_t)B, (int32_t)T, qp, kp, vp, w, init, &st.st, o.p, s); }));
    return o.release();
  });
}
// (q, k, v, conv_w, state, group, alpha, softmax_scale, init_state, out, stream)
PyObject* prefill_grouped(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Plan* p = (Plan*)self;
  return method(n, 11, [&] {
    const at::Tensor& q = lead(a[0], 4, "q");
    const int64_t B = q.size(0), T = q.size(2);
    const Shape shp = {B, p->H, T, p->d};
    StateArg st(p, a[4], B);
    const void *qp = ptr(a[0], p->io, shp, "q"), *kp = ptr(a[1], p->io, shp, "k"), *vp = ptr(a[2], p->io, shp, "v");
    const float* w = (const float*)ptr(a[3], at::kFloat, {p->H, p->d, p->W}, "conv_w");
    const int32_t group = (int32_t)integer(a[5]);
    const float alpha = real(a[6]), scale = real(a[7]);
    const int init = truth(a[8]);
    Out o(a[9], q, p->io, shp, "o");
    void* s = stream_of(a[10]);
    check("la_prefill_grouped", unlocked([&] {
            return la_prefill_grouped(p->ctx, (int32_t)B, (int32_t)T, qp, kp, vp, w, group, alpha, scale, init, &st.st, o.p, s);
          }));
    return o.release();
  });
}
// (q, k, v, conv_w, state, out, stream)
PyObject* decode_step(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Plan* p = (Plan*)self;
  return method(n, 7, [&] {
    const at::Tensor& q = lead(a[0], 3, "q");
    const int64_t B = q.size(0);
    const Shape shp = {B, p->H, p->d};
    StateArg st(p, a[4], B);
    const void *qp = ptr(a[0], p->io, shp, "q"), *kp = ptr(a[1], p->io, shp, "k"), *vp = ptr(a[2], p->io, shp, "v");
    const float* w = (const float*)ptr(a[3], at::kFloat, {p->H, p->d, p->W}, "conv_w");
    Out o(a[5], q, p->io, shp, "o");
    void* s = stream_of(a[6]);
    check("la_decode_step", unlocked([&] { return la_decode_step(p->ctx, (int32_t)B, qp, kp, vp, w, &st.st, o.p, s); }));
    return o.release();
  });
}
// (q, k, v, parent, conv_w, state, out, stream)
PyObject* verify_tree(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Plan* p = (Plan*)self;
  return method(n, 8, [&] {
    const at::Tensor& q = lead(a[0], 4, "q");
    const int64_t B = q.size(0), N = q.size(2);
    const Shape shp = {B, p->H, N, p->d};
    StateArg st(p, a[5], B);
    const void *qp = ptr(a[0], p->io, shp, "q"), *kp = ptr(a[1], p->io, shp, "k"), *vp = ptr(a[2], p->io, shp, "v");
    const int32_t* parent = (const int32_t*)ptr(a[3], at::kInt, {B, N}, "parent");
    const float* w = (const float*)ptr(a[4], at::kFloat, {p->H, p->d, p->W}, "conv_w");
    Out o(a[6], q, p->io, shp, "o");
    void* s = stream_of(a[7]);
    check("la_verify_tree",
          unlocked([&] { return la_verify_tree(p->ctx, (int32_t)B, (int32_t)N, qp, kp, vp, parent, w, &st.st, o.p, s); }));
    return o.release();
  });
}
// (k, v, parent, accept_node, state, path_out, commit_len, stream)
PyObject* commit(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Plan* p = (Plan*)self;
  return method(n, 8, [&] {
    const at::Tensor& k = lead(a[0], 4, "k");
    const int64_t B = k.size(0), N = k.size(2);
    const Shape shp = {B, p->H, N, p->d};
    StateArg st(p, a[4], B);
    const void *kp = ptr(a[0], p->io, shp, "k"), *vp = ptr(a[1], p->io, shp, "v");
    const int32_t* parent = (const int32_t*)ptr(a[2], at::kInt, {B, N}, "parent");
    const int32_t* accept = (const int32_t*)ptr(a[3], at::kInt, {B}, "accept_node");
    // Buffers made here have no earlier contents to keep: the kernel fills them for skipped sequences too (-1 and 0),
    // which takes the place of two fill launches.
    const int fresh = (a[5] == Py_None ? LA_FRESH_PATH : 0) | (a[6] == Py_None ? LA_FRESH_LEN : 0);
    Pool pool;
    const int64_t room = Pool::padded(B * p->max_depth) + Pool::padded(B);
    Out path(a[5], k, {B, p->max_depth}, "path_out", pool, room), len(a[6], k, {B}, "commit_len", pool, room);
    void* s = stream_of(a[7]);
    check("la_commit", unlocked([&] {
            return la_commit_fresh(p->ctx, (int32_t)B, (int32_t)N, kp, vp, parent, accept, &st.st, (int32_t*)path.p,
                                   (int32_t*)len.p, fresh, s);
          }));
    return pair(path, len);
  });
}
// (parent, draft_token, pred_root, pred, accept_node, accept_len, next_token, stream)
PyObject* accept_greedy(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Plan* p = (Plan*)self;
  return method(n, 8, [&] {
    const at::Tensor& par = lead(a[0], 2, "parent");
    const int64_t B = par.size(0), N = par.size(1);
    const int32_t* parent = (const int32_t*)ptr(a[0], at::kInt, {B, N}, "parent");
    const int32_t* draft = (const int32_t*)ptr(a[1], at::kInt, {B, N}, "draft_token");
    const int32_t* root = (const int32_t*)ptr(a[2], at::kInt, {B}, "pred_root");
    const int32_t* pred = (const int32_t*)ptr(a[3], at::kInt, {B, N}, "pred");
    Pool pool;
    const int64_t room = 3 * Pool::padded(B);
    Out node(a[4], par, {B}, "accept_node", pool, room), len(a[5], par, {B}, "accept_len", pool, room),
        next(a[6], par, {B}, "next_token", pool, room);
    void* s = stream_of(a[7]);
    check("la_accept_greedy", unlocked([&] {
            return la_accept_greedy(p->ctx, (int32_t)B, (int32_t)N, parent, draft, root, pred, (int32_t*)node.p, (int32_t*)len.p,
                                    (int32_t*)next.p, s);
          }));
    PyObject* t = PyTuple_New(3);
    if (!t) throw Raised();
    PyTuple_SET_ITEM(t, 0, node.release());
    PyTuple_SET_ITEM(t, 1, len.release());
    PyTuple_SET_ITEM(t, 2, next.release());
    return t;
  });
}
// (parent, score, thresh, accept_node, accept_len, stream)
PyObject* accept_threshold(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Plan* p = (Plan*)self;
  return method(n, 6, [&] {
    const at::Tensor& par = lead(a[0], 2, "parent");
    const int64_t B = par.size(0), N = par.size(1);
    const int32_t* parent = (const int32_t*)ptr(a[0], at::kInt, {B, N}, "parent");
    const float* score = (const float*)ptr(a[1], at::kFloat, {B, N}, "score");
    const float* thresh = (const float*)ptr(a[2], at::kFloat, {B, N}, "thresh");
    Pool pool;
    const int64_t room = 2 * Pool::padded(B);
    Out node(a[3], par, {B}, "accept_node", pool, room), len(a[4], par, {B}, "accept_len", pool, room);
    void* s = stream_of(a[5]);
    check("la_accept_threshold", unlocked([&] {
            return la_accept_threshold(p->ctx, (int32_t)B, (int32_t)N, parent, score, thresh, (int32_t*)node.p, (int32_t*)len.p, s);
          }));
    return pair(node, len);
  });
}

PyObject* plan_new(PyTypeObject* type, PyObject* args, PyObject*) {
  unsigned long long handle;
  long long H, d, W, max_depth;
  int bf16;
  if (!PyArg_ParseTuple(args, "KLLLLp", &handle, &H, &d, &W, &max_depth, &bf16)) return nullptr;
  Plan* p = (Plan*)type->tp_alloc(type, 0);
  if (!p) return nullptr;
  p->ctx = reinterpret_cast<la_ctx*>((uintptr_t)handle);
  p->H = H;
  p->d = d;
  p->W = W;
  p->max_depth = max_depth;
  p->io = bf16 ? at::kBFloat16 : at::kFloat;
  return (PyObject*)p;
}
void plan_dealloc(PyObject* self) { Py_TYPE(self)->tp_free(self); }
PyObject* plan_close(PyObject* self, PyObject*) {   // calls after this get LA_ERR_INVALID_ARG, like a null handle
  ((Plan*)self)->ctx = nullptr;
  Py_RETURN_NONE;
}
#define LA_FAST(f) {#f, (PyCFunction)(void (*)(void)) f, METH_FASTCALL, nullptr}
PyMethodDef plan_methods[] = {LA_FAST(prefill), LA_FAST(prefill_grouped), LA_FAST(decode_step), LA_FAST(verify_tree),
                              LA_FAST(commit), LA_FAST(accept_greedy), LA_FAST(accept_threshold),
                              {"close", plan_close, METH_NOARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyTypeObject PlanType = {PyVarObject_HEAD_INIT(nullptr, 0)};

PyObject* set_error(PyObject*, PyObject* cls) {
  Py_INCREF(cls);
  Py_XDECREF(g_error);
  g_error = cls;
  Py_RETURN_NONE;
}
PyMethodDef module_methods[] = {{"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, module_methods};

}  // namespace

PyMODINIT_FUNC PyInit__host(void) {
  s_S = PyUnicode_InternFromString("S");
  s_z = PyUnicode_InternFromString("z");
  s_win = PyUnicode_InternFromString("win");
  s_pos = PyUnicode_InternFromString("pos");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  g_error = PyExc_RuntimeError;
  Py_INCREF(g_error);
  PlanType.tp_name = "_host.Plan";
  PlanType.tp_basicsize = sizeof(Plan);
  PlanType.tp_flags = Py_TPFLAGS_DEFAULT;
  PlanType.tp_new = plan_new;
  PlanType.tp_dealloc = plan_dealloc;
  PlanType.tp_methods = plan_methods;
  if (PyType_Ready(&PlanType) < 0) return nullptr;
  PyObject* m = PyModule_Create(&module_def);
  if (!m) return nullptr;
  Py_INCREF(&PlanType);
  if (PyModule_AddObject(m, "Plan", (PyObject*)&PlanType) < 0) return nullptr;
  return m;
}
