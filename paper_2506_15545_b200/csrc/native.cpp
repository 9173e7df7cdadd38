// CPython extension behind binding.py: turns torch tensors into device pointers, sizes and a stream handle and calls
// the C ABI (include/rattn.h).  It holds no arithmetic and no fallback.
//
// Why it exists: a decode step occupies the GPU for 10 - 25 us, and marshalling it through ctypes (a structure of 40
// fields filled by Python attribute stores, half a dozen Python calls per tensor) took longer than that, so small calls
// were bound by the host: 32 us for a prologue plus a decode step of one sequence, of which the GPU needed 23.
//
// The library is not linked: binding.py loads librattn.so (or another build of it) and hands over the addresses of its
// entry points, so that both sides use one instance of it.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>

#include <cstring>

#include "rattn.h"

namespace {

struct Entry {
  decltype(&rattn_forward) forward;
  decltype(&rattn_forward_static) forward_static;
  decltype(&rattn_forward_ex) forward_ex;
  decltype(&rattn_backward) backward;
  decltype(&rattn_backward_ex) backward_ex;
  decltype(&rattn_decode_step) decode_step;
  decltype(&rattn_decode_step_ex) decode_step_ex;
  decltype(&rattn_qk_prologue) qk_prologue;
  decltype(&rattn_qk_prologue_backward) qk_prologue_backward;
  decltype(&rattn_qk_prologue_workspace_bytes) qk_prologue_workspace_bytes;
} E;
PyObject* g_error = nullptr;                 // RattnError(code, where)

// A Python exception is set; unwinds to the entry function, which returns NULL.
struct Raised {};
[[noreturn]] void raise(PyObject* type, const char* text) {
  PyErr_SetString(type, text);
  throw Raised{};
}
void check(int code, const char* where) {
  if (code == RATTN_OK) return;
  PyObject* e = PyObject_CallFunction(g_error, "is", code, where);
  if (e) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  throw Raised{};
}

// Positional arguments of one call, read in order.
struct Args {
  PyObject* const* at;
  PyObject* const* end;
  PyObject* next() {
    if (at == end) raise(PyExc_TypeError, "too few arguments");
    return *at++;
  }
  // a contiguous CUDA tensor; None gives an undefined tensor where `optional`
  at::Tensor tensor(bool optional) {
    PyObject* o = next();
    if (o == Py_None && optional) return at::Tensor();
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch tensor");
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) raise(PyExc_ValueError, "tensors must be contiguous CUDA tensors");
    return t;
  }
  at::Tensor tensor() { return tensor(false); }
  at::Tensor maybe() { return tensor(true); }
  long integer() {
    const long v = PyLong_AsLong(next());
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return v;
  }
  // what ctypes did with an integer field or argument: the low 32 bits
  int32_t i32() { return static_cast<int32_t>(integer()); }
  float real() {
    const double v = PyFloat_AsDouble(next());
    if (v == -1.0 && PyErr_Occurred()) throw Raised{};
    return static_cast<float>(v);
  }
  bool flag() {
    const int v = PyObject_IsTrue(next());
    if (v < 0) throw Raised{};
    return v != 0;
  }
  // None: torch's current stream of the current device; else an object with a cuda_stream attribute
  void* stream() {
    PyObject* o = next();
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw Raised{};
    void* s = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!s && PyErr_Occurred()) throw Raised{};
    return s;
  }
};

template <typename T = void>
T* ptr(const at::Tensor& t) { return t.defined() ? static_cast<T*>(t.data_ptr()) : nullptr; }

int dtype_code(const at::Tensor& t) {
  if (t.scalar_type() == at::kBFloat16) return RATTN_BF16;
  if (t.scalar_type() == at::kFloat) return RATTN_F32;
  raise(PyExc_TypeError, "unsupported dtype: bfloat16 or float32 is expected");
}

// An uninitialised contiguous tensor on t's device.  Straight to the CUDA factory: through the dispatcher each of a
// step's three results cost 1.4 us.
at::Tensor fresh(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& t) {
  return at::Tensor(at::detail::empty_cuda(sizes, type, t.device(), c10::nullopt));
}
at::Tensor like(const at::Tensor& t) { return fresh(t.sizes(), t.scalar_type(), t); }
at::Tensor or_like(at::Tensor given, const at::Tensor& t) { return given.defined() ? given : like(t); }

PyObject* wrap(const at::Tensor& t) {
  if (!t.defined()) Py_RETURN_NONE;
  return THPVariable_Wrap(t);
}

void need_dim(const at::Tensor& t, int n) {
  if (t.dim() != n) raise(PyExc_ValueError, n == 4 ? "a four-dimensional tensor is expected" : "a three-dimensional tensor is expected");
}

// B, H_q, H_kv, T, d of q, k in either layout; three-dimensional q, k are a decode step's token
void set_shape(rattn_params* p, const at::Tensor& q, const at::Tensor& k, int layout) {
  const int n = q.dim() == 3 ? 3 : 4;
  need_dim(q, n);
  need_dim(k, n);
  p->B = (int32_t)q.size(0);
  p->d = (int32_t)q.size(n - 1);
  if (n == 3) {
    p->H_q = (int32_t)q.size(1); p->T = 1; p->H_kv = (int32_t)k.size(1);
  } else {
    const int hd = layout == RATTN_LAYOUT_BTHD ? 2 : 1;
    p->H_q = (int32_t)q.size(hd); p->T = (int32_t)q.size(3 - hd); p->H_kv = (int32_t)k.size(hd);
  }
}

template <typename F>
int released(F&& call) {                     // the library call itself runs without the interpreter lock
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = call();
  Py_END_ALLOW_THREADS
  return rc;
}

template <PyObject* (*F)(Args)>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  try {
    return F(Args{args, args + n});
  } catch (const Raised&) {
  } catch (...) {                            // as torch's own functions raise it: callers catch torch.OutOfMemoryError
    torch::translate_exception_to_python(std::current_exception());
  }
  return nullptr;
}

PyObject* forward(Args a) {
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor();
  const int w = a.i32();
  const at::Tensor given = a.maybe();
  void* s = a.stream();
  need_dim(q, 4);
  need_dim(k, 4);
  const at::Tensor out = or_like(given, q);
  check(released([&] {
          return E.forward(ptr(q), ptr(k), ptr(v), (int)q.size(0), (int)q.size(1), (int)k.size(1), (int)q.size(2),
                           (int)q.size(3), w, ptr(out), s);
        }), "rattn_forward");
  return wrap(out);
}

PyObject* forward_static(Args a) {
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor();
  const int w = a.i32();
  const float scale = a.real();
  const at::Tensor given = a.maybe();
  void* s = a.stream();
  need_dim(q, 4);
  need_dim(k, 4);
  const at::Tensor out = or_like(given, q);
  check(released([&] {
          return E.forward_static(ptr(q), ptr(k), ptr(v), (int)q.size(0), (int)q.size(1), (int)k.size(1),
                                  (int)q.size(2), (int)q.size(3), w, scale, ptr(out), s);
        }), "rattn_forward_static");
  return wrap(out);
}

PyObject* forward_ex(Args a) {
  rattn_params p;
  std::memset(&p, 0, sizeof(p));
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor();
  p.w = a.i32();
  p.scale = a.real();
  p.eps = a.real();
  const at::Tensor gs = a.maybe(), gr = a.maybe();
  p.mode = a.i32();
  const at::Tensor ws = a.maybe();
  const bool save = a.flag();
  const at::Tensor state_out = a.maybe(), kro = a.maybe(), vro = a.maybe(), given = a.maybe();
  p.flags = (uint32_t)a.i32() | (save ? RATTN_FLAG_SAVE_RESIDUALS : 0u);
  p.feature_map = a.i32();
  const at::Tensor state_in = a.maybe(), kri = a.maybe(), vri = a.maybe();
  p.pos0 = a.i32();
  const at::Tensor lens = a.maybe();
  p.layout = a.i32();
  void* s = a.stream();
  const at::Tensor out = or_like(given, q);
  p.q = ptr(q); p.k = ptr(k); p.v = ptr(v); p.out = ptr(out);
  set_shape(&p, q, k, p.layout);
  p.dtype = dtype_code(q);
  p.gamma_swa = ptr<float>(gs); p.gamma_rla = ptr<float>(gr);
  if (ws.defined()) { p.workspace = ptr(ws); p.workspace_bytes = ws.nbytes(); }
  p.state_out = ptr<float>(state_out); p.k_ring_out = ptr(kro); p.v_ring_out = ptr(vro);
  p.state_in = ptr<float>(state_in); p.k_ring_in = ptr(kri); p.v_ring_in = ptr(vri);
  p.seq_lens = ptr<int32_t>(lens);
  check(released([&] { return E.forward_ex(&p, s); }), "rattn_forward_ex");
  return wrap(out);
}

PyObject* three(const at::Tensor& x, const at::Tensor& y, const at::Tensor& z) {
  return Py_BuildValue("(NNN)", wrap(x), wrap(y), wrap(z));
}

PyObject* backward(Args a) {
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor(), dout = a.tensor(), ws = a.tensor();
  const int w = a.i32();
  const at::Tensor dq_ = a.maybe(), dk_ = a.maybe(), dv_ = a.maybe();
  void* s = a.stream();
  need_dim(q, 4);
  need_dim(k, 4);
  const at::Tensor dq = or_like(dq_, q), dk = or_like(dk_, k), dv = or_like(dv_, v);
  check(released([&] {
          return E.backward(ptr(q), ptr(k), ptr(v), ptr(dout), ptr(ws), ws.nbytes(), (int)q.size(0), (int)q.size(1),
                            (int)k.size(1), (int)q.size(2), (int)q.size(3), w, ptr(dq), ptr(dk), ptr(dv), s);
        }), "rattn_backward");
  return three(dq, dk, dv);
}

PyObject* backward_ex(Args a) {
  rattn_params p;
  std::memset(&p, 0, sizeof(p));
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor(), dout = a.tensor();
  p.w = a.i32();
  const at::Tensor ws = a.maybe();
  p.scale = a.real();
  p.eps = a.real();
  const at::Tensor gs = a.maybe(), gr = a.maybe();
  p.mode = a.i32();
  const at::Tensor dq_ = a.maybe(), dk_ = a.maybe(), dv_ = a.maybe(), dgs = a.maybe(), dgr = a.maybe();
  p.flags = (uint32_t)a.i32();
  p.feature_map = a.i32();
  p.layout = a.i32();
  void* s = a.stream();
  const at::Tensor dq = or_like(dq_, q), dk = or_like(dk_, k), dv = or_like(dv_, v);
  p.q = ptr(q); p.k = ptr(k); p.v = ptr(v); p.out = ptr(dq);
  set_shape(&p, q, k, p.layout);
  p.dtype = dtype_code(q);
  p.gamma_swa = ptr<float>(gs); p.gamma_rla = ptr<float>(gr);
  if (ws.defined()) { p.workspace = ptr(ws); p.workspace_bytes = ws.nbytes(); }
  p.dout = ptr(dout); p.dq = ptr(dq); p.dk = ptr(dk); p.dv = ptr(dv);
  p.dgamma_swa = ptr<float>(dgs); p.dgamma_rla = ptr<float>(dgr);
  check(released([&] { return E.backward_ex(&p, s); }), "rattn_backward_ex");
  return three(dq, dk, dv);
}

PyObject* decode_step(Args a) {
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor(), kr = a.tensor(), vr = a.tensor(), state = a.tensor();
  const int pos = a.i32();
  const at::Tensor given = a.maybe();
  void* s = a.stream();
  need_dim(q, 3);
  need_dim(kr, 4);
  const at::Tensor out = or_like(given, q);
  check(released([&] {
          return E.decode_step(ptr(q), ptr(k), ptr(v), ptr(kr), ptr(vr), ptr<float>(state), pos, (int)q.size(0),
                               (int)q.size(1), (int)k.size(1), (int)q.size(2), (int)kr.size(2), ptr(out), s);
        }), "rattn_decode_step");
  return wrap(out);
}

PyObject* decode_step_ex(Args a) {
  rattn_params p;
  std::memset(&p, 0, sizeof(p));
  const at::Tensor q = a.tensor(), k = a.tensor(), v = a.tensor(), kr = a.tensor(), vr = a.tensor(), state = a.tensor();
  const int pos = a.i32();
  p.scale = a.real();
  p.eps = a.real();
  const at::Tensor gs = a.maybe(), gr = a.maybe(), given = a.maybe();
  p.feature_map = a.i32();
  const at::Tensor pos_dev = a.maybe();
  p.flags = (uint32_t)a.i32();
  void* s = a.stream();
  need_dim(kr, 4);
  const at::Tensor out = or_like(given, q);
  p.q = ptr(q); p.k = ptr(k); p.v = ptr(v); p.out = ptr(out);
  set_shape(&p, q, k, RATTN_LAYOUT_BHTD);
  p.w = (int32_t)kr.size(2);
  p.dtype = dtype_code(q);
  p.gamma_swa = ptr<float>(gs); p.gamma_rla = ptr<float>(gr);
  p.pos = ptr<int32_t>(pos_dev);
  check(released([&] { return E.decode_step_ex(&p, ptr(kr), ptr(vr), ptr<float>(state), pos, s); }),
        "rattn_decode_step_ex");
  return wrap(out);
}

// the part of the parameter block that both directions of the prologue share; q, k, gains and pos are read from `a`
struct Qk {
  rattn_qk_params p;
  at::Tensor q, k, q_gain, k_gain, pos;
};
void read_qk(Args& a, Qk* x) {
  std::memset(&x->p, 0, sizeof(x->p));
  x->q_gain = a.maybe();
  x->k_gain = a.maybe();
  PyObject* theta = a.next();
  double th = 0.0;
  if (theta != Py_None) {
    th = PyFloat_AsDouble(theta);
    if (th == -1.0 && PyErr_Occurred()) throw Raised{};
  }
  x->p.theta = static_cast<float>(th);
  x->p.eps = a.real();
  x->p.pos0 = a.i32();
  x->pos = a.maybe();
  x->p.layout = a.i32();
  need_dim(x->q, 4);
  const int hd = x->p.layout == RATTN_LAYOUT_BTHD ? 2 : 1;
  x->p.q = ptr(x->q);
  x->p.B = (int32_t)x->q.size(0); x->p.d = (int32_t)x->q.size(3);
  x->p.H_q = (int32_t)x->q.size(hd); x->p.T = (int32_t)x->q.size(3 - hd);
  if (x->k.defined()) {
    need_dim(x->k, 4);
    x->p.k = ptr(x->k);
    x->p.H_kv = (int32_t)x->k.size(hd);
  }
  x->p.q_gain = ptr<float>(x->q_gain); x->p.k_gain = ptr<float>(x->k_gain);
  x->p.dtype = dtype_code(x->q);
  x->p.pos = ptr<int32_t>(x->pos);
}

PyObject* qk_prologue(Args a) {
  Qk x;
  x.q = a.tensor();
  x.k = a.maybe();
  read_qk(a, &x);
  const bool inplace = a.flag();
  void* s = a.stream();
  const at::Tensor q_out = inplace ? x.q : like(x.q), k_out = !x.k.defined() || inplace ? x.k : like(x.k);
  x.p.q_out = ptr(q_out); x.p.k_out = ptr(k_out);
  check(released([&] { return E.qk_prologue(&x.p, s); }), "rattn_qk_prologue");
  return Py_BuildValue("(NN)", wrap(q_out), wrap(k_out));
}

PyObject* qk_prologue_backward(Args a) {
  Qk x;
  x.q = a.tensor();
  x.k = a.maybe();
  const at::Tensor dq_out = a.tensor(), dk_out = a.maybe();
  read_qk(a, &x);
  const bool gain_grads = a.flag();
  at::Tensor ws = a.maybe();
  void* s = a.stream();
  const at::Tensor dq = like(x.q), dk = x.k.defined() ? like(x.k) : at::Tensor();
  at::Tensor dqg, dkg;
  if (gain_grads) {
    dqg = fresh({x.q.size(3)}, at::kFloat, x.q);
    if (x.k.defined()) dkg = fresh({x.q.size(3)}, at::kFloat, x.q);
    if (!ws.defined()) {
      const size_t n = E.qk_prologue_workspace_bytes(x.p.B, x.p.H_q, x.p.H_kv, x.p.T, x.p.d);
      ws = fresh({(int64_t)n}, at::kByte, x.q);
    }
  }
  const size_t nbytes = ws.defined() ? (size_t)ws.numel() : 0;
  check(released([&] {
          return E.qk_prologue_backward(&x.p, ptr(dq_out), ptr(dk_out), ptr(dq), ptr(dk), ptr<float>(dqg),
                                        ptr<float>(dkg), ptr(ws), nbytes, s);
        }), "rattn_qk_prologue_backward");
  return Py_BuildValue("(NNNN)", wrap(dq), wrap(dk), wrap(dqg), wrap(dkg));
}

// bind(error class, addresses of the entry points in the order of `Entry`)
PyObject* bind(Args a) {
  PyObject* err = a.next();
  Py_INCREF(err);
  Py_XSETREF(g_error, err);
  void* at[10];
  for (void*& f : at) {
    f = PyLong_AsVoidPtr(a.next());
    if (!f) raise(PyExc_ValueError, "an entry point is missing");
  }
  static_assert(sizeof(at) == sizeof(E), "one address per entry point");
  std::memcpy(&E, at, sizeof(E));
  Py_RETURN_NONE;
}

#define METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<name>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(bind), METHOD(forward), METHOD(forward_static), METHOD(forward_ex), METHOD(backward),
                         METHOD(backward_ex), METHOD(decode_step), METHOD(decode_step_ex), METHOD(qk_prologue),
                         METHOD(qk_prologue_backward), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
