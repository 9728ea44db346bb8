// Call path of the Python binding for the compute entry points: checks the tensors, allocates what the
// caller left out, looks up the current stream and calls the C ABI.  binding.py keeps the signatures and
// hands everything over positionally; the addresses of the C functions come from the library it loaded
// (bind()), so this module does not link against it.
//
// Why native: a small forward runs for 10 to 15 us on the device, and the same steps written in Python
// (attribute look-ups on four tensors, argument conversion by ctypes, the stream look-up) took about as
// long on the host, so back-to-back calls waited for the host.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>

#include <optional>
#include <string>

#include "ap.h"

namespace {

struct Error {};  // a Python exception has been set

struct Entry {
  decltype(&ap_accumulate_attention) accumulate;
  decltype(&ap_accumulate_attention_entmax15) accumulate_entmax;
  decltype(&ap_build_mask) build_mask;
  decltype(&ap_build_mask_layer) build_mask_layer;
  decltype(&ap_build_mask_ex) build_mask_ex;
  decltype(&ap_build_mask_workspace_bytes) build_mask_workspace;
  decltype(&ap_sparse_attention_fwd) fwd;
  decltype(&ap_sparse_attention_entmax15_fwd) fwd_entmax;
  decltype(&ap_sparse_attention_bwd) bwd;
  decltype(&ap_sparse_attention_bwd_workspace_bytes) bwd_workspace;
};
Entry g_fn;
PyObject *g_check = nullptr;  // binding._check(status, name): raises ApError

[[noreturn]] void fail(PyObject *type, const std::string &msg) {
  PyErr_SetString(type, msg.c_str());
  throw Error{};
}

const at::Tensor &tensor(PyObject *o, const char *name) {
  if (!THPVariable_Check(o)) fail(PyExc_TypeError, std::string(name) + " must be a torch tensor");
  return THPVariable_Unpack(o);
}

const at::Tensor &device_tensor(PyObject *o, const char *name) {
  const at::Tensor &t = tensor(o, name);
  if (!t.is_cuda() || !t.is_contiguous()) fail(PyExc_ValueError, std::string(name) + " must be a contiguous CUDA tensor");
  return t;
}

// optional tensor: its address, or null for None
void *address(PyObject *o, const char *name) { return o == Py_None ? nullptr : tensor(o, name).data_ptr(); }

double number(PyObject *o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Error{};
  return v;
}
int truth(PyObject *o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw Error{};
  return v;
}
ap_tiles *tiles_at(PyObject *o) {  // address of the descriptor as an integer, or None
  if (o == Py_None) return nullptr;
  void *p = PyLong_AsVoidPtr(o);
  if (!p && PyErr_Occurred()) throw Error{};
  return static_cast<ap_tiles *>(p);
}
void *stream_of(PyObject *o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw Error{};
  void *p = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (!p && PyErr_Occurred()) throw Error{};
  return p;
}

ap_dtype dtype_code(const at::Tensor &t) {
  switch (t.scalar_type()) {
    case at::kFloat: return AP_F32;
    case at::kBFloat16: return AP_BF16;
    case at::kHalf: return AP_F16;
    default: fail(PyExc_TypeError, std::string("dtype must be float32, bfloat16 or float16, got ") + c10::toString(t.scalar_type()));
  }
}

PyObject *done(ap_status st, const char *name, PyObject *result) {  // takes over the reference to result
  if (st != AP_OK) {
    Py_DECREF(result);
    PyObject *r = PyObject_CallFunction(g_check, "is", (int)st, name);
    Py_XDECREF(r);
    if (r) PyErr_Format(PyExc_RuntimeError, "%s failed", name);
    return nullptr;
  }
  return result;
}
PyObject *none() { return Py_NewRef(Py_None); }

void want(Py_ssize_t n, Py_ssize_t expected) {
  if (n != expected) fail(PyExc_TypeError, "wrong number of arguments");
}

// The interpreter lock is released while f allocates and launches: a launch waits where the stream's queue is full.  f uses C++
// values only.
template <class F>
auto unlocked(F f) {
  struct Lock {
    PyThreadState *state = PyEval_SaveThread();
    ~Lock() { PyEval_RestoreThread(state); }
  } lock;
  return f();
}

// Memory for a call on `stream`.  Where that is not the current stream, the memory is allocated for `stream`: it is not
// handed out again before the call's kernels have run, nor does the call use memory that earlier work of the current
// stream still reads.  What the caller gets to see is also held for the current stream.
class Memory {
 public:
  Memory(const at::Tensor &like, void *stream) : current_(c10::cuda::getCurrentCUDAStream(like.device().index())) {
    if (current_.stream() != stream)
      guard_.emplace(c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(stream), like.device().index()));
  }
  at::Tensor output(const at::Tensor &like) const {
    at::Tensor t = at::empty_like(like);
    if (guard_) t.record_stream(current_.unwrap());
    return t;
  }
  at::Tensor bytes(size_t n, const at::Tensor &like) const {
    return at::empty({(int64_t)n}, like.options().dtype(at::kByte));
  }

 private:
  c10::cuda::CUDAStream current_;
  std::optional<c10::cuda::CUDAStreamGuard> guard_;
};

struct Shape {
  int B, H, Lq, Lk, d;
};
// Q[B,H,Lq,d] against K[B,H,Lk,d] of the same type
Shape shape_of(const at::Tensor &q, const at::Tensor &k) {
  if (q.dim() != 4 || k.dim() != 4 || k.size(0) != q.size(0) || k.size(1) != q.size(1) || k.size(3) != q.size(3) ||
      k.scalar_type() != q.scalar_type())
    fail(PyExc_ValueError, "shape/dtype mismatch");
  return Shape{(int)q.size(0), (int)q.size(1), (int)q.size(2), (int)k.size(2), (int)q.size(3)};
}
void like(const at::Tensor &t, const at::Tensor &ref) {
  if (t.sizes() != ref.sizes() || t.scalar_type() != ref.scalar_type()) fail(PyExc_ValueError, "shape/dtype mismatch");
}

template <class F>
PyObject *guarded(F f) {
  try {
    return f();
  } catch (const Error &) {
    return nullptr;
  } catch (...) {  // to the exceptions that torch's own functions raise (out of memory among them)
    torch::translate_exception_to_python(std::current_exception());
    return nullptr;
  }
}

// (acc, Q, K, bias, causal, scale, stream)
template <bool kEntmax>
PyObject *py_accumulate(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    want(n, 7);
    const at::Tensor &acc = device_tensor(a[0], "acc"), &q = device_tensor(a[1], "Q"), &k = device_tensor(a[2], "K");
    const Shape s = shape_of(q, k);
    auto scores = [&](const at::Tensor &t) {
      return t.dim() == 3 && t.size(0) == s.H && t.size(1) == s.Lq && t.size(2) == s.Lk && t.scalar_type() == at::kFloat;
    };
    if (!scores(acc)) fail(PyExc_ValueError, "shape/dtype mismatch");
    const float *bias = nullptr;
    if (a[3] != Py_None) {
      const at::Tensor &b = device_tensor(a[3], "bias");
      if (!scores(b)) fail(PyExc_ValueError, "bias must be float32 [H,Lq,Lk]");
      bias = static_cast<const float *>(b.data_ptr());
    }
    float *out = static_cast<float *>(acc.data_ptr());
    const void *pq = q.data_ptr(), *pk = k.data_ptr();
    const ap_dtype dt = dtype_code(q);
    const int causal = truth(a[4]);
    const float scale = (float)number(a[5]);
    void *stream = stream_of(a[6]);
    const auto fn = kEntmax ? g_fn.accumulate_entmax : g_fn.accumulate;
    const ap_status st =
        unlocked([&] { return fn(out, pq, pk, bias, s.B, s.H, s.Lq, s.Lk, s.d, dt, causal, scale, stream); });
    return done(st, kEntmax ? "ap_accumulate_attention_entmax15" : "ap_accumulate_attention", none());
  });
}

// (rule, acc, keep_frac, causal, keep_diag, flags, mask, tiles, nnz_per_head, workspace, stream)
// rule: 0 = per head, 1 = per layer, 2 = by flags
PyObject *py_build_mask(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    want(n, 11);
    const long rule = PyLong_AsLong(a[0]), flags = PyLong_AsLong(a[5]);
    if (PyErr_Occurred()) throw Error{};
    const at::Tensor &acc = device_tensor(a[1], "acc");
    if (acc.dim() != 3) fail(PyExc_ValueError, "acc must be [H,Lq,Lk]");
    if (acc.scalar_type() != at::kFloat) fail(PyExc_ValueError, "acc must be float32");
    const int H = (int)acc.size(0), Lq = (int)acc.size(1), Lk = (int)acc.size(2);
    at::Tensor ws;
    if (a[9] != Py_None) ws = tensor(a[9], "workspace");
    const float *in = static_cast<const float *>(acc.data_ptr());
    const double keep = number(a[2]);
    const int causal = truth(a[3]), diag = truth(a[4]);
    uint8_t *mask = static_cast<uint8_t *>(address(a[6], "mask"));
    ap_tiles *tiles = tiles_at(a[7]);
    int64_t *nnz = static_cast<int64_t *>(address(a[8], "nnz_per_head"));
    void *s = stream_of(a[10]);
    const auto fn = rule == 1 ? g_fn.build_mask_layer : g_fn.build_mask;
    const ap_status st = unlocked([&] {
      if (!ws.defined()) ws = Memory(acc, s).bytes(g_fn.build_mask_workspace(H, Lq, Lk), acc);
      void *p = ws.data_ptr();
      const size_t n = (size_t)ws.numel();
      return rule == 2 ? g_fn.build_mask_ex(in, H, Lq, Lk, keep, causal, diag, (int)flags, mask, tiles, nnz, p, n, s)
                       : fn(in, H, Lq, Lk, keep, causal, diag, mask, tiles, nnz, p, n, s);
    });
    return done(st, rule == 2 ? "ap_build_mask_ex" : rule == 1 ? "ap_build_mask_layer" : "ap_build_mask", none());
  });
}

// (Q, K, V, tiles, O, scale, stream) -> O
template <bool kEntmax>
PyObject *py_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    want(n, 7);
    const at::Tensor &q = device_tensor(a[0], "Q"), &k = device_tensor(a[1], "K"), &v = device_tensor(a[2], "V");
    const Shape s = shape_of(q, k);
    like(v, k);
    at::Tensor o;
    if (a[4] != Py_None) o = device_tensor(a[4], "O");
    const void *pq = q.data_ptr(), *pk = k.data_ptr(), *pv = v.data_ptr();
    ap_tiles *tiles = tiles_at(a[3]);
    const ap_dtype dt = dtype_code(q);
    const float scale = (float)number(a[5]);
    void *stream = stream_of(a[6]);
    const auto fn = kEntmax ? g_fn.fwd_entmax : g_fn.fwd;
    const ap_status st = unlocked([&] {
      if (!o.defined()) o = Memory(q, stream).output(q);
      return fn(pq, pk, pv, tiles, o.data_ptr(), s.B, s.H, s.Lq, s.Lk, s.d, dt, scale, stream);
    });
    PyObject *out = a[4] == Py_None ? THPVariable_Wrap(std::move(o)) : Py_NewRef(a[4]);
    if (!out) return nullptr;
    return done(st, kEntmax ? "ap_sparse_attention_entmax15_fwd" : "ap_sparse_attention_fwd", out);
  });
}

// (Q, K, V, O, dO, tiles, dQ, dK, dV, scale, workspace, stream) -> (dQ, dK, dV)
PyObject *py_bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    want(n, 12);
    const at::Tensor &q = device_tensor(a[0], "Q"), &k = device_tensor(a[1], "K"), &v = device_tensor(a[2], "V"),
                     &o = device_tensor(a[3], "O"), &g = device_tensor(a[4], "dO");
    const Shape s = shape_of(q, k);
    like(v, k), like(o, q), like(g, q);
    at::Tensor dq, dk, dv, ws;
    if (a[6] != Py_None) dq = device_tensor(a[6], "dQ");
    if (a[7] != Py_None) dk = device_tensor(a[7], "dK");
    if (a[8] != Py_None) dv = device_tensor(a[8], "dV");
    if (a[10] != Py_None) ws = tensor(a[10], "workspace");
    const void *pq = q.data_ptr(), *pk = k.data_ptr(), *pv = v.data_ptr(), *po = o.data_ptr(), *pg = g.data_ptr();
    ap_tiles *tiles = tiles_at(a[5]);
    const ap_dtype dt = dtype_code(q);
    const float scale = (float)number(a[9]);
    void *stream = stream_of(a[11]);
    const ap_status st = unlocked([&] {
      {
        const Memory memory(q, stream);
        if (!dq.defined()) dq = memory.output(q);
        if (!dk.defined()) dk = memory.output(k);
        if (!dv.defined()) dv = memory.output(v);
        if (!ws.defined()) ws = memory.bytes(g_fn.bwd_workspace(s.B, s.H, s.Lq, s.Lk), q);
      }
      return g_fn.bwd(pq, pk, pv, po, pg, tiles, dq.data_ptr(), dk.data_ptr(), dv.data_ptr(), s.B, s.H, s.Lq, s.Lk, s.d, dt,
                      scale, ws.data_ptr(), (size_t)ws.numel(), stream);
    });
    PyObject *out = Py_BuildValue("(NNN)", THPVariable_Wrap(dq), THPVariable_Wrap(dk), THPVariable_Wrap(dv));
    if (!out) return nullptr;
    return done(st, "ap_sparse_attention_bwd", out);
  });
}

// ({name: address}, check)
PyObject *py_bind(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded([&]() -> PyObject * {
    want(n, 2);
    auto look = [&](const char *name, auto &slot) {
      PyObject *o = PyDict_GetItemString(a[0], name);
      void *p = o ? PyLong_AsVoidPtr(o) : nullptr;
      if (!p) fail(PyExc_ImportError, std::string("no address for ") + name);
      slot = reinterpret_cast<std::remove_reference_t<decltype(slot)>>(p);
    };
    look("ap_accumulate_attention", g_fn.accumulate);
    look("ap_accumulate_attention_entmax15", g_fn.accumulate_entmax);
    look("ap_build_mask", g_fn.build_mask);
    look("ap_build_mask_layer", g_fn.build_mask_layer);
    look("ap_build_mask_ex", g_fn.build_mask_ex);
    look("ap_build_mask_workspace_bytes", g_fn.build_mask_workspace);
    look("ap_sparse_attention_fwd", g_fn.fwd);
    look("ap_sparse_attention_entmax15_fwd", g_fn.fwd_entmax);
    look("ap_sparse_attention_bwd", g_fn.bwd);
    look("ap_sparse_attention_bwd_workspace_bytes", g_fn.bwd_workspace);
    Py_XSETREF(g_check, Py_NewRef(a[1]));
    return none();
  });
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)), METH_FASTCALL, nullptr
PyMethodDef g_methods[] = {{"bind", FAST(py_bind)},
                           {"accumulate", FAST(py_accumulate<false>)},
                           {"accumulate_entmax15", FAST(py_accumulate<true>)},
                           {"build_mask", FAST(py_build_mask)},
                           {"fwd", FAST(py_fwd<false>)},
                           {"fwd_entmax15", FAST(py_fwd<true>)},
                           {"bwd", FAST(py_bwd)},
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_ap_call", "Native call path of the binding.", -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

// The torch whose headers this was compiled with: binding.py loads it beside no other, build.py looks for it in the file.
PyMODINIT_FUNC PyInit__ap_call(void) {
  PyObject *m = PyModule_Create(&g_module);
  if (m && PyModule_AddStringConstant(m, "built_for", "torch " AP_TORCH_VERSION) < 0) Py_CLEAR(m);
  return m;
}
