// The compute calls of the Python binding: argument marshalling in C.
//
// A call on a few tokens takes 2-20 us on the GPU; assembled in Python (ctypes structures, one
// data_ptr() at a time through the interpreter, a size query, torch.cuda.current_stream()) it took the
// host 18-32 us, so the GPU waited for the next launch.  Here the same steps, in the same order,
// are calls of the interpreter's C API: w8a8_linear on one token 18.2 -> 8.3 us a call, the
// 37-token bf16 linear 21.8 -> 10.3, the 16-token W8A8 one 21.5 -> 13.5 (now the GPU's time).
//
// The module holds no state of a call: descriptors are built from the tensors on every call.  Library
// functions are reached through the addresses that init() gets from the binding, which has loaded the
// library; errors are raised by the binding's own check.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstring>

#include "../../include/w8a8.h"

namespace {

struct Api {
  decltype(&w8a8_linear_workspace_size) linear_ws;
  decltype(&w8a8_linear_bf16_workspace_size) bf16_ws;
  decltype(&w8a8_ffn_workspace_size) ffn_ws;
  decltype(&w8a8_lm_head_workspace_size) head_ws;
  decltype(&w8a8_linear) linear;
  decltype(&w8a8_linear_bf16) bf16;
  decltype(&w8a8_ffn_block) ffn;
  decltype(&w8a8_fp8_linear) fp8_linear;
  decltype(&w8a8_fp8_ffn_block) fp8_ffn;
  decltype(&w8a8_lm_head) head;
} g_api;

// Python objects used by every call (owned by the module for the process's life).
PyObject *g_empty, *g_bf16, *g_f32, *g_i32, *g_raw_stream, *g_device, *g_check, *g_default_ws, *g_ws_table, *g_ws_type;
// interned names
PyObject *s_data_ptr, *s_shape, *s_is_cuda, *s_is_contiguous, *s_numel, *s_device, *s_wq, *s_s_w, *s_inv_delta, *s_wq_f16,
    *s_buf, *s_get, *s_cuda_stream, *s_hidden, *s_inter, *s_vocab, *s_gate_up, *s_down, *s_gate_up_bf16, *s_down_bf16,
    *s_q, *s_bf16;
PyObject* g_kw_empty;  // ("dtype", "device")

// An owned reference.
struct Ref {
  PyObject* p;
  explicit Ref(PyObject* o = nullptr) : p(o) {}
  Ref(const Ref&) = delete;
  Ref& operator=(const Ref&) = delete;
  ~Ref() { Py_XDECREF(p); }
  explicit operator bool() const { return p != nullptr; }
  PyObject* give() {
    PyObject* o = p;
    p = nullptr;
    return o;
  }
};

PyObject* call0(PyObject* self, PyObject* name) { return PyObject_CallMethodNoArgs(self, name); }

bool as_int(PyObject* o, long long* out) {  // takes the reference
  Ref r(o);
  if (!r) return false;
  *out = PyLong_AsLongLong(r.p);
  return !(*out == -1 && PyErr_Occurred());
}
// data_ptr() of a tensor; NULL for None
template <class T>
bool ptr_of(PyObject* t, T** out) {
  *out = nullptr;
  if (t == Py_None) return true;
  Ref r(call0(t, s_data_ptr));
  if (!r) return false;
  const unsigned long long v = PyLong_AsUnsignedLongLong(r.p);
  if (v == (unsigned long long)-1 && PyErr_Occurred()) return false;
  *out = reinterpret_cast<T*>(static_cast<uintptr_t>(v));
  return true;
}
template <class T>
bool ptr_attr(PyObject* o, PyObject* name, T** out) {
  Ref a(PyObject_GetAttr(o, name));
  return a && ptr_of(a.p, out);
}
bool int_attr(PyObject* o, PyObject* name, int32_t* out) {
  long long v;
  if (!as_int(PyObject_GetAttr(o, name), &v)) return false;
  *out = (int32_t)v;
  return true;
}
// the first n extents of a tensor
bool shape_of(PyObject* t, int n, long long* out) {
  Ref s(PyObject_GetAttr(t, s_shape));
  if (!s) return false;
  for (int i = 0; i < n; ++i)
    if (!as_int(PySequence_GetItem(s.p, i), out + i)) return false;
  return true;
}
// the extents of a matrix: a tensor of more dimensions is refused, not read as its first two
bool matrix_shape(PyObject* t, long long* out) {
  Ref s(PyObject_GetAttr(t, s_shape));
  if (!s) return false;
  const Py_ssize_t dims = PySequence_Size(s.p);
  if (dims < 0) return false;
  if (dims > 2) {
    PyErr_Format(PyExc_ValueError, "a matrix expected, not a tensor of %zd dimensions", dims);
    return false;
  }
  return shape_of(t, 2, out);
}
// The binding's rule for an input: a contiguous CUDA tensor.
bool check_bits(PyObject* t) {
  Ref c(PyObject_GetAttr(t, s_is_cuda));
  if (!c) return false;
  bool ok = PyObject_IsTrue(c.p) == 1;
  if (ok) {
    Ref k(call0(t, s_is_contiguous));
    if (!k) return false;
    ok = PyObject_IsTrue(k.p) == 1;
  }
  if (!ok && !PyErr_Occurred()) PyErr_SetString(PyExc_AssertionError, "tensors must be contiguous CUDA tensors");
  return ok;
}

template <class W>
bool weight_desc(PyObject* w, W* d) {  // everything but the fp16 copy
  Ref wq(PyObject_GetAttr(w, s_wq));
  long long nk[2];
  if (!wq || !shape_of(wq.p, 2, nk) || !ptr_of(wq.p, &d->wq)) return false;
  d->n = (int32_t)nk[0];
  d->k = (int32_t)nk[1];
  return ptr_attr(w, s_s_w, &d->s_w) && ptr_attr(w, s_inv_delta, &d->inv_delta);
}
bool qweight(PyObject* w, w8a8_qweight* d) { return weight_desc(w, d) && ptr_attr(w, s_wq_f16, &d->wq_f16); }
bool qweight_attr(PyObject* o, PyObject* name, w8a8_qweight* d) {  // zeros where the attribute is None
  Ref w(PyObject_GetAttr(o, name));
  if (!w) return false;
  if (w.p == Py_None) {
    std::memset(d, 0, sizeof(*d));
    return true;
  }
  return qweight(w.p, d);
}

// torch.empty(rows, cols, dtype=dtype, device=like.device); cols < 0: one dimension
PyObject* new_empty(PyObject* like, long long rows, long long cols, PyObject* dtype) {
  Ref dev(PyObject_GetAttr(like, s_device)), r(PyLong_FromLongLong(rows)), c(PyLong_FromLongLong(cols));
  if (!dev || !r || !c) return nullptr;
  if (cols < 0) {
    PyObject* args[4] = {r.p, dtype, dev.p, nullptr};
    return PyObject_Vectorcall(g_empty, args, 1, g_kw_empty);
  }
  PyObject* args[4] = {r.p, c.p, dtype, dev.p};
  return PyObject_Vectorcall(g_empty, args, 2, g_kw_empty);
}

bool check(const char* name, w8a8_status st) {
  if (st == W8A8_OK) return true;
  Ref r(PyObject_CallFunction(g_check, "si", name, (int)st));
  if (r) PyErr_SetString(PyExc_RuntimeError, "status check passed an error");
  return false;
}

// The buffer of `ws` (None: the current device's default workspace), grown to `need` bytes.
struct Buf {
  Ref t;
  void* ptr = nullptr;
  size_t bytes = 0;
};
bool workspace(PyObject* ws, size_t need, Buf* b) {
  Ref own;
  if (ws == Py_None) {
    Ref dev(PyObject_CallNoArgs(g_device));
    if (!dev) return false;
    PyObject* known = PyDict_GetItemWithError(g_ws_table, dev.p);
    if (!known && PyErr_Occurred()) return false;
    Py_XINCREF(known);
    own.p = known ? known : PyObject_CallNoArgs(g_default_ws);
    if (!own) return false;
    ws = own.p;
  }
  long long have = -1;
  if ((PyObject*)Py_TYPE(ws) == g_ws_type) {  // what get() does while the buffer is large enough
    b->t.p = PyObject_GetAttr(ws, s_buf);
    if (!b->t || !as_int(call0(b->t.p, s_numel), &have)) return false;
  }
  if (have < 0 || (size_t)have < need) {
    Ref n(PyLong_FromSize_t(need));
    if (!n) return false;
    Py_CLEAR(b->t.p);
    b->t.p = PyObject_CallMethodOneArg(ws, s_get, n.p);
    if (!b->t || !as_int(call0(b->t.p, s_numel), &have)) return false;
  }
  b->bytes = (size_t)have;
  return ptr_of(b->t.p, &b->ptr);
}
bool stream_of(PyObject* stream, void** out) {
  Ref v;
  if (stream == Py_None) {
    Ref dev(PyObject_CallNoArgs(g_device));
    if (!dev) return false;
    v.p = PyObject_CallOneArg(g_raw_stream, dev.p);
  } else {
    v.p = PyObject_GetAttr(stream, s_cuda_stream);
  }
  if (!v) return false;
  const unsigned long long s = PyLong_AsUnsignedLongLong(v.p);
  if (s == (unsigned long long)-1 && PyErr_Occurred()) return false;
  *out = reinterpret_cast<void*>(static_cast<uintptr_t>(s));
  return true;
}
bool nargs_are(Py_ssize_t n, Py_ssize_t want, const char* name) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "%s takes %zd arguments", name, want);
  return false;
}

// The library call without the interpreter lock (a full launch queue blocks).
template <class F>
w8a8_status unlocked(F f) {
  w8a8_status st;
  Py_BEGIN_ALLOW_THREADS st = f();
  Py_END_ALLOW_THREADS return st;
}

// (w, X, bias, out, ws, stream) -> Y
template <class W, class Fill, class Run>
PyObject* linear_call(PyObject* const* a, const char* name, Fill fill, Run run) {
  W d;
  long long M;
  size_t need = 0;
  if (!fill(a[0], &d) || !shape_of(a[1], 1, &M)) return nullptr;
  Ref y;
  if (a[3] == Py_None) {
    y.p = new_empty(a[1], M, d.n, g_bf16);
    if (!y) return nullptr;
  } else {
    Py_INCREF(a[3]);
    y.p = a[3];
  }
  if (!check("w8a8_linear_workspace_size", g_api.linear_ws((int)M, d.n, d.k, &need))) return nullptr;
  Buf b;
  const uint16_t* X;
  const float* bias;
  uint16_t* Y;
  void* st;
  if (!workspace(a[4], need, &b) || !check_bits(a[1]) || !ptr_of(a[1], &X) || !ptr_of(a[2], &bias) || !ptr_of(y.p, &Y) ||
      !stream_of(a[5], &st))
    return nullptr;
  if (!check(name, unlocked([&] { return run(&d, X, (int)M, bias, Y, b.ptr, b.bytes, st); }))) return nullptr;
  return y.give();
}

PyObject* py_linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs_are(n, 6, "linear")) return nullptr;
  return linear_call<w8a8_qweight>(a, "w8a8_linear", qweight,
                                   [](const w8a8_qweight* w, const uint16_t* X, int M, const float* bias, uint16_t* Y,
                                      void* ws, size_t bytes, void* st) {
                                     return g_api.linear(w, X, M, bias, Y, nullptr, ws, bytes, st);
                                   });
}
PyObject* py_fp8_linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs_are(n, 6, "fp8_linear")) return nullptr;
  return linear_call<w8a8_fp8_weight>(a, "w8a8_fp8_linear", weight_desc<w8a8_fp8_weight>,
                                      [](const w8a8_fp8_weight* w, const uint16_t* X, int M, const float* bias, uint16_t* Y,
                                         void* ws, size_t bytes, void* st) {
                                        return g_api.fp8_linear(w, X, M, bias, Y, nullptr, nullptr, ws, bytes, st);
                                      });
}

// (W, X, bias, out, ws, stream) -> Y
PyObject* py_linear_bf16(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs_are(n, 6, "linear_bf16")) return nullptr;
  long long nk[2], M;
  size_t need = 0;
  if (!matrix_shape(a[0], nk) || !shape_of(a[1], 1, &M)) return nullptr;
  Ref y;
  if (a[3] == Py_None) {
    y.p = new_empty(a[1], M, nk[0], g_bf16);
    if (!y) return nullptr;
  } else {
    Py_INCREF(a[3]);
    y.p = a[3];
  }
  const int N = (int)nk[0], K = (int)nk[1];
  if (!check("w8a8_linear_bf16_workspace_size", g_api.bf16_ws((int)M, N, K, &need))) return nullptr;
  Buf b;
  const uint16_t *W, *X;
  const float* bias;
  uint16_t* Y;
  void* st;
  if (!workspace(a[4], need, &b) || !check_bits(a[0]) || !ptr_of(a[0], &W) || !check_bits(a[1]) || !ptr_of(a[1], &X) ||
      !ptr_of(a[2], &bias) || !ptr_of(y.p, &Y) || !stream_of(a[5], &st))
    return nullptr;
  if (!check("w8a8_linear_bf16", unlocked([&] { return g_api.bf16(W, N, K, X, (int)M, bias, Y, b.ptr, b.bytes, st); })))
    return nullptr;
  return y.give();
}

// Shared part of the FFN calls: Y, and h when wanted.
struct FfnOut {
  Ref y, h;
  const uint16_t* X;
  uint16_t *Y, *H;
  void* st;
  Buf b;
  long long M;
};
bool ffn_out(PyObject* X, bool want_h, PyObject* out, PyObject* ws, PyObject* stream, int32_t hidden, int32_t inter,
             FfnOut* o) {
  size_t need = 0;
  if (!shape_of(X, 1, &o->M)) return false;
  if (out == Py_None) {
    o->y.p = new_empty(X, o->M, hidden, g_bf16);
    if (!o->y) return false;
  } else {
    Py_INCREF(out);
    o->y.p = out;
  }
  o->H = nullptr;
  if (want_h) {
    o->h.p = new_empty(X, o->M, inter, g_bf16);
    if (!o->h || !ptr_of(o->h.p, &o->H)) return false;
  }
  return check("w8a8_ffn_workspace_size", g_api.ffn_ws((int)o->M, hidden, inter, &need)) && workspace(ws, need, &o->b) &&
         check_bits(X) && ptr_of(X, &o->X) && ptr_of(o->y.p, &o->Y) && stream_of(stream, &o->st);
}
PyObject* ffn_result(FfnOut* o) {
  if (!o->h) return o->y.give();
  return PyTuple_Pack(2, o->y.p, o->h.p);
}

// (f, precision, X, want_h, out, ws, stream) -> Y or (Y, h)
PyObject* py_ffn_block(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs_are(n, 7, "ffn_block")) return nullptr;
  w8a8_ffn_weights d;
  long long prec;
  if (!as_int(PyNumber_Long(a[1]), &prec)) return nullptr;
  const int want_h = PyObject_IsTrue(a[3]);
  FfnOut o;
  if (want_h < 0 || !int_attr(a[0], s_hidden, &d.hidden) || !int_attr(a[0], s_inter, &d.inter) ||
      !qweight_attr(a[0], s_gate_up, &d.gate_up) || !qweight_attr(a[0], s_down, &d.down) ||
      !ptr_attr(a[0], s_gate_up_bf16, &d.gate_up_bf16) || !ptr_attr(a[0], s_down_bf16, &d.down_bf16) ||
      !ffn_out(a[2], want_h, a[4], a[5], a[6], d.hidden, d.inter, &o))
    return nullptr;
  if (!check("w8a8_ffn_block", unlocked([&] {
               return g_api.ffn(&d, (int)prec, o.X, (int)o.M, o.Y, o.H, o.b.ptr, o.b.bytes, o.st);
             })))
    return nullptr;
  return ffn_result(&o);
}

// (f, X, want_h, out, ws, stream) -> Y or (Y, h)
PyObject* py_fp8_ffn_block(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs_are(n, 6, "fp8_ffn_block")) return nullptr;
  w8a8_fp8_ffn_weights d;
  const int want_h = PyObject_IsTrue(a[2]);
  Ref gu(PyObject_GetAttr(a[0], s_gate_up)), dn(PyObject_GetAttr(a[0], s_down));
  FfnOut o;
  if (want_h < 0 || !gu || !dn || !int_attr(a[0], s_hidden, &d.hidden) || !int_attr(a[0], s_inter, &d.inter) ||
      !weight_desc(gu.p, &d.gate_up) || !weight_desc(dn.p, &d.down) ||
      !ffn_out(a[1], want_h, a[3], a[4], a[5], d.hidden, d.inter, &o))
    return nullptr;
  if (!check("w8a8_fp8_ffn_block", unlocked([&] {
               return g_api.fp8_ffn(&d, o.X, (int)o.M, o.Y, o.H, o.b.ptr, o.b.bytes, o.st);
             })))
    return nullptr;
  return ffn_result(&o);
}

// (head, precision, X, want_logits, logits, top1, ws, stream) -> (logits or None, top1)
PyObject* py_lm_head(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs_are(n, 8, "lm_head")) return nullptr;
  w8a8_head_weights d;
  long long prec;
  if (!as_int(PyNumber_Long(a[1]), &prec)) return nullptr;
  const int want = PyObject_IsTrue(a[3]);
  long long M;
  size_t need = 0;
  if (want < 0 || !int_attr(a[0], s_vocab, &d.vocab) || !int_attr(a[0], s_hidden, &d.hidden) ||
      !qweight_attr(a[0], s_q, &d.q) || !ptr_attr(a[0], s_bf16, &d.bf16) || !shape_of(a[2], 1, &M))
    return nullptr;
  Ref lg, tp;
  float* L = nullptr;
  int32_t* T;
  if (want) {
    if (a[4] == Py_None) {
      lg.p = new_empty(a[2], M, d.vocab, g_f32);
      if (!lg) return nullptr;
    } else {
      Py_INCREF(a[4]);
      lg.p = a[4];
    }
    if (!ptr_of(lg.p, &L)) return nullptr;
  } else {
    Py_INCREF(Py_None);
    lg.p = Py_None;
  }
  if (a[5] == Py_None) {
    tp.p = new_empty(a[2], M, -1, g_i32);
    if (!tp) return nullptr;
  } else {
    Py_INCREF(a[5]);
    tp.p = a[5];
  }
  Buf b;
  const uint16_t* X;
  void* st;
  if (!check("w8a8_lm_head_workspace_size", g_api.head_ws((int)M, d.vocab, d.hidden, &need)) || !workspace(a[6], need, &b) ||
      !check_bits(a[2]) || !ptr_of(a[2], &X) || !ptr_of(tp.p, &T) || !stream_of(a[7], &st))
    return nullptr;
  if (!check("w8a8_lm_head",
             unlocked([&] { return g_api.head(&d, (int)prec, X, (int)M, L, T, b.ptr, b.bytes, st); })))
    return nullptr;
  return PyTuple_Pack(2, lg.p, tp.p);
}

// (addresses: dict name -> int, check, default_workspace, workspace table, Workspace)
PyObject* py_init(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!nargs_are(n, 5, "init")) return nullptr;
  auto address = [&](const char* name, void* slot) {
    PyObject* v = PyDict_GetItemString(a[0], name);
    const unsigned long long p = v ? PyLong_AsUnsignedLongLong(v) : 0ull;
    if (!v || p == 0 || PyErr_Occurred()) {
      if (!PyErr_Occurred()) PyErr_Format(PyExc_KeyError, "no address of %s", name);
      return false;
    }
    std::memcpy(slot, &p, sizeof(void*));
    return true;
  };
  static_assert(sizeof(unsigned long long) == sizeof(void*), "64-bit addresses");
  if (!address("w8a8_linear_workspace_size", &g_api.linear_ws) ||
      !address("w8a8_linear_bf16_workspace_size", &g_api.bf16_ws) ||
      !address("w8a8_ffn_workspace_size", &g_api.ffn_ws) || !address("w8a8_lm_head_workspace_size", &g_api.head_ws) ||
      !address("w8a8_linear", &g_api.linear) || !address("w8a8_linear_bf16", &g_api.bf16) ||
      !address("w8a8_ffn_block", &g_api.ffn) || !address("w8a8_fp8_linear", &g_api.fp8_linear) ||
      !address("w8a8_fp8_ffn_block", &g_api.fp8_ffn) || !address("w8a8_lm_head", &g_api.head))
    return nullptr;
  Ref torch(PyImport_ImportModule("torch")), c(PyImport_ImportModule("torch._C"));
  if (!torch || !c) return nullptr;
  struct {
    PyObject** to;
    PyObject* from;
    const char* name;
  } items[] = {{&g_empty, torch.p, "empty"},
               {&g_bf16, torch.p, "bfloat16"},
               {&g_f32, torch.p, "float32"},
               {&g_i32, torch.p, "int32"},
               {&g_raw_stream, c.p, "_cuda_getCurrentRawStream"},
               {&g_device, c.p, "_cuda_getDevice"}};
  for (auto& it : items)
    if (!(*it.to = PyObject_GetAttrString(it.from, it.name))) return nullptr;
  g_check = Py_NewRef(a[1]);
  g_default_ws = Py_NewRef(a[2]);
  g_ws_table = Py_NewRef(a[3]);
  g_ws_type = Py_NewRef(a[4]);
  struct {
    PyObject** to;
    const char* name;
  } names[] = {{&s_data_ptr, "data_ptr"}, {&s_shape, "shape"}, {&s_is_cuda, "is_cuda"},
               {&s_is_contiguous, "is_contiguous"}, {&s_numel, "numel"}, {&s_device, "device"}, {&s_wq, "wq"},
               {&s_s_w, "s_w"}, {&s_inv_delta, "inv_delta"}, {&s_wq_f16, "wq_f16"}, {&s_buf, "buf"}, {&s_get, "get"},
               {&s_cuda_stream, "cuda_stream"}, {&s_hidden, "hidden"}, {&s_inter, "inter"}, {&s_vocab, "vocab"},
               {&s_gate_up, "gate_up"}, {&s_down, "down"}, {&s_gate_up_bf16, "gate_up_bf16"},
               {&s_down_bf16, "down_bf16"}, {&s_q, "q"}, {&s_bf16, "bf16"}};
  for (auto& it : names)
    if (!(*it.to = PyUnicode_InternFromString(it.name))) return nullptr;
  if (!(g_kw_empty = Py_BuildValue("(ss)", "dtype", "device"))) return nullptr;
  Py_RETURN_NONE;
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL
PyMethodDef g_methods[] = {{"init", FAST(py_init), "Set the library's addresses and the binding's helpers."},
                           {"linear", FAST(py_linear), "w8a8_linear"},
                           {"linear_bf16", FAST(py_linear_bf16), "w8a8_linear_bf16"},
                           {"ffn_block", FAST(py_ffn_block), "w8a8_ffn_block"},
                           {"fp8_linear", FAST(py_fp8_linear), "w8a8_fp8_linear"},
                           {"fp8_ffn_block", FAST(py_fp8_ffn_block), "w8a8_fp8_ffn_block"},
                           {"lm_head", FAST(py_lm_head), "w8a8_lm_head"},
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_calls", "Compute calls of the binding.", -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&g_module); }
