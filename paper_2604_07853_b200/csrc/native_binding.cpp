// Marshalling of the hot calls between Python and the C ABI: tensors in, pointers and sizes to
// libqarl.so, output tensors back, with the checks and results of the ctypes wrappers it replaces.  A
// decode-sized call was bound by those: us of host time per call, ctypes -> here, on a B200 host:
// dense projection of one token 23.6 -> 6.7 (GPU work 11.8), router + expert layer of one token
// 55 -> 12.3, TBPO loss 40 -> 15.  What is left is the launches themselves.
//
// Every function takes the Context object first: its `_hv` (address of the qarl_ctx), `_ws` (the cached
// scratch tensor, replaced here when a call needs a larger one) and `_check` (raises on a status).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/qarl.h"

namespace {

PyObject *s_hv, *s_ws, *s_check, *s_r, *s_w, *s_J, *s_flags, *s_grad, *s_loss, *s_gate_up, *s_h, *s_index[3];

struct Fail {};  // a Python exception is set

[[noreturn]] void fail(const char* what) {
  if (!PyErr_Occurred()) PyErr_SetString(PyExc_AssertionError, what);
  throw Fail{};
}
void expect(bool ok, const char* what) {
  if (!ok) fail(what);
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a torch.Tensor, got %s", Py_TYPE(o)->tp_name);
    throw Fail{};
  }
  return THPVariable_Unpack(o);
}
const at::Tensor& cuda_tensor(PyObject* o, at::ScalarType type, const char* what) {
  const at::Tensor& t = tensor(o);
  expect(t.scalar_type() == type && t.is_cuda(), what);
  return t;
}
const at::Tensor& dense(PyObject* o, at::ScalarType type, const char* what) {
  const at::Tensor& t = cuda_tensor(o, type, what);
  expect(t.is_contiguous(), what);
  return t;
}
bool truth(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw Fail{};
  return v == 1;
}
void* ptr(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
template <typename T>
T* ptr_as(PyObject* o) { return static_cast<T*>(ptr(o)); }

// The tensor a mapping (or a sequence, with an int key) holds under `key`: a reference of its own.
at::Tensor item(PyObject* o, PyObject* key) {
  PyObject* v = PyObject_GetItem(o, key);
  if (!v) throw Fail{};
  at::Tensor t;
  if (THPVariable_Check(v)) t = THPVariable_Unpack(v);
  else PyErr_Format(PyExc_TypeError, "expected a torch.Tensor, got %s", Py_TYPE(v)->tp_name);
  Py_DECREF(v);
  if (!t.defined()) throw Fail{};
  return t;
}

at::Tensor empty(at::IntArrayRef shape, at::ScalarType type, const at::Tensor& like) {
  return at::detail::empty_cuda(shape, type, like.device(), std::nullopt);
}
// the caller's output tensor, or a new one
at::Tensor output(PyObject* given, at::IntArrayRef shape, at::ScalarType type, const at::Tensor& like) {
  return given == Py_None ? empty(shape, type, like) : tensor(given);
}

struct Call {
  PyObject* self;
  qarl_ctx* ctx;
  void* stream;
  explicit Call(PyObject* ctx_object) : self(ctx_object) {
    PyObject* h = PyObject_GetAttr(self, s_hv);
    if (!h) throw Fail{};
    ctx = static_cast<qarl_ctx*>(PyLong_AsVoidPtr(h));  // null once closed: the library refuses it
    Py_DECREF(h);
    if (!ctx && PyErr_Occurred()) throw Fail{};
    stream = c10::cuda::getCurrentCUDAStream().stream();
  }
  // the caller's workspace, or the context's cached scratch, grown if it is too small
  at::Tensor workspace(PyObject* given, size_t bytes, const at::Tensor& like) {
    if (given != Py_None) return tensor(given);
    PyObject* o = PyObject_GetAttr(self, s_ws);
    if (!o) throw Fail{};
    at::Tensor t;
    if (THPVariable_Check(o)) t = THPVariable_Unpack(o);
    Py_DECREF(o);
    if (!t.defined() || static_cast<size_t>(t.numel()) < bytes) {
      t = empty({static_cast<int64_t>(std::max<size_t>(bytes, 256))}, at::kByte, like);
      PyObject* n = THPVariable_Wrap(t);
      const int rc = n ? PyObject_SetAttr(self, s_ws, n) : -1;
      Py_XDECREF(n);
      if (rc != 0) throw Fail{};
    }
    return t;
  }
  // runs the library call without the GIL and raises on an error status
  template <typename F>
  void run(F&& f) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    if (rc == QARL_OK) return;
    PyObject* n = PyLong_FromLong(rc);
    PyObject* r = n ? PyObject_CallMethodOneArg(self, s_check, n) : nullptr;
    Py_XDECREF(n);
    Py_XDECREF(r);
    fail("a library call failed");
  }
};

// The argument the caller gave, or the tensor made in its place (new reference).
PyObject* wrap(const at::Tensor& t) {
  PyObject* o = THPVariable_Wrap(t);
  if (!o) throw Fail{};
  return o;
}
PyObject* wrap_or(PyObject* given, const at::Tensor& t) { return given == Py_None ? wrap(t) : Py_NewRef(given); }
PyObject* none_or(const at::Tensor& t) { return t.defined() ? wrap(t) : Py_NewRef(Py_None); }

// A tuple that takes over the references.
template <typename... O>
PyObject* tuple_of(O*... o) {
  PyObject* t = PyTuple_New(sizeof...(o));
  if (!t) throw Fail{};
  Py_ssize_t i = 0;
  (PyTuple_SET_ITEM(t, i++, o), ...);
  return t;
}

template <typename F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F&& f) {
  if (n != want) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return nullptr;
  }
  try {
    return f();
  } catch (const Fail&) {
    return nullptr;
  } catch (...) {  // torch's errors keep their types (torch.OutOfMemoryError, IndexError, ...)
    if (!PyErr_Occurred()) torch::translate_exception_to_python(std::current_exception());
    return nullptr;
  }
}

// weights [E, N, K] or [N, K]
struct WeightShape {
  int64_t E, N, K;
  explicit WeightShape(const at::Tensor& w) {
    expect(w.dim() == 2 || w.dim() == 3, "weights are [N, K] or [E, N, K]");
    E = w.dim() == 3 ? w.size(0) : 1;
    N = w.size(-2);
    K = w.size(-1);
  }
};

void quantize_weight_call(Call& c, const at::Tensor& w, const WeightShape& s, void* codes, void* scales, void* pub_codes,
                          void* pub_scales) {
  void* wp = w.data_ptr();
  c.run([&] {
    return qarl_quantize_weight_publish(c.ctx, wp, s.E, s.N, s.K, static_cast<uint8_t*>(codes), static_cast<float*>(scales),
                                        static_cast<uint8_t*>(pub_codes), static_cast<float*>(pub_scales), c.stream);
  });
}

// (self, w, codes, scales) -> (codes, scales)
PyObject* quantize_weight(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 4, [&]() -> PyObject* {
    Call c(a[0]);
    const at::Tensor& w = dense(a[1], at::kBFloat16, "w: a contiguous bf16 CUDA tensor");
    const WeightShape s(w);
    at::Tensor codes = output(a[2], w.sizes(), at::kByte, w);
    at::Tensor scales = a[3] != Py_None ? tensor(a[3])
                        : w.dim() == 3  ? empty({s.E, s.N / 128, s.K / 128}, at::kFloat, w)
                                        : empty({s.N / 128, s.K / 128}, at::kFloat, w);
    quantize_weight_call(c, w, s, codes.data_ptr(), scales.data_ptr(), nullptr, nullptr);
    return tuple_of(wrap_or(a[2], codes), wrap_or(a[3], scales));
  });
}

// (self, w, codes, scales, pub_codes, pub_scales) -> (codes, scales); the buffers are the caller's
PyObject* quantize_weight_publish(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 6, [&]() -> PyObject* {
    Call c(a[0]);
    const at::Tensor& w = dense(a[1], at::kBFloat16, "w: a contiguous bf16 CUDA tensor");
    quantize_weight_call(c, w, WeightShape(w), ptr(a[2]), ptr(a[3]), ptr(a[4]), ptr(a[5]));
    return tuple_of(Py_NewRef(a[2]), Py_NewRef(a[3]));
  });
}

// (self, x, codes, scales) -> (codes, scales)
PyObject* quantize_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 4, [&]() -> PyObject* {
    Call c(a[0]);
    const at::Tensor& x = cuda_tensor(a[1], at::kBFloat16, "x: a bf16 CUDA tensor");
    expect(x.dim() == 2 && x.stride(1) == 1, "x: [M, K] with dense rows");
    const int64_t M = x.size(0), K = x.size(1), ldx = M > 1 ? x.stride(0) : K;
    at::Tensor codes = output(a[2], {M, K}, at::kByte, x);
    at::Tensor scales = output(a[3], {M, K / 128}, at::kFloat, x);
    void *xp = x.data_ptr(), *cp = codes.data_ptr(), *sp = scales.data_ptr();
    c.run([&] {
      return qarl_quantize_act(c.ctx, xp, M, K, ldx, static_cast<uint8_t*>(cp), static_cast<float*>(sp), c.stream);
    });
    return tuple_of(wrap_or(a[2], codes), wrap_or(a[3], scales));
  });
}

// (self, x, w_codes, w_scales, out, want_f32) -> y, or (y, y32)
PyObject* linear_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 6, [&]() -> PyObject* {
    Call c(a[0]);
    const at::Tensor& x = dense(a[1], at::kBFloat16, "x: a contiguous bf16 CUDA tensor");
    expect(x.dim() == 2, "x: [M, K]");
    const int64_t M = x.size(0), K = x.size(1), N = tensor(a[2]).size(0);
    const bool want_f32 = truth(a[5]);
    at::Tensor y = output(a[4], {M, N}, at::kBFloat16, x);
    at::Tensor y32;
    if (want_f32) y32 = empty({M, N}, at::kFloat, x);
    at::Tensor ws = c.workspace(Py_None, qarl_linear_workspace_bytes(M, N, K), x);
    const size_t ws_bytes = static_cast<size_t>(ws.numel());
    void *xp = x.data_ptr(), *wc = ptr(a[2]), *wsc = ptr(a[3]), *yp = y.data_ptr(), *wp = ws.data_ptr();
    void* y32p = want_f32 ? y32.data_ptr() : nullptr;
    c.run([&] {
      return qarl_linear_fwd(c.ctx, xp, M, K, static_cast<uint8_t*>(wc), static_cast<float*>(wsc), N, yp,
                             static_cast<float*>(y32p), wp, ws_bytes, c.stream);
    });
    return want_f32 ? tuple_of(wrap_or(a[4], y), wrap(y32)) : wrap_or(a[4], y);
  });
}

// The routed-expert layer's tensors, common to the FP8 and the 4-bit forms.
struct LayerArgs {
  int64_t M, H, I, E, k;
  void *x, *ids, *wts;
  LayerArgs(PyObject* xo, PyObject* ido, PyObject* wto, const at::Tensor& w13) {
    const at::Tensor& xt = dense(xo, at::kBFloat16, "x: a contiguous bf16 CUDA tensor");
    const at::Tensor& it = cuda_tensor(ido, at::kInt, "topk_ids: an int32 CUDA tensor");
    const at::Tensor& wt = cuda_tensor(wto, at::kFloat, "topk_weights: a float32 CUDA tensor");
    expect(xt.dim() == 2 && it.dim() >= 2 && w13.dim() == 3, "x [M, H], topk_ids [M, k], w13 [E, 2I, .]");
    M = xt.size(0);
    H = xt.size(1);
    k = it.size(1);
    E = w13.size(0);
    I = w13.size(1) / 2;
    x = xt.data_ptr();
    ids = it.data_ptr();
    wts = wt.data_ptr();
  }
};

// (self, x, ids, wts, w13_codes, w13_scales, w2_codes, w2_scales, out, workspace, save) -> out; save: None or a mapping
// with the tensors gate_up and h
PyObject* moe_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 11, [&]() -> PyObject* {
    Call c(a[0]);
    const LayerArgs l(a[1], a[2], a[3], tensor(a[4]));
    const at::Tensor& x = tensor(a[1]);
    at::Tensor y = output(a[8], {l.M, l.H}, at::kBFloat16, x);
    at::Tensor ws = c.workspace(a[9], a[9] != Py_None ? 0 : qarl_moe_workspace_bytes(l.M, l.H, l.I, l.E, l.k), x);
    const size_t ws_bytes = static_cast<size_t>(ws.numel());
    void *c13 = ptr(a[4]), *s13 = ptr(a[5]), *c2 = ptr(a[6]), *s2 = ptr(a[7]), *yp = y.data_ptr(), *wp = ws.data_ptr();
    qarl_moe_debug dbg{};
    const bool save = a[10] != Py_None;
    at::Tensor gate_up, h;
    if (save) {
      dbg.gate_up_bf16 = (gate_up = item(a[10], s_gate_up)).data_ptr();
      dbg.h_bf16 = (h = item(a[10], s_h)).data_ptr();
    }
    c.run([&] {
      return qarl_moe_fwd(c.ctx, l.x, static_cast<int32_t*>(l.ids), static_cast<float*>(l.wts), l.M, l.H, l.I, l.E, l.k,
                          static_cast<uint8_t*>(c13), static_cast<float*>(s13), static_cast<uint8_t*>(c2),
                          static_cast<float*>(s2), yp, wp, ws_bytes, save ? &dbg : nullptr, c.stream);
    });
    return wrap_or(a[8], y);
  });
}

// (self, parts, x, ids, wts, w13, w2, out, workspace) -> out; w13 and w2 are (packed, scales, zeros) with parts = 3
// (integer codes), (packed, scales) with parts = 2 (e2m1).  The method that calls says which: what else the caller's
// tuples hold is not looked at, as in the methods' debug forms.
PyObject* moe_fwd_4bit(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 9, [&]() -> PyObject* {
    Call c(a[0]);
    const int parts = static_cast<int>(PyLong_AsLong(a[1]));
    at::Tensor w[2][3];  // (held until the call returns: a sequence may make its items on request)
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < parts; ++j) w[i][j] = item(a[5 + i], s_index[j]);
    const LayerArgs l(a[2], a[3], a[4], w[0][0]);
    const at::Tensor& x = tensor(a[2]);
    at::Tensor y = output(a[7], {l.M, l.H}, at::kBFloat16, x);
    at::Tensor ws = c.workspace(a[8], a[8] != Py_None ? 0 : qarl_moe_w4a16_workspace_bytes(l.M, l.H, l.I, l.E, l.k), x);
    const size_t ws_bytes = static_cast<size_t>(ws.numel());
    void *yp = y.data_ptr(), *wp = ws.data_ptr();
    const int32_t* ids = static_cast<int32_t*>(l.ids);
    const float* wts = static_cast<float*>(l.wts);
    void* d[2][3];
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < 3; ++j) d[i][j] = j < parts ? w[i][j].data_ptr() : nullptr;
    uint8_t *p13 = static_cast<uint8_t*>(d[0][0]), *p2 = static_cast<uint8_t*>(d[1][0]);
    uint8_t *z13 = static_cast<uint8_t*>(d[0][2]), *z2 = static_cast<uint8_t*>(d[1][2]);
    c.run([&] {
      return parts == 3 ? qarl_moe_fwd_w4a16(c.ctx, l.x, ids, wts, l.M, l.H, l.I, l.E, l.k, p13, d[0][1], z13, p2, d[1][1],
                                             z2, yp, wp, ws_bytes, nullptr, c.stream)
                        : qarl_moe_fwd_fp4a16(c.ctx, l.x, ids, wts, l.M, l.H, l.I, l.E, l.k, p13, d[0][1], p2, d[1][1], yp,
                                              wp, ws_bytes, nullptr, c.stream);
    });
    return wrap_or(a[7], y);
  });
}

// (self, x, w_router, k) -> (logits, ids, weights)
PyObject* router_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 4, [&]() -> PyObject* {
    Call c(a[0]);
    const at::Tensor& x = dense(a[1], at::kBFloat16, "x: a contiguous bf16 CUDA tensor");
    const at::Tensor& w = dense(a[2], at::kBFloat16, "w_router: a contiguous bf16 CUDA tensor");
    expect(x.dim() == 2 && w.dim() >= 1, "x [M, H], w_router [E, H]");
    const int64_t k = PyLong_AsLongLong(a[3]);
    if (k == -1 && PyErr_Occurred()) throw Fail{};
    const int64_t M = x.size(0), H = x.size(1), E = w.size(0);
    at::Tensor logits = empty({M, E}, at::kFloat, x), ids = empty({M, k}, at::kInt, x), wts = empty({M, k}, at::kFloat, x);
    void *xp = x.data_ptr(), *wp = w.data_ptr(), *lp = logits.data_ptr(), *ip = ids.data_ptr(), *tp = wts.data_ptr();
    c.run([&] {
      return qarl_router_fwd(c.ctx, xp, M, H, wp, E, k, static_cast<float*>(lp), static_cast<int32_t*>(ip),
                             static_cast<float*>(tp), c.stream);
    });
    return tuple_of(wrap(logits), wrap(ids), wrap(wts));
  });
}

// (self, dy, x, w, want_dx_f32, dx, dw) -> (dx or None, dx32 or None, dw or None)
PyObject* linear_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 7, [&]() -> PyObject* {
    Call c(a[0]);
    const at::Tensor& dy = dense(a[1], at::kBFloat16, "dy: a contiguous bf16 CUDA tensor");
    const at::Tensor& x = dense(a[2], at::kBFloat16, "x: a contiguous bf16 CUDA tensor");
    const at::Tensor& w = dense(a[3], at::kBFloat16, "w: a contiguous bf16 CUDA tensor");
    expect(dy.dim() == 2 && x.dim() == 2 && w.dim() == 2, "dy [M, N], x [M, K], w [N, K]");
    const int64_t M = dy.size(0), N = dy.size(1), K = x.size(1);
    expect(x.size(0) == M && w.size(0) == N && w.size(1) == K, "dy [M, N], x [M, K], w [N, K]");
    const bool f32 = truth(a[4]), want_dx = truth(a[5]), want_dw = truth(a[6]);
    at::Tensor dx, dx32, dw;
    if (want_dx) dx = empty({M, K}, at::kBFloat16, dy);
    if (want_dx && f32) dx32 = empty({M, K}, at::kFloat, dy);
    if (want_dw) dw = empty({N, K}, at::kFloat, dy);
    auto at_of = [](const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; };
    void *dyp = dy.data_ptr(), *xp = x.data_ptr(), *wp = w.data_ptr(), *dxp = at_of(dx), *dx32p = at_of(dx32), *dwp = at_of(dw);
    c.run([&] {
      return qarl_linear_bwd(c.ctx, dyp, xp, wp, M, N, K, dxp, static_cast<float*>(dx32p), static_cast<float*>(dwp), c.stream);
    });
    return tuple_of(none_or(dx), none_or(dx32), none_or(dw));
  });
}

// (self, lp_cur, lp_old_learner, lp_old_sampler, offsets, adv, eps_h, delta_l, delta_h, cap, want_grad, out, workspace)
// -> dict(r, w, J, flags, grad, loss)
PyObject* tbpo_loss(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 13, [&]() -> PyObject* {
    Call c(a[0]);
    const at::Tensor& cur = dense(a[1], at::kFloat, "lp_cur: a contiguous float32 CUDA tensor");
    const at::Tensor& old_l = dense(a[2], at::kFloat, "lp_old_learner: a contiguous float32 CUDA tensor");
    const at::Tensor& old_s = dense(a[3], at::kFloat, "lp_old_sampler: a contiguous float32 CUDA tensor");
    const at::Tensor& off = cuda_tensor(a[4], at::kLong, "offsets: an int64 CUDA tensor");
    const at::Tensor& adv = dense(a[5], at::kFloat, "adv: a contiguous float32 CUDA tensor");
    const int64_t B = adv.size(0), T = cur.size(0);
    double prm[4];
    for (int i = 0; i < 4; ++i) {
      prm[i] = PyFloat_AsDouble(a[6 + i]);
      if (prm[i] == -1.0 && PyErr_Occurred()) throw Fail{};
    }
    const qarl_tbpo_params params{prm[0], prm[1], prm[2], prm[3]};
    struct Output {
      PyObject* key;
      at::ScalarType type;
      int64_t n;
    };
    const Output outputs[6] = {{s_r, at::kDouble, B},  {s_w, at::kDouble, B},   {s_J, at::kDouble, B},
                               {s_flags, at::kInt, B}, {s_grad, at::kFloat, T}, {s_loss, at::kDouble, 1}};
    at::Tensor t[6];
    void* p[6] = {};
    const bool given = a[11] != Py_None;
    const bool want_grad = !given && truth(a[10]);
    for (int i = 0; i < 6; ++i) {
      if (!given) {
        if (outputs[i].key != s_grad || want_grad) t[i] = empty({outputs[i].n}, outputs[i].type, cur);
      } else {  // any mapping; an entry may be None (no gradient)
        PyObject* v = PyObject_GetItem(a[11], outputs[i].key);
        if (!v) throw Fail{};
        const bool none = v == Py_None;
        if (THPVariable_Check(v)) t[i] = THPVariable_Unpack(v);
        Py_DECREF(v);
        if (!none && !t[i].defined()) fail("out: a mapping of tensors, as an earlier call returned it");
      }
      if (t[i].defined()) p[i] = t[i].data_ptr();
    }
    at::Tensor ws = c.workspace(a[12], a[12] != Py_None ? 0 : qarl_tbpo_workspace_bytes(B, T), cur);
    const size_t ws_bytes = static_cast<size_t>(ws.numel());
    void *p0 = cur.data_ptr(), *p1 = old_l.data_ptr(), *p2 = old_s.data_ptr(), *po = off.data_ptr(), *pa = adv.data_ptr(),
         *wp = ws.data_ptr();
    c.run([&] {
      return qarl_tbpo_loss(c.ctx, static_cast<float*>(p0), static_cast<float*>(p1), static_cast<float*>(p2),
                            static_cast<int64_t*>(po), static_cast<float*>(pa), B, T, &params, static_cast<double*>(p[0]),
                            static_cast<double*>(p[1]), static_cast<double*>(p[2]), static_cast<int32_t*>(p[3]),
                            static_cast<float*>(p[4]), static_cast<double*>(p[5]), wp, ws_bytes, c.stream);
    });
    if (given) return Py_NewRef(a[11]);
    PyObject* out = PyDict_New();
    if (!out) throw Fail{};
    for (int i = 0; i < 6; ++i) {
      PyObject* v = t[i].defined() ? THPVariable_Wrap(t[i]) : Py_NewRef(Py_None);
      const int rc = v ? PyDict_SetItem(out, outputs[i].key, v) : -1;
      Py_XDECREF(v);
      if (rc != 0) {
        Py_DECREF(out);
        throw Fail{};
      }
    }
    return out;
  });
}

#define FAST(name, doc) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name)), METH_FASTCALL, doc}
PyMethodDef methods[] = {
    FAST(quantize_weight, "qarl_quantize_weight"),         FAST(quantize_weight_publish, "qarl_quantize_weight_publish"),
    FAST(quantize_act, "qarl_quantize_act"),               FAST(linear_fwd, "qarl_linear_fwd"),
    FAST(moe_fwd, "qarl_moe_fwd"),                         FAST(moe_fwd_4bit, "qarl_moe_fwd_w4a16 / qarl_moe_fwd_fp4a16"),
    FAST(router_fwd, "qarl_router_fwd"),                   FAST(linear_bwd, "qarl_linear_bwd"),
    FAST(tbpo_loss, "qarl_tbpo_loss"),                     {nullptr, nullptr, 0, nullptr}};
#undef FAST

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Marshalling of the hot calls of libqarl.so.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  struct {
    PyObject** at;
    const char* text;
  } names[] = {{&s_hv, "_hv"}, {&s_ws, "_ws"}, {&s_check, "_check"}, {&s_r, "r"},      {&s_w, "w"},
               {&s_J, "J"},    {&s_flags, "flags"}, {&s_grad, "grad"},  {&s_loss, "loss"},   {&s_gate_up, "gate_up"},
               {&s_h, "h"}};
  for (auto& s : names)
    if (!(*s.at = PyUnicode_InternFromString(s.text))) return nullptr;
  for (long i = 0; i < 3; ++i)
    if (!(s_index[i] = PyLong_FromLong(i))) return nullptr;
  return PyModule_Create(&module);
}
