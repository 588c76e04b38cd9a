// Native argument marshalling of the Python binding: torch tensors -> the C
// ABI's structs -> the call. The same checks and errors as api.py documents;
// a call's 15 segments took 45 to 80 us through ctypes (shape, strides, type
// and address of every tensor, each an interpreted call), longer than many of
// the kernels they describe; here 1 to 2 us.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "refadapt.h"

namespace {

// A Python error is set; unwinds to the entry point, which returns NULL.
struct Raised {};

[[noreturn]] void raise(PyObject* type, const char* msg) {
  PyErr_SetString(type, msg);
  throw Raised{};
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a tensor, got %R", o);
    throw Raised{};
  }
  return THPVariable_Unpack(o);
}

// Device address of a tensor, NULL for None.
void* address(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }

long long integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw Raised{};
  return v;
}
int32_t integer32(PyObject* o) { return int32_t(integer(o)); }
// int(o): any number, or its text.
int32_t as_int32(PyObject* o) {
  PyObject* v = PyNumber_Long(o);
  if (!v) throw Raised{};
  const long long x = PyLong_AsLongLong(v);
  Py_DECREF(v);
  if (x == -1 && PyErr_Occurred()) throw Raised{};
  return int32_t(x);
}
double real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Raised{};
  return v;
}

PyObject* shape_of(PyObject* o) {
  PyObject* s = PyObject_GetAttrString(o, "shape");
  PyObject* t = s ? PySequence_Tuple(s) : nullptr;
  Py_XDECREF(s);
  if (!t) throw Raised{};
  return t;
}

// ra_seg of a [B, H, n, d] bf16 CUDA tensor; None: absent, n query rows.
ra_seg seg(PyObject* o, int64_t n = 0) {
  if (o == Py_None) return ra_seg{nullptr, 0, 0, 0, int32_t(n), 0};
  const at::Tensor& t = tensor(o);
  if (t.dim() != 4 || t.scalar_type() != at::kBFloat16 || !t.is_cuda() || (t.size(3) > 1 && t.stride(3) != 1)) {
    PyObject* shape = shape_of(o);
    PyObject* dtype = PyObject_GetAttrString(o, "dtype");
    PyObject* device = PyObject_GetAttrString(o, "device");
    if (dtype && device)
      PyErr_Format(PyExc_ValueError,
                   "expected a [B, H, n, d] bf16 CUDA tensor with contiguous last axis, got %S %S %S", shape, dtype,
                   device);
    Py_DECREF(shape);
    Py_XDECREF(dtype);
    Py_XDECREF(device);
    throw Raised{};
  }
  return ra_seg{t.numel() > 0 ? t.data_ptr() : nullptr, t.stride(0), t.stride(1), t.stride(2), int32_t(t.size(2)), 0};
}

struct Rows {
  void* ptr;
  int64_t stride_s, stride_r, rows, samples;
};
// A [B, rows, F] CUDA tensor with contiguous last axis.
Rows rows_of(PyObject* o, const char* what) {
  const at::Tensor& t = tensor(o);
  if (t.dim() != 3 || !t.is_cuda() || (t.size(2) > 1 && t.stride(2) != 1)) {
    PyObject* shape = shape_of(o);
    PyErr_Format(PyExc_ValueError, "%s: expected a [B, rows, F] CUDA tensor with contiguous last axis, got %S", what,
                 shape);
    Py_DECREF(shape);
    throw Raised{};
  }
  return Rows{t.numel() > 0 ? t.data_ptr() : nullptr, t.stride(0), t.stride(1), t.size(1), t.size(0)};
}

// B, H and d of a [B, H, n, d] tensor.
struct Dims {
  int32_t B, H, d;
};
Dims dims_of(PyObject* o) {
  const at::Tensor& t = tensor(o);
  if (t.dim() != 4) raise(PyExc_ValueError, "expected a tensor of four dimensions [B, H, n, d]");
  return Dims{int32_t(t.size(0)), int32_t(t.size(1)), int32_t(t.size(3))};
}
int64_t rows4(PyObject* o) {
  const at::Tensor& t = tensor(o);
  if (t.dim() < 3) raise(PyExc_IndexError, "tuple index out of range");
  return t.size(2);
}

// Items of a sequence of at least `want` entries.
struct Seq {
  PyObject* fast;
  Seq(PyObject* o, Py_ssize_t want) : fast(PySequence_Fast(o, "expected a sequence")) {
    if (!fast) throw Raised{};
    if (size() < want) {
      Py_DECREF(fast);
      raise(PyExc_IndexError, "tuple index out of range");
    }
  }
  Seq(const Seq&) = delete;
  ~Seq() { Py_DECREF(fast); }
  Py_ssize_t size() const { return PySequence_Fast_GET_SIZE(fast); }
  PyObject* operator[](Py_ssize_t i) const { return PySequence_Fast_GET_ITEM(fast, i); }
};

// A segment's dict (any mapping): need() raises KeyError, get() gives None.
struct Map {
  PyObject* dict;
  explicit Map(PyObject* o) : dict(nullptr) {
    if (PyDict_Check(o)) {
      dict = o;
      Py_INCREF(dict);
      return;
    }
    dict = PyDict_New();
    if (!dict || PyDict_Update(dict, o) != 0) {
      Py_XDECREF(dict);
      throw Raised{};
    }
  }
  Map(const Map&) = delete;
  ~Map() { Py_DECREF(dict); }
  PyObject* get(PyObject* key) const {
    PyObject* v = PyDict_GetItemWithError(dict, key);
    if (!v && PyErr_Occurred()) throw Raised{};
    return v ? v : Py_None;
  }
  bool has(PyObject* key) const {
    const int v = PyDict_Contains(dict, key);
    if (v < 0) throw Raised{};
    return v != 0;
  }
  PyObject* need(PyObject* key) const {
    PyObject* v = PyDict_GetItemWithError(dict, key);
    if (!v) {
      if (!PyErr_Occurred()) PyErr_SetObject(PyExc_KeyError, key);
      throw Raised{};
    }
    return v;
  }
};

bool truth(PyObject* o) {
  const int v = PyObject_IsTrue(o);
  if (v < 0) throw Raised{};
  return v != 0;
}

// Interned names of the segments' entries.
struct Names {
  PyObject *h, *x, *shift, *scale, *gated, *a, *w, *bias, *out, *resid, *gate, *q, *k, *v, *q_norm, *k_norm, *pos_offset;
} N;

// Stream argument: None is the calling thread's current stream.
void* stream_of(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  return reinterpret_cast<void*>(uintptr_t(integer(o)));
}

template <class F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F f) {
  if (n != want) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return nullptr;
  }
  try {
    return PyLong_FromLong(long(f()));
  } catch (const Raised&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

template <class F>
ra_status released(F f) {
  ra_status s;
  Py_BEGIN_ALLOW_THREADS;
  s = f();
  Py_END_ALLOW_THREADS;
  return s;
}

// joint_attn(q, k, v, o, mass_partial, mode, softmax_scale, ref_logit_bias, mass_rows, err_word, mass_row_stride,
//            ref_fresh, a_b, step, stream)
PyObject* joint_attn(PyObject*, PyObject* const* g, Py_ssize_t n) {
  return guarded(n, 15, [&] {
    const Seq q(g[0], 3), k(g[1], 3), v(g[2], 3), o(g[3], 3);
    ra_attn_args a;
    std::memset(&a, 0, sizeof(a));
    const Dims dm = dims_of(k[2]);
    a.B = dm.B, a.H = dm.H, a.d = dm.d;
    for (int r = 0; r < 3; ++r) {
      const int64_t n_q = rows4(q[r] != Py_None ? q[r] : k[r]);
      a.q[r] = seg(q[r], n_q);
      a.k[r] = seg(k[r]);
      a.v[r] = seg(v[r]);
      a.o[r] = seg(o[r], n_q);
    }
    a.mass_partial = static_cast<float*>(address(g[4]));
    a.mode = static_cast<const int32_t*>(address(g[5]));
    a.softmax_scale = float(real(g[6]));
    a.ref_logit_bias = static_cast<const float*>(address(g[7]));
    a.mass_rows = integer32(g[8]);
    a.err_word = static_cast<int32_t*>(address(g[9]));
    a.mass_row_stride = integer32(g[10]);
    if (g[11] != Py_None) {
      const Seq f(g[11], 0);
      if (f.size() != 3) raise(PyExc_ValueError, "ref_fresh: expected (q, k, v)");
      a.ref_fresh_q = seg(f[0]);
      a.ref_fresh_k = seg(f[1]);
      a.ref_fresh_v = seg(f[2]);
      a.a_b = static_cast<int32_t*>(address(g[12]));
      a.step = integer32(g[13]);
    }
    void* st = stream_of(g[14]);
    return released([&] { return refadapt_joint_attn(&a, st); });
  });
}

size_t bytes_of(PyObject* o) {
  const at::Tensor& t = tensor(o);
  return size_t(t.numel()) * size_t(t.element_size());
}

// q_delta(q_cur, q_prev, d_out, workspace, eps, stream)
PyObject* q_delta(PyObject*, PyObject* const* g, Py_ssize_t n) {
  return guarded(n, 6, [&] {
    const Dims dm = dims_of(g[0]);
    const ra_seg c = seg(g[0]), p = seg(g[1]);
    float* d_out = static_cast<float*>(address(g[2]));
    void* ws = address(g[3]);
    const size_t ws_bytes = bytes_of(g[3]);
    const float eps = float(real(g[4]));
    void* st = stream_of(g[5]);
    return released([&] { return refadapt_q_delta(&c, &p, dm.B, dm.H, dm.d, eps, d_out, ws, ws_bytes, st); });
  });
}

// head: t, b, state, mode_out, theta, delta_max; tail: mass_partial_prev, mass_row_count, forced_boundary, gbar_out,
// m_out, cue
ra_gate_args gate_args(PyObject* const* head, int32_t B, int32_t H, PyObject* q_delta, PyObject* const* tail) {
  ra_gate_args a;
  std::memset(&a, 0, sizeof(a));
  a.t = integer32(head[0]);
  a.b = integer32(head[1]);
  a.state = static_cast<ra_state*>(address(head[2]));
  a.mode_out = static_cast<int32_t*>(address(head[3]));
  a.theta = real(head[4]);
  a.delta_max = integer32(head[5]);
  a.B = B;
  a.H = H;
  a.q_delta = static_cast<const float*>(address(q_delta));
  a.mass_partial_prev = static_cast<const float*>(address(tail[0]));
  if (tail[0] != Py_None) {
    const at::Tensor& m = tensor(tail[0]);
    if (m.dim() < 1) raise(PyExc_IndexError, "tuple index out of range");
    a.mass_partial_len = int32_t(m.size(-1));
  }
  a.mass_row_count = integer32(tail[1]);
  a.forced_boundary = integer32(tail[2]);
  a.gbar_out = static_cast<float*>(address(tail[3]));
  a.m_out = static_cast<float*>(address(tail[4]));
  a.cue = integer32(tail[5]);
  return a;
}

// gate(<head>, B, H, q_delta, <tail>, stream)
PyObject* gate(PyObject*, PyObject* const* g, Py_ssize_t n) {
  return guarded(n, 16, [&] {
    const ra_gate_args a = gate_args(g, integer32(g[6]), integer32(g[7]), g[8], g + 9);
    void* st = stream_of(g[15]);
    return released([&] { return refadapt_gate(&a, st); });
  });
}

// q_delta_gate(q_cur, q_prev, d_out, workspace, eps, stream, <head>, <tail>)
PyObject* q_delta_gate(PyObject*, PyObject* const* g, Py_ssize_t n) {
  return guarded(n, 18, [&] {
    const Dims dm = dims_of(g[0]);
    const ra_seg c = seg(g[0]), p = seg(g[1]);
    float* d_out = static_cast<float*>(address(g[2]));
    void* ws = address(g[3]);
    const size_t ws_bytes = bytes_of(g[3]);
    const float eps = float(real(g[4]));
    const ra_gate_args a = gate_args(g + 6, dm.B, dm.H, g[2], g + 12);
    void* st = stream_of(g[5]);
    return released([&] { return refadapt_q_delta_gate(&c, &p, dm.B, dm.H, dm.d, eps, d_out, ws, ws_bytes, &a, st); });
  });
}

[[noreturn]] void too_many_segments() { raise(PyExc_IndexError, "invalid index"); }

// ln_modulate(segs, C, eps, mode, stream)
PyObject* ln_modulate(PyObject*, PyObject* const* g, Py_ssize_t n) {
  return guarded(n, 5, [&] {
    const Seq segs(g[0], 0);
    ra_lnmod_args a;
    std::memset(&a, 0, sizeof(a));
    for (Py_ssize_t i = 0; i < segs.size(); ++i) {
      if (i >= 3) too_many_segments();
      const Map sd(segs[i]);
      ra_lnmod_seg& s = a.seg[i];
      const Rows h = rows_of(sd.need(N.h), "h"), x = rows_of(sd.need(N.x), "x");
      if (h.rows != x.rows) raise(PyExc_ValueError, "h and x rows differ");
      a.B = int32_t(h.samples);
      s.h = h.ptr, s.h_stride_s = h.stride_s, s.h_stride_r = h.stride_r;
      s.x = x.ptr, s.x_stride_s = x.stride_s, s.x_stride_r = x.stride_r;
      const at::Tensor &shift = tensor(sd.need(N.shift)), &scale = tensor(sd.need(N.scale));
      s.shift = static_cast<const float*>(shift.data_ptr());
      s.scale = static_cast<const float*>(scale.data_ptr());
      s.mod_stride_s = shift.stride(0);
      if (scale.stride(0) != s.mod_stride_s) raise(PyExc_ValueError, "shift and scale must share a row stride");
      s.rows = int32_t(h.rows);
      s.gated = truth(sd.get(N.gated));
    }
    if (segs.size() == 0) raise(PyExc_TypeError, "refadapt_ln_modulate: no segments");
    a.n_seg = int32_t(segs.size());
    a.C = integer32(g[1]);
    a.eps = float(real(g[2]));
    a.mode = static_cast<const int32_t*>(address(g[3]));
    void* st = stream_of(g[4]);
    return released([&] { return refadapt_ln_modulate(&a, st); });
  });
}

// gemm(segs, N, K, epilogue, mode, rope, H, d, norm_eps, err_word, tile_mode, stream)
PyObject* gemm(PyObject*, PyObject* const* g, Py_ssize_t n) {
  return guarded(n, 12, [&] {
    const Seq segs(g[0], 0);
    ra_gemm_args a;
    std::memset(&a, 0, sizeof(a));
    a.N = integer32(g[1]);
    a.K = integer32(g[2]);
    a.epilogue = integer32(g[3]);
    for (Py_ssize_t i = 0; i < segs.size(); ++i) {
      if (i >= 3) too_many_segments();
      const Map sd(segs[i]);
      ra_gemm_seg& s = a.seg[i];
      const Rows ar = rows_of(sd.need(N.a), "a");
      a.B = int32_t(ar.samples);
      s.a = ar.ptr, s.a_stride_s = ar.stride_s, s.a_stride_r = ar.stride_r, s.rows = int32_t(ar.rows);
      s.gated = truth(sd.get(N.gated));
      PyObject* wo = sd.need(N.w);
      const at::Tensor& w = tensor(wo);
      if (w.dim() != 2 || w.size(0) != a.N || w.size(1) != a.K || !w.is_contiguous() ||
          w.scalar_type() != at::kBFloat16) {
        PyObject* shape = shape_of(wo);
        PyErr_Format(PyExc_ValueError, "w: expected a contiguous [N, K] = [%d, %d] bf16 tensor, got %S", int(a.N),
                     int(a.K), shape);
        Py_DECREF(shape);
        throw Raised{};
      }
      s.w = w.data_ptr();
      s.bias = static_cast<const float*>(address(sd.get(N.bias)));
      if (PyObject* out = sd.get(N.out); out != Py_None) {
        const Rows r = rows_of(out, "out");
        s.out = r.ptr, s.out_stride_s = r.stride_s, s.out_stride_r = r.stride_r;
      }
      if (PyObject* res = sd.get(N.resid); res != Py_None) {
        const Rows r = rows_of(res, "resid");
        s.resid = r.ptr, s.resid_stride_s = r.stride_s, s.resid_stride_r = r.stride_r;
      }
      if (PyObject* gt = sd.get(N.gate); gt != Py_None) {
        const at::Tensor& t = tensor(gt);
        s.gate = static_cast<const float*>(t.data_ptr());
        s.gate_stride_s = t.stride(0);
      }
      if (a.epilogue == RA_EPI_QKV) {
        s.q_out = seg(sd.need(N.q));
        s.k_out = seg(sd.need(N.k));
        s.v_out = seg(sd.need(N.v));
        s.q_norm = static_cast<const float*>(address(sd.need(N.q_norm)));
        s.k_norm = static_cast<const float*>(address(sd.need(N.k_norm)));
        s.pos_offset = sd.has(N.pos_offset) ? as_int32(sd.need(N.pos_offset)) : 0;
      }
    }
    if (segs.size() == 0) raise(PyExc_TypeError, "refadapt_gemm: no segments");
    a.n_seg = int32_t(segs.size());
    a.mode = static_cast<const int32_t*>(address(g[4]));
    a.rope = static_cast<const float*>(address(g[5]));
    a.rope_len = g[5] != Py_None ? int32_t(tensor(g[5]).size(0)) : 0;
    a.H = integer32(g[6]);
    a.d = integer32(g[7]);
    a.norm_eps = float(real(g[8]));
    a.err_word = static_cast<int32_t*>(address(g[9]));
    a.tile_mode = integer32(g[10]);
    void* st = stream_of(g[11]);
    return released([&] { return refadapt_gemm(&a, st); });
  });
}

#define RA_METHOD(f) \
  {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {RA_METHOD(joint_attn), RA_METHOD(q_delta), RA_METHOD(gate),   RA_METHOD(q_delta_gate),
                         RA_METHOD(ln_modulate), RA_METHOD(gemm),   {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
  const struct {
    PyObject** slot;
    const char* name;
  } names[] = {{&N.h, "h"},       {&N.x, "x"},         {&N.shift, "shift"},   {&N.scale, "scale"},
               {&N.gated, "gated"}, {&N.a, "a"},         {&N.w, "w"},           {&N.bias, "bias"},
               {&N.out, "out"},   {&N.resid, "resid"}, {&N.gate, "gate"},     {&N.q, "q"},
               {&N.k, "k"},       {&N.v, "v"},         {&N.q_norm, "q_norm"}, {&N.k_norm, "k_norm"},
               {&N.pos_offset, "pos_offset"}};
  for (const auto& e : names)
    if (!(*e.slot = PyUnicode_InternFromString(e.name))) return nullptr;
  return PyModule_Create(&module);
}
