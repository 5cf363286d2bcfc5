// Argument marshalling of binding.py: the objects of the Python layer (AttnParams, QTensor, torch tensors)
// into the structs and pointers of the C ABI.  Every function takes positional arguments, calls one entry
// point with the interpreter lock released and returns its status.  With ctypes the same marshalling took
// 12 us of a 16 us forward call (structs built field by field, a Python call per pointer and for the
// stream); the GPU side of a small problem is shorter than that.
#include <Python.h>

#include <torch/csrc/autograd/python_variable.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/ops/empty.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>

#include "../../include/attn_fp8.h"

// What this file was compiled for, found in the module's bytes by build.py and binding.py before they load it.
extern "C" __attribute__((used, visibility("default"))) const char attn_marshal_built_for[] = "marshal built for: " MARSHAL_BUILT_FOR;

namespace {

struct Names {
  PyObject *batch, *seqlen, *heads_q, *heads_kv, *head_dim_qk, *head_dim_v, *causal, *softmax_scale, *precision, *delta_mode,
      *seqlen_k, *q_start, *keys_valid;
  PyObject *row_codes, *row_scales, *col_codes, *col_scales, *shape;
  PyObject *data_ptr, *numel, *cuda_stream;
} names;

struct Failed {};                                     // a Python exception is set

void fail(PyObject* type, const char* message) {
  PyErr_SetString(type, message);
  throw Failed{};
}

// An attribute, held for the length of a scope.
struct Attr {
  PyObject* o;
  Attr(PyObject* of, PyObject* name) : o(PyObject_GetAttr(of, name)) { if (!o) throw Failed{}; }
  explicit Attr(PyObject* owned) : o(owned) { if (!o) throw Failed{}; }
  ~Attr() { Py_DECREF(o); }
  Attr(const Attr&) = delete;
};

int64_t integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw Failed{};
  return v;
}
// A field of a struct, as ctypes stores it: by __index__ (a float is refused, not truncated), the low 32 bits.
int32_t int32(PyObject* o) {
  const unsigned long v = PyLong_AsUnsignedLongMask(o);
  if (v == static_cast<unsigned long>(-1) && PyErr_Occurred()) throw Failed{};
  return static_cast<int32_t>(v);
}
int32_t int_field(PyObject* of, PyObject* name) {
  Attr a(of, name);
  return int32(a.o);
}
// what int() and float() make of a value
int32_t as_int(PyObject* o) {
  Attr n(PyNumber_Long(o));
  return int32(n.o);
}
float as_float(PyObject* o) {
  Attr n(PyNumber_Float(o));
  return static_cast<float>(PyFloat_AS_DOUBLE(n.o));
}

// Device pointer of a tensor (null for None).
void* pointer(PyObject* o) {
  if (o == Py_None) return nullptr;
  if (THPVariable_Check(o)) return THPVariable_Unpack(o).data_ptr();
  Attr p(PyObject_CallMethodNoArgs(o, names.data_ptr));
  void* v = PyLong_AsVoidPtr(p.o);
  if (!v && PyErr_Occurred()) throw Failed{};
  return v;
}
size_t elements(PyObject* o) {
  if (o == Py_None) return 0;
  if (THPVariable_Check(o)) return static_cast<size_t>(THPVariable_Unpack(o).numel());
  Attr n(PyObject_CallMethodNoArgs(o, names.numel));
  return static_cast<size_t>(integer(n.o));
}
void* pointer_field(PyObject* of, PyObject* name) {
  Attr a(of, name);
  return pointer(a.o);
}

attn_qtensor_t operand(PyObject* o) {
  attn_qtensor_t t;
  t.row_codes = static_cast<uint8_t*>(pointer_field(o, names.row_codes));
  t.row_scales = static_cast<uint8_t*>(pointer_field(o, names.row_scales));
  t.col_codes = static_cast<uint8_t*>(pointer_field(o, names.col_codes));
  t.col_scales = static_cast<uint8_t*>(pointer_field(o, names.col_scales));
  return t;
}

attn_params_t parameters(PyObject* o) {
  attn_params_t p;
  p.batch = int_field(o, names.batch);
  p.seqlen = int_field(o, names.seqlen);
  p.heads_q = int_field(o, names.heads_q);
  p.heads_kv = int_field(o, names.heads_kv);
  p.head_dim_qk = int_field(o, names.head_dim_qk);
  p.head_dim_v = int_field(o, names.head_dim_v);
  Attr causal(o, names.causal), scale(o, names.softmax_scale);
  p.causal = as_int(causal.o);
  p.softmax_scale = as_float(scale.o);
  p.precision = int_field(o, names.precision);
  p.delta_mode = int_field(o, names.delta_mode);
  p.seqlen_k = int_field(o, names.seqlen_k);
  p.q_start = int_field(o, names.q_start);
  p.keys_valid = int_field(o, names.keys_valid);
  return p;
}

// None: the current stream of the current device.
void* stream_of(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  Attr s(o, names.cuda_stream);
  void* v = PyLong_AsVoidPtr(s.o);
  if (!v && PyErr_Occurred()) throw Failed{};
  return v;
}

// A contiguous CUDA tensor [B, H, N, d] of one of the source types, as a quantiser job.
attn_quantize_job_t source(PyObject* o, const char* not_tensor, const char* not_type) {
  if (!THPVariable_Check(o)) fail(PyExc_ValueError, not_tensor);
  const at::Tensor& x = THPVariable_Unpack(o);
  if (!x.is_cuda() || !x.is_contiguous() || x.dim() != 4) fail(PyExc_ValueError, not_tensor);
  attn_quantize_job_t j = {};
  if (x.scalar_type() == at::kBFloat16) j.src_dtype = ATTN_SRC_BF16;
  else if (x.scalar_type() == at::kFloat) j.src_dtype = ATTN_SRC_FP32;
  else fail(PyExc_ValueError, not_type);
  j.src = x.data_ptr();
  j.B = static_cast<int32_t>(x.size(0));
  j.H = static_cast<int32_t>(x.size(1));
  j.N = static_cast<int32_t>(x.size(2));
  j.d = static_cast<int32_t>(x.size(3));
  return j;
}
void check_shape(PyObject* qtensor, const attn_quantize_job_t& j, const char* message) {
  Attr shape(qtensor, names.shape);
  Attr t(PySequence_Tuple(shape.o));
  const int32_t want[4] = {j.B, j.H, j.N, j.d};
  bool same = PyTuple_GET_SIZE(t.o) == 4;
  for (int i = 0; same && i < 4; ++i) {
    Attr n(PyLong_FromLong(want[i]));
    const int equal = PyObject_RichCompareBool(PyTuple_GET_ITEM(t.o, i), n.o, Py_EQ);
    if (equal < 0) throw Failed{};
    same = equal;
  }
  if (!same) fail(PyExc_ValueError, message);
}

// Whether a kernel launched here may stand in for torch operations on `o`: a plain CUDA tensor, with nothing that follows
// or replaces the operations (a trace, a dispatch or function mode, a functorch level, a tensor subclass, a tangent, a
// lazy conjugate, negative or zero).  Whatever does has to see torch's own operations.
bool plain(PyObject* o) {
  using c10::DispatchKey;
  static constexpr c10::DispatchKeySet kTensor({DispatchKey::CUDA, DispatchKey::AutogradCUDA, DispatchKey::AutocastCUDA, DispatchKey::ADInplaceOrView});
  static constexpr c10::DispatchKeySet kThread({DispatchKey::BackendSelect, DispatchKey::ADInplaceOrView});
  if (!THPVariable_CheckExact(o)) return false;
  const at::Tensor& x = THPVariable_Unpack(o);
  return kTensor.has_all(x.key_set()) && kThread.has_all(c10::impl::tls_local_dispatch_key_set().included_) &&
         !at::impl::torch_function_mode_enabled() && !x._fw_grad(0).defined();
}

template <class F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F&& body) {
  try {
    if (n != want) fail(PyExc_TypeError, "wrong number of arguments");
    return body();
  } catch (const Failed&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

template <class F>
PyObject* status_of(F&& call) {
  attn_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

// (params, q, k, v, o, lse, workspace, stream)
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 8, [&] {
    const attn_params_t p = parameters(a[0]);
    const attn_qtensor_t q = operand(a[1]), k = operand(a[2]), v = operand(a[3]);
    void *o = pointer(a[4]), *lse = pointer(a[5]), *ws = pointer(a[6]), *st = stream_of(a[7]);
    const size_t bytes = elements(a[6]);
    return status_of([&] { return attn_fp8_fwd(&p, q, k, v, o, static_cast<float*>(lse), ws, bytes, st); });
  });
}

// (params, q, k, v, o, lse, stream)
PyObject* fwd_noalloc(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 7, [&] {
    const attn_params_t p = parameters(a[0]);
    const attn_qtensor_t q = operand(a[1]), k = operand(a[2]), v = operand(a[3]);
    void *o = pointer(a[4]), *lse = pointer(a[5]), *st = stream_of(a[6]);
    return status_of([&] { return attn_fp8_fwd_noalloc(&p, q, k, v, o, static_cast<float*>(lse), st); });
  });
}

// (params, q, k, v, dO, dO_bf16, o_bf16, lse, delta, workspace, stream)
PyObject* bwd_delta(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 11, [&] {
    const attn_params_t p = parameters(a[0]);
    const attn_qtensor_t q = operand(a[1]), k = operand(a[2]), v = operand(a[3]), dO = operand(a[4]);
    void *dOb = pointer(a[5]), *o = pointer(a[6]), *lse = pointer(a[7]), *delta = pointer(a[8]), *ws = pointer(a[9]);
    void* st = stream_of(a[10]);
    const size_t bytes = elements(a[9]);
    return status_of([&] {
      return attn_fp8_bwd_delta(&p, q, k, v, dO, dOb, o, static_cast<const float*>(lse), static_cast<float*>(delta), ws, bytes, st);
    });
  });
}

// (params, q, k, v, dO, lse, delta, dq, dk, dv, rowsum, rowabs, workspace, stream)
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 14, [&] {
    const attn_params_t p = parameters(a[0]);
    const attn_qtensor_t q = operand(a[1]), k = operand(a[2]), v = operand(a[3]), dO = operand(a[4]);
    const float *lse = static_cast<float*>(pointer(a[5])), *delta = static_cast<float*>(pointer(a[6]));
    void *dq = pointer(a[7]), *dk = pointer(a[8]), *dv = pointer(a[9]), *rs = pointer(a[10]), *ra = pointer(a[11]);
    void *ws = pointer(a[12]), *st = stream_of(a[13]);
    const size_t bytes = elements(a[12]);
    return status_of([&] {
      return attn_fp8_bwd(&p, q, k, v, dO, lse, delta, dq, dk, dv, static_cast<float*>(rs), static_cast<float*>(ra), ws, bytes, st);
    });
  });
}

// (params, q, k, v, dO, lse, delta, dq, rowsum, rowabs, workspace, stream)
PyObject* bwd_dq(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 12, [&] {
    const attn_params_t p = parameters(a[0]);
    const attn_qtensor_t q = operand(a[1]), k = operand(a[2]), v = operand(a[3]), dO = operand(a[4]);
    const float *lse = static_cast<float*>(pointer(a[5])), *delta = static_cast<float*>(pointer(a[6]));
    void *dq = pointer(a[7]), *rs = pointer(a[8]), *ra = pointer(a[9]), *ws = pointer(a[10]), *st = stream_of(a[11]);
    const size_t bytes = elements(a[10]);
    return status_of([&] {
      return attn_fp8_bwd_dq(&p, q, k, v, dO, lse, delta, dq, static_cast<float*>(rs), static_cast<float*>(ra), ws, bytes, st);
    });
  });
}

// (params, q, k, v, dO, lse, delta, dk, dv, workspace, stream)
PyObject* bwd_dkdv(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 11, [&] {
    const attn_params_t p = parameters(a[0]);
    const attn_qtensor_t q = operand(a[1]), k = operand(a[2]), v = operand(a[3]), dO = operand(a[4]);
    const float *lse = static_cast<float*>(pointer(a[5])), *delta = static_cast<float*>(pointer(a[6]));
    void *dk = pointer(a[7]), *dv = pointer(a[8]), *ws = pointer(a[9]), *st = stream_of(a[10]);
    const size_t bytes = elements(a[9]);
    return status_of([&] { return attn_fp8_bwd_dkdv(&p, q, k, v, dO, lse, delta, dk, dv, ws, bytes, st); });
  });
}

const char* kOneSource = "src must be a contiguous CUDA tensor [B, H, N, d]";
const char* kOneType = "src must be bfloat16 or float32";
const char* kOneOut = "out was allocated for another shape";

// (src, out, stream)
PyObject* quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 3, [&] {
    attn_quantize_job_t j = source(a[0], kOneSource, kOneType);
    check_shape(a[1], j, kOneOut);
    j.out = operand(a[1]);
    void* st = stream_of(a[2]);
    return status_of([&] { return attn_fp8_quantize(j.src, j.src_dtype, j.B, j.H, j.N, j.d, j.out, st); });
  });
}

// (srcs, outs, workspace, stream)
PyObject* quantize_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 4, [&] {
    Attr srcs(PySequence_Fast(a[0], "srcs must be a sequence")), outs(PySequence_Fast(a[1], "outs must be a sequence"));
    const Py_ssize_t count = PySequence_Fast_GET_SIZE(srcs.o);
    attn_quantize_job_t jobs[ATTN_QUANTIZE_MAX_JOBS] = {};
    for (Py_ssize_t i = 0; i < count && i < PySequence_Fast_GET_SIZE(outs.o); ++i) {
      attn_quantize_job_t j = source(PySequence_Fast_GET_ITEM(srcs.o, i), "every source must be a contiguous CUDA tensor [B, H, N, d]",
                                     "sources must be bfloat16 or float32");
      PyObject* out = PySequence_Fast_GET_ITEM(outs.o, i);
      check_shape(out, j, "an output was allocated for another shape");
      j.out = operand(out);
      if (i < ATTN_QUANTIZE_MAX_JOBS) jobs[i] = j;    // (more are refused by the entry point)
    }
    void *ws = pointer(a[2]), *st = stream_of(a[3]);
    const size_t bytes = elements(a[2]);
    return status_of([&] { return attn_fp8_quantize_batch(jobs, static_cast<int32_t>(count), ws, bytes, st); });
  });
}

// (src, cos, sin, scale, mean, out, stream)
PyObject* quantize_fused(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 7, [&] {
    const attn_quantize_job_t j = source(a[0], kOneSource, kOneType);
    for (int i = 1; i <= 2; ++i) {
      if (a[i] == Py_None) continue;
      const bool tensor = THPVariable_Check(a[i]);
      if (!tensor || THPVariable_Unpack(a[i]).scalar_type() != at::kFloat || !THPVariable_Unpack(a[i]).is_contiguous() ||
          THPVariable_Unpack(a[i]).dim() != 2 || THPVariable_Unpack(a[i]).size(0) != j.N || THPVariable_Unpack(a[i]).size(1) != j.d / 2)
        fail(PyExc_ValueError, "rotary tables must be contiguous float32 [N, d/2]");
    }
    const float *cos = static_cast<float*>(pointer(a[1])), *sin = static_cast<float*>(pointer(a[2]));
    const float scale = as_float(a[3]);
    float* mean = static_cast<float*>(pointer(a[4]));
    const attn_qtensor_t out = operand(a[5]);
    void* st = stream_of(a[6]);
    return status_of([&] {
      return attn_fp8_quantize_fused(j.src, j.src_dtype, j.B, j.H, j.N, j.d, cos, sin, scale, mean, out, st);
    });
  });
}

// (src, row_out or None, col_out or None, stream)
PyObject* prepare_bf16(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 4, [&] {
    const attn_quantize_job_t j = source(a[0], kOneSource, kOneType);
    attn_qtensor_t out = {};
    out.row_codes = static_cast<uint8_t*>(pointer(a[1]));
    out.col_codes = static_cast<uint8_t*>(pointer(a[2]));
    void* st = stream_of(a[3]);
    return status_of([&] { return attn_fp8_prepare_bf16(j.src, j.src_dtype, j.B, j.H, j.N, j.d, out, st); });
  });
}

// (src, want_row, want_col): new buffers (row_codes, row_scales, col_codes, col_scales) for the quantised src
PyObject* new_operand(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 3, [&]() -> PyObject* {
    const attn_quantize_job_t j = source(a[0], kOneSource, kOneType);
    const int row = PyObject_IsTrue(a[1]), col = PyObject_IsTrue(a[2]);
    if (row < 0 || col < 0) throw Failed{};
    const auto u8 = THPVariable_Unpack(a[0]).options().dtype(at::kByte).requires_grad(false);
    const auto bytes = [&](int64_t rows, int64_t cols) { return static_cast<int64_t>(attn_fp8_scale_bytes(j.B, j.H, rows, cols)); };
    PyObject* t[4] = {nullptr, nullptr, nullptr, nullptr};
    if (row) {
      t[0] = THPVariable_Wrap(at::empty({j.B, j.H, j.N, j.d}, u8));
      t[1] = THPVariable_Wrap(at::empty({bytes(j.N, j.d)}, u8));
    }
    if (col) {
      t[2] = THPVariable_Wrap(at::empty({j.B, j.H, j.d, j.N}, u8));
      t[3] = THPVariable_Wrap(at::empty({bytes(j.d, j.N)}, u8));
    }
    for (PyObject*& o : t)
      if (!o) { o = Py_None; Py_INCREF(o); }
    return Py_BuildValue("(NNNN)", t[0], t[1], t[2], t[3]);
  });
}

// (x, multiple): the padded tensor, or None where there is nothing to pad or the kernel does not apply (the caller goes on
// with torch then)
PyObject* pad_tokens(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 2, [&]() -> PyObject* {
    if (!plain(a[0]) || !PyLong_Check(a[1])) Py_RETURN_NONE;
    const at::Tensor& x = THPVariable_Unpack(a[0]);
    const int64_t multiple = integer(a[1]);
    if (multiple <= 0 || multiple > INT32_MAX || !x.is_contiguous() || x.dim() != 4 || x.size(2) % multiple == 0) Py_RETURN_NONE;
    const int64_t rows = (x.size(2) / multiple + 1) * multiple;
    if (x.requires_grad() || x.numel() == 0 ||
        (x.size(3) * x.element_size()) % 16 || reinterpret_cast<uintptr_t>(x.data_ptr()) % 16 || x.size(0) * x.size(1) > INT32_MAX ||
        rows > INT32_MAX || x.size(3) * x.element_size() / 16 * rows > INT32_MAX ||     // the kernel counts a slab's pieces in 32 bits
        x.get_device() != c10::cuda::current_device())
      Py_RETURN_NONE;
    at::Tensor out = at::empty({x.size(0), x.size(1), rows, x.size(3)}, x.options());
    const attn_status_t st = attn_fp8_pad_tokens(x.data_ptr(), static_cast<int32_t>(x.element_size()), static_cast<int32_t>(x.size(0)),
                                                 static_cast<int32_t>(x.size(1)), static_cast<int32_t>(x.size(2)),
                                                 static_cast<int32_t>(x.size(3)), static_cast<int32_t>(rows), out.data_ptr(),
                                                 c10::cuda::getCurrentCUDAStream().stream());
    if (st != ATTN_OK) fail(PyExc_RuntimeError, attn_fp8_last_error());
    return THPVariable_Wrap(out);
  });
}

// (parts): the buffers (row_codes, row_scales, col_codes, col_scales) of the QTensors of consecutive tokens put together,
// or None where the kernel does not apply (the caller concatenates with torch then)
PyObject* concat(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 1, [&]() -> PyObject* {
    Attr parts(PySequence_Fast(a[0], "parts must be a sequence"));
    const Py_ssize_t count = PySequence_Fast_GET_SIZE(parts.o);
    PyObject* const field[4] = {names.row_codes, names.row_scales, names.col_codes, names.col_scales};
    constexpr Py_ssize_t kMost = 256;
    if (count < 1 || count > kMost) Py_RETURN_NONE;
    int64_t b = 0, h = 0, d = 0, total = 0, tokens[kMost];
    for (Py_ssize_t i = 0; i < count; ++i) {
      Attr shape(PySequence_Fast_GET_ITEM(parts.o, i), names.shape);
      Attr t(PySequence_Tuple(shape.o));
      if (PyTuple_GET_SIZE(t.o) != 4) Py_RETURN_NONE;
      const int64_t s[4] = {integer(PyTuple_GET_ITEM(t.o, 0)), integer(PyTuple_GET_ITEM(t.o, 1)), integer(PyTuple_GET_ITEM(t.o, 2)),
                            integer(PyTuple_GET_ITEM(t.o, 3))};
      if (i == 0) { b = s[0]; h = s[1]; d = s[3]; }
      if (s[0] != b || s[1] != h || s[3] != d || s[2] <= 0 || s[2] % 128) Py_RETURN_NONE;
      tokens[i] = s[2];
      total += s[2];
    }
    // rows and bytes per row and token of the four byte tensors
    const int64_t c = (d + 127) / 128, rows[4] = {b * h, b * h, b * h * d, b * h * c};
    const auto width = [&](int f, int64_t n) { return f == 0 ? n * d : f == 1 ? n / 128 * c * 512 : f == 2 ? n : n / 128 * 512; };
    if (b <= 0 || h <= 0 || d <= 0 || d % 16) Py_RETURN_NONE;
    const int64_t dims[4][4] = {{b, h, total, d}, {}, {b, h, d, total}, {}};
    at::Tensor out[4];
    attn_copy_job_t jobs[ATTN_COPY_MAX_JOBS];
    int n_jobs = 0;
    void* const stream = c10::cuda::getCurrentCUDAStream().stream();
    const auto flush = [&] {
      if (n_jobs && attn_fp8_copy_batch(jobs, n_jobs, stream) != ATTN_OK) fail(PyExc_RuntimeError, attn_fp8_last_error());
      n_jobs = 0;
    };
    // all tensors are looked at before the first launch
    for (int pass = 0; pass < 2; ++pass) {
      for (int f = 0; f < 4; ++f) {
        int64_t at_bytes = 0;
        for (Py_ssize_t i = 0; i < count; ++i) {
          Attr o(PySequence_Fast_GET_ITEM(parts.o, i), field[f]);
          if (o.o == Py_None) {
            if (i && out[f].defined()) Py_RETURN_NONE;
            continue;
          }
          if (!plain(o.o)) Py_RETURN_NONE;
          const at::Tensor& x = THPVariable_Unpack(o.o);
          const int64_t w = width(f, tokens[i]);
          if (pass == 0) {
            if (x.get_device() != c10::cuda::current_device() || x.scalar_type() != at::kByte || !x.is_contiguous() ||
                x.numel() != rows[f] * w || reinterpret_cast<uintptr_t>(x.data_ptr()) % 16 || (i && !out[f].defined()))
              Py_RETURN_NONE;
            if (i == 0)
              out[f] = f % 2 == 0 ? at::empty({dims[f][0], dims[f][1], dims[f][2], dims[f][3]}, x.options())
                                  : at::empty({rows[f] * width(f, total)}, x.options());
          } else {
            jobs[n_jobs++] = attn_copy_job_t{x.data_ptr(), static_cast<uint8_t*>(out[f].data_ptr()) + at_bytes, rows[f], w, width(f, total)};
            if (n_jobs == ATTN_COPY_MAX_JOBS) flush();
            at_bytes += w;
          }
        }
      }
    }
    flush();
    PyObject* t[4];
    for (int f = 0; f < 4; ++f) {
      if (out[f].defined()) t[f] = THPVariable_Wrap(out[f]);
      else { t[f] = Py_None; Py_INCREF(Py_None); }
    }
    return Py_BuildValue("(NNNN)", t[0], t[1], t[2], t[3]);
  });
}

PyMethodDef methods[] = {
#define ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(name)), METH_FASTCALL, nullptr}
    ENTRY(fwd), ENTRY(fwd_noalloc), ENTRY(bwd_delta), ENTRY(bwd), ENTRY(bwd_dq), ENTRY(bwd_dkdv), ENTRY(quantize),
    ENTRY(quantize_batch), ENTRY(quantize_fused), ENTRY(prepare_bf16), ENTRY(new_operand), ENTRY(pad_tokens), ENTRY(concat),
#undef ENTRY
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
#define NAME(n) if (!(names.n = PyUnicode_InternFromString(#n))) return nullptr
  NAME(batch); NAME(seqlen); NAME(heads_q); NAME(heads_kv); NAME(head_dim_qk); NAME(head_dim_v); NAME(causal);
  NAME(softmax_scale); NAME(precision); NAME(delta_mode); NAME(seqlen_k); NAME(q_start); NAME(keys_valid);
  NAME(row_codes); NAME(row_scales); NAME(col_codes); NAME(col_scales); NAME(shape);
  NAME(data_ptr); NAME(numel); NAME(cuda_stream);
#undef NAME
  return PyModule_Create(&module);
}
