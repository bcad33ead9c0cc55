// CPython binding of the library's per-step calls for PyTorch tensors (module _mq_torch; mq.py is its only user).
//
// A small layer's call is two or three launches of a few microseconds of GPU work, so what it costs is the host: marshalled in
// Python through ctypes (argument structures, size queries, two to three torch.empty, the stream object) a quantizer call took
// 17.1 us and a weight gradient 26.8 us of host time, 4.3 and 8.8 us of them in the library.  Here the same steps run natively:
// sizes come from the library, buffers from at::empty on the operands' device and the call's stream (see Launch), and the
// interpreter lock is released around large allocations and the library call.  Nothing is kept between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <limits>
#include <optional>

#include "mq.h"

namespace {

PyObject* g_error = nullptr;   // mq.MqError
PyObject *s_codes, *s_scales, *s_fmt, *s_role, *s_block, *s_tscale, *s_stream;

struct PyFail {};   // a Python exception is set

PyObject* fail_status(const char* call, int status) {
  PyObject* args = Py_BuildValue("(si)", call, status);
  if (args) { PyErr_SetObject(g_error, args); Py_DECREF(args); }
  return nullptr;
}
void check(const char* call, mq_status st) {
  if (st != MQ_OK) { fail_status(call, st); throw PyFail{}; }
}
void require(bool ok, const char* what) {
  if (!ok) { PyErr_SetString(PyExc_AssertionError, what); throw PyFail{}; }
}
// an integer argument: an int, or an object that stands for one; no float and no text
long to_long(PyObject* o) {
  PyObject* n = PyNumber_Index(o);
  if (!n) throw PyFail{};
  const long v = PyLong_AsLong(n);
  Py_DECREF(n);
  if (v == -1 && PyErr_Occurred()) throw PyFail{};
  return v;
}
// an extent of the layer: whatever int() takes
long extent_of(PyObject* o) {
  if (PyLong_CheckExact(o)) return to_long(o);
  PyObject* n = PyNumber_Long(o);
  if (!n) throw PyFail{};
  const long v = PyLong_AsLong(n);
  Py_DECREF(n);
  if (v == -1 && PyErr_Occurred()) throw PyFail{};
  return v;
}
const at::Tensor& tensor_of(PyObject* o) {
  if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor"); throw PyFail{}; }
  return THPVariable_Unpack(o);
}
mq_conv_desc desc_of(PyObject* o) {
  mq_conv_desc d;
  int* f = &d.N;
  PyObject* seq = PySequence_Fast(o, "the layer descriptor is a sequence of eleven integers");
  if (!seq) throw PyFail{};
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
  bool ok = n == 11;
  if (!ok) PyErr_SetString(PyExc_TypeError, "the layer descriptor is a sequence of eleven integers");
  try {
    for (Py_ssize_t i = 0; ok && i < n; ++i) f[i] = (int)extent_of(PySequence_Fast_GET_ITEM(seq, i));
  } catch (PyFail&) { ok = false; }
  Py_DECREF(seq);
  if (!ok) throw PyFail{};
  d.block_size = 32;
  return d;
}
int out_extent(int in, int pad, int k, int stride) {
  if (stride == 0) { PyErr_SetString(PyExc_ZeroDivisionError, "stride is zero"); throw PyFail{}; }
  const int num = in + 2 * pad - k;
  return (num >= 0 ? num / stride : -((-num + stride - 1) / stride)) + 1;
}
int dtype_code(at::ScalarType t) {
  if (t == at::kFloat) return MQ_F32;
  if (t == at::kBFloat16) return MQ_BF16;
  PyErr_SetString(PyExc_KeyError, "element type of an unquantized tensor: torch.float32 or torch.bfloat16");
  throw PyFail{};
}
cudaStream_t stream_of(PyObject* o) {
  PyObject* v = PyObject_GetAttr(o, s_stream);
  if (!v) throw PyFail{};
  const unsigned long long p = PyLong_AsUnsignedLongLong(v);
  Py_DECREF(v);
  if (p == (unsigned long long)-1 && PyErr_Occurred()) throw PyFail{};
  const auto s = reinterpret_cast<cudaStream_t>(p);
  return s == cudaStreamLegacy ? nullptr : s;
}
// the interpreter lock is not held while one of these lives
class Unlocked {
 public:
  Unlocked() : state_(PyEval_SaveThread()) {}
  ~Unlocked() { PyEval_RestoreThread(state_); }
  Unlocked(const Unlocked&) = delete;
  Unlocked& operator=(const Unlocked&) = delete;

 private:
  PyThreadState* state_;
};
// Where a call runs: the operands' device, and PyTorch's current stream there or the one the caller names.  What the call
// allocates comes from the pool of ITS stream, for PyTorch's allocator orders a block's uses by the stream it was given out
// for: a block of another stream's pool might still be in use there when the kernels write it, and a workspace dropped at the
// end of the call be given out there while they run.
class Launch {
 public:
  void* stream = nullptr;
  Launch(PyObject* given, const at::Device& dev) {
    if (dev.is_cuda() && dev.index() != c10::cuda::current_device()) device_.emplace(dev);
    if (given == Py_None) { stream = c10::cuda::getCurrentCUDAStream().stream(); return; }
    const cudaStream_t s = stream_of(given);
    stream = s;
    if (!dev.is_cuda()) return;
    const c10::cuda::CUDAStream current = c10::cuda::getCurrentCUDAStream();
    if (current.stream() == s) return;
    pool_.emplace(c10::cuda::getStreamFromExternal(s, dev.index()));
    callers_ = current;
  }
  // A result leaves with the caller, who may read it on the current stream (ordered after the call's) and drop it: its block
  // then waits for that stream too before it is given out again.
  void hand_out(const at::Tensor& t) const {
    if (callers_ && t.defined() && t.is_cuda()) c10::cuda::CUDACachingAllocator::recordStream(t.storage().data_ptr(), *callers_);
  }

 private:
  std::optional<c10::cuda::CUDAGuard> device_;
  std::optional<c10::cuda::CUDAStreamGuard> pool_;
  std::optional<c10::cuda::CUDAStream> callers_;
};
at::Tensor fresh(at::IntArrayRef shape, at::ScalarType t, const at::Device& dev, bool fill) {
  int64_t n = (int64_t)c10::elementSize(t);
  for (const int64_t v : shape) n *= v;
  std::optional<Unlocked> u;
  if (n >= 1 << 20 || fill) u.emplace();     // (large blocks may take a cudaMalloc, or a wait for one; small ones cost less than the lock)
  at::Tensor r = at::empty(shape, at::TensorOptions().dtype(t).device(dev));
  if (fill) {
    if (at::isFloatingType(t)) r.fill_(std::numeric_limits<double>::quiet_NaN()); else r.fill_(0xA5);
  }
  return r;
}

// A stored tensor (mq.QTensor) as the library sees it.  The attribute objects are held until the call is done.
struct Stored {
  mq_qtensor q{};
  PyObject* held[3] = {nullptr, nullptr, nullptr};
  std::optional<at::Device> device;
  explicit Stored(PyObject* o) {
    try {
      held[0] = get(o, s_codes); held[1] = get(o, s_scales); held[2] = get(o, s_tscale);
      const at::Tensor &c = tensor_of(held[0]), &s = tensor_of(held[1]);
      q.codes = c.data_ptr(); q.codes_bytes = (size_t)c.numel();
      q.scales = static_cast<uint8_t*>(s.data_ptr()); q.scales_bytes = (size_t)s.numel();
      if (held[2] != Py_None) q.tensor_scale = static_cast<float*>(tensor_of(held[2]).data_ptr());
      q.fmt = num(o, s_fmt); q.role = num(o, s_role); q.block = num(o, s_block);
      device = c.device();
    } catch (...) { drop(); throw; }
  }
  ~Stored() { drop(); }
  Stored(const Stored&) = delete;
  Stored& operator=(const Stored&) = delete;

 private:
  void drop() { for (auto& h : held) { Py_XDECREF(h); h = nullptr; } }
  static PyObject* get(PyObject* o, PyObject* name) {
    PyObject* v = PyObject_GetAttr(o, name);
    if (!v) throw PyFail{};
    return v;
  }
  static int num(PyObject* o, PyObject* name) {
    PyObject* v = get(o, name);
    int r = 0;
    try { r = (int)to_long(v); } catch (...) { Py_DECREF(v); throw; }
    Py_DECREF(v);
    return r;
  }
};
// A stored tensor to be created for a result
struct Created {
  at::Tensor codes, scales, tscale;
  mq_qtensor q{};
  Created(size_t cb, size_t sb, int fmt, int role, int block, const at::Device& dev, bool fill) {
    codes = fresh({(int64_t)cb}, at::kByte, dev, fill);
    scales = fresh({(int64_t)sb}, at::kByte, dev, fill);
    if (block == MQ_BLOCK_TS16) { tscale = fresh({2}, at::kFloat, dev, fill); q.tensor_scale = tscale.data_ptr<float>(); }
    q.codes = codes.data_ptr(); q.codes_bytes = cb;
    q.scales = scales.data_ptr<uint8_t>(); q.scales_bytes = sb;
    q.fmt = fmt; q.role = role; q.block = block;
  }
  PyObject* to_python(const Launch& l) {   // (codes, scales, tensor scale or None)
    l.hand_out(codes); l.hand_out(scales); l.hand_out(tscale);
    PyObject* t = Py_None;
    if (tscale.defined()) t = THPVariable_Wrap(tscale); else Py_INCREF(t);
    return Py_BuildValue("(NNN)", THPVariable_Wrap(codes), THPVariable_Wrap(scales), t);
  }
};

// the caller's workspace, or one of `need` bytes
struct Workspace {
  at::Tensor own;
  void* ptr = nullptr;
  size_t bytes = 0;
  Workspace(PyObject* given, size_t need, const at::Device& dev, bool fill) {
    if (given != Py_None) {
      const at::Tensor& t = tensor_of(given);
      ptr = t.data_ptr(); bytes = (size_t)t.numel() * t.element_size();
    } else if (need > 0) {
      own = fresh({(int64_t)need}, at::kByte, dev, fill);
      ptr = own.data_ptr(); bytes = need;
    }
  }
};

template <typename F>
mq_status unlocked(F&& f) {
  Unlocked u;
  return f();
}

template <typename F>
PyObject* guarded(Py_ssize_t nargs, Py_ssize_t want, F&& f) {
  if (nargs != want) { PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs); return nullptr; }
  try {
    return f();
  } catch (PyFail&) {
    return nullptr;
  } catch (...) {   // PyTorch's own errors (out of memory among them) become its Python exceptions
    torch::translate_exception_to_python(std::current_exception());
  }
  return nullptr;
}

// quantize(kind, desc, role, fmt, block, src, src_layout, out, seed, amax, stream, fill); kind 0 mq_quantize, 1 mq_quantize_sr, 2 mq_quantize_ts
PyObject* py_quantize(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 12, [&]() -> PyObject* {
    const long kind = to_long(a[0]);
    const mq_conv_desc d = desc_of(a[1]);
    const int role = (int)to_long(a[2]), fmt = (int)to_long(a[3]), block = (int)to_long(a[4]), layout = (int)to_long(a[6]);
    const at::Tensor& src = tensor_of(a[5]);
    const bool fill = PyObject_IsTrue(a[11]) == 1;
    require(src.is_cuda(), "src is a CUDA tensor");
    require(src.scalar_type() == at::kFloat || src.scalar_type() == at::kBFloat16, "src is float32 or bfloat16");
    require(src.is_contiguous(), "src is contiguous");
    const Launch launch(a[10], src.device());
    std::optional<Stored> given;
    std::optional<Created> made;
    if (a[7] != Py_None) given.emplace(a[7]);
    else {
      size_t cb = 0, sb = 0;
      check("mq_qtensor_sizes", mq_qtensor_sizes(&d, role, fmt, block, &cb, &sb));
      made.emplace(cb, sb, fmt, role, block, src.device(), fill);
    }
    mq_qtensor* q = given ? &given->q : &made->q;
    unsigned long long seed = 0;
    if (a[8] != Py_None) {
      PyObject* n = PyNumber_Long(a[8]);
      if (!n) throw PyFail{};
      seed = PyLong_AsUnsignedLongLongMask(n);
      Py_DECREF(n);
      if (PyErr_Occurred()) throw PyFail{};
    }
    const float* amax = a[9] != Py_None ? static_cast<const float*>(tensor_of(a[9]).data_ptr()) : nullptr;
    const bool sr = a[8] != Py_None;
    void* s = launch.stream;
    const void* p = src.data_ptr();
    const int dt = dtype_code(src.scalar_type());
    if (kind == 2) check("mq_quantize_ts", unlocked([&] { return mq_quantize_ts(&d, p, dt, layout, q, amax, sr ? &seed : nullptr, s); }));
    else if (kind == 1) check("mq_quantize_sr", unlocked([&] { return mq_quantize_sr(&d, p, dt, layout, q, seed, s); }));
    else check("mq_quantize", unlocked([&] { return mq_quantize(&d, p, dt, layout, q, s); }));
    if (given) Py_RETURN_NONE;
    return made->to_python(launch);
  });
}

// im2col(desc, xq, out_codes, out_scales, stream, fill)
PyObject* py_im2col(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 6, [&]() -> PyObject* {
    const mq_conv_desc d = desc_of(a[0]);
    Stored x(a[1]);
    const bool fill = PyObject_IsTrue(a[5]) == 1;
    const Launch launch(a[4], *x.device);
    size_t cb = 0, sb = 0;
    check("mq_im2col_sizes", mq_im2col_sizes(&d, x.q.fmt, x.q.block, &cb, &sb));
    at::Tensor codes = a[2] != Py_None ? tensor_of(a[2]) : fresh({(int64_t)cb}, at::kByte, *x.device, fill);
    at::Tensor scales = a[3] != Py_None ? tensor_of(a[3]) : fresh({(int64_t)sb}, at::kByte, *x.device, fill);
    check("mq_cbf_im2col", unlocked([&] { return mq_cbf_im2col(&d, &x.q, codes.data_ptr(), static_cast<uint8_t*>(scales.data_ptr()), launch.stream); }));
    if (a[2] == Py_None) launch.hand_out(codes);
    if (a[3] == Py_None) launch.hand_out(scales);
    return Py_BuildValue("(NN)", THPVariable_Wrap(codes), THPVariable_Wrap(scales));
  });
}

// conv(op, desc, qa, qb, out, layout, workspace, stream, dtype, fill): op as mq_op
PyObject* py_conv(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 10, [&]() -> PyObject* {
    const int op = (int)to_long(a[0]), layout = (int)to_long(a[5]);
    const mq_conv_desc d = desc_of(a[1]);
    Stored qa(a[2]), qb(a[3]);
    const bool fill = PyObject_IsTrue(a[9]) == 1;
    const Launch launch(a[7], *qa.device);
    at::Tensor out;
    if (a[4] != Py_None) out = tensor_of(a[4]);
    else {
      if (a[8] != Py_None && !THPDtype_Check(a[8])) { PyErr_SetString(PyExc_TypeError, "dtype is a torch.dtype"); throw PyFail{}; }
      const at::ScalarType t = a[8] != Py_None ? reinterpret_cast<THPDtype*>(a[8])->scalar_type : c10::get_default_dtype_as_scalartype();
      int64_t n, c, h, w;   // logical NCHW (weight gradient: OIHW) extents
      if (op == MQ_OP_BWD_WEIGHT) { n = d.C_out; c = d.C_in; h = d.Kh; w = d.Kw; }
      else if (op == MQ_OP_BWD_DATA) { n = d.N; c = d.C_in; h = d.H; w = d.W; }
      else { n = d.N; c = d.C_out; h = out_extent(d.H, d.pad_h, d.Kh, d.stride_h); w = out_extent(d.W, d.pad_w, d.Kw, d.stride_w); }
      if (layout == MQ_NCHW) out = fresh({n, c, h, w}, t, *qa.device, fill);
      else if (op == MQ_OP_BWD_WEIGHT) out = fresh({n, h, w, c}, t, *qa.device, fill);
      else out = fresh({h, w, n, c}, t, *qa.device, fill);
    }
    size_t need = 0;
    check("mq_workspace_size", mq_workspace_size(&d, op, qa.q.fmt, qb.q.fmt, qa.q.block, &need));
    Workspace ws(a[6], need, *qa.device, fill);
    const int dt = dtype_code(out.scalar_type());
    void* s = launch.stream;
    void* o = out.data_ptr();
    if (op == MQ_OP_FWD) check("mq_conv_fwd", unlocked([&] { return mq_conv_fwd(&d, &qa.q, &qb.q, o, dt, layout, ws.ptr, ws.bytes, s); }));
    else if (op == MQ_OP_BWD_DATA) check("mq_conv_bwd_data", unlocked([&] { return mq_conv_bwd_data(&d, &qa.q, &qb.q, o, dt, layout, ws.ptr, ws.bytes, s); }));
    else check("mq_conv_bwd_weight", unlocked([&] { return mq_conv_bwd_weight(&d, &qa.q, &qb.q, o, dt, layout, ws.ptr, ws.bytes, s); }));
    if (a[4] == Py_None) launch.hand_out(out);
    return THPVariable_Wrap(out);
  });
}

// conv_emit(op, desc, qa, qb, fmt, act, amax, out, workspace, stream, fill): the quantizing producer epilogue; amax: None = MX
// tiles of element format fmt, else the paper's own format with that supplied maximum
PyObject* py_conv_emit(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  return guarded(nargs, 11, [&]() -> PyObject* {
    const int op = (int)to_long(a[0]), fmt = (int)to_long(a[4]), act = (int)to_long(a[5]);
    const mq_conv_desc d = desc_of(a[1]);
    const bool ts = a[6] != Py_None, fill = PyObject_IsTrue(a[10]) == 1;
    const float* amax = nullptr;
    if (ts) {
      const at::Tensor& t = tensor_of(a[6]);
      require(t.is_cuda() && t.scalar_type() == at::kFloat && t.numel() >= 1, "amax_in is a float32 CUDA tensor of at least one element");
      amax = t.data_ptr<float>();
    }
    Stored qa(a[2]), qb(a[3]);
    const Launch launch(a[9], *qa.device);
    std::optional<Stored> given;
    std::optional<Created> made;
    if (a[7] != Py_None) given.emplace(a[7]);
    else {
      // the next tensor: N x C_out x Ho x Wo (forward) or N x C_in x H x W (input gradient)
      const bool fwd = op == MQ_OP_FWD;
      const int64_t P = fwd ? (int64_t)out_extent(d.H, d.pad_h, d.Kh, d.stride_h) * out_extent(d.W, d.pad_w, d.Kw, d.stride_w) : (int64_t)d.H * d.W;
      const int64_t cp = ((fwd ? d.C_out : d.C_in) + 31) / 32 * 32;
      const int64_t cb = P * d.N * cp * (fmt == MQ_E2M1 ? 4 : 8) / 8;
      const int64_t sb = ts ? P * ((d.N + 15) / 16) * (cp / 16) : P * ((d.N + 31) / 32) * (cp / 32);
      made.emplace((size_t)cb, (size_t)sb, fmt, fwd ? MQ_ROLE_X : MQ_ROLE_DY, ts ? MQ_BLOCK_TS16 : MQ_BLOCK_TILE32, *qa.device, fill);
    }
    mq_qtensor* q = given ? &given->q : &made->q;
    size_t need = 0;
    if (ts) check("mq_conv_ts_workspace_size", mq_conv_ts_workspace_size(&d, op, &need));
    else check("mq_conv_mx_workspace_size", mq_conv_mx_workspace_size(&d, op, qa.q.fmt, qb.q.fmt, &need));
    Workspace ws(a[8], need, *qa.device, fill);
    void* s = launch.stream;
    if (ts && op == MQ_OP_FWD) check("mq_conv_fwd_ts", unlocked([&] { return mq_conv_fwd_ts(&d, &qa.q, &qb.q, act, amax, q, ws.ptr, ws.bytes, s); }));
    else if (ts) check("mq_conv_bwd_data_ts", unlocked([&] { return mq_conv_bwd_data_ts(&d, &qa.q, &qb.q, amax, q, ws.ptr, ws.bytes, s); }));
    else if (op == MQ_OP_FWD) check("mq_conv_fwd_mx", unlocked([&] { return mq_conv_fwd_mx(&d, &qa.q, &qb.q, act, q, ws.ptr, ws.bytes, s); }));
    else check("mq_conv_bwd_data_mx", unlocked([&] { return mq_conv_bwd_data_mx(&d, &qa.q, &qb.q, q, ws.ptr, ws.bytes, s); }));
    if (given) Py_RETURN_NONE;
    return made->to_python(launch);
  });
}

PyObject* py_set_error(PyObject*, PyObject* cls) {
  Py_INCREF(cls);
  Py_XSETREF(g_error, cls);
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"quantize", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_quantize)), METH_FASTCALL, nullptr},
    {"im2col", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_im2col)), METH_FASTCALL, nullptr},
    {"conv", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_conv)), METH_FASTCALL, nullptr},
    {"conv_emit", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_conv_emit)), METH_FASTCALL, nullptr},
    {"set_error", py_set_error, METH_O, "set_error(cls): the exception class of failed calls, made as cls(call, status)"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mq_torch", "native marshalling of libmq's calls for torch tensors", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__mq_torch() {
  s_codes = PyUnicode_InternFromString("codes"); s_scales = PyUnicode_InternFromString("scales");
  s_fmt = PyUnicode_InternFromString("fmt"); s_role = PyUnicode_InternFromString("role"); s_block = PyUnicode_InternFromString("block");
  s_tscale = PyUnicode_InternFromString("tensor_scale"); s_stream = PyUnicode_InternFromString("cuda_stream");
  g_error = PyExc_RuntimeError;
  Py_INCREF(g_error);
  return PyModule_Create(&module);
}
