// Marshalling of the hot entry points in native code: checks of the tensors, allocation of the results and the call into
// the C ABI, for binding.py.  No arithmetic of the path lives here; the library's functions come in as addresses, so this
// module is tied to whichever libfp4attn.so binding.py has loaded.
//
// Why: a step of the smallest problems is four kernels of 2-8 us each, and the same marshalling in Python (ctypes, size
// queries, torch.empty, stream look-up) took about 15 us per call: B=1, H=2, N=256 ran at 66 us per step, all of it host
// time.
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>

#include "../../include/fp4attn.h"

namespace {

struct Api {
  decltype(&fp4attn_status_string) status_string;
  decltype(&fp4attn_packed_bytes) packed_bytes;
  decltype(&fp4attn_scale_bytes) scale_bytes;
  decltype(&fp4attn_quantize_workspace_bytes) quantize_workspace_bytes;
  decltype(&fp4attn_quantize) quantize;
  decltype(&fp4attn_quantize_mxfp4_rule) quantize_mxfp4_rule;
  decltype(&fp4attn_quantize_nvfp4_per_head_workspace_bytes) per_head_workspace_bytes;
  decltype(&fp4attn_quantize_nvfp4_per_head) per_head;
  decltype(&fp4attn_quantize_v_e4m3_workspace_bytes) e4m3_workspace_bytes;
  decltype(&fp4attn_quantize_v_e4m3) e4m3;
  decltype(&fp4attn_fwd) fwd;
};
Api g_api;
PyObject* g_error = nullptr;                            // Fp4AttnError
enum { A_PACKED, A_SCALES, A_G, A_FMT, A_ROLE, A_SHAPE, A_PER_HEAD, A_COUNT };
PyObject* g_names[A_COUNT];
constexpr int kFmtE4m3 = 2;                             // QuantizedOperand.fmt of an E4M3 V

PyObject* fail(int rc, const char* what) {
  PyErr_Format(g_error, "%s: %s (status %d)", what, g_api.status_string(rc), rc);
  return nullptr;
}
PyObject* assertion(const char* what) {
  PyErr_SetString(PyExc_AssertionError, what);
  return nullptr;
}
fp4attn_stream_t stream() { return reinterpret_cast<fp4attn_stream_t>(c10::cuda::getCurrentCUDAStream().stream()); }
at::Tensor device_empty(at::IntArrayRef size, at::ScalarType type, c10::Device device) {
  return at::Tensor(at::detail::empty_cuda(size, type, device, std::nullopt));
}
// The results of one call.  An allocation costs about as much host time as the rest of a call's marshalling, so up to
// kShareBytes they are pieces of one (a step of B=1, H=2, N=256: 19.9 -> 17.0 us); beyond that (where the kernels take longer anyway) each has memory of its own, so that
// keeping one alone does not keep them all.
struct Results {
  static constexpr size_t kShareBytes = 1 << 20, kMost = 4;
  struct Piece {
    int64_t sizes[4];
    int dims;
    at::ScalarType type;
    at::Tensor tensor;
  } piece[kMost];
  int n = 0;
  at::Tensor& add(std::initializer_list<int64_t> sizes, at::ScalarType type) {
    Piece& p = piece[n++];
    p.dims = (int)sizes.size();
    p.type = type;
    std::copy(sizes.begin(), sizes.end(), p.sizes);
    return p.tensor;
  }
  void allocate(c10::Device device) {
    int64_t at[kMost + 1] = {0}, count[kMost];
    for (int i = 0; i < n; ++i) {
      count[i] = 1;
      for (int k = 0; k < piece[i].dims; ++k) count[i] *= piece[i].sizes[k];
      at[i + 1] = at[i] + ((count[i] * (int64_t)c10::elementSize(piece[i].type) + 511) & ~511ll);   // as the allocator aligns
    }
    if (at[n] > (int64_t)kShareBytes) {
      for (int i = 0; i < n; ++i) piece[i].tensor = device_empty(at::IntArrayRef(piece[i].sizes, piece[i].dims), piece[i].type, device);
      return;
    }
    // straight from the caching allocator: a tensor of its own for the block would only be taken apart again
    const c10::cuda::OptionalCUDAGuard guard(device);
    c10::Allocator* const pool = c10::cuda::CUDACachingAllocator::get();
    const c10::Storage block(c10::Storage::use_byte_size_t(), (size_t)at[n], pool->allocate((size_t)at[n]), pool, /*resizable=*/true);
    for (int i = 0; i < n; ++i) {
      piece[i].tensor = at::detail::make_tensor<c10::TensorImpl>(c10::Storage(block), c10::DispatchKeySet(c10::DispatchKey::CUDA), c10::scalarTypeToTypeMeta(piece[i].type));
      c10::TensorImpl* impl = piece[i].tensor.unsafeGetTensorImpl();
      impl->set_sizes_contiguous(at::IntArrayRef(piece[i].sizes, piece[i].dims));
      impl->set_storage_offset(at[i] / (int64_t)c10::elementSize(piece[i].type));
    }
  }
};
// What a Python caller's `None if o is None else o.data_ptr()` gives: a null pointer for None, and an error for what has no
// memory (an argument that is not a tensor must not pass for one that was left out).
bool data_of(PyObject* o, void** ptr) {
  *ptr = nullptr;
  if (o == Py_None) return true;
  if (THPVariable_Check(o)) {
    *ptr = THPVariable_Unpack(o).data_ptr();
    return true;
  }
  PyObject* p = PyObject_CallMethod(o, "data_ptr", nullptr);
  if (p) *ptr = PyLong_AsVoidPtr(p);
  Py_XDECREF(p);
  return !PyErr_Occurred();
}
bool numel_of(PyObject* o, size_t* n) {
  if (THPVariable_Check(o)) {
    *n = (size_t)THPVariable_Unpack(o).numel();
    return true;
  }
  PyObject* p = PyObject_CallMethod(o, "numel", nullptr);
  if (p) *n = PyLong_AsSize_t(p);
  Py_XDECREF(p);
  return !PyErr_Occurred();
}

struct Input {
  const at::Tensor* t = nullptr;
  int B = 0, H = 0, N = 0, d = 0;
  bool take(PyObject* o) {
    if (!THPVariable_Check(o)) return false;
    t = &THPVariable_Unpack(o);
    if (!t->is_cuda() || t->scalar_type() != at::kBFloat16 || t->dim() != 4 || !t->is_contiguous()) return false;
    const auto s = t->sizes();
    for (int i = 0; i < 4; ++i)
      if (s[i] > INT32_MAX) return false;
    B = (int)s[0]; H = (int)s[1]; N = (int)s[2]; d = (int)s[3];
    return true;
  }
  PyObject* shape() const { return Py_BuildValue("(iiii)", B, H, N, d); }
};
const char* kInputRule = "x must be a contiguous CUDA bfloat16 tensor [B, H, N, d]";

// (packed, scales, G or None, shape)
PyObject* result(const at::Tensor& packed, const at::Tensor* scales, const at::Tensor* G, const Input& in) {
  PyObject* g = G ? THPVariable_Wrap(*G) : Py_NewRef(Py_None);
  PyObject* s = scales ? THPVariable_Wrap(*scales) : Py_NewRef(Py_None);
  return Py_BuildValue("(NNNN)", THPVariable_Wrap(packed), s, g, in.shape());
}

// whole numbers; `convert`: whatever int() takes
bool ints(PyObject* const* args, Py_ssize_t n, int* out, bool convert = false) {
  for (Py_ssize_t i = 0; i < n; ++i) {
    if (!convert && !PyLong_Check(args[i])) {
      PyErr_Format(PyExc_TypeError, "int expected instead of %s instance", Py_TYPE(args[i])->tp_name);
      return false;
    }
    PyObject* o = PyLong_Check(args[i]) ? Py_NewRef(args[i]) : PyNumber_Long(args[i]);
    const long v = o ? PyLong_AsLong(o) : -1;
    Py_XDECREF(o);
    if (v == -1 && PyErr_Occurred()) return false;
    out[i] = (int)v;
  }
  return true;
}
bool number(PyObject* o, float* out) {                  // whatever float() takes
  PyObject* f = PyNumber_Float(o);
  if (f) *out = (float)PyFloat_AsDouble(f);
  Py_XDECREF(f);
  return f != nullptr;
}
// A call into the library, which may block on a full launch queue, without the interpreter lock (nothing in it may touch a
// Python object).
template <class F>
int unlocked(F call) {
  struct Unlock {
    PyThreadState* ts = PyEval_SaveThread();
    ~Unlock() { PyEval_RestoreThread(ts); }
  } guard;
  return call();
}

#define FP4_TRY try {
#define FP4_CATCH                                                                              \
  }                                                                                            \
  catch (const c10::OutOfMemoryError& e) {                                                     \
    PyErr_SetString(out_of_memory_class(), e.what_without_backtrace());                   \
    return nullptr;                                                                            \
  }                                                                                            \
  catch (const std::exception& e) {                                                            \
    PyErr_SetString(PyExc_RuntimeError, e.what());                                             \
    return nullptr;                                                                            \
  }
PyObject* out_of_memory_class() {                       // torch.OutOfMemoryError
  static PyObject* cls = [] {
    PyObject* torch = PyImport_ImportModule("torch");
    PyObject* c = torch ? PyObject_GetAttrString(torch, "OutOfMemoryError") : nullptr;
    Py_XDECREF(torch);
    return c ? c : PyExc_RuntimeError;
  }();
  return cls;
}

// quantize(x, fmt, role, workspace)
PyObject* py_quantize(PyObject*, PyObject* const* args, Py_ssize_t n) {
  FP4_TRY
  int a[2];
  Input in;
  if (n != 4 || !in.take(args[0])) return assertion(kInputRule);
  if (!ints(args + 1, 2, a)) return nullptr;
  const int fmt = a[0], role = a[1];
  const size_t nb = g_api.packed_bytes(in.B, in.H, in.N, in.d), ns = g_api.scale_bytes(fmt, role, in.B, in.H, in.N, in.d);
  void* const any = reinterpret_cast<void*>(1);
  if (!nb || !ns) {                                     // unsupported: the library says why, before it looks at a pointer's use
    const int rc = unlocked([&] { return g_api.quantize(in.t->data_ptr(), fmt, role, in.B, in.H, in.N, in.d, any, any, nullptr, nullptr, 0, stream()); });
    if (rc) return fail(rc, "fp4attn_quantize");
    PyErr_SetString(g_error, "fp4attn_quantize: unsupported arguments");
    return nullptr;
  }
  const size_t nw = args[3] == Py_None ? g_api.quantize_workspace_bytes(fmt, role, in.B, in.H, in.N, in.d) : 0;
  Results r;
  at::Tensor none, &packed = r.add({(int64_t)nb}, at::kByte), &scales = r.add({(int64_t)ns}, at::kByte);
  at::Tensor& G = fmt == FP4ATTN_FMT_NVFP4 ? r.add({1}, at::kFloat) : none;
  at::Tensor& ws = nw ? r.add({(int64_t)nw}, at::kByte) : none;
  void* wptr = nullptr;
  size_t wbytes = nw;
  if (args[3] != Py_None && (!data_of(args[3], &wptr) || !numel_of(args[3], &wbytes))) return nullptr;
  r.allocate(in.t->device());
  if (nw) wptr = ws.data_ptr();
  const int rc = unlocked([&] { return g_api.quantize(in.t->data_ptr(), fmt, role, in.B, in.H, in.N, in.d, packed.data_ptr(), scales.data_ptr(),
                                G.defined() ? G.data_ptr<float>() : nullptr, wptr, wbytes, stream()); });
  if (rc) return fail(rc, "fp4attn_quantize");
  return result(packed, &scales, G.defined() ? &G : nullptr, in);
  FP4_CATCH
}

// quantize_mxfp4_rule(x, role, scale_rule)
PyObject* py_rule(PyObject*, PyObject* const* args, Py_ssize_t n) {
  FP4_TRY
  int a[2];
  Input in;
  if (n != 3 || !in.take(args[0])) return assertion(kInputRule);
  if (!ints(args + 1, 2, a)) return nullptr;
  const size_t nb = g_api.packed_bytes(in.B, in.H, in.N, in.d), ns = g_api.scale_bytes(FP4ATTN_FMT_MXFP4, a[0], in.B, in.H, in.N, in.d);
  void* const any = reinterpret_cast<void*>(1);
  if (!nb || !ns) {
    const int rc = unlocked([&] { return g_api.quantize_mxfp4_rule(in.t->data_ptr(), a[0], a[1], in.B, in.H, in.N, in.d, any, any, stream()); });
    if (rc) return fail(rc, "fp4attn_quantize_mxfp4_rule");
    PyErr_SetString(g_error, "fp4attn_quantize_mxfp4_rule: unsupported arguments");
    return nullptr;
  }
  Results r;
  at::Tensor &packed = r.add({(int64_t)nb}, at::kByte), &scales = r.add({(int64_t)ns}, at::kByte);
  r.allocate(in.t->device());
  const int rc = unlocked([&] { return g_api.quantize_mxfp4_rule(in.t->data_ptr(), a[0], a[1], in.B, in.H, in.N, in.d, packed.data_ptr(), scales.data_ptr(), stream()); });
  if (rc) return fail(rc, "fp4attn_quantize_mxfp4_rule");
  return result(packed, &scales, nullptr, in);
  FP4_CATCH
}

// quantize_nvfp4_per_head(x, role)
PyObject* py_per_head(PyObject*, PyObject* const* args, Py_ssize_t n) {
  FP4_TRY
  int role;
  Input in;
  if (n != 2 || !in.take(args[0])) return assertion(kInputRule);
  if (!ints(args + 1, 1, &role)) return nullptr;
  const size_t nb = g_api.packed_bytes(in.B, in.H, in.N, in.d), ns = g_api.scale_bytes(FP4ATTN_FMT_NVFP4, role, in.B, in.H, in.N, in.d);
  const size_t nw = g_api.per_head_workspace_bytes(in.B, in.H, in.N, in.d);
  void* const any = reinterpret_cast<void*>(1);
  if (!nb || !ns || !nw) {
    const int rc = unlocked([&] { return g_api.per_head(in.t->data_ptr(), role, in.B, in.H, in.N, in.d, any, any, reinterpret_cast<float*>(any), nullptr, 0, stream()); });
    if (rc) return fail(rc, "fp4attn_quantize_nvfp4_per_head");
    PyErr_SetString(g_error, "fp4attn_quantize_nvfp4_per_head: unsupported arguments");
    return nullptr;
  }
  Results r;
  at::Tensor &packed = r.add({(int64_t)nb}, at::kByte), &scales = r.add({(int64_t)ns}, at::kByte);
  at::Tensor &G = r.add({(int64_t)in.B * in.H}, at::kFloat), &ws = r.add({(int64_t)nw}, at::kByte);
  r.allocate(in.t->device());
  const int rc = unlocked([&] { return g_api.per_head(in.t->data_ptr(), role, in.B, in.H, in.N, in.d, packed.data_ptr(), scales.data_ptr(), G.data_ptr<float>(),
                                ws.data_ptr(), nw, stream()); });
  if (rc) return fail(rc, "fp4attn_quantize_nvfp4_per_head");
  return result(packed, &scales, &G, in);
  FP4_CATCH
}

// quantize_v_e4m3(x); scales comes back empty
PyObject* py_e4m3(PyObject*, PyObject* const* args, Py_ssize_t n) {
  FP4_TRY
  Input in;
  if (n != 1 || !in.take(args[0])) return assertion(kInputRule);
  const size_t nw = g_api.e4m3_workspace_bytes(in.B, in.H, in.N, in.d);
  void* const any = reinterpret_cast<void*>(1);
  if (!nw) {
    const int rc = unlocked([&] { return g_api.e4m3(in.t->data_ptr(), in.B, in.H, in.N, in.d, any, reinterpret_cast<float*>(any), nullptr, 0, stream()); });
    if (rc) return fail(rc, "fp4attn_quantize_v_e4m3");
    PyErr_SetString(g_error, "fp4attn_quantize_v_e4m3: unsupported arguments");
    return nullptr;
  }
  Results r;
  at::Tensor &out = r.add({in.t->numel()}, at::kByte), &scales = r.add({0}, at::kByte);
  at::Tensor &G = r.add({(int64_t)in.B * in.H}, at::kFloat), &ws = r.add({(int64_t)nw}, at::kByte);
  r.allocate(in.t->device());
  const int rc = unlocked([&] { return g_api.e4m3(in.t->data_ptr(), in.B, in.H, in.N, in.d, out.data_ptr(), G.data_ptr<float>(), ws.data_ptr(), nw, stream()); });
  if (rc) return fail(rc, "fp4attn_quantize_v_e4m3");
  return result(out, &scales, &G, in);
  FP4_CATCH
}

// What fp4attn_fwd reads of a QuantizedOperand.  The tensors stay alive through the operand, which the caller holds.
struct Operand {
  void *packed = nullptr, *scales = nullptr, *G = nullptr;
  c10::Device device{c10::kCPU};
  int fmt = 0, shape[4] = {0, 0, 0, 0};
  bool per_head = false;
  bool take(PyObject* o) {
    PyObject* v[A_COUNT] = {};
    bool ok = true;
    for (int i = 0; i < A_COUNT && ok; ++i) {
      if (i == A_ROLE) continue;
      v[i] = PyObject_GetAttr(o, g_names[i]);
      ok = v[i] != nullptr;
    }
    if (ok && !PyTuple_Check(v[A_SHAPE])) {
      PyObject* const t = PySequence_Tuple(v[A_SHAPE]);
      Py_SETREF(v[A_SHAPE], t);
      ok = t != nullptr;
    }
    if (ok && (!THPVariable_Check(v[A_PACKED]) || PyTuple_GET_SIZE(v[A_SHAPE]) != 4)) {
      PyErr_SetString(PyExc_TypeError, "fp4attn_fwd takes QuantizedOperand arguments");
      ok = false;
    }
    if (ok) {
      const at::Tensor& t = THPVariable_Unpack(v[A_PACKED]);
      packed = t.data_ptr();
      device = t.device();
      if (!data_of(v[A_SCALES], &scales) || !data_of(v[A_G], &G)) ok = false;
      fmt = ok ? (int)PyLong_AsLong(v[A_FMT]) : 0;
      per_head = ok && PyObject_IsTrue(v[A_PER_HEAD]) == 1;
      for (int i = 0; ok && i < 4; ++i) shape[i] = (int)PyLong_AsLong(PyTuple_GET_ITEM(v[A_SHAPE], i));
      ok = ok && !PyErr_Occurred();
    }
    for (int i = 0; i < A_COUNT; ++i) Py_XDECREF(v[i]);
    return ok;
  }
};

// fwd(q, k, v, softmax_scale, out, lse, status, p_map, affine_a, affine_b, p_scale_rule, causal, exact_pairs, schedule, seq_len,
//     fixed_reference) -> (out, lse)
PyObject* py_fwd(PyObject*, PyObject* const* args, Py_ssize_t n) {
  FP4_TRY
  if (n != 16) return assertion("fwd takes 16 arguments");
  Operand q, k, v;
  if (!q.take(args[0]) || !k.take(args[1]) || !v.take(args[2])) return nullptr;
  const int B = q.shape[0], H = q.shape[1], N = q.shape[2], d = q.shape[3], Hkv = k.shape[1];
  bool same = k.shape[0] == B && k.shape[2] == N && k.shape[3] == d && Hkv > 0 && H % Hkv == 0;
  for (int i = 0; i < 4; ++i) same = same && k.shape[i] == v.shape[i];
  if (!same || q.fmt != k.fmt || (v.fmt != FP4ATTN_FMT_MXFP4 && v.fmt != kFmtE4m3))
    return assertion("K and V must have one shape, Q the same but for the heads, whose number K's divides; Q and K one format, V MXFP4 or E4M3");
  if (q.per_head != k.per_head) return assertion("Q and K must both carry per-head factors, or neither");
  const bool fp8 = v.fmt == kFmtE4m3;
  PyObject* const seq = args[14];
  if (seq != Py_None) {
    if (!THPVariable_Check(seq)) return assertion("seq_len must be a contiguous CUDA int32 tensor of B counts");
    const at::Tensor& t = THPVariable_Unpack(seq);
    if (!t.is_cuda() || t.scalar_type() != at::kInt || t.numel() != B || !t.is_contiguous())
      return assertion("seq_len must be a contiguous CUDA int32 tensor of B counts");
  }
  fp4attn_operands ops = {};
  ops.q = q.packed; ops.k = k.packed; ops.v = v.packed;
  ops.q_sf = q.scales; ops.k_sf = k.scales; ops.v_sf = fp8 ? nullptr : v.scales;
  ops.q_G = (const float*)q.G; ops.k_G = (const float*)k.G;
  ops.qk_fmt = q.fmt;
  ops.kv_heads = Hkv;
  ops.g_per_head = q.per_head ? 1 : 0;
  ops.pv_fmt = fp8 ? FP4ATTN_PV_E4M3 : FP4ATTN_PV_MXFP4;
  ops.v_G = fp8 ? (const float*)v.G : nullptr;
  void *seq_len, *out_ptr, *lse_ptr, *status;
  if (!number(args[3], &ops.softmax_scale) || !number(args[8], &ops.affine_a) || !number(args[9], &ops.affine_b) ||
      !ints(args + 7, 1, &ops.p_map, true) || !ints(args + 10, 1, &ops.p_scale_rule, true) ||
      !ints(args + 12, 1, &ops.exact_pairs, true) || !ints(args + 13, 1, &ops.schedule, true) || !data_of(seq, &seq_len) ||
      !data_of(args[4], &out_ptr) || !data_of(args[5], &lse_ptr) || !data_of(args[6], &status))
    return nullptr;
  if ((ops.causal = PyObject_IsTrue(args[11])) < 0) return nullptr;
  ops.seq_len = (const int*)seq_len;
  if (args[15] != Py_None) {
    ops.row_reference = FP4ATTN_REFERENCE_FIXED;
    if (!ints(args + 15, 1, &ops.fixed_reference, true)) return nullptr;
  }
  THPObjectPtr out(Py_NewRef(args[4])), lse(Py_NewRef(args[5]));        // given back on every way out, an exception's too
  if (out.get() == Py_None || lse.get() == Py_None) {
    Results r;
    at::Tensor none, &o = out.get() == Py_None ? r.add({B, H, N, d}, at::kBFloat16) : none, &l = lse.get() == Py_None ? r.add({B, H, N}, at::kFloat) : none;
    r.allocate(q.device);
    if (o.defined()) { out_ptr = o.data_ptr(); out = THPVariable_Wrap(o); }
    if (l.defined()) { lse_ptr = l.data_ptr(); lse = THPVariable_Wrap(l); }
    if (!out || !lse) return nullptr;
  }
  const int rc = unlocked([&] { return g_api.fwd(&ops, B, H, N, d, out_ptr, (float*)lse_ptr, (int*)status, stream()); });
  if (rc) return fail(rc, "fp4attn_fwd");
  return Py_BuildValue("(NN)", out.release(), lse.release());
  FP4_CATCH
}

// init(error class, status_string, packed_bytes, ..., fwd): addresses of the library's functions, in Api's order
PyObject* py_init(PyObject*, PyObject* const* args, Py_ssize_t n) {
  constexpr Py_ssize_t kFunctions = sizeof(Api) / sizeof(void*);
  if (n != 1 + kFunctions) return assertion("init takes the error class and one address per function");
  void* p[kFunctions];
  for (Py_ssize_t i = 0; i < kFunctions; ++i) {
    p[i] = PyLong_AsVoidPtr(args[1 + i]);
    if (!p[i]) return PyErr_Occurred() ? nullptr : assertion("a function's address is 0");
  }
  memcpy(static_cast<void*>(&g_api), p, sizeof p);
  Py_XSETREF(g_error, Py_NewRef(args[0]));
  Py_RETURN_NONE;
}

#define FP4_METHOD(NAME, FN) {NAME, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(FN)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FP4_METHOD("init", py_init), FP4_METHOD("quantize", py_quantize), FP4_METHOD("quantize_mxfp4_rule", py_rule),
                         FP4_METHOD("quantize_nvfp4_per_head", py_per_head), FP4_METHOD("quantize_v_e4m3", py_e4m3),
                         FP4_METHOD("fwd", py_fwd), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fp4attn_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__fp4attn_native() {
  const char* names[A_COUNT] = {"packed", "scales", "G", "fmt", "role", "shape", "per_head"};
  for (int i = 0; i < A_COUNT; ++i)
    if (!(g_names[i] = PyUnicode_InternFromString(names[i]))) return nullptr;
  return PyModule_Create(&module);
}
