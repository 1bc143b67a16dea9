// Python side of the C ABI: reads pointers, strides and the current stream straight from the tensors and calls the entry
// point whose address it is given (the library, or the test build of it).
//
// A decoding step makes one call per layer and short prefixes take ~10 us of device time each, so what a call costs on
// the host decides how long the step takes.  Measured for one attention call of the 8B layer shape, enqueue only: 12.2 us
// with the arguments marshalled in Python (8.4 of them Python and ctypes), 5.4 us with this module (launches and tensor maps included).
//
// Every function holds no state; arguments are checked on each call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <initializer_list>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/specext.h"

namespace {

// Thrown with the Python error already set.
struct PyFailure {};

[[noreturn]] void fail(const char* what) {
  PyErr_SetString(PyExc_ValueError, what);
  throw PyFailure();
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor");
    throw PyFailure();
  }
  return THPVariable_Unpack(o);
}
const at::Tensor& cuda_tensor(PyObject* o) {
  const at::Tensor& t = tensor(o);
  if (!t.is_cuda()) fail("specext operates on CUDA tensors only (there is no CPU path)");
  return t;
}
void* ptr(PyObject* o) { return cuda_tensor(o).data_ptr(); }
void* ptr_or_null(PyObject* o) { return o == Py_None ? nullptr : ptr(o); }

template <typename T>
T* typed(PyObject* o, at::ScalarType type, const char* what) {
  const at::Tensor& t = cuda_tensor(o);
  if (t.scalar_type() != type) fail(what);
  return static_cast<T*>(t.data_ptr());
}
int32_t* i32(PyObject* o, const char* what) { return typed<int32_t>(o, at::kInt, what); }
float* f32(PyObject* o, const char* what) { return typed<float>(o, at::kFloat, what); }

void same_strides(PyObject* a, PyObject* b, const char* what) {
  if (tensor(a).strides() != tensor(b).strides()) fail(what);
}
const at::Tensor& bf16_3d(PyObject* o, const char* what) {
  const at::Tensor& t = tensor(o);
  if (t.scalar_type() != at::kBFloat16 || t.dim() != 3 || t.stride(2) != 1) fail(what);
  return t;
}
const at::Tensor& draft_kv(PyObject* o) {
  const at::Tensor& t = cuda_tensor(o);
  if (t.scalar_type() != at::kBFloat16 || t.dim() != 4 || t.stride(3) != 1)
    fail("draft K/V must be bf16 [layers][tokens][heads][dim]");
  return t;
}

long long integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) throw PyFailure();
  return v;
}
int32_t int32(PyObject* o) {
  const long long v = integer(o);
  if (v < INT32_MIN || v > INT32_MAX) {
    PyErr_SetString(PyExc_OverflowError, "value does not fit an int32");
    throw PyFailure();
  }
  return static_cast<int32_t>(v);
}
float real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyFailure();
  return static_cast<float>(v);
}
// Whether `t` holds the product of the factors (none of them negative), which may not fit 64 bits.
bool holds(const at::Tensor& t, std::initializer_list<int64_t> factors) {
  int64_t need = 1;
  for (const int64_t f : factors)
    if (f == 0) return true;
  for (const int64_t f : factors)
    if (__builtin_mul_overflow(need, f, &need)) return false;
  return t.numel() >= need;
}
template <typename F>
F entry(PyObject* address) {
  return reinterpret_cast<F>(static_cast<uintptr_t>(integer(address)));
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The descriptor is a ctypes structure; its memory is reached through the buffer protocol.
struct Desc {
  Py_buffer b;
  explicit Desc(PyObject* o, bool writable = false) {
    if (PyObject_GetBuffer(o, &b, writable ? PyBUF_WRITABLE : PyBUF_SIMPLE) != 0) throw PyFailure();
    if (b.len != (Py_ssize_t)sizeof(specext_attn_desc)) {
      PyBuffer_Release(&b);
      PyErr_SetString(PyExc_TypeError, "expected an AttnDesc");
      throw PyFailure();
    }
  }
  ~Desc() { PyBuffer_Release(&b); }
  specext_attn_desc* get() const { return static_cast<specext_attn_desc*>(b.buf); }
};

template <typename Body>
PyObject* guarded(Py_ssize_t nargs, Py_ssize_t want, Body&& body) {
  if (nargs != want) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs);
    return nullptr;
  }
  try {
    return body();
  } catch (const PyFailure&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}
// Runs the entry point without the interpreter lock.  `call` holds plain values only: what a tensor's accessors throw (a
// wrapped tensor has no data pointer) has to be thrown before, while the lock is held.
template <typename Call>
PyObject* released(Call&& call) {
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

constexpr const char* kStrides = "V tensors must have the strides of the matching K tensors";
constexpr const char* kAttnTypes = "parent/device_status must be int32 and lse fp32";

// (desc, Q, K_prefix, K_tree, O, prefix_len, chunk_size, softmax_scale, want_chunk_score): fills desc from the tensors'
// shapes and strides (V tensors share K's).
PyObject* fill_desc(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 9, [&]() -> PyObject* {
    const at::Tensor& Q = bf16_3d(a[1], "Q must be a bf16 [.][heads][head_dim] tensor with contiguous head_dim");
    const at::Tensor& K = bf16_3d(a[2], "K_prefix must be a bf16 [.][heads][head_dim] tensor with contiguous head_dim");
    const at::Tensor& Kt = bf16_3d(a[3], "K_tree must be a bf16 [.][heads][head_dim] tensor with contiguous head_dim");
    const at::Tensor& O = bf16_3d(a[4], "O must be a bf16 [.][heads][head_dim] tensor with contiguous head_dim");
    Desc d(a[0], true);
    specext_attn_desc& x = *d.get();
    x.n_tree = (int32_t)Q.size(0);
    x.n_q_heads = (int32_t)Q.size(1);
    x.head_dim = (int32_t)Q.size(2);
    x.n_kv_heads = (int32_t)Kt.size(1);
    x.prefix_len = int32(a[5]);
    x.chunk_size = int32(a[6]);
    x.softmax_scale = real(a[7]);
    const int want = PyObject_IsTrue(a[8]);
    if (want < 0) throw PyFailure();
    x.want_chunk_score = want;
    x.q_stride_t = Q.stride(0);
    x.q_stride_h = Q.stride(1);
    x.kv_stride_l = K.stride(0);
    x.kv_stride_h = K.stride(1);
    x.tkv_stride_t = Kt.stride(0);
    x.tkv_stride_h = Kt.stride(1);
    x.o_stride_t = O.stride(0);
    x.o_stride_h = O.stride(1);
    Py_RETURN_NONE;
  });
}

// (entry, desc, Q, K_prefix, V_prefix, K_tree, V_tree, parent, O, lse, chunk_score, workspace, device_status)
PyObject* verify_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 13, [&]() -> PyObject* {
    same_strides(a[4], a[3], kStrides);
    same_strides(a[6], a[5], kStrides);
    const Desc d(a[1]);
    const int32_t* parent = i32(a[7], kAttnTypes);
    float* lse = f32(a[9], kAttnTypes);
    float* score = a[10] == Py_None ? nullptr : f32(a[10], "chunk_score must be fp32");
    int32_t* status = i32(a[12], kAttnTypes);
    void* ws = ptr(a[11]);
    const size_t ws_bytes = tensor(a[11]).nbytes();
    const auto fn = entry<decltype(&specext_verify_attn)>(a[0]);
    void *Q = ptr(a[2]), *Kp = ptr(a[3]), *Vp = ptr(a[4]), *Kt = ptr(a[5]), *Vt = ptr(a[6]), *O = ptr(a[8]);
    void* st = stream();
    return released([&] { return fn(d.get(), Q, Kp, Vp, Kt, Vt, parent, O, lse, score, ws, ws_bytes, status, st); });
  });
}

// (entry, desc, Q, K_cache, V_cache, n_tokens, K_tree, V_tree, parent, O, lse, workspace, device_status)
PyObject* draft_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 13, [&]() -> PyObject* {
    constexpr const char* types = "parent/device_status/n_tokens must be int32 and lse fp32";
    same_strides(a[4], a[3], kStrides);
    same_strides(a[7], a[6], kStrides);
    const Desc d(a[1]);
    const int32_t* n_tokens = i32(a[5], types);
    const int32_t* parent = i32(a[8], types);
    float* lse = f32(a[10], types);
    int32_t* status = i32(a[12], types);
    void* ws = ptr(a[11]);
    const size_t ws_bytes = tensor(a[11]).nbytes();
    const auto fn = entry<decltype(&specext_draft_attn)>(a[0]);
    void *Q = ptr(a[2]), *K = ptr(a[3]), *V = ptr(a[4]), *Kt = ptr(a[6]), *Vt = ptr(a[7]), *O = ptr(a[9]);
    void* st = stream();
    return released([&] { return fn(d.get(), Q, K, V, n_tokens, Kt, Vt, parent, O, lse, ws, ws_bytes, status, st); });
  });
}

// (entry, Q, K, V, O, lse, device_status, softmax_scale)
PyObject* prefill_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 8, [&]() -> PyObject* {
    const at::Tensor& Q = bf16_3d(a[1], "Q must be a bf16 [.][heads][head_dim] tensor with contiguous head_dim");
    const at::Tensor& K = bf16_3d(a[2], "K must be a bf16 [.][heads][head_dim] tensor with contiguous head_dim");
    const at::Tensor& V = bf16_3d(a[3], "V must be a bf16 [.][heads][head_dim] tensor with contiguous head_dim");
    const at::Tensor& O = bf16_3d(a[4], "O must be a bf16 [.][heads][head_dim] tensor with contiguous head_dim");
    constexpr const char* types = "K and V must share strides; lse must be fp32 and device_status int32";
    if (K.strides() != V.strides()) fail(types);
    float* lse = f32(a[5], types);
    int32_t* status = i32(a[6], types);
    const at::Tensor& lse_t = tensor(a[5]);
    const int64_t L = Q.size(0), Hq = Q.size(1);
    if (K.size(0) < L || O.sizes() != Q.sizes() || lse_t.numel() < Hq * L || !lse_t.is_contiguous())
      fail("shapes: K, V [>=L][Hkv][D], O like Q, lse contiguous [Hq][L]");
    specext_attn_desc d = {};
    d.n_q_heads = (int32_t)Hq;
    d.n_kv_heads = (int32_t)K.size(1);
    d.head_dim = (int32_t)Q.size(2);
    d.prefix_len = (int32_t)L;
    d.n_tree = 1;
    d.chunk_size = 32;
    d.softmax_scale = real(a[7]);
    d.q_stride_t = Q.stride(0);
    d.q_stride_h = Q.stride(1);
    d.kv_stride_l = d.tkv_stride_t = K.stride(0);
    d.kv_stride_h = d.tkv_stride_h = K.stride(1);
    d.o_stride_t = O.stride(0);
    d.o_stride_h = O.stride(1);
    const auto fn = entry<decltype(&specext_prefill_attn)>(a[0]);
    void *q = ptr(a[1]), *k = ptr(a[2]), *v = ptr(a[3]), *o = ptr(a[4]);
    void* st = stream();
    return released([&] { return fn(&d, q, k, v, o, lse, status, st); });
  });
}

// (entry, chunk_score, n_tree, n_chunks, row, prefix_len, chunk_size, k, n_sink, n_recent, draft_K, draft_V, idx,
//  n_selected, K_out, V_out, n_tokens_out, device_status); chunk_score holds at least n_tree x n_chunks contiguous values
PyObject* select_gather(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded(n, 18, [&]() -> PyObject* {
    const float* score = f32(a[1], "chunk_score must be a contiguous fp32 [n_tree][n_chunks] tensor");
    const int32_t n_tree = int32(a[2]), n_chunks = int32(a[3]);
    const at::Tensor& cs = tensor(a[1]);
    if (!cs.is_contiguous() || cs.numel() < (int64_t)n_tree * n_chunks)
      fail("chunk_score must be a contiguous fp32 [n_tree][n_chunks] tensor");
    const int32_t row = int32(a[4]), L = int32(a[5]), C = int32(a[6]), k = int32(a[7]);
    const int32_t n_sink = int32(a[8]), n_recent = int32(a[9]);
    const at::Tensor &dK = draft_kv(a[10]), &dV = draft_kv(a[11]);
    if (dK.strides() != dV.strides()) fail("draft K and V must share strides");
    int32_t* idx = i32(a[12], "idx and n_selected must be int32");
    int32_t* n_selected = i32(a[13], "idx and n_selected must be int32");
    if (tensor(a[12]).numel() < (k < n_chunks ? k : n_chunks)) fail("idx is too small");
    const at::Tensor &Ko = cuda_tensor(a[14]), &Vo = cuda_tensor(a[15]);
    const int64_t nl = dK.size(0), H = dK.size(2), D = dK.size(3);
    const std::initializer_list<int64_t> out = {nl, k < 0 ? 0 : k, C < 0 ? 0 : C, H, D};   // (negative: refused by the library)
    if (!Ko.is_contiguous() || !Vo.is_contiguous() || !holds(Ko, out) || !holds(Vo, out))
      fail("K_out/V_out must be contiguous and hold [layers][k*C][H][D]");
    int32_t* n_tokens = static_cast<int32_t*>(ptr(a[16]));
    int32_t* status = static_cast<int32_t*>(ptr_or_null(a[17]));
    const auto fn = entry<decltype(&specext_select_gather)>(a[0]);
    void *k_in = dK.data_ptr(), *v_in = dV.data_ptr(), *k_out = Ko.data_ptr(), *v_out = Vo.data_ptr();
    const int64_t s_layer = dK.stride(0), s_l = dK.stride(1), s_h = dK.stride(2);
    void* st = stream();
    return released([&] {
      return fn(score, n_tree, n_chunks, row, L, C, k, n_sink, n_recent, k_in, v_in, (int32_t)nl, (int32_t)H, (int32_t)D,
                s_layer, s_l, s_h, idx, n_selected, k_out, v_out, n_tokens, status, st);
    });
  });
}

PyObject* current_stream(PyObject*, PyObject*) {
  return guarded(0, 0, [&]() -> PyObject* { return PyLong_FromVoidPtr(stream()); });
}

PyMethodDef kMethods[] = {
    {"fill_desc", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fill_desc)), METH_FASTCALL, nullptr},
    {"verify_attn", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(verify_attn)), METH_FASTCALL, nullptr},
    {"draft_attn", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(draft_attn)), METH_FASTCALL, nullptr},
    {"prefill_attn", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(prefill_attn)), METH_FASTCALL, nullptr},
    {"select_gather", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(select_gather)), METH_FASTCALL, nullptr},
    {"current_stream", current_stream, METH_NOARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (SPX_BUILT_FOR: the torch and the Python whose headers this was compiled with; the module is loaded by no other)
PyMODINIT_FUNC PyInit__binding() {
  PyObject* m = PyModule_Create(&kModule);
  if (m && PyModule_AddStringConstant(m, "built_for", SPX_BUILT_FOR) != 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
