// The calls of a serving loop (encode, append, the attention calls) from Python tensors to the C ABI without ctypes: one
// vectorcall per entry point that checks shapes and dtypes, reads the data pointers and the current stream, and calls the
// library.  A ctypes call with seventeen arguments, its pointer conversions and the stream lookup cost 8 to 10 us, more
// than the kernels of a short step; this path costs below 1 us.  Every function returns the library's status code.
//
// Arguments common to all: `stream` is None (PyTorch's current stream) or an object with a cuda_stream attribute,
// `paging` 0, the address of a struct pq_paging, or a tuple (page table tensor, tokens per page, pages of the pool).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/polarquant.h"

namespace {

struct PyError {};   // a Python exception has been set

[[noreturn]] void fail(PyObject* type, const char* text) {
  PyErr_SetString(type, text);
  throw PyError();
}
void check(bool ok, const char* text) {
  if (!ok) fail(PyExc_AssertionError, text);
}
const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a tensor");
  return THPVariable_Unpack(o);
}
const at::Tensor* tensor_or_none(PyObject* o) { return o == Py_None ? nullptr : &tensor(o); }
template <class T = void>
T* ptr(const at::Tensor& t) {
  return static_cast<T*>(t.data_ptr());
}
int32_t i32(PyObject* o) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) throw PyError();
  if (v < INT32_MIN || v > INT32_MAX) fail(PyExc_OverflowError, "value does not fit in 32 bits");
  return (int32_t)v;
}
float f32(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyError();
  return (float)v;
}
template <class T>
const T* address(PyObject* o) {
  void* p = PyLong_AsVoidPtr(o);
  if (p == nullptr && PyErr_Occurred()) throw PyError();
  return static_cast<const T*>(p);
}
// The paging of a call, read before the interpreter lock is released.
class PagingArg {
 public:
  explicit PagingArg(PyObject* o) {
    if (PyTuple_Check(o)) {
      check(PyTuple_GET_SIZE(o) == 3, "paging is (page table, tokens per page, pages)");
      const at::Tensor& table = tensor(PyTuple_GET_ITEM(o, 0));
      check(table.scalar_type() == at::kInt && table.is_contiguous() && table.dim() == 2, "the page table must be a contiguous int32 tensor [batch, pages]");
      paging_ = {ptr<int32_t>(table), i32(PyTuple_GET_ITEM(o, 1)), (int32_t)table.size(1), i32(PyTuple_GET_ITEM(o, 2))};
      paged_ = true;
    } else if (const auto* p = address<pq_paging>(o)) {
      paging_ = *p;
      paged_ = true;
    }
  }
  const pq_paging* get() const { return paged_ ? &paging_ : nullptr; }

 private:
  pq_paging paging_ = {};
  bool paged_ = false;
};
void* stream_of(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
  if (v == nullptr) throw PyError();
  void* p = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  if (p == nullptr && PyErr_Occurred()) throw PyError();
  return p;
}
int32_t dtype_code(const at::Tensor& t) {
  if (t.scalar_type() == at::kFloat) return PQ_DTYPE_F32;
  if (t.scalar_type() == at::kBFloat16) return PQ_DTYPE_BF16;
  fail(PyExc_TypeError, "unsupported dtype (float32 and bfloat16 are taken)");
}

// Calls the library without the interpreter lock, as ctypes does: a launch may block on a full queue, and the first call of a kernel loads
// it.  The arguments have been evaluated by then; the caller's frame holds the tensors.
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};
template <class... Params, class... Args>
int32_t call(int32_t (*fn)(Params...), Args... args) {
  const Unlocked unlocked;
  return fn(args...);
}

// Runs `body` with `n` arguments checked and every exception turned into a Python one.
template <class Body>
PyObject* entry(Py_ssize_t got, Py_ssize_t want, Body body) {
  if (got != want) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
    return nullptr;
  }
  try {
    return PyLong_FromLong(body());
  } catch (const PyError&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

void check_rows(const at::Tensor& K, const at::Tensor& V) {   // packed rows [tokens, heads, d]
  check(K.dim() == 3 && V.sizes() == K.sizes() && V.scalar_type() == K.scalar_type() && K.stride(2) == 1 && V.strides() == K.strides(),
        "K and V must be [tokens, kv heads, head_dim] of one dtype with the same strides and contiguous vectors");
}
void check_query(const at::Tensor& q, const at::Tensor& out, int64_t dim) {
  check(q.dim() == dim && q.is_contiguous() && out.is_contiguous() && out.sizes() == q.sizes() && out.scalar_type() == q.scalar_type(),
        "q and out must be contiguous tensors of one shape and dtype");
}

// encode(S, tables, K, V, cu_seqlens, cache, lens, capacity, status, paging, stream)
PyObject* encode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return entry(n, 11, [&]() -> int32_t {
    const at::Tensor &K = tensor(a[2]), &V = tensor(a[3]), &cu = tensor(a[4]);
    check_rows(K, V);
    const PagingArg paging(a[9]);
    const pq_paging* pg = paging.get();
    const int32_t d = (int32_t)K.size(2), h = (int32_t)K.size(1), total = (int32_t)K.size(0), batch = (int32_t)cu.numel() - 1;
    if (pg != nullptr)
      return call(pq_encode_kv_paged, d, h, ptr<float>(tensor(a[0])), ptr(tensor(a[1])), ptr(K), ptr(V), dtype_code(K), K.stride(0),
                                K.stride(1), ptr<int32_t>(cu), batch, total, ptr(tensor(a[5])), ptr<int32_t>(tensor(a[6])), pg,
                                ptr<int32_t>(tensor(a[8])), stream_of(a[10]));
    return call(pq_encode_kv, d, h, ptr<float>(tensor(a[0])), ptr(tensor(a[1])), ptr(K), ptr(V), dtype_code(K), K.stride(0), K.stride(1),
                        ptr<int32_t>(cu), batch, total, ptr(tensor(a[5])), ptr<int32_t>(tensor(a[6])), i32(a[7]),
                        ptr<int32_t>(tensor(a[8])), stream_of(a[10]));
  });
}

// append(S, tables, k_new, v_new, cache, lens, capacity, status, paging, stream)
PyObject* append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return entry(n, 10, [&]() -> int32_t {
    const at::Tensor &k = tensor(a[2]), &v = tensor(a[3]);
    check(k.dim() == 3 && k.is_contiguous() && v.is_contiguous() && v.sizes() == k.sizes() && v.scalar_type() == k.scalar_type(),
          "k_new and v_new must be contiguous [batch, kv heads, head_dim] of one dtype");
    const PagingArg paging(a[8]);
    const pq_paging* pg = paging.get();
    const int32_t d = (int32_t)k.size(2), h = (int32_t)k.size(1), batch = (int32_t)k.size(0);
    if (pg != nullptr)
      return call(pq_append_kv_paged, d, h, ptr<float>(tensor(a[0])), ptr(tensor(a[1])), ptr(k), ptr(v), dtype_code(k), batch,
                                ptr(tensor(a[4])), ptr<int32_t>(tensor(a[5])), pg, ptr<int32_t>(tensor(a[7])), stream_of(a[9]));
    return call(pq_append_kv, d, h, ptr<float>(tensor(a[0])), ptr(tensor(a[1])), ptr(k), ptr(v), dtype_code(k), batch, ptr(tensor(a[4])),
                        ptr<int32_t>(tensor(a[5])), i32(a[6]), ptr<int32_t>(tensor(a[7])), stream_of(a[9]));
  });
}

// attend(S, tables, q, cache, lens, n_kv_heads, capacity, max_len, scale, out, lse or None, workspace, status, paging, stream):
// q [batch, heads, d], or [batch, queries, heads, d] for the causal last positions of every sequence
PyObject* attend(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return entry(n, 15, [&]() -> int32_t {
    const at::Tensor &q = tensor(a[2]), &out = tensor(a[9]);
    const bool multi = q.dim() == 4;
    check_query(q, out, multi ? 4 : 3);
    const at::Tensor* lse = tensor_or_none(a[10]);
    const PagingArg paging(a[13]);
    const pq_paging* pg = paging.get();
    const int32_t d = (int32_t)q.size(-1), hq = (int32_t)q.size(-2), batch = (int32_t)q.size(0), hkv = i32(a[5]), cap = i32(a[6]),
                  most = i32(a[7]);
    const float scale = f32(a[8]);
    const float* S = ptr<float>(tensor(a[0]));
    const void *tables = ptr(tensor(a[1])), *cache = ptr(tensor(a[3]));
    const int32_t* lens = ptr<int32_t>(tensor(a[4]));
    void *ws = ptr(tensor(a[11])), *stream = stream_of(a[14]);
    int32_t* status = ptr<int32_t>(tensor(a[12]));
    if (lse != nullptr) {
      check(!multi && lse->scalar_type() == at::kFloat && lse->is_contiguous() && lse->dim() == 2 && lse->size(0) == batch && lse->size(1) == hq,
            "lse must be a contiguous float32 tensor [batch, query heads]");
      return call(pq_decode_attention_lse, d, hq, hkv, S, tables, ptr(q), dtype_code(q), cache, lens, batch, cap, pg, most, scale, ptr(out),
                                     ptr<float>(*lse), ws, status, stream);
    }
    if (multi) {
      const int32_t nq = (int32_t)q.size(1);
      if (pg != nullptr)
        return call(pq_multi_query_attention_paged, d, hq, hkv, S, tables, ptr(q), dtype_code(q), cache, lens, batch, nq, pg, most, scale,
                                              ptr(out), ws, status, stream);
      return call(pq_multi_query_attention, d, hq, hkv, S, tables, ptr(q), dtype_code(q), cache, lens, batch, nq, cap, most, scale, ptr(out),
                                      ws, status, stream);
    }
    if (pg != nullptr)
      return call(pq_decode_attention_paged, d, hq, hkv, S, tables, ptr(q), dtype_code(q), cache, lens, batch, pg, most, scale, ptr(out), ws,
                                       status, stream);
    return call(pq_decode_attention, d, hq, hkv, S, tables, ptr(q), dtype_code(q), cache, lens, batch, cap, most, scale, ptr(out), ws, status,
                               stream);
  });
}

// general_encode(cfg, S, boundaries, K, V, cu_seqlens, cache, lens, capacity, status, stream)
PyObject* general_encode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return entry(n, 11, [&]() -> int32_t {
    const at::Tensor &K = tensor(a[3]), &V = tensor(a[4]), &cu = tensor(a[5]);
    check_rows(K, V);
    const auto* cfg = address<pq_general_config>(a[0]);
    check(cfg != nullptr && K.size(2) == cfg->head_dim, "K and V must have the configuration's head_dim");
    return call(pq_general_encode_kv, cfg, (int32_t)K.size(1), ptr<float>(tensor(a[1])), ptr<double>(tensor(a[2])), ptr(K), ptr(V),
                                dtype_code(K), K.stride(0), K.stride(1), ptr<int32_t>(cu), (int32_t)cu.numel() - 1,
                                (int32_t)K.size(0), ptr(tensor(a[6])), ptr<int32_t>(tensor(a[7])), i32(a[8]),
                                ptr<int32_t>(tensor(a[9])), stream_of(a[10]));
  });
}

// general_attend(cfg, n_kv_heads, S, centroids, q, cache, lens, capacity, scale, out, status, stream)
PyObject* general_attend(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return entry(n, 12, [&]() -> int32_t {
    const at::Tensor &q = tensor(a[4]), &out = tensor(a[9]);
    check(q.dim() == 3 && q.is_contiguous() && out.is_contiguous() && out.numel() >= q.numel() && out.scalar_type() == q.scalar_type(),
          "q must be [batch, heads, head_dim], out of its dtype with room for as many values, both contiguous");
    const auto* cfg = address<pq_general_config>(a[0]);
    check(cfg != nullptr && q.size(2) == cfg->head_dim, "q must have the configuration's head_dim");
    return call(pq_general_decode_attention, cfg, (int32_t)q.size(1), i32(a[1]), ptr<float>(tensor(a[2])), ptr<double>(tensor(a[3])), ptr(q),
                                       dtype_code(q), ptr(tensor(a[5])), ptr<int32_t>(tensor(a[6])), (int32_t)q.size(0), i32(a[7]),
                                       f32(a[8]), ptr(out), ptr<int32_t>(tensor(a[10])), stream_of(a[11]));
  });
}

// angle_histograms(S, K, V, hist, status, stream): hist int64 [levels, bins], counts are added
PyObject* angle_histograms(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return entry(n, 6, [&]() -> int32_t {
    const at::Tensor &K = tensor(a[1]), &V = tensor(a[2]), &hist = tensor(a[3]);
    check_rows(K, V);
    check(hist.scalar_type() == at::kLong && hist.is_contiguous() && hist.dim() == 2 && hist.size(0) == PQ_N_LEVELS,
          "hist must be a contiguous int64 tensor [levels, bins]");
    return call(pq_angle_histograms, (int32_t)K.size(2), (int32_t)K.size(1), ptr<float>(tensor(a[0])), ptr(K), ptr(V), dtype_code(K),
                               K.stride(0), K.stride(1), (int32_t)K.size(0), (int32_t)hist.size(1), ptr<uint64_t>(hist),
                               ptr<int32_t>(tensor(a[4])), stream_of(a[5]));
  });
}

// tail_attend(q, k_tail, v_tail, tail_lens, scale, out, lse or None, status, n_splits, stream)
PyObject* tail_attend(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return entry(n, 10, [&]() -> int32_t {
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]), &out = tensor(a[5]);
    const at::Tensor* lse = tensor_or_none(a[6]);
    const int32_t splits = i32(a[8]);
    check(q.dim() == 3 && q.is_contiguous() && out.is_contiguous() && out.scalar_type() == q.scalar_type(),
          "q and out must be contiguous tensors of one dtype");
    check(k.dim() == 4 && k.is_contiguous() && v.is_contiguous() && k.sizes() == v.sizes() && k.scalar_type() == v.scalar_type() &&
              k.size(0) == q.size(0) && k.size(3) == q.size(2),
          "the window must be contiguous [batch, tokens, kv heads, head_dim]");
    check(out.numel() == splits * q.numel() && (lse == nullptr || lse->numel() == splits * q.size(0) * q.size(1)),
          "out and lse must hold n_splits parts");
    return call(pq_tail_attention, (int32_t)q.size(2), (int32_t)q.size(1), (int32_t)k.size(2), ptr(q), dtype_code(q), ptr(k), ptr(v),
                             dtype_code(k), ptr<int32_t>(tensor(a[3])), (int32_t)q.size(0), (int32_t)k.size(1), splits, f32(a[4]),
                             ptr(out), lse == nullptr ? nullptr : ptr<float>(*lse), ptr<int32_t>(tensor(a[7])), stream_of(a[9]));
  });
}

// merge(parts_out, parts_lse, out, lse_out or None, status, stream)
PyObject* merge(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return entry(n, 6, [&]() -> int32_t {
    const at::Tensor &parts = tensor(a[0]), &lse = tensor(a[1]), &out = tensor(a[2]);
    const at::Tensor* lse_out = tensor_or_none(a[3]);
    check(parts.dim() == 4 && parts.is_contiguous() && lse.is_contiguous() && out.is_contiguous(), "contiguous tensors are taken");
    check(lse.scalar_type() == at::kFloat && lse.dim() == 3 && lse.sizes() == parts.sizes().slice(0, 3) &&
              out.sizes() == parts.sizes().slice(1, 3),
          "parts_out [parts, batch, heads, head_dim], parts_lse float32 [parts, batch, heads], out [batch, heads, head_dim]");
    return call(pq_merge_attention, (int32_t)parts.size(3), (int32_t)parts.size(2), (int32_t)parts.size(1), (int32_t)parts.size(0), ptr(parts),
                              dtype_code(parts), ptr<float>(lse), ptr(out), dtype_code(out),
                              lse_out == nullptr ? nullptr : ptr<float>(*lse_out), ptr<int32_t>(tensor(a[4])), stream_of(a[5]));
  });
}

PyMethodDef kMethods[] = {
    {"angle_histograms", (PyCFunction)(void (*)(void))angle_histograms, METH_FASTCALL, nullptr},
    {"tail_attend", (PyCFunction)(void (*)(void))tail_attend, METH_FASTCALL, nullptr},
    {"merge", (PyCFunction)(void (*)(void))merge, METH_FASTCALL, nullptr},
    {"encode", (PyCFunction)(void (*)(void))encode, METH_FASTCALL, nullptr},
    {"append", (PyCFunction)(void (*)(void))append, METH_FASTCALL, nullptr},
    {"attend", (PyCFunction)(void (*)(void))attend, METH_FASTCALL, nullptr},
    {"general_encode", (PyCFunction)(void (*)(void))general_encode, METH_FASTCALL, nullptr},
    {"general_attend", (PyCFunction)(void (*)(void))general_attend, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_pq_binding", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pq_binding(void) { return PyModule_Create(&kModule); }
