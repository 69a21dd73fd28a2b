// Argument marshalling of the Python binding in C++: tensors to pointers and sizes, then the C call.
//
// What bounds it: a call's launches cost 2-4 us of host time, and marshalling the same arguments in
// Python (shape tuples, a ctypes structure, the current stream) cost another 9 us, more than most
// of the kernels take.  With it here a whole cross-attention call costs 2.3 us (11.3 before) and a
// verification call of two launches 3.8 us (13.6).
//
// Each function takes the arguments of binding.py's function of the same name by position and
// returns the C function's status, or -1 for a call that it does not take.  It takes plain CUDA
// tensors of the documented shapes and types, plain int and float values, and a stream that is
// None, an int or a torch.cuda.Stream; everything else, and everything wrong, goes to the Python
// code, which accepts or refuses it.  Nothing is kept from one call to the next.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>
#include <cstdint>

#include "glide.h"

namespace {

PyObject* g_stream_type = nullptr;  // torch.cuda.Stream

struct NotTaken {};

// One call's arguments, read from left to right; the first unusual one throws NotTaken.
class Args {
 public:
  Args(PyObject* const* v, Py_ssize_t n, Py_ssize_t want) : v_(v) {
    if (n != want) throw NotTaken{};
  }

  const at::Tensor& tensor(at::ScalarType type) {
    const at::Tensor& t = any_tensor();
    if (t.scalar_type() != type) throw NotTaken{};
    return t;
  }
  // contiguous, of this shape
  const at::Tensor& tensor(at::ScalarType type, std::initializer_list<int64_t> shape) {
    const at::Tensor& t = tensor(type);
    if (t.sizes() != at::IntArrayRef(shape) || !t.is_contiguous()) throw NotTaken{};
    return t;
  }
  // a cache or the queries: bf16 or fp32, contiguous, no size beyond 32 bits
  const at::Tensor& data() {
    const at::Tensor& t = any_tensor();
    if ((t.scalar_type() != at::kBFloat16 && t.scalar_type() != at::kFloat) || !t.is_contiguous()) throw NotTaken{};
    for (int64_t s : t.sizes())
      if (s > INT_MAX) throw NotTaken{};
    return t;
  }
  const at::Tensor& any_tensor() {
    PyObject* o = *v_++;
    if (!THPVariable_CheckExact(o)) throw NotTaken{};
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || !t.has_storage()) throw NotTaken{};
    return t;
  }
  bool none() {
    if (*v_ != Py_None) return false;
    ++v_;
    return true;
  }
  int32_t i32() { return static_cast<int32_t>(integer(INT_MIN, INT_MAX)); }
  uint32_t u32() { return static_cast<uint32_t>(integer(0, UINT_MAX)); }
  float f32() {
    PyObject* o = *v_;
    if (!PyFloat_CheckExact(o)) return static_cast<float>(integer(-(1 << 24), 1 << 24));
    ++v_;
    return static_cast<float>(PyFloat_AS_DOUBLE(o));
  }
  glide_stream_t stream() {
    PyObject* o = *v_++;
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    if (PyLong_CheckExact(o)) return handle(o);
    if (reinterpret_cast<PyObject*>(Py_TYPE(o)) != g_stream_type) throw NotTaken{};
    struct Ref {
      PyObject* o;
      ~Ref() { Py_XDECREF(o); }
    } h{PyObject_GetAttrString(o, "cuda_stream")};
    if (h.o == nullptr || !PyLong_CheckExact(h.o)) throw NotTaken{};
    return handle(h.o);
  }

 private:
  long long integer(long long lo, long long hi) {
    PyObject* o = *v_++;
    if (!PyLong_CheckExact(o)) throw NotTaken{};
    int over = 0;
    const long long x = PyLong_AsLongLongAndOverflow(o, &over);
    if (over != 0 || x < lo || x > hi) throw NotTaken{};
    return x;
  }
  static glide_stream_t handle(PyObject* o) {
    void* p = PyLong_AsVoidPtr(o);
    if (PyErr_Occurred()) throw NotTaken{};
    return static_cast<glide_stream_t>(p);
  }
  PyObject* const* v_;
};

template <class T>
T* ptr(const at::Tensor& t) {
  return static_cast<T*>(t.data_ptr());
}
int32_t* ints(const at::Tensor& t) { return ptr<int32_t>(t); }

// Runs `body`, which throws before its C call or returns that call's status; the GIL is given up
// around the C call alone, as ctypes does.
template <class F>
PyObject* call(F body) {
  long status = -1;
  try {
    status = body();
  } catch (...) {
    PyErr_Clear();
  }
  return PyLong_FromLong(status);
}
template <class F>
long without_gil(F f) {
  PyThreadState* s = PyEval_SaveThread();
  const long status = f();
  PyEval_RestoreThread(s);
  return status;
}

int32_t dim(const at::Tensor& t, int i) { return static_cast<int32_t>(t.size(i)); }

// queries [B, rows, H, D] and caches [B, H_kv, S_cap, D]
glide_attn_desc describe(const at::Tensor& q, const at::Tensor& K, const at::Tensor& V) {
  if (K.dim() != 4 || q.dim() != 4 || V.sizes() != K.sizes() || K.scalar_type() != V.scalar_type() ||
      q.scalar_type() != K.scalar_type() || q.size(0) != K.size(0) || q.size(3) != K.size(3))
    throw NotTaken{};
  glide_attn_desc d{};
  d.B = dim(K, 0);
  d.H = dim(q, 2);
  d.D = dim(K, 3);
  d.S_cap = dim(K, 2);
  d.dtype = K.scalar_type() == at::kBFloat16 ? GLIDE_BF16 : GLIDE_F32;
  d.H_kv = dim(K, 1) == d.H ? 0 : dim(K, 1);
  return d;
}
// What the kernels read and write as dense rows behind the pointer: the result, of the queries'
// shape, and the lengths of d.B sequences.
void check_dense(const at::Tensor& out, const at::Tensor& q, const at::Tensor& len, const glide_attn_desc& d) {
  if (out.sizes() != q.sizes() || !out.is_contiguous() || len.numel() < d.B || !len.is_contiguous()) throw NotTaken{};
}
void options(glide_attn_desc& d, Args& a) {
  d.scale = a.f32();
  d.flags = a.u32();
  d.max_ctas = a.i32();
}

// q, K, V, kv_len, max_kv_len, out, workspace (not where kNoAlloc), scale, flags, max_ctas, stream
template <bool kNoAlloc>
PyObject* cross_attn(PyObject*, PyObject* const* v, Py_ssize_t n) {
  return call([&] {
    Args a(v, n, kNoAlloc ? 10 : 11);
    const at::Tensor &q = a.data(), &K = a.data(), &V = a.data(), &len = a.tensor(at::kInt);
    glide_attn_desc d = describe(q, K, V);
    const int32_t most = a.i32();
    const at::Tensor& out = a.tensor(at::kFloat);
    if (q.size(1) != 1) throw NotTaken{};
    check_dense(out, q, len, d);
    void* ws = nullptr;
    size_t bytes = 0;
    if constexpr (!kNoAlloc) {
      const at::Tensor& w = a.any_tensor();
      ws = w.data_ptr();
      bytes = w.nbytes();
    }
    options(d, a);
    const glide_stream_t stream = a.stream();
    const void *pq = q.data_ptr(), *pk = K.data_ptr(), *pv = V.data_ptr();
    const int32_t* pl = ints(len);
    float* po = ptr<float>(out);
    return without_gil([&] {
      return long(kNoAlloc ? glide_cross_attn_noalloc(&d, pq, pk, pv, pl, most, po, stream)
                           : glide_cross_attn(&d, pq, pk, pv, pl, most, po, ws, bytes, stream));
    });
  });
}

// q, parent_idx, K, V, kv_len, max_kv_len, out, workspace, scale, flags, max_ctas, stream
PyObject* verify_attn(PyObject*, PyObject* const* v, Py_ssize_t n) {
  return call([&] {
    Args a(v, n, 12);
    const at::Tensor &q = a.data(), &parent = a.tensor(at::kInt), &K = a.data(), &V = a.data();
    const at::Tensor& len = a.tensor(at::kInt);
    glide_attn_desc d = describe(q, K, V);
    const int32_t most = a.i32(), nodes = dim(q, 1);
    const at::Tensor &out = a.tensor(at::kFloat), &w = a.any_tensor();
    if (parent.dim() != 2 || parent.size(0) != d.B || parent.size(1) != nodes || !parent.is_contiguous())
      throw NotTaken{};
    check_dense(out, q, len, d);
    options(d, a);
    const glide_stream_t stream = a.stream();
    const void *pq = q.data_ptr(), *pk = K.data_ptr(), *pv = V.data_ptr();
    const int32_t *pp = ints(parent), *pl = ints(len);
    float* po = ptr<float>(out);
    void* ws = w.data_ptr();
    const size_t bytes = w.nbytes();
    return without_gil(
        [&] { return long(tree_verify_attn(&d, pq, nodes, pp, pk, pv, pl, most, po, ws, bytes, stream)); });
  });
}

// q, K, V, seq_len, L, out, workspace, scale, max_ctas, stream
PyObject* block_attn(PyObject*, PyObject* const* v, Py_ssize_t n) {
  return call([&] {
    Args a(v, n, 10);
    const at::Tensor &q = a.data(), &K = a.data(), &V = a.data(), &len = a.tensor(at::kInt);
    glide_attn_desc d = describe(q, K, V);
    const int32_t L = a.i32(), T = dim(q, 1);
    const at::Tensor &out = a.tensor(at::kFloat), &w = a.any_tensor();
    if (len.dim() != 1 || len.size(0) != d.B) throw NotTaken{};
    check_dense(out, q, len, d);
    d.scale = a.f32();
    d.max_ctas = a.i32();
    const glide_stream_t stream = a.stream();
    const void *pq = q.data_ptr(), *pk = K.data_ptr(), *pv = V.data_ptr();
    const int32_t* pl = ints(len);
    float* po = ptr<float>(out);
    void* ws = w.data_ptr();
    const size_t bytes = w.nbytes();
    return without_gil(
        [&] { return long(glide_block_cross_attn(&d, pq, T, L, pk, pv, pl, po, ws, bytes, stream)); });
  });
}

// draft_tokens, parent_idx, target_logits, path, length, bonus, workspace, stream
PyObject* accept(PyObject*, PyObject* const* v, Py_ssize_t n) {
  return call([&] {
    Args a(v, n, 8);
    const at::Tensor &tok = a.tensor(at::kInt), &parent = a.tensor(at::kInt), &logits = a.data();
    if (logits.dim() != 3 || logits.scalar_type() != at::kFloat) throw NotTaken{};
    const int32_t B = dim(logits, 0), nodes = dim(logits, 1), V = dim(logits, 2);
    const at::IntArrayRef rows = logits.sizes().slice(0, 2);
    const at::Tensor &path = a.tensor(at::kInt, {B, nodes}), &length = a.tensor(at::kInt, {B}),
                     &bonus = a.tensor(at::kInt, {B}), &w = a.any_tensor();
    if (tok.sizes() != rows || parent.sizes() != rows || !tok.is_contiguous() || !parent.is_contiguous())
      throw NotTaken{};
    const glide_stream_t stream = a.stream();
    const int32_t *pt = ints(tok), *pp = ints(parent);
    const float* pg = ptr<float>(logits);
    int32_t *pa = ints(path), *pl = ints(length), *pb = ints(bonus);
    void* ws = w.data_ptr();
    const size_t bytes = w.nbytes();
    return without_gil([&] { return long(tree_accept(pt, pp, pg, B, nodes, V, pa, pl, pb, ws, bytes, stream)); });
  });
}

// probs, root_token, max_tokens, draft_tokens, parent_idx, n_nodes, workspace, conf, fixed_k, stream
PyObject* expand(PyObject*, PyObject* const* v, Py_ssize_t n) {
  return call([&] {
    Args a(v, n, 10);
    const at::Tensor& probs = a.data();
    if (probs.dim() != 3 || probs.scalar_type() != at::kFloat) throw NotTaken{};
    const int32_t B = dim(probs, 0), gamma = dim(probs, 1), V = dim(probs, 2);
    const at::Tensor& root = a.tensor(at::kInt, {B});
    const int32_t most = a.i32();
    const int64_t nodes = int64_t(most) + 1;
    const at::Tensor &tok = a.tensor(at::kInt, {B, nodes}), &parent = a.tensor(at::kInt, {B, nodes}),
                     &count = a.tensor(at::kInt, {B}), &w = a.any_tensor();
    float* conf = a.none() ? nullptr : ptr<float>(a.tensor(at::kFloat, {B, gamma}));
    const int32_t k = a.i32();
    const glide_stream_t stream = a.stream();
    const float* pp = ptr<float>(probs);
    const int32_t* pr = ints(root);
    int32_t *pt = ints(tok), *pa = ints(parent), *pn = ints(count);
    void* ws = w.data_ptr();
    const size_t bytes = w.nbytes();
    return without_gil(
        [&] { return long(cape_expand(pp, pr, B, gamma, V, most, k, pt, pa, pn, conf, ws, bytes, stream)); });
  });
}

// K, V, kv_len, path, length, new_kv_len, stream
PyObject* compact(PyObject*, PyObject* const* v, Py_ssize_t n) {
  return call([&] {
    Args a(v, n, 7);
    const at::Tensor &K = a.data(), &V = a.data();
    const int64_t rank = K.dim();
    if ((rank != 4 && rank != 5) || K.sizes() != V.sizes() || K.scalar_type() != V.scalar_type()) throw NotTaken{};
    const int o = static_cast<int>(rank) - 4;
    glide_attn_desc d{};
    d.B = dim(K, o);
    d.H = dim(K, o + 1);
    d.S_cap = dim(K, o + 2);
    d.D = dim(K, o + 3);
    d.dtype = K.scalar_type() == at::kBFloat16 ? GLIDE_BF16 : GLIDE_F32;
    const int32_t layers = o ? dim(K, 0) : 1;
    const int64_t stride = int64_t(d.B) * d.H * d.S_cap * d.D;
    const at::Tensor &len = a.tensor(at::kInt, {d.B}), &path = a.tensor(at::kInt);
    if (path.dim() != 2 || path.size(0) != d.B || path.size(1) > INT_MAX || !path.is_contiguous()) throw NotTaken{};
    const int32_t nodes = dim(path, 1);
    const at::Tensor &length = a.tensor(at::kInt, {d.B}), &fresh = a.tensor(at::kInt, {d.B});
    const glide_stream_t stream = a.stream();
    void *pk = K.data_ptr(), *pv = V.data_ptr();
    const int32_t *pl = ints(len), *pp = ints(path), *pn = ints(length);
    int32_t* po = ints(fresh);
    return without_gil(
        [&] { return long(glide_kv_compact(&d, layers, stride, pk, pv, pl, nodes, pp, pn, po, stream)); });
  });
}

// draft_tokens, draft_probs, target_logits, uniforms, n_accepted, next_token, workspace, stream
PyObject* sample(PyObject*, PyObject* const* v, Py_ssize_t n) {
  return call([&] {
    Args a(v, n, 8);
    const at::Tensor& tok = a.tensor(at::kInt);
    if (tok.dim() != 2 || tok.size(0) > INT_MAX || tok.size(1) >= INT_MAX || !tok.is_contiguous()) throw NotTaken{};
    const int32_t B = dim(tok, 0), gamma = dim(tok, 1);
    const at::Tensor &probs = a.data(), &logits = a.data();
    if (probs.dim() != 3 || logits.dim() != 3 || probs.scalar_type() != at::kFloat ||
        logits.scalar_type() != at::kFloat)
      throw NotTaken{};
    const int32_t V = dim(logits, 2);
    if (probs.sizes() != at::IntArrayRef({B, gamma, V}) || logits.sizes() != at::IntArrayRef({B, int64_t(gamma) + 1, V}))
      throw NotTaken{};
    const at::Tensor &u = a.tensor(at::kFloat, {B, int64_t(gamma) + 1}), &acc = a.tensor(at::kInt, {B}),
                     &next = a.tensor(at::kInt, {B}), &w = a.any_tensor();
    const glide_stream_t stream = a.stream();
    const int32_t* pt = ints(tok);
    const float *pp = ptr<float>(probs), *pg = ptr<float>(logits), *pu = ptr<float>(u);
    int32_t *pa = ints(acc), *pn = ints(next);
    void* ws = w.data_ptr();
    const size_t bytes = w.nbytes();
    return without_gil([&] { return long(spec_sample_accept(pt, pp, pg, pu, B, gamma, V, pa, pn, ws, bytes, stream)); });
  });
}

#define FN(name, f) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {FN("cross_attn", cross_attn<false>),
                          FN("cross_attn_noalloc", cross_attn<true>),
                          FN("verify_attn", verify_attn),
                          FN("block_attn", block_attn),
                          FN("accept", accept),
                          FN("expand", expand),
                          FN("compact", compact),
                          FN("sample", sample),
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_glidecall", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__glidecall() {
  PyObject* m = PyImport_ImportModule("torch.cuda");
  if (m == nullptr) return nullptr;
  g_stream_type = PyObject_GetAttrString(m, "Stream");  // held for the process's life, as the module is
  Py_DECREF(m);
  return g_stream_type == nullptr ? nullptr : PyModule_Create(&kModule);
}
