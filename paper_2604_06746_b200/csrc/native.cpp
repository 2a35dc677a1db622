// CPython side of the binding's calls: checks the tensors, reads their pointers and strides, calls the C ABI.  (Through
// ctypes and tensor attributes a call cost 6 us beside its launches, and the argument block of a prefill of 32
// layers 42 us; here 1 us and 3 us.)  Every function returns the library's status, checks raise AssertionError, and
// the interpreter lock is released while the library runs.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "structkv.h"

namespace {

struct PyError {};                                         // a Python exception is set
[[noreturn]] void fail(PyObject* type, const char* what) {
  PyErr_SetString(type, what);
  throw PyError{};
}
void require(bool ok, const char* what) { if (!ok) fail(PyExc_AssertionError, what); }

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) fail(PyExc_TypeError, "a tensor is expected");
  return THPVariable_Unpack(o);
}
template <typename T = void>
T* pointer(PyObject* o) { return o == Py_None ? nullptr : (T*)tensor(o).data_ptr(); }
long long integer(PyObject* o) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) {
    // numpy integers and the like
    PyErr_Clear();
    PyObject* i = PyNumber_Index(o);
    if (!i) throw PyError{};
    const long long w = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (w == -1 && PyErr_Occurred()) throw PyError{};
    return w;
  }
  return v;
}
int int_of(PyObject* o) {
  const long long v = integer(o);
  if (v < INT_MIN || v > INT_MAX) fail(PyExc_OverflowError, "an int of 32 bits is expected");
  return (int)v;
}
float real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyError{};
  return (float)v;
}
structkv_ctx* context(PyObject* o) { return o == Py_None ? nullptr : (structkv_ctx*)integer(o); }
// A torch stream, or None for the current one.
void* stream_of(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw PyError{};
  void* st = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (!st && PyErr_Occurred()) throw PyError{};
  return st;
}
at::ScalarType dtype_of(PyObject* code) { return integer(code) == STRUCTKV_BF16 ? at::kBFloat16 : at::kFloat; }
bool rows_of(const at::Tensor& t, at::ScalarType type) { return t.scalar_type() == type && t.is_contiguous(); }
int64_t dim_of(const at::Tensor& t, int64_t i) {
  if (i >= t.dim()) fail(PyExc_IndexError, "a tensor has too few dimensions");
  return t.size(i);
}
int64_t step_of(const at::Tensor& t, int64_t i) {
  dim_of(t, i);
  return t.stride(i);
}
// [batch, n], or [n] as a batch of one.
struct Vectors { long long stride; int batch, n; const float* p; };
Vectors vectors_of(PyObject* o) {
  const at::Tensor& t = tensor(o);
  require(t.dim() == 1 || t.dim() == 2, "scores: [n] or [batch, n]");
  require(t.scalar_type() == at::kFloat && t.stride(t.dim() - 1) == 1, "scores: rows of float32");
  const int64_t n = t.size(t.dim() - 1);
  return {t.dim() == 2 ? t.stride(0) : n, t.dim() == 2 ? (int)t.size(0) : 1, (int)n, (const float*)t.data_ptr()};
}
// src [n_slabs, n_rows, row...]
struct Source { const void* p; long long slab_bytes, row_stride_bytes; int row_bytes, slabs, rows; };
Source source_of(const at::Tensor& t, bool whole_rows) {
  int64_t row = 1;
  for (int64_t i = 2; i < t.dim(); ++i) row *= t.size(i);
  const int64_t es = t.element_size();
  dim_of(t, 1);
  if (whole_rows && t.dim() > 2) {
    if (t.size(0) == 0 || t.size(1) == 0) fail(PyExc_IndexError, "src: no rows");
    int64_t z = 1;
    for (int64_t i = t.dim() - 1; i >= 2 && row > 0; --i) {
      if (t.size(i) == 1) continue;
      require(t.stride(i) == z, "src: rows are contiguous");
      z *= t.size(i);
    }
  }
  return {t.data_ptr(), t.stride(0) * es, t.stride(1) * es, (int)(row * es), (int)t.size(0), (int)t.size(1)};
}

template <typename F>
PyObject* call(F f) {
  structkv_status s;
  Py_BEGIN_ALLOW_THREADS
  s = f();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(s);
}
// Entry points take positional arguments; C++ and Python errors leave as Python exceptions.
using Body = PyObject* (*)(PyObject* const* a);
template <Body body, int N>
PyObject* entry(PyObject*, PyObject* const* a, Py_ssize_t n) {
  try {
    if (n != N) fail(PyExc_TypeError, "wrong number of arguments");
    return body(a);
  } catch (const PyError&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// ctx, dtype, q_window, k, scale, s_out, metrics_out, c_inout, lam, head_cols_out, flags, stream
PyObject* score_layer(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const at::ScalarType dt = dtype_of(a[1]);
  const at::Tensor &q = tensor(a[2]), &k = tensor(a[3]);
  require(q.is_contiguous() && step_of(k, 2) == 1 && k.scalar_type() == dt && q.scalar_type() == dt,
          "q_window: contiguous, k: unit stride along the head dimension, both of the context's dtype");
  const float scale = real(a[4]), lam = real(a[8]);
  float *s = pointer<float>(a[5]), *m = pointer<float>(a[6]), *ci = pointer<float>(a[7]), *hc = pointer<float>(a[9]);
  const unsigned flags = (unsigned)integer(a[10]);
  void *st = stream_of(a[11]), *qp = q.data_ptr(), *kp = k.data_ptr();
  const long long s0 = k.stride(0), s1 = k.stride(1);
  const int n = (int)k.size(1);
  return call([&] { return structkv_score_layer(c, qp, kp, s0, s1, n, scale, lam, s, ci, hc, m, flags, st); });
}
// ctx, scores, budget, window, idx_out, stream
PyObject* select(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const Vectors v = vectors_of(a[1]);
  const int budget = int_of(a[2]), window = int_of(a[3]);
  const at::Tensor& idx = tensor(a[4]);
  require(rows_of(idx, at::kInt) && idx.numel() == (int64_t)v.batch * budget, "idx_out: contiguous int32 [batch, budget]");
  int* const ip = (int*)idx.data_ptr();
  void* const st = stream_of(a[5]);
  return call([&] { return structkv_select(c, v.p, v.stride, v.batch, v.n, budget, window, ip, st); });
}
// ctx, src, idx, dst, stream
PyObject* compact(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const at::Tensor &idx = tensor(a[2]), &dst = tensor(a[3]);
  require(rows_of(idx, at::kInt) && dst.is_contiguous(), "idx: contiguous int32, dst: contiguous");
  const Source s = source_of(tensor(a[1]), true);
  const int* const ip = (const int*)idx.data_ptr();
  const int n = (int)idx.numel();
  void *dp = dst.data_ptr(), *st = stream_of(a[4]);
  return call([&] { return structkv_compact(c, s.p, s.slab_bytes, s.row_stride_bytes, s.row_bytes, s.slabs, s.rows, ip, n, dp, st); });
}
// ctx, src, idx, dst, stream
PyObject* compact_per_slab(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const at::Tensor &src = tensor(a[1]), &idx = tensor(a[2]), &dst = tensor(a[3]);
  require(idx.scalar_type() == at::kInt && idx.dim() == 2 && idx.stride(1) == 1 && dst.is_contiguous(),
          "idx: int32 [n_slabs, n_idx] with unit stride, dst: contiguous");
  require(idx.size(0) == dim_of(src, 0), "idx: a list per slab");
  const Source s = source_of(src, false);
  const int* const ip = (const int*)idx.data_ptr();
  const long long is = idx.stride(0);
  const int n = (int)idx.size(1);
  void *dp = dst.data_ptr(), *st = stream_of(a[4]);
  return call([&] { return structkv_compact_per_slab(c, s.p, s.slab_bytes, s.row_stride_bytes, s.row_bytes, s.slabs, s.rows, ip, is, n, dp, st); });
}
// ctx, n_q_heads, n_kv_heads, head_cols, out, stream
PyObject* group_saliency(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const at::Tensor &cols = tensor(a[3]), &out = tensor(a[4]);
  require(step_of(cols, 1) == 1 && cols.scalar_type() == at::kFloat && out.is_contiguous(), "head_cols: rows of float32, out: contiguous");
  require(cols.size(0) == integer(a[1]) && out.dim() == 2 && out.size(0) == integer(a[2]) && out.size(1) == cols.size(1),
          "head_cols [H, n], out [H_kv, n]");
  const float* const p = (const float*)cols.data_ptr();
  const long long stride = cols.stride(0);
  const int n = (int)cols.size(1);
  float* const op = (float*)out.data_ptr();
  void* const st = stream_of(a[5]);
  return call([&] { return structkv_group_saliency(c, p, stride, n, op, st); });
}
// ctx, scores, block_size, out, stream
PyObject* block_scores(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const Vectors v = vectors_of(a[1]);
  const int bs = int_of(a[2]);
  if (bs == 0) fail(PyExc_ZeroDivisionError, "block_size is 0");
  const at::Tensor& out = tensor(a[3]);
  // (rounded as the quotient of Python integers is)
  const int64_t up = (int64_t)v.n + bs - 1, per = up >= 0 == bs > 0 || up % bs == 0 ? up / bs : up / bs - 1;
  require(rows_of(out, at::kFloat) && out.numel() == v.batch * per, "out: contiguous float32 [batch, ceil(n / block_size)]");
  float* const op = (float*)out.data_ptr();
  void* const st = stream_of(a[4]);
  return call([&] { return structkv_block_scores(c, v.p, v.stride, v.batch, v.n, bs, op, st); });
}
// ctx, scores, idx, out, stream
PyObject* mass_recovery(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const Vectors v = vectors_of(a[1]);
  const at::Tensor &idx = tensor(a[2]), &out = tensor(a[3]);
  require(rows_of(idx, at::kInt) && out.scalar_type() == at::kFloat && out.numel() == v.batch,
          "idx: contiguous int32, out: float32 [batch]");
  const int* const ip = (const int*)idx.data_ptr();
  const int n = (int)idx.numel();
  float* const op = (float*)out.data_ptr();
  void* const st = stream_of(a[4]);
  return call([&] { return structkv_mass_recovery(c, v.p, v.stride, v.batch, v.n, ip, n, op, st); });
}
// ctx, s_hist, pivot, lam, c_out, stream
PyObject* accumulate(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const at::Tensor& s = tensor(a[1]);
  const int n = (int)dim_of(s, 1), pivot = int_of(a[2]);
  const float lam = real(a[3]);
  const float* const p = (const float*)s.data_ptr();
  const long long stride = s.stride(0);
  float* const out = pointer<float>(a[4]);
  void* const st = stream_of(a[5]);
  return call([&] { return structkv_accumulate(c, p, stride, pivot, n, lam, out, st); });
}

bool fits(const at::Tensor& t, at::IntArrayRef shape, at::ScalarType type) { return t.sizes() == shape && rows_of(t, type); }

// Fills the argument block at address a[0] (its per-layer arrays exist) in; False: the tensors are not in the form of the
// one-call path.  block, layers, hidden, positions, s_hist, head_cols, metrics, c_running, c_star, i_kv, i_struct, kv_out,
// hidden_out, pos_out, layers_workspace, (n_q_heads, n_kv_heads, n_keys, head_dim, window, kv_budget, struct_budget, l_limit),
// dtype, lam, weights
PyObject* fill_prefill(PyObject* const* a) {
  structkv_prefill_args& p = *(structkv_prefill_args*)PyLong_AsVoidPtr(a[0]);
  if (PyErr_Occurred()) throw PyError{};
  if (!PyTuple_Check(a[15]) || PyTuple_GET_SIZE(a[15]) != 8) fail(PyExc_TypeError, "eight sizes are expected");
  auto size = [&](int i) { return integer(PyTuple_GET_ITEM(a[15], i)); };
  const int64_t H = size(0), Hkv = size(1), N = size(2), d = size(3), B = size(5), rows = size(6), L = p.n_layers;
  const at::ScalarType dt = dtype_of(a[16]);
  static PyObject *const key_q = PyUnicode_InternFromString("q_win"), *const key_k = PyUnicode_InternFromString("k"),
                  *const key_kv = PyUnicode_InternFromString("kv"), *const key_scale = PyUnicode_InternFromString("scale");
  auto get = [&](PyObject* dict, PyObject* key, bool needed) {   // borrowed from the dict
    PyObject* v = PyDict_GetItemWithError(dict, key);
    if (!v && PyErr_Occurred()) throw PyError{};
    if (!v && needed) { PyErr_SetObject(PyExc_KeyError, key); throw PyError{}; }
    return v;
  };
  PyObject* const seq = PySequence_Fast(a[1], "layers: a sequence of dicts");
  if (!seq) throw PyError{};
  struct Release { PyObject* o; ~Release() { Py_DECREF(o); } } release{seq};
  if (PySequence_Fast_GET_SIZE(seq) != L) Py_RETURN_FALSE;
  const int64_t kv_shape[4] = {2, Hkv, N, d};
  int64_t k_stride[3] = {0, 0, 0}, kv_stride[4] = {0, 0, 0, 0};
  at::IntArrayRef k_shape;
  std::vector<int64_t> k_sizes;
  for (int64_t l = 0; l < L; ++l) {
    PyObject* const layer = PySequence_Fast_GET_ITEM(seq, l);
    if (!PyDict_Check(layer)) Py_RETURN_FALSE;             // other mappings go step by step
    PyObject *const kvo = get(layer, key_kv, false), *const ko = get(layer, key_k, true), *const qo = get(layer, key_q, true);
    if (!kvo || kvo == Py_None) Py_RETURN_FALSE;
    const at::Tensor &kv = tensor(kvo), &k = tensor(ko), &q = tensor(qo);
    if (l == 0) {
      if (kv.sizes() != at::IntArrayRef(kv_shape, 4) || k.dim() != 3 || k.stride(2) != 1 || k.size(1) != N) Py_RETURN_FALSE;
      k_sizes = k.sizes().vec();
      k_shape = k_sizes;
      for (int i = 0; i < 3; ++i) k_stride[i] = k.stride(i);
      for (int i = 0; i < 4; ++i) kv_stride[i] = kv.stride(i);
    }
    if (k.sizes() != k_shape || k.strides() != at::IntArrayRef(k_stride, 3) || kv.sizes() != at::IntArrayRef(kv_shape, 4) ||
        kv.strides() != at::IntArrayRef(kv_stride, 4) || k.scalar_type() != dt || q.scalar_type() != dt || kv.scalar_type() != dt ||
        !q.is_contiguous())
      Py_RETURN_FALSE;
    ((const void**)p.q_windows)[l] = q.data_ptr();
    ((const void**)p.ks)[l] = k.data_ptr();
    ((const void**)p.kv_srcs)[l] = kv.data_ptr();
    ((float*)p.scales)[l] = real(get(layer, key_scale, true));
  }
  const at::Tensor &s_hist = tensor(a[4]), &head_cols = tensor(a[5]), &metrics = tensor(a[6]), &c_run = tensor(a[7]),
                   &c_star = tensor(a[8]), &i_kv = tensor(a[9]), &i_struct = tensor(a[10]), &kv_out = tensor(a[11]);
  if (!(fits(s_hist, {L, N}, at::kFloat) && fits(head_cols, {L, H, N}, at::kFloat) && fits(metrics, {L, 3}, at::kFloat) &&
        fits(c_run, {N}, at::kFloat) && fits(c_star, {N}, at::kFloat) && fits(i_kv, {L, B}, at::kInt) &&
        fits(i_struct, {rows}, at::kInt) && fits(kv_out, {L, 2, Hkv, B, d}, dt)))
    Py_RETURN_FALSE;
  p.hidden = p.positions = nullptr;
  p.hidden_dst = p.positions_dst = nullptr;
  if (a[2] != Py_None) {
    if (a[12] == Py_None) Py_RETURN_FALSE;
    const at::Tensor &h = tensor(a[2]), &ho = tensor(a[12]);
    if (h.dim() != 2 || h.stride(1) != 1 || h.size(0) != N || h.scalar_type() != ho.scalar_type() || !ho.is_contiguous() ||
        ho.sizes() != at::IntArrayRef({rows, h.size(1)}))
      Py_RETURN_FALSE;
    const at::Tensor &pos = tensor(a[3]), &po = tensor(a[13]);
    if (pos.dim() != 1 || pos.size(0) != N || pos.scalar_type() != at::kInt || !fits(po, {rows}, at::kInt)) Py_RETURN_FALSE;
    const int64_t es = h.element_size(), ps = pos.element_size();
    p.hidden = h.data_ptr();
    p.hidden_row_stride_bytes = h.stride(0) * es;
    p.hidden_row_bytes = (int)(h.size(1) * es);
    p.hidden_dst = ho.data_ptr();
    p.positions = pos.data_ptr();
    p.position_row_stride_bytes = pos.stride(0) * ps;
    p.position_row_bytes = (int)ps;
    p.positions_dst = po.data_ptr();
  }
  if (Hkv > 1 && kv_stride[0] != Hkv * kv_stride[1]) Py_RETURN_FALSE;   // the 2 H_kv slabs have no common stride
  const int64_t es = kv_out.element_size();
  p.n_keys = (int)N;
  p.lambda = real(a[17]);
  p.l_limit = (int)size(7);
  p.window = (int)size(4);
  p.k_stride_head = k_stride[0];
  p.k_stride_token = k_stride[1];
  p.s_out = (float*)s_hist.data_ptr();
  p.s_layer_stride = N;
  p.c_out = (float*)c_run.data_ptr();
  p.head_cols = (float*)head_cols.data_ptr();
  p.head_cols_layer_stride = H * N;
  p.metrics = (float*)metrics.data_ptr();
  p.layers_workspace = nullptr;
  p.layers_workspace_bytes = 0;
  if (a[14] != Py_None) {
    p.layers_workspace = tensor(a[14]).data_ptr();
    p.layers_workspace_bytes = (size_t)tensor(a[14]).numel();
  }
  PyObject* const ws = PySequence_Fast(a[18], "weights: three numbers");
  if (!ws) throw PyError{};
  Release release_w{ws};
  if (PySequence_Fast_GET_SIZE(ws) > 3) fail(PyExc_IndexError, "weights: three numbers");
  for (int i = 0; i < 3; ++i) p.weights[i] = i < PySequence_Fast_GET_SIZE(ws) ? real(PySequence_Fast_GET_ITEM(ws, i)) : 0.f;
  p.kv_budget = (int)B;
  p.struct_budget = (int)rows;
  p.i_kv = (int*)i_kv.data_ptr();
  p.i_struct = (int*)i_struct.data_ptr();
  p.c_star = (float*)c_star.data_ptr();
  p.kv_slab_stride_bytes = kv_stride[Hkv > 1 ? 1 : 0] * es;
  p.kv_row_stride_bytes = kv_stride[2] * es;
  p.kv_row_bytes = (int)(d * es);
  p.kv_slabs = (int)(2 * Hkv);
  p.kv_rows = (int)N;
  p.kv_dst = kv_out.data_ptr();
  p.kv_dst_layer_stride_bytes = 2 * Hkv * B * d * es;
  Py_RETURN_TRUE;
}
// ctx, address of a filled block, stream: (status, pivot, [T_l])
PyObject* prefill(PyObject* const* a) {
  structkv_ctx* const c = context(a[0]);
  const structkv_prefill_args* const p = (const structkv_prefill_args*)PyLong_AsVoidPtr(a[1]);
  if (PyErr_Occurred()) throw PyError{};
  void* const st = stream_of(a[2]);
  std::vector<float> t((size_t)(p->n_layers > 0 ? p->n_layers : 0));
  int pivot = 0;
  structkv_status s;
  Py_BEGIN_ALLOW_THREADS
  s = structkv_prefill(c, p, &pivot, t.data(), st);
  Py_END_ALLOW_THREADS
  PyObject* const list = PyList_New((Py_ssize_t)t.size());
  if (!list) throw PyError{};
  for (size_t i = 0; i < t.size(); ++i) {
    PyObject* const v = PyFloat_FromDouble(t[i]);
    if (!v) { Py_DECREF(list); throw PyError{}; }
    PyList_SET_ITEM(list, (Py_ssize_t)i, v);
  }
  return Py_BuildValue("iiN", (int)s, pivot, list);
}

#define ENTRY(f, n) {#f, (PyCFunction)(void (*)())entry<f, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY(score_layer, 12), ENTRY(select, 6), ENTRY(compact, 5), ENTRY(compact_per_slab, 5),
                         ENTRY(group_saliency, 6), ENTRY(block_scores, 5), ENTRY(mass_recovery, 5), ENTRY(accumulate, 6),
                         ENTRY(fill_prefill, 19), ENTRY(prefill, 3), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// Read from the file by the build, which compiles this again for another torch or python.
extern "C" __attribute__((used)) const char structkv_native_for[] = STRUCTKV_NATIVE_FOR;

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
