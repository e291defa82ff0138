// Native half of the binding's argument marshalling: the per-layer records of a call, read from the
// Python objects in one pass.  Each torch attribute read from Python costs about 0.12 us and a layer
// needs a dozen; with a hundred layers that was most of a step's host time (2.3 us per layer in
// Python, 0.3 us here).  step() fills the whole record of dp_step_enqueue and makes the call: the step of
// one small layer, bound by the host, takes 31 us call by call; it took 49 with the record filled in
// Python.  No device work of its own, nothing is kept between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <exception>
#include <memory>
#include <type_traits>
#include <vector>

#include "../../include/dp_ghost.h"

namespace {

// an owned reference, released also where torch throws
struct Decref { void operator()(PyObject* o) const { Py_DECREF(o); } };
using Ref = std::unique_ptr<PyObject, Decref>;

// dp_dtype of a tensor, kOther if it has none; *kind: that of the tensors seen before, kNone at first
constexpr int32_t kNone = -1, kOther = -2;
int32_t dtype_of(const at::Tensor& t) {
  return t.scalar_type() == at::kFloat ? int32_t(DP_F32) : t.scalar_type() == at::kBFloat16 ? int32_t(DP_BF16) : kOther;
}
bool same_dtype(const at::Tensor& t, int32_t* kind) {
  const int32_t k = dtype_of(t);
  if (k == kOther || (*kind != kNone && *kind != k)) return false;
  *kind = k;
  return true;
}

// base pointer and leading dimension of a (..., ld) CUDA tensor whose leading axes are densely packed and whose
// type is *kind; false: the caller's Python check words the complaint
bool rows(PyObject* o, const void** ptr, int64_t* ld, int64_t* cols, int32_t* kind) {
  if (!THPVariable_Check(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  const auto st = t.strides();
  const size_t n = st.size();
  if (!t.is_cuda() || n < 2 || st[n - 1] != 1 || !same_dtype(t, kind)) return false;
  if (n == 3 && st[0] != t.size(1) * st[1]) return false;
  *ptr = t.const_data_ptr();
  *ld = st[n - 2];
  *cols = t.size(int64_t(n) - 1);
  return true;
}

// integer attribute; None gives `otherwise`
bool integer(PyObject* o, const char* name, int64_t otherwise, int64_t* out) {
  const Ref v(PyObject_GetAttrString(o, name));
  if (!v) { PyErr_Clear(); return false; }
  *out = v.get() == Py_None ? otherwise : PyLong_AsLongLong(v.get());
  if (PyErr_Occurred()) { PyErr_Clear(); return false; }
  return true;
}

bool attr_rows(PyObject* o, const char* name, const void** ptr, int64_t* ld, int64_t* cols, int32_t* kind) {
  const Ref v(PyObject_GetAttrString(o, name));
  if (!v) { PyErr_Clear(); return false; }
  return rows(v.get(), ptr, ld, cols, kind);
}

bool linear_record(dp_linear_desc& L, PyObject* o, int32_t* kind) {
  int64_t ca = 0, cg = 0, d = 0, p = 0, mode = 0;
  const bool ok = attr_rows(o, "A", &L.A, &L.lda, &ca, kind) && attr_rows(o, "G", &L.G, &L.ldg, &cg, kind) &&
                  integer(o, "d", ca, &d) && integer(o, "p", cg, &p) && integer(o, "mode", 0, &mode);
  L.d = int32_t(d); L.p = int32_t(p); L.mode = int32_t(mode); L.mode_used = -1;
  return ok;
}

bool vector_record(dp_vector_desc& v, PyObject* o, int32_t* kind) {
  int64_t cols = 0, other = 0, p = 0;
  bool ok = attr_rows(o, "G", &v.G, &v.ldg, &cols, kind) && integer(o, "p", cols, &p);
  const Ref x(PyObject_GetAttrString(o, "X"));
  if (!x) { PyErr_Clear(); return false; }
  if (x.get() != Py_None) ok = ok && rows(x.get(), &v.X, &v.ldx, &other, kind);
  v.p = int32_t(p);
  return ok;
}

// f(record, object, kind) over a sequence -> bytearray of records, or None if a tensor is not usable or the
// tensors are not all of one type
template <typename Rec, typename F>
PyObject* records(PyObject* arg, F f) {
  const Ref seq(PySequence_Fast(arg, "a sequence"));
  if (!seq) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq.get());
  Ref out(PyByteArray_FromStringAndSize(nullptr, n * Py_ssize_t(sizeof(Rec))));
  if (!out) return nullptr;
  auto* rec = reinterpret_cast<Rec*>(PyByteArray_AS_STRING(out.get()));
  memset(static_cast<void*>(rec), 0, size_t(n) * sizeof(Rec));
  bool ok = true;
  int32_t kind = kNone;
  for (Py_ssize_t k = 0; k < n && ok; ++k) ok = f(rec[k], PySequence_Fast_GET_ITEM(seq.get(), k), &kind);
  if (!ok) Py_RETURN_NONE;
  return out.release();
}

// linears(sequence of Linear) -> dp_linear_desc[]
PyObject* linears(PyObject*, PyObject* arg) {
  return records<dp_linear_desc>(arg, linear_record);
}

// vectors(sequence of Vector) -> dp_vector_desc[]
PyObject* vectors(PyObject*, PyObject* arg) {
  return records<dp_vector_desc>(arg, vector_record);
}

// outputs(sequence of CUDA tensors) -> bytearray: n pointers, then n leading strides; or None
PyObject* outputs(PyObject*, PyObject* arg) {
  const Ref seq(PySequence_Fast(arg, "a sequence of tensors"));
  if (!seq) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq.get());
  Ref out(PyByteArray_FromStringAndSize(nullptr, 16 * n));
  if (!out) return nullptr;
  auto* w = reinterpret_cast<int64_t*>(PyByteArray_AS_STRING(out.get()));
  for (Py_ssize_t k = 0; k < n; ++k) {
    PyObject* o = PySequence_Fast_GET_ITEM(seq.get(), k);
    if (!THPVariable_Check(o) || !THPVariable_Unpack(o).is_cuda()) Py_RETURN_NONE;
    const at::Tensor& t = THPVariable_Unpack(o);
    w[k] = reinterpret_cast<int64_t>(t.mutable_data_ptr());
    w[n + k] = t.dim() > 0 ? t.stride(0) : 0;
  }
  return out.release();
}

// f(index, object) over a sequence; false: it said no, or it is no sequence of n objects
template <typename F>
bool each(PyObject* arg, Py_ssize_t n, F f) {
  const Ref seq(PySequence_Fast(arg, "a sequence"));
  if (!seq) { PyErr_Clear(); return false; }
  bool ok = PySequence_Fast_GET_SIZE(seq.get()) == n;
  for (Py_ssize_t k = 0; k < n && ok; ++k) ok = f(k, PySequence_Fast_GET_ITEM(seq.get(), k));
  return ok;
}

// a CUDA tensor, or nullptr for None; false: neither
bool device_tensor(PyObject* o, const at::Tensor** t) {
  *t = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) return false;
  *t = &THPVariable_Unpack(o);
  return (*t)->is_cuda();
}

// address to read from (P const) or to write to: a tensor that shares its memory until it is written to
// (copy-on-write) gets its own first
template <typename P>
P* pointer(const at::Tensor* t) {
  if (!t) return nullptr;
  if constexpr (std::is_const_v<P>) return static_cast<P*>(t->const_data_ptr());
  else return static_cast<P*>(t->mutable_data_ptr());
}

bool output_list(PyObject* arg, Py_ssize_t n, std::vector<float*>& ptr, std::vector<int64_t>& ld) {
  ptr.resize(size_t(n)); ld.resize(size_t(n));
  return each(arg, n, [&](Py_ssize_t k, PyObject* o) {
    const at::Tensor* t;
    if (!device_tensor(o, &t) || !t || t->scalar_type() != at::kFloat) return false;
    ptr[size_t(k)] = pointer<float>(t);
    ld[size_t(k)] = t->dim() > 0 ? t->stride(0) : 0;
    return true;
  });
}

bool word_list(PyObject* arg, Py_ssize_t n, std::vector<uint32_t>& w) {
  w.resize(size_t(n));
  return each(arg, n, [&](Py_ssize_t k, PyObject* o) {
    w[size_t(k)] = uint32_t(PyLong_AsUnsignedLongMask(o));
    if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    return true;
  });
}

// step(address of dp_step_enqueue, layers, outs, ids of outs, vectors, vector outs, their ids,
//      (17 tensors or None), (stream or None, side stream, 4 events, seed, V, d, tied, noise, step, wte id,
//      wpe id, phases), C, sigma) -> status, with mode_used set on the layers; None: some argument is not
// usable and the caller's Python checks say which
PyObject* step(PyObject*, PyObject* const* a, Py_ssize_t na) {
  if (na != 11) { PyErr_SetString(PyExc_TypeError, "step takes 11 arguments"); return nullptr; }
  using Enqueue = dp_status (*)(const dp_step_desc*, int32_t);
  const Enqueue enqueue = reinterpret_cast<Enqueue>(PyLong_AsVoidPtr(a[0]));
  if (!enqueue || PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }
  const Py_ssize_t n = PyObject_Length(a[1]), nv = PyObject_Length(a[4]);
  if (n < 0 || nv < 0) { PyErr_Clear(); Py_RETURN_NONE; }
  std::vector<dp_linear_desc> layers(static_cast<size_t>(n));
  std::vector<dp_vector_desc> vectors(static_cast<size_t>(nv));
  std::vector<float*> outs, vouts;
  std::vector<int64_t> ldos, unused;
  std::vector<uint32_t> ids, vids;
  const at::Tensor* t[17];
  int64_t v[15];
  int32_t layer_kind = kNone, vector_kind = kNone, embed_kind = kNone;
  memset(static_cast<void*>(layers.data()), 0, layers.size() * sizeof(dp_linear_desc));
  memset(static_cast<void*>(vectors.data()), 0, vectors.size() * sizeof(dp_vector_desc));
  bool ok = each(a[1], n, [&](Py_ssize_t k, PyObject* o) { return linear_record(layers[size_t(k)], o, &layer_kind); }) &&
            output_list(a[2], n, outs, ldos) && word_list(a[3], n, ids) &&
            each(a[4], nv, [&](Py_ssize_t k, PyObject* o) { return vector_record(vectors[size_t(k)], o, &vector_kind); }) &&
            output_list(a[5], nv, vouts, unused) && word_list(a[6], nv, vids) &&
            each(a[7], 17, [&](Py_ssize_t k, PyObject* o) { return device_tensor(o, &t[k]); }) &&
            each(a[8], 15, [&](Py_ssize_t k, PyObject* o) {
              if (k == 0 && o == Py_None) v[k] = reinterpret_cast<int64_t>(c10::cuda::getCurrentCUDAStream().stream());
              else v[k] = int64_t(PyLong_AsUnsignedLongLongMask(o));
              if (PyErr_Occurred()) { PyErr_Clear(); return false; }
              return true;
            });
  enum { IDS, G_EMB, POS_IDS, WTE, WPE, SQ, CLIP, NORMS, CROSS, SIDE_SQ, PERM, SEG, POS_PERM, POS_SEG, WS, SIDE_WS, STATUS };
  const void* g = nullptr;
  int64_t ldg = 0, cols = 0;
  PyObject* tensors = a[7];
  ok = ok && PyTuple_Check(tensors) && rows(PyTuple_GET_ITEM(tensors, G_EMB), &g, &ldg, &cols, &embed_kind);
  ok = ok && t[IDS] && t[IDS]->dim() == 2 && t[WTE] && t[WTE]->dim() == 2 && (!t[WPE] || t[WPE]->dim() == 2) && t[WS] &&
       t[SIDE_WS];
  for (int k : {IDS, POS_IDS, PERM, SEG, POS_PERM, POS_SEG, STATUS}) ok = ok && (!t[k] || t[k]->scalar_type() == at::kInt);
  for (int k : {WTE, WPE, SQ, CLIP, NORMS, CROSS, SIDE_SQ}) ok = ok && (!t[k] || t[k]->scalar_type() == at::kFloat);
  const double C = PyFloat_AsDouble(a[9]), sigma = PyFloat_AsDouble(a[10]);
  if (PyErr_Occurred()) { PyErr_Clear(); ok = false; }
  if (!ok) Py_RETURN_NONE;
  dp_step_desc S;
  memset(&S, 0, sizeof(S));
  if (n) { S.layers = layers.data(); S.outs = outs.data(); S.ldos = ldos.data(); }
  S.tensor_ids = ids.data();
  if (nv) { S.vectors = vectors.data(); S.vector_outs = vouts.data(); }
  S.vector_ids = vids.data();
  S.ids = pointer<const int32_t>(t[IDS]); S.G_emb = g; S.ldge = ldg;
  S.pos_ids = pointer<const int32_t>(t[POS_IDS]);
  S.wte = pointer<float>(t[WTE]); S.ld_wte = t[WTE]->stride(0);
  S.wpe = pointer<float>(t[WPE]); S.ld_wpe = t[WPE] ? t[WPE]->stride(0) : 0;
  S.sq = pointer<float>(t[SQ]); S.clip = pointer<float>(t[CLIP]); S.norms = pointer<float>(t[NORMS]);
  S.cross = pointer<float>(t[CROSS]); S.side_sq = pointer<float>(t[SIDE_SQ]);
  S.perm = pointer<int32_t>(t[PERM]); S.seg = pointer<int32_t>(t[SEG]);
  S.pos_perm = pointer<int32_t>(t[POS_PERM]); S.pos_seg = pointer<int32_t>(t[POS_SEG]);
  S.ws = pointer<void>(t[WS]); S.ws_bytes = size_t(t[WS]->nbytes());
  S.side_ws = pointer<void>(t[SIDE_WS]); S.side_ws_bytes = size_t(t[SIDE_WS]->nbytes());
  S.dev_status = pointer<int32_t>(t[STATUS]);
  S.stream = reinterpret_cast<void*>(v[0]); S.side_stream = reinterpret_cast<void*>(v[1]);
  for (int k = 0; k < 4; ++k) S.events[k] = reinterpret_cast<void*>(v[2 + k]);
  S.seed = uint64_t(v[6]);
  S.layer_dtype = layer_kind == kNone ? embed_kind : layer_kind;           // no layers, no vectors: nothing to read
  S.vector_dtype = vector_kind == kNone ? embed_kind : vector_kind;
  S.embed_dtype = embed_kind;
  S.n_layers = int32_t(n); S.n_vectors = int32_t(nv);
  S.B = int32_t(t[IDS]->size(0)); S.T = int32_t(t[IDS]->size(1)); S.V = int32_t(v[7]); S.d = int32_t(v[8]);
  S.pos_rows = t[WPE] ? int32_t(t[WPE]->size(0)) : 0;
  S.tied = int32_t(v[9]); S.with_noise = int32_t(v[10]); S.C = float(C); S.sigma = float(sigma);
  S.step = uint32_t(v[11]); S.wte_id = uint32_t(v[12]); S.wpe_id = uint32_t(v[13]);
  const int32_t phases = int32_t(v[14]);
  dp_status st;
  {
    struct Unlocked {
      PyThreadState* state = PyEval_SaveThread();
      ~Unlocked() { PyEval_RestoreThread(state); }
    } unlocked;
    st = enqueue(&S, phases);
  }
  if (st == DP_OK && (phases & DP_STEP_NORMS))
    each(a[1], n, [&](Py_ssize_t k, PyObject* o) {
      PyObject* m = PyLong_FromLong(layers[size_t(k)].mode_used);
      const bool set = m && PyObject_SetAttrString(o, "mode_used", m) == 0;
      Py_XDECREF(m);
      if (!set) PyErr_Clear();
      return set;
    });
  return PyLong_FromLong(long(st));
}

// What torch throws for tensors without strides or memory of their own (nested ones, those inside vmap) becomes a
// Python exception: past the C entry it would end the process.
template <PyObject* (*F)(PyObject*, PyObject*)>
PyObject* guarded(PyObject* self, PyObject* arg) {
  try {
    return F(self, arg);
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}
PyObject* guarded_step(PyObject* self, PyObject* const* a, Py_ssize_t na) {
  try {
    return step(self, a, na);
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyMethodDef methods[] = {{"step", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded_step)), METH_FASTCALL, nullptr},
                         {"linears", guarded<linears>, METH_O, nullptr},
                         {"vectors", guarded<vectors>, METH_O, nullptr},
                         {"outputs", guarded<outputs>, METH_O, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
  PyObject* m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "torch_version", DP_TORCH_VERSION) < 0) { Py_DECREF(m); return nullptr; }
  return m;
}
