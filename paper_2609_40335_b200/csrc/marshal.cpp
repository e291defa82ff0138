// Native half of the binding's argument marshalling: the per-layer records of a call, read from the
// Python objects in one pass.  Each torch attribute read from Python costs about 0.12 us and a layer
// needs a dozen; with a hundred layers that was most of a step's host time (2.3 us per layer in
// Python, 0.3 us here).  No device work, nothing is kept between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "../../include/dp_ghost.h"

namespace {

// base pointer and leading dimension of a (..., ld) CUDA tensor whose leading axes are densely packed;
// false: the caller's Python check words the complaint
bool rows(PyObject* o, const void** ptr, int64_t* ld, int64_t* cols) {
  if (!THPVariable_Check(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  const auto st = t.strides();
  const size_t n = st.size();
  if (!t.is_cuda() || n < 2 || st[n - 1] != 1) return false;
  if (n == 3 && st[0] != t.size(1) * st[1]) return false;
  *ptr = t.const_data_ptr();
  *ld = st[n - 2];
  *cols = t.size(int64_t(n) - 1);
  return true;
}

// integer attribute; None gives `otherwise`
bool integer(PyObject* o, const char* name, int64_t otherwise, int64_t* out) {
  PyObject* v = PyObject_GetAttrString(o, name);
  if (!v) { PyErr_Clear(); return false; }
  *out = v == Py_None ? otherwise : PyLong_AsLongLong(v);
  Py_DECREF(v);
  if (PyErr_Occurred()) { PyErr_Clear(); return false; }
  return true;
}

bool attr_rows(PyObject* o, const char* name, const void** ptr, int64_t* ld, int64_t* cols) {
  PyObject* v = PyObject_GetAttrString(o, name);
  if (!v) { PyErr_Clear(); return false; }
  const bool ok = rows(v, ptr, ld, cols);
  Py_DECREF(v);
  return ok;
}

// f(record, object) over a sequence -> bytearray of records, or None if a tensor is not usable
template <typename Rec, typename F>
PyObject* records(PyObject* arg, F f) {
  PyObject* seq = PySequence_Fast(arg, "a sequence");
  if (!seq) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
  PyObject* out = PyByteArray_FromStringAndSize(nullptr, n * Py_ssize_t(sizeof(Rec)));
  if (!out) { Py_DECREF(seq); return nullptr; }
  auto* rec = reinterpret_cast<Rec*>(PyByteArray_AS_STRING(out));
  memset(static_cast<void*>(rec), 0, size_t(n) * sizeof(Rec));
  bool ok = true;
  for (Py_ssize_t k = 0; k < n && ok; ++k) ok = f(rec[k], PySequence_Fast_GET_ITEM(seq, k));
  Py_DECREF(seq);
  if (!ok) { Py_DECREF(out); Py_RETURN_NONE; }
  return out;
}

// linears(sequence of Linear) -> dp_linear_desc[]
PyObject* linears(PyObject*, PyObject* arg) {
  return records<dp_linear_desc>(arg, [](dp_linear_desc& L, PyObject* o) {
    int64_t ca = 0, cg = 0, d = 0, p = 0, mode = 0;
    const bool ok = attr_rows(o, "A", &L.A, &L.lda, &ca) && attr_rows(o, "G", &L.G, &L.ldg, &cg) &&
                    integer(o, "d", ca, &d) && integer(o, "p", cg, &p) && integer(o, "mode", 0, &mode);
    L.d = int32_t(d); L.p = int32_t(p); L.mode = int32_t(mode); L.mode_used = -1;
    return ok;
  });
}

// vectors(sequence of Vector) -> dp_vector_desc[]
PyObject* vectors(PyObject*, PyObject* arg) {
  return records<dp_vector_desc>(arg, [](dp_vector_desc& v, PyObject* o) {
    int64_t cols = 0, other = 0, p = 0;
    bool ok = attr_rows(o, "G", &v.G, &v.ldg, &cols) && integer(o, "p", cols, &p);
    PyObject* x = PyObject_GetAttrString(o, "X");
    if (!x) { PyErr_Clear(); return false; }
    if (x != Py_None) ok = ok && rows(x, &v.X, &v.ldx, &other);
    Py_DECREF(x);
    v.p = int32_t(p);
    return ok;
  });
}

// outputs(sequence of CUDA tensors) -> bytearray: n pointers, then n leading strides; or None
PyObject* outputs(PyObject*, PyObject* arg) {
  PyObject* seq = PySequence_Fast(arg, "a sequence of tensors");
  if (!seq) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
  PyObject* out = PyByteArray_FromStringAndSize(nullptr, 16 * n);
  if (!out) { Py_DECREF(seq); return nullptr; }
  auto* w = reinterpret_cast<int64_t*>(PyByteArray_AS_STRING(out));
  bool ok = true;
  for (Py_ssize_t k = 0; k < n; ++k) {
    PyObject* o = PySequence_Fast_GET_ITEM(seq, k);
    ok = THPVariable_Check(o) && THPVariable_Unpack(o).is_cuda();
    if (!ok) break;
    const at::Tensor& t = THPVariable_Unpack(o);
    w[k] = reinterpret_cast<int64_t>(t.const_data_ptr());
    w[n + k] = t.dim() > 0 ? t.stride(0) : 0;
  }
  Py_DECREF(seq);
  if (!ok) { Py_DECREF(out); Py_RETURN_NONE; }
  return out;
}

PyMethodDef methods[] = {{"linears", linears, METH_O, nullptr},
                         {"vectors", vectors, METH_O, nullptr},
                         {"outputs", outputs, METH_O, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&module); }
