// Marshalling of verify()'s arguments from torch tensors to lantern_verify_ex, natively.  The binding does the same through ctypes, where
// a call of two launches cost 16.4 us of host time, more than the GPU needs for it; here it only recognises
// calls that need nothing but their pointers taken (all outputs and the workspace given, tensors of the right types on the current
// device) and answers None to everything else, which the binding then handles itself, errors included.
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>

#include "lantern.h"

namespace {

using VerifyFn = decltype(&lantern_verify_ex);
VerifyFn g_verify = nullptr;

// bind(address of lantern_verify_ex)
PyObject* bind(PyObject*, PyObject* address) {
  void* p = PyLong_AsVoidPtr(address);
  if (!p && PyErr_Occurred()) return nullptr;
  g_verify = reinterpret_cast<VerifyFn>(p);
  Py_RETURN_NONE;
}

// The pointer of an optional tensor; false if it is anything but a contiguous one of that type on that device.
bool pointer(PyObject* o, at::ScalarType type, int device, void** out) {
  *out = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_CheckExact(o)) return false;   // (a subclass may have no memory of its own)
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_cuda() || t.get_device() != device || t.scalar_type() != type || !t.is_contiguous()) return false;
  *out = t.data_ptr();
  return true;
}
bool attribute(PyObject* o, PyObject* name, at::ScalarType type, int device, void** out) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (!v) {
    PyErr_Clear();
    return false;
  }
  const bool ok = pointer(v, type, device, out);   // (the attribute keeps the tensor alive)
  Py_DECREF(v);
  return ok;
}

// names of VerifyOutputs' fields
enum { LEN, TOKEN, PATH, STATUS, QA, PX, M, FIELDS };
PyObject* g_names[FIELDS];

// verify(target, draft, cfg_scale, T, tokens, parents, neighbors, delta, uniforms, out, workspace, divergence, top_k) -> status or None
PyObject* call_verify(PyObject* const* a, Py_ssize_t n) {
  if (n != 13 || !g_verify) Py_RETURN_NONE;
  if (!THPVariable_CheckExact(a[0]) || !THPVariable_CheckExact(a[6]) || !THPVariable_CheckExact(a[10]) || !PyLong_CheckExact(a[11]) || !PyLong_CheckExact(a[12]))
    Py_RETURN_NONE;
  double scalar[3];
  const int at_scalar[3] = {2, 3, 7};
  for (int i = 0; i < 3; ++i) {
    PyObject* v = a[at_scalar[i]];
    if (PyFloat_CheckExact(v)) scalar[i] = PyFloat_AS_DOUBLE(v);
    else if (PyLong_CheckExact(v)) scalar[i] = PyLong_AsDouble(v);
    else Py_RETURN_NONE;
  }
  const long divergence = PyLong_AsLong(a[11]), top_k = PyLong_AsLong(a[12]);
  if (PyErr_Occurred() || top_k != static_cast<int>(top_k)) {
    PyErr_Clear();
    Py_RETURN_NONE;
  }
  const at::Tensor& target = THPVariable_Unpack(a[0]);
  const at::Tensor& neighbors = THPVariable_Unpack(a[6]);
  const at::Tensor& workspace = THPVariable_Unpack(a[10]);
  if (!target.is_cuda() || target.dim() != 4 || neighbors.dim() != 2) Py_RETURN_NONE;
  const int device = target.get_device();
  const at::ScalarType type = target.scalar_type();
  const int64_t C = target.size(0), B = target.size(1), R = target.size(2), V = target.size(3), k = neighbors.size(1);
  if ((type != at::kBFloat16 && type != at::kFloat) || (C != 1 && C != 2) || R < 1 || neighbors.size(0) != V || B > INT32_MAX || V > INT32_MAX ||
      R > INT32_MAX || device != c10::cuda::current_device())
    Py_RETURN_NONE;
  const bool sampling = scalar[1] != 0.0;
  if (sampling && (a[8] == Py_None || (a[1] == Py_None && R > 1))) Py_RETURN_NONE;
  void *p_target, *p_draft, *p_tokens, *p_parents, *p_neighbors, *p_uniforms, *p_out[FIELDS], *p_workspace;
  if (!pointer(a[0], type, device, &p_target) || !pointer(a[1], type, device, &p_draft) || !pointer(a[4], at::kInt, device, &p_tokens) ||
      !pointer(a[5], at::kInt, device, &p_parents) || !pointer(a[6], at::kInt, device, &p_neighbors) ||
      !pointer(a[8], at::kFloat, device, &p_uniforms) || !pointer(a[10], at::kByte, device, &p_workspace))
    Py_RETURN_NONE;
  for (int f = 0; f < FIELDS; ++f)
    if (!attribute(a[9], g_names[f], f == QA || f == PX ? at::kFloat : at::kInt, device, &p_out[f])) Py_RETURN_NONE;
  const size_t workspace_bytes = static_cast<size_t>(workspace.numel());
  lantern_status rc;
  cudaStream_t stream = c10::cuda::getCurrentCUDAStream(device).stream();
  Py_BEGIN_ALLOW_THREADS
  rc = g_verify(p_target, p_draft, type == at::kBFloat16 ? LANTERN_BF16 : LANTERN_F32, static_cast<float>(scalar[0]), C == 2,
                static_cast<float>(scalar[1]), static_cast<const int32_t*>(p_tokens), static_cast<const int32_t*>(p_parents),
                static_cast<const int32_t*>(p_neighbors), static_cast<int>(k), static_cast<float>(scalar[2]), static_cast<int>(divergence),
                static_cast<int>(top_k), static_cast<const float*>(p_uniforms), static_cast<int>(B), static_cast<int>(R - 1), static_cast<int>(V),
                static_cast<int32_t*>(p_out[LEN]), static_cast<int32_t*>(p_out[TOKEN]), static_cast<int32_t*>(p_out[PATH]),
                static_cast<int32_t*>(p_out[STATUS]), static_cast<float*>(p_out[QA]), static_cast<float*>(p_out[PX]),
                static_cast<int32_t*>(p_out[M]), p_workspace, workspace_bytes, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

PyObject* verify(PyObject*, PyObject* const* a, Py_ssize_t n) {
  try {
    return call_verify(a, n);
  } catch (...) {   // (a tensor without memory that can be read, say: the binding finds out)
    PyErr_Clear();
    Py_RETURN_NONE;
  }
}

PyMethodDef kMethods[] = {
    {"bind", bind, METH_O, nullptr},
    {"verify", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(verify)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_call", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call() {
  const char* names[FIELDS] = {"accept_len", "next_token", "accept_path", "status", "node_qa", "node_px", "node_m"};
  for (int f = 0; f < FIELDS; ++f) {
    g_names[f] = PyUnicode_InternFromString(names[f]);
    if (!g_names[f]) return nullptr;
  }
  return PyModule_Create(&kModule);
}
