// CPython extension behind binding.py: the two calls of the hot path with their arguments taken straight from the tensor
// objects.  Through ctypes a call is 30 to 60 Python-level operations (attributes, strides as a struct, data pointers, argument
// conversion), and a small call is all host time: append of 2 heads x 256 tokens 5.7 us, of which 2.4 on the GPU.
//
// It marshals and nothing else: the C entry points come in by address (bind), a call that is not the plain one - a tensor
// subclass, another dtype or layout, an integer-like object, whatever raises - is answered with kNotPlain, and binding.py takes
// its ctypes route, which checks and raises as it always has.
#include <Python.h>
#include <torch/csrc/autograd/python_variable.h>

#include "kvq.h"

namespace {

constexpr long long kNotPlain = -1000;               // not a status of kvq.h

decltype(&kvq_quantize_append) g_append;
decltype(&kvq_attn_workspace_bytes) g_workspace_bytes;
decltype(&kvq_attn_corrected) g_attn;

// A plain CUDA BF16 tensor [batch, heads, tokens, head_dim] with unit inner stride, or nullptr.
const at::Tensor* plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (t.scalar_type() != at::kBFloat16 || !t.is_cuda() || t.dim() != 4 || t.stride(3) != 1) return nullptr;
  return &t;
}
kvq_strides strides_of(const at::Tensor& t) { return {t.stride(0), t.stride(1), t.stride(2)}; }

// Device pointer of an optional tensor; false if the object is neither None nor a plain tensor.
bool optional_ptr(PyObject* o, void** out) {
  *out = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_CheckExact(o)) return false;
  *out = THPVariable_Unpack(o).data_ptr();
  return true;
}
// Integers as ctypes takes them: Python ints only, cut to the width of the parameter.
bool integer(PyObject* o, long long* out) {
  if (!PyLong_Check(o)) return false;
  *out = (long long)PyLong_AsUnsignedLongLongMask(o);
  return true;
}

PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  long long p[3];
  for (int i = 0; i < 3; ++i)
    if (n != 3 || !integer(a[i], &p[i])) { PyErr_SetString(PyExc_TypeError, "bind(append, workspace_bytes, attn): addresses"); return nullptr; }
  g_append = reinterpret_cast<decltype(g_append)>(p[0]);
  g_workspace_bytes = reinterpret_cast<decltype(g_workspace_bytes)>(p[1]);
  g_attn = reinterpret_cast<decltype(g_attn)>(p[2]);
  Py_RETURN_NONE;
}

// append(desc address, position, k, v, stream) -> status or kNotPlain
PyObject* append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  long long desc, pos, stream, r = kNotPlain;
  try {
    if (n == 5 && g_append && integer(a[0], &desc) && integer(a[1], &pos) && integer(a[4], &stream)) {
      const at::Tensor *k = plain(a[2]), *v = plain(a[3]);
      if (k && v && k->sizes() == v->sizes() && k->strides() == v->strides()) {
        const void *kp = k->data_ptr(), *vp = v->data_ptr();
        const kvq_strides st = strides_of(*k);
        const int64_t tokens = k->size(2);
        Py_BEGIN_ALLOW_THREADS
        r = g_append(reinterpret_cast<const kvq_cache_desc*>(desc), pos, kp, vp, st, tokens, reinterpret_cast<void*>(stream));
        Py_END_ALLOW_THREADS
      }
    }
  } catch (...) { r = kNotPlain; }
  return PyLong_FromLongLong(r);
}

// attn(desc address, begin, cached, q, k, v, out, scale, flags, lse, mass, status, workspace, stream)
// -> status, or the bytes of workspace the call needs and did not bring, or kNotPlain
PyObject* attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
  long long desc, begin, cached, flags, stream, r = kNotPlain;
  try {
    if (n == 14 && g_attn && integer(a[0], &desc) && integer(a[1], &begin) && integer(a[2], &cached) && PyFloat_CheckExact(a[7]) &&
        integer(a[8], &flags) && integer(a[13], &stream)) {
      const at::Tensor *q = plain(a[3]), *k = plain(a[4]), *v = plain(a[5]), *out = plain(a[6]);
      void *lse, *mass, *status;
      if (q && k && v && out && k->sizes() == v->sizes() && k->strides() == v->strides() && optional_ptr(a[9], &lse) &&
          optional_ptr(a[10], &mass) && optional_ptr(a[11], &status) && (a[12] == Py_None || THPVariable_CheckExact(a[12]))) {
        const kvq_cache_desc* d = reinterpret_cast<const kvq_cache_desc*>(desc);
        const int64_t m = q->size(2), n_cur = k->size(2);
        size_t need = 0;
        r = g_workspace_bytes(d, cached, m, n_cur, (uint32_t)flags, &need);
        if (r == KVQ_OK) {
          void* ws = nullptr;
          size_t have = 0;
          if (need && a[12] != Py_None) {
            const at::Tensor& w = THPVariable_Unpack(a[12]);
            have = (size_t)w.numel();
            if (have >= need) ws = w.data_ptr();
          }
          if (need && !ws) {
            r = (long long)need;
          } else {
            const void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr();
            void* op = out->data_ptr();
            const kvq_strides qs = strides_of(*q), ks = strides_of(*k), os = strides_of(*out);
            const float scale = (float)PyFloat_AS_DOUBLE(a[7]);
            Py_BEGIN_ALLOW_THREADS
            r = g_attn(d, begin, cached, qp, qs, kp, vp, ks, m, n_cur, op, os, scale, (uint32_t)flags, static_cast<float*>(lse),
                       static_cast<float*>(mass), ws, have, static_cast<int32_t*>(status), reinterpret_cast<void*>(stream));
            Py_END_ALLOW_THREADS
          }
        }
      }
    }
  } catch (...) { r = kNotPlain; }
  return PyLong_FromLongLong(r);
}

PyMethodDef methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&bind)), METH_FASTCALL, nullptr},
    {"append", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&append)), METH_FASTCALL, nullptr},
    {"attn", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&attn)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_py_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// Nothing of torch's layout is touched here: binding.py looks at built_for (the torch and the Python of the headers above) before it
// calls anything else.
PyMODINIT_FUNC PyInit__py_call(void) {
  PyObject* m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "built_for", KVQ_BUILT_FOR) < 0) { Py_DECREF(m); return nullptr; }
  return m;
}
