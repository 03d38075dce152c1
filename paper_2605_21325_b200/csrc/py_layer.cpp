// The marshalling of binding.gdn_forward in native code: shape checks, the two outputs, the workspace and the call, for the ordinary case of
// plain contiguous CUDA tensors on the current stream.  Whatever else comes (other types, other devices, arguments that convert) makes it return None, and the
// Python body of gdn_forward takes the call, with its conversions and its errors.
//
// A decode step is one kernel of 5.7 us; eight data pointers, a descriptor, two allocations and two calls through ctypes took 12.9 us of host time for it.
#include <torch/extension.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>

#include <climits>
#include <vector>

#include "tri_inv.h"

namespace {

using WorkspaceFn = int (*)(const tri_inv_desc*, int, size_t*);
using ForwardFn = int (*)(const void*, const void*, const void*, const float*, const float*, const float*, void*, float*, float, void*, size_t,
                          const tri_inv_desc*, int, void*);
WorkspaceFn g_workspace = nullptr;
ForwardFn g_forward = nullptr;

PyObject* bind(PyObject*, PyObject* args) {   // the addresses of tri_inv_gdn_forward_workspace and tri_inv_gdn_forward in the loaded library
  unsigned long long w = 0, f = 0;
  if (!PyArg_ParseTuple(args, "KK", &w, &f)) return nullptr;
  g_workspace = reinterpret_cast<WorkspaceFn>(w);
  g_forward = reinterpret_cast<ForwardFn>(f);
  Py_RETURN_NONE;
}

bool plain(PyObject* o, int dims) {
  if (!THPVariable_CheckExact(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.is_cuda() && t.layout() == at::kStrided && t.is_contiguous() && (dims == 0 || t.dim() == dims);
}
bool whole(PyObject* o, long lo, long hi, long* out) {
  if (!PyLong_CheckExact(o)) return false;
  int over = 0;
  *out = PyLong_AsLongAndOverflow(o, &over);
  return !over && *out >= lo && *out <= hi;
}

// (Q, K, V, beta, g, C, scale, S0, method, cu_seqlens) -> (O, S), None (not an ordinary call), or the failing call's status (+ 256: the workspace query's)
PyObject* gdn_forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  long C = 0, method = 0;
  if (n != 10 || !g_forward || !plain(a[0], 0) || !plain(a[1], 4) || !plain(a[2], 4) || !plain(a[3], 0) || !plain(a[4], 0) || !whole(a[5], INT_MIN, INT_MAX, &C) ||
      !PyFloat_CheckExact(a[6]) || !(a[7] == Py_None || plain(a[7], 0)) || !whole(a[8], INT_MIN, INT_MAX, &method))
    Py_RETURN_NONE;
  const at::Tensor &Q = THPVariable_Unpack(a[0]), &K = THPVariable_Unpack(a[1]), &V = THPVariable_Unpack(a[2]), &beta = THPVariable_Unpack(a[3]), &g = THPVariable_Unpack(a[4]);
  const bool f32 = K.scalar_type() == at::kFloat;
  if (!f32 && K.scalar_type() != at::kBFloat16) Py_RETURN_NONE;
  for (int i = 0; i < 4; ++i)
    if (K.size(i) > INT_MAX || V.size(i) > INT_MAX) Py_RETURN_NONE;
  tri_inv_desc d{};
  d.B = (int32_t)K.size(0); d.T = (int32_t)K.size(1); d.H = (int32_t)K.size(2); d.d_k = (int32_t)K.size(3); d.d_v = (int32_t)V.size(3);
  d.C = (int32_t)C;
  d.kv_dtype = f32 ? TRI_INV_F32 : TRI_INV_BF16;
  int64_t n_seqs = d.B;
  std::vector<int32_t> cu;
  if (a[9] != Py_None) {
    const bool list = PyList_CheckExact(a[9]);
    if (!list && !PyTuple_CheckExact(a[9])) Py_RETURN_NONE;
    const Py_ssize_t m = list ? PyList_GET_SIZE(a[9]) : PyTuple_GET_SIZE(a[9]);
    if (m < 1 || m > INT_MAX) Py_RETURN_NONE;
    cu.resize(m);
    for (Py_ssize_t i = 0; i < m; ++i) {
      long x = 0;
      if (!whole(list ? PyList_GET_ITEM(a[9], i) : PyTuple_GET_ITEM(a[9], i), INT_MIN, INT_MAX, &x)) Py_RETURN_NONE;
      cu[i] = (int32_t)x;
    }
    d.cu_seqlens = cu.data();
    d.n_seqs = (int32_t)(m - 1);
    n_seqs = m - 1;
  }
  size_t need = 0;
  int rc = g_workspace(&d, (int)method, &need);
  if (rc) return PyLong_FromLong(rc + 256);
  at::Tensor O = at::empty_like(V), S = at::empty({n_seqs, d.H, d.d_k, d.d_v}, K.options().dtype(at::kFloat)), work;
  if (need) work = at::empty({(int64_t)need}, K.options().dtype(at::kByte));
  const float* S0 = a[7] == Py_None ? nullptr : (const float*)THPVariable_Unpack(a[7]).data_ptr();
  const void *q = Q.data_ptr(), *k = K.data_ptr(), *v = V.data_ptr();
  const float *b = (const float*)beta.data_ptr(), *gg = (const float*)g.data_ptr();
  void *o = O.data_ptr(), *s = S.data_ptr(), *w = need ? work.data_ptr() : nullptr;
  void* stream = c10::cuda::getCurrentCUDAStream().stream();
  const float scale = (float)PyFloat_AS_DOUBLE(a[6]);
  Py_BEGIN_ALLOW_THREADS
  rc = g_forward(q, k, v, b, gg, S0, o, (float*)s, scale, w, need, &d, (int)method, stream);
  Py_END_ALLOW_THREADS
  if (rc) return PyLong_FromLong(rc);
  PyObject* out = PyTuple_New(2);
  if (!out) return nullptr;
  PyTuple_SET_ITEM(out, 0, THPVariable_Wrap(std::move(O)));
  PyTuple_SET_ITEM(out, 1, THPVariable_Wrap(std::move(S)));
  return out;
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, nullptr},
                         {"gdn_forward", (PyCFunction)(void (*)(void))gdn_forward, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
