// The forward's arguments from Python objects to the C entry point.  A scoring request of 48 samples is one launch
// of 2 us; handing twelve arguments over through ctypes and asking tensors for their addresses from Python took longer
// than that (5.3 us a call in all, 2.6 this way).
#define PY_SSIZE_T_CLEAN
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "antdt.h"

namespace {

using Fwd = decltype(&antdt_embbag_fwd);
Fwd g_fwd = nullptr;  // bound once, when the library is loaded
constexpr long kNotPlain = -1;

bool plain(PyObject* o) { return THPVariable_CheckExact(o) && THPVariable_Unpack(o).is_contiguous(); }

// embbag_fwd(table, row_ids, bag_offsets, pooled, dev_status or None, stream or None) -> status, or kNotPlain
// without a call where an argument is not a plain contiguous tensor: the caller's general way then says what is wrong.
PyObject* embbag_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 6 || !g_fwd || !plain(a[0]) || !plain(a[1]) || !plain(a[2]) || !plain(a[3]) || (a[4] != Py_None && !plain(a[4])))
    return PyLong_FromLong(kNotPlain);
  const at::Tensor &table = THPVariable_Unpack(a[0]), &ids = THPVariable_Unpack(a[1]), &off = THPVariable_Unpack(a[2]),
                   &pooled = THPVariable_Unpack(a[3]);
  const auto type = table.scalar_type();
  if (table.dim() != 2 || (type != at::kFloat && type != at::kBFloat16)) return PyLong_FromLong(kNotPlain);
  void* stream = nullptr;
  if (a[5] == Py_None) {
    stream = c10::cuda::getCurrentCUDAStream(c10::cuda::current_device()).stream();
  } else {
    PyObject* s = PyObject_GetAttrString(a[5], "cuda_stream");
    if (!s) return nullptr;
    stream = PyLong_AsVoidPtr(s);
    Py_DECREF(s);
    if (!stream && PyErr_Occurred()) return nullptr;
  }
  int32_t* const status = a[4] == Py_None ? nullptr : static_cast<int32_t*>(THPVariable_Unpack(a[4]).data_ptr());
  const int64_t dim = table.size(1), nnz = ids.numel(), n_bags = off.numel() - 1;
  const void* const t = table.const_data_ptr();
  const int32_t* const i = static_cast<const int32_t*>(ids.const_data_ptr());
  const int64_t* const o = static_cast<const int64_t*>(off.const_data_ptr());
  float* const p = static_cast<float*>(pooled.data_ptr());
  int32_t rc;
  Py_BEGIN_ALLOW_THREADS;
  rc = g_fwd(t, type == at::kBFloat16 ? ANTDT_BF16 : ANTDT_F32, table.size(0), (int32_t)dim, i, nnz, o, n_bags, p, status,
             stream);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(rc);
  END_HANDLE_TH_ERRORS
}

PyObject* bind(PyObject*, PyObject* address) {  // of antdt_embbag_fwd in the library that is loaded
  void* p = PyLong_AsVoidPtr(address);
  if (!p) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_ValueError, "no address");
  g_fwd = reinterpret_cast<Fwd>(p);
  Py_RETURN_NONE;
}

PyMethodDef kMethods[] = {
    {"embbag_fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(embbag_fwd)), METH_FASTCALL, nullptr},
    {"bind", bind, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, kMethods};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
  PyObject* m = PyModule_Create(&kModule);
  // the torch it was built against: with another one it is not used
  if (m && PyModule_AddStringConstant(m, "torch_version", ANTDT_TORCH) < 0) Py_CLEAR(m);
  return m;
}
