// The matmul entry points' way from Python tensors to the C ABI: what binding.py does through ctypes, for plain calls.
//
// A small matmul takes 2 us on the device and 2 to launch; reading the tensors' attributes one by one from Python and marshalling eight
// arguments through ctypes took as long again (1 x 1024 x 1024, host-bound: 4.9 us a call, 2.8 with this and the plans remembered).
// matmul() and gemv_host() take the address of the library's function and the type that a descriptor must have, and return the
// library's return code, or None for anything that is not a plain call; binding.py then takes its own way, which also raises what there
// is to raise.  Nothing is kept between calls.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/razer.h"

namespace {

typedef int (*MatmulFn)(const razer_desc*, const void*, const void*, int, void*, void*, size_t, void*);
typedef int (*HostFn)(const razer_desc*, const void*, const void*, int, void*, void*, void*, void*, size_t, void*);

// The descriptor behind binding.RazerDesc (a ctypes structure: its memory through the buffer protocol).
struct Desc {
  Py_buffer view;
  bool held = false;
  const razer_desc* get(PyObject* type, PyObject* o) {
    if (reinterpret_cast<PyObject*>(Py_TYPE(o)) != type) return nullptr;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) {
      PyErr_Clear();
      return nullptr;
    }
    held = true;
    return view.len == (Py_ssize_t)sizeof(razer_desc) ? static_cast<const razer_desc*>(view.buf) : nullptr;
  }
  ~Desc() {
    if (held) PyBuffer_Release(&view);
  }
};

// Plain torch.Tensor or Parameter objects only: a subclass may have attributes of its own.
bool plain(PyObject* o) { return THPVariable_CheckExact(o); }
const at::Tensor& tensor(PyObject* o) { return THPVariable_Unpack(o); }
bool dense(const at::Tensor& t) { return t.has_storage() && t.layout() == at::kStrided; }

void* address(PyObject* o) {
  void* p = PyLong_Check(o) ? PyLong_AsVoidPtr(o) : nullptr;
  if (PyErr_Occurred()) PyErr_Clear();
  return p;
}

// matmul(function, descriptor type, desc, packed, x, y, workspace)
PyObject* matmul(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 7 || !plain(a[3]) || !plain(a[4]) || !plain(a[5]) || !plain(a[6])) Py_RETURN_NONE;
  const MatmulFn fn = reinterpret_cast<MatmulFn>(address(a[0]));
  if (!fn) Py_RETURN_NONE;
  try {
    const at::Tensor &packed = tensor(a[3]), &x = tensor(a[4]), &y = tensor(a[5]), &ws = tensor(a[6]);
    Desc d;
    const razer_desc* desc = d.get(a[1], a[2]);
    if (!desc || !dense(packed) || !dense(x) || !dense(y) || !dense(ws) || !x.is_cuda() || x.scalar_type() != at::kBFloat16 || x.dim() < 2 ||
        !x.is_contiguous() || x.size(1) != desc->K || x.size(0) > INT32_MAX)
      Py_RETURN_NONE;
    const int M = (int)x.size(0);
    void *p = packed.data_ptr(), *px = x.data_ptr(), *py = y.data_ptr(), *pw = ws.data_ptr(), *st = c10::cuda::getCurrentCUDAStream().stream();
    const size_t bytes = (size_t)ws.numel();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn(desc, p, px, M, py, pw, bytes, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
  } catch (const std::exception&) {
    Py_RETURN_NONE;
  }
}

// gemv_host(function, descriptor type, desc, packed, x_host, y_host, x_stage, y_stage, workspace)
PyObject* gemv_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 9) Py_RETURN_NONE;
  for (int i = 3; i < 9; ++i)
    if (!plain(a[i])) Py_RETURN_NONE;
  const HostFn fn = reinterpret_cast<HostFn>(address(a[0]));
  if (!fn) Py_RETURN_NONE;
  try {
    Desc d;
    const razer_desc* desc = d.get(a[1], a[2]);
    if (!desc) Py_RETURN_NONE;
    void* p[6];
    for (int i = 0; i < 6; ++i) {
      const at::Tensor& t = tensor(a[i + 3]);
      if (!dense(t) || ((i == 1 || i == 2) && t.is_cuda())) Py_RETURN_NONE;
      p[i] = t.data_ptr();
    }
    const at::Tensor& x = tensor(a[4]);
    if (x.dim() < 1 || x.size(0) > INT32_MAX) Py_RETURN_NONE;
    const int M = (int)x.size(0);
    const size_t bytes = (size_t)tensor(a[8]).numel();
    void* st = c10::cuda::getCurrentCUDAStream().stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn(desc, p[0], p[1], M, p[2], p[3], p[4], p[5], bytes, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
  } catch (const std::exception&) {
    Py_RETURN_NONE;
  }
}

PyMethodDef methods[] = {{"matmul", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(matmul)), METH_FASTCALL, nullptr},
                         {"gemv_host", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(gemv_host)), METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "razer_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_razer_call() { return PyModule_Create(&module); }
