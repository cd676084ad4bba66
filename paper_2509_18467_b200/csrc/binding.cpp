// CPython module behind api.py: turns torch tensors into the device pointers of a C entry point and calls it. A decode step
// takes thirteen tensors; marshalling them through ctypes objects cost 25 us of host time per call, more than the kernels of
// a small step, and about a microsecond here.
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/torch.h>

#include <cstdint>

namespace {

constexpr int MAX_PTRS = 20;

// None and empty tensors are NULL, anything else must be a contiguous CUDA tensor. False with a Python error set otherwise.
bool argument(PyObject* o, void** out) {
  *out = nullptr;
  if (o == Py_None) return true;
  if (!THPVariable_Check(o)) {
    PyErr_SetString(PyExc_TypeError, "expected a tensor or None");
    return false;
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  if (t.numel() == 0) return true;
  if (!t.is_cuda() || !t.is_contiguous()) {
    PyErr_SetString(PyExc_AssertionError, "tensors must be contiguous CUDA tensors");
    return false;
  }
  *out = t.data_ptr();
  return true;
}

template <size_t... I>
int call_n(void* fn, const void* p, void* const* a, void* ws, size_t nb, void* st, void* ds, std::index_sequence<I...>) {
  using F = int (*)(const void*, decltype((void)I, (void*)nullptr)..., void*, size_t, void*, void*);
  return reinterpret_cast<F>(fn)(p, a[I]..., ws, nb, st, ds);
}

// call(fn, params, ws_fn, op, args, ws, stream, dev_status, nint = 0) -> status
//   fn: address of an entry point fn(params, args..., ws, ws_bytes, stream, dev_status)
//   args: tensors or None, behind `nint` integers that are passed as they are (sizes, the address of a host array)
//   ws_fn(params, op): its scratch bytes; op = -1: ws_fn is that number itself
//   ws: scratch tensor, or None to take it from torch's allocator for the duration of the call
//   stream: cudaStream_t as an integer, or None for the current stream of the current device
// The library's call runs without the interpreter lock: it stands while the device's launch queue is full or a kernel's module
// is loaded, and other Python threads go on meanwhile.
PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs < 8 || nargs > 9 || !PyTuple_Check(args[4])) {
    PyErr_SetString(PyExc_TypeError, "call(fn, params, ws_fn, op, args, ws, stream, dev_status, nint = 0)");
    return nullptr;
  }
  void* fn = PyLong_AsVoidPtr(args[0]);
  const void* p = PyLong_AsVoidPtr(args[1]);
  const size_t ws_arg = PyLong_AsSize_t(args[2]);
  const int op = (int)PyLong_AsLong(args[3]);
  const Py_ssize_t nint = nargs > 8 ? PyLong_AsSsize_t(args[8]) : 0;
  if (PyErr_Occurred()) return nullptr;
  const Py_ssize_t n = PyTuple_GET_SIZE(args[4]);
  if (n < 1 || n > MAX_PTRS || nint < 0 || nint > n) {
    PyErr_SetString(PyExc_TypeError, "number of arguments");
    return nullptr;
  }
  void* a[MAX_PTRS];
  for (Py_ssize_t i = 0; i < nint; ++i) {
    a[i] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(args[4], i));
    if (PyErr_Occurred()) return nullptr;
  }
  for (Py_ssize_t i = nint; i < n; ++i)
    if (!argument(PyTuple_GET_ITEM(args[4], i), &a[i])) return nullptr;
  void *ws = nullptr, *ds = nullptr, *st = nullptr;
  if (!argument(args[5], &ws) || !argument(args[7], &ds)) return nullptr;
  size_t nb = 0;
  at::Tensor scratch;
  try {
    if (args[5] != Py_None) {
      nb = THPVariable_Unpack(args[5]).nbytes();
    } else {
      nb = op < 0 ? ws_arg : reinterpret_cast<size_t (*)(const void*, int)>(ws_arg)(p, op);
      if (nb) {
        c10::Device dev(c10::kCUDA);
        for (Py_ssize_t i = nint; i < n; ++i)
          if (THPVariable_Check(PyTuple_GET_ITEM(args[4], i))) {
            dev = THPVariable_Unpack(PyTuple_GET_ITEM(args[4], i)).device();
            break;
          }
        scratch = at::empty({(int64_t)nb}, at::TensorOptions().dtype(at::kByte).device(dev));
        ws = scratch.data_ptr();
      }
    }
    if (args[6] != Py_None) st = PyLong_AsVoidPtr(args[6]);
    else if (c10::cuda::device_count() > 0) st = c10::cuda::getCurrentCUDAStream().stream();
    // the scratch goes back to the allocator when this call returns, and the allocator hands it on in the order of the current
    // stream: on another one it has to know how long the block is in use
    if (scratch.defined()) {
      const c10::DeviceIndex dev = scratch.device().index();
      if (st != (void*)c10::cuda::getCurrentCUDAStream(dev).stream())
        scratch.record_stream(c10::cuda::getStreamFromExternal((cudaStream_t)st, dev).unwrap());
    }
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
  if (PyErr_Occurred()) return nullptr;
  int r = 0;
  Py_BEGIN_ALLOW_THREADS
  switch (n) {
#define N(k) case k: r = call_n(fn, p, a, ws, nb, st, ds, std::make_index_sequence<k>{}); break;
    N(1) N(2) N(3) N(4) N(5) N(6) N(7) N(8) N(9) N(10) N(11) N(12) N(13) N(14) N(15) N(16) N(17) N(18) N(19) N(20)
#undef N
  }
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(r);
}

// empty(like, dtype, sizes...) -> tensor on like's device; dtype: 0 fp32, 1 bf16
PyObject* empty(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs < 3 || nargs > 7 || !THPVariable_Check(args[0])) {
    PyErr_SetString(PyExc_TypeError, "empty(like, dtype, sizes...)");
    return nullptr;
  }
  int64_t sz[5];
  for (Py_ssize_t i = 2; i < nargs; ++i) sz[i - 2] = PyLong_AsLongLong(args[i]);
  const long dt = PyLong_AsLong(args[1]);
  if (PyErr_Occurred()) return nullptr;
  try {
    return THPVariable_Wrap(at::empty(at::IntArrayRef(sz, (size_t)nargs - 2),
                                      at::TensorOptions().dtype(dt ? at::kBFloat16 : at::kFloat).device(THPVariable_Unpack(args[0]).device())));
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyMethodDef methods[] = {
    {"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call an entry point of the CUDA library"},
    {"empty", (PyCFunction)(void (*)(void))empty, METH_FASTCALL, "uninitialised tensor"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&module); }
