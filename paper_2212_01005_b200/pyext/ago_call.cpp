// The host path of one Subgraph.run call, native: tensors -> device pointers -> ago_subgraph_run.
//
// A run of a small subgraph takes 5 to 10 us on the GPU; marshalled in Python (pointer arrays built with ctypes, the
// current stream and the output allocated through torch's Python layer) the call itself took 12.5 to 16 us, so every
// small subgraph was bound by the host. Here the pointers are read from the tensors, the output comes from torch's
// allocator and the stream from its current-stream query without leaving C++. No computation, no device memory of
// its own, nothing kept between calls but the handle's constants.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <ATen/record_function.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <string>
#include <vector>

namespace {

// The C entry points, taken from the library that the ctypes binding loaded (struct layouts stay on that side).
using RunFn = int (*)(void*, const void* const*, const void* const*, void* const*, void*);
using ErrFn = int (*)(const char**);

constexpr int kMaxPtrs = 64;          // more than a handle has inputs (AGO_MAX_INPUTS) or weights (one per operator, AGO_MAX_OPS = 32)
constexpr int kErrInvalidArg = 1, kErrCuda = 6;

struct Runner {
  PyObject_HEAD
  vectorcallfunc vectorcall;
  void* handle;
  RunFn run;
  ErrFn last_error;
  PyObject* error;                    // the exception class raised for a status
  std::vector<int64_t>* shape;        // output
  at::ScalarType dtype;
  int64_t workspace_bytes;
  Py_ssize_t num_inputs, num_weights;
};

PyObject* raise(Runner* r, int status, const char* msg) {
  PyObject* e = PyObject_CallFunction(r->error, "is", status, msg);
  if (e) { PyErr_SetObject(r->error, e); Py_DECREF(e); }
  return nullptr;
}

// Device pointer of a tensor; of any other object, what its data_ptr() returns.
bool pointer_of(PyObject* o, const void** p) {
  if (THPVariable_Check(o)) { *p = THPVariable_Unpack(o).const_data_ptr(); return true; }
  PyObject* v = PyObject_CallMethod(o, "data_ptr", nullptr);
  if (!v) return false;
  *p = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

// Device of a tensor; of any other object, what its `device` names ("cuda:0").
bool device_of(PyObject* o, at::Device* dev) {
  if (THPVariable_Check(o)) { *dev = THPVariable_Unpack(o).device(); return true; }
  PyObject* d = PyObject_GetAttrString(o, "device");
  PyObject* name = d ? PyObject_Str(d) : nullptr;
  Py_XDECREF(d);
  const char* text = name ? PyUnicode_AsUTF8(name) : nullptr;
  const bool ok = text != nullptr;
  if (ok) *dev = at::Device(std::string(text));
  Py_XDECREF(name);
  return ok;
}

// A stream given as an address or as a ctypes pointer.
bool stream_of(PyObject* o, void** stream) {
  PyObject* v = PyLong_Check(o) ? Py_NewRef(o) : PyObject_GetAttrString(o, "value");
  if (!v) return false;
  *stream = v == Py_None ? nullptr : PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

// The output tensor, as at::empty makes it. Where nothing takes part in a factory call (no dispatch mode, transform, tracer or
// autocast on this thread, no deterministic fill, no profiler that records operators) and the device is the current one, without the
// dispatcher's way there: 0.3 us of a call's host time, which is what a small subgraph takes (fp32 depthwise stage 2 x 9 x 9 x 64
// 3.95 -> 3.6 us, depthwise pair 3.25 -> 2.95). The allocator needs torch's CUDA state, which nothing but this call may have asked
// for where all inputs are another library's arrays: initialised here as at::empty does it (a flag once that is done).
at::Tensor make_output(const Runner* r, at::Device dev) {
  const auto tls = c10::impl::tls_local_dispatch_key_set();
  if ((tls.included_ - c10::default_included_set).empty() && !at::globalContext().deterministicAlgorithms() && !at::hasCallbacks() &&
      dev.index() == c10::cuda::current_device()) {
    at::globalContext().lazyInitDevice(c10::DeviceType::CUDA);
    return at::Tensor(at::detail::empty_generic(*r->shape, c10::cuda::CUDACachingAllocator::get(), c10::DispatchKeySet(c10::DispatchKey::CUDA),
                                                r->dtype, std::nullopt));
  }
  return at::empty(*r->shape, at::TensorOptions().dtype(r->dtype).device(dev));
}

// Pointers of the first `need` tensors of a sequence. The tensors outlive the call: the caller holds the sequence.
bool pointers_of(Runner* r, PyObject* seq, Py_ssize_t need, const char* what, const void** out) {
  PyObject* fast = PySequence_Fast(seq, "inputs and weights are sequences of tensors");
  if (!fast) return false;
  PyObject** items = PySequence_Fast_ITEMS(fast);
  bool ok = need <= kMaxPtrs && PySequence_Fast_GET_SIZE(fast) >= need;
  if (!ok) raise(r, kErrInvalidArg, what);
  for (Py_ssize_t i = 0; ok && i < need; ++i) ok = pointer_of(items[i], out + i);
  Py_DECREF(fast);
  return ok;
}

// runner(inputs, weights, out, stream, workspace) -> output tensor, or None when the workspace has to be attached first
PyObject* call(PyObject* self, PyObject* const* args, size_t nargsf, PyObject* kw) {
  Runner* r = reinterpret_cast<Runner*>(self);
  if (PyVectorcall_NARGS(nargsf) != 5 || (kw && PyTuple_GET_SIZE(kw) != 0)) {
    PyErr_SetString(PyExc_TypeError, "runner(inputs, weights, out, stream, workspace)");
    return nullptr;
  }
  try {
    PyObject* first = PySequence_GetItem(args[0], 0);
    if (!first) return nullptr;
    at::Device dev(at::kCPU);
    const bool has_device = device_of(first, &dev);
    Py_DECREF(first);
    if (!has_device) return nullptr;
    if (!dev.is_cuda()) return raise(r, kErrCuda, "inputs must be CUDA tensors: this library has no CPU path");
    if (!dev.has_index()) dev.set_index(c10::cuda::current_device());
    if (r->workspace_bytes > 0) {
      if (args[4] == Py_None || !THPVariable_Check(args[4])) Py_RETURN_NONE;
      const at::Tensor& ws = THPVariable_Unpack(args[4]);
      if (ws.numel() < r->workspace_bytes || ws.device() != dev) Py_RETURN_NONE;
    }
    const void* in[kMaxPtrs];
    const void* w[kMaxPtrs];
    void* out[1];
    if (!pointers_of(r, args[0], r->num_inputs, "fewer inputs than the subgraph has", in)) return nullptr;
    if (!pointers_of(r, args[1], r->num_weights, "fewer weights than the subgraph has", w)) return nullptr;
    void* stream;
    if (args[3] == Py_None) stream = static_cast<void*>(c10::cuda::getCurrentCUDAStream(dev.index()).stream());
    else if (!stream_of(args[3], &stream)) return nullptr;
    PyObject* result;
    if (args[2] == Py_None) {
      at::Tensor t = make_output(r, dev);
      out[0] = t.mutable_data_ptr();
      result = THPVariable_Wrap(std::move(t));
      if (!result) return nullptr;
    } else {
      if (THPVariable_Check(args[2])) {
        out[0] = THPVariable_Unpack(args[2]).mutable_data_ptr();
      } else {
        const void* p;
        if (!pointer_of(args[2], &p)) return nullptr;
        out[0] = const_cast<void*>(p);
      }
      result = Py_NewRef(args[2]);
    }
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = r->run(r->handle, in, w, out, stream);
    Py_END_ALLOW_THREADS
    if (status != 0) {
      const char* msg = nullptr;
      const int code = r->last_error(&msg);
      Py_DECREF(result);
      return raise(r, code, msg ? msg : "");
    }
    return result;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

void dealloc(PyObject* self) {
  Runner* r = reinterpret_cast<Runner*>(self);
  delete r->shape;
  Py_XDECREF(r->error);
  Py_TYPE(self)->tp_free(self);
}

PyTypeObject RunnerType = {PyVarObject_HEAD_INIT(nullptr, 0)};

// make_runner(run, last_error, error class, handle, shape, is_fp32, workspace bytes, inputs, weights)
PyObject* make_runner(PyObject*, PyObject* a) {
  unsigned long long run, err, handle;
  PyObject *cls, *shape;
  int fp32;
  long long ws, ni, nw;
  if (!PyArg_ParseTuple(a, "KKOKO!pLLL", &run, &err, &cls, &handle, &PyTuple_Type, &shape, &fp32, &ws, &ni, &nw)) return nullptr;
  Runner* r = PyObject_New(Runner, &RunnerType);
  if (!r) return nullptr;
  r->vectorcall = call;
  r->handle = reinterpret_cast<void*>(static_cast<uintptr_t>(handle));
  r->run = reinterpret_cast<RunFn>(static_cast<uintptr_t>(run));
  r->last_error = reinterpret_cast<ErrFn>(static_cast<uintptr_t>(err));
  r->error = Py_NewRef(cls);
  r->shape = new std::vector<int64_t>();
  for (Py_ssize_t i = 0; i < PyTuple_GET_SIZE(shape); ++i) r->shape->push_back(PyLong_AsLongLong(PyTuple_GET_ITEM(shape, i)));
  r->dtype = fp32 ? at::kFloat : at::kBFloat16;
  r->workspace_bytes = ws;
  r->num_inputs = (Py_ssize_t)ni; r->num_weights = (Py_ssize_t)nw;
  if (PyErr_Occurred()) { Py_DECREF(r); return nullptr; }
  return reinterpret_cast<PyObject*>(r);
}

PyMethodDef methods[] = {{"make_runner", make_runner, METH_VARARGS, "A callable that runs one handle."}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_ago_call", "Native host path of Subgraph.run.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__ago_call(void) {
  RunnerType.tp_name = "_ago_call.Runner";
  RunnerType.tp_basicsize = sizeof(Runner);
  RunnerType.tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL;
  RunnerType.tp_vectorcall_offset = offsetof(Runner, vectorcall);
  RunnerType.tp_call = PyVectorcall_Call;
  RunnerType.tp_dealloc = dealloc;
  if (PyType_Ready(&RunnerType) < 0) return nullptr;
  return PyModule_Create(&module);
}
