// The binding's calls on torch tensors, in native code: argument checks, output and workspace tensors, the current
// stream, one call into the library.  The product of one token with a 4096 x 4096 layer takes the GPU 6 us; the same
// marshalling in Python with ctypes took 12.5, so a serving loop waited for its own calls (now about 4).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/CUDAContext.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>

#include "../../include/gwq.h"

bool gwq_takes_decode(const gwq_packed* P, gwq_dtype xd, int M);
cudaError_t gwq_copy_arrays(int count, const void* const* from, void* const* to, const size_t* bytes, cudaStream_t stream);

namespace {

PyObject* g_error = nullptr;   // binding.GwqError(status, where)

// Thrown where a Python exception has been set.
struct python_error {};
[[noreturn]] void fail(PyObject* type, const char* text) {
  PyErr_SetString(type, text);
  throw python_error();
}

[[noreturn]] void fail_status(gwq_status st, const char* where) {
  PyObject* e = g_error ? PyObject_CallFunction(g_error, "is", (int)st, where) : nullptr;
  if (e) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  } else if (!PyErr_Occurred()) {
    PyErr_SetString(PyExc_RuntimeError, where);
  }
  throw python_error();
}
void check(gwq_status st, const char* where) {
  if (st != GWQ_OK) fail_status(st, where);
}

// Runs f; what it throws becomes a Python exception.
template <class F>
PyObject* guarded(F f) {
  try {
    return f();
  } catch (const python_error&) {
  } catch (const c10::Error& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
  }
  return nullptr;
}

// The library call without the interpreter lock, as ctypes makes it.
struct no_gil {
  PyThreadState* state = PyEval_SaveThread();
  ~no_gil() { PyEval_RestoreThread(state); }
};

const at::Tensor& tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
    throw python_error();
  }
  return THPVariable_Unpack(o);
}

const at::Tensor& cuda_tensor(PyObject* o, const char* name) {
  const at::Tensor& t = tensor(o, name);
  if (!t.is_cuda()) {
    PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor (no CPU path exists)", name);
    throw python_error();
  }
  if (!t.is_contiguous()) {
    PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
    throw python_error();
  }
  return t;
}

gwq_dtype dtype_code(at::ScalarType t) {
  if (t == at::kHalf) return GWQ_F16;
  if (t == at::kBFloat16) return GWQ_BF16;
  if (t == at::kFloat) return GWQ_F32;
  PyErr_Format(PyExc_TypeError, "unsupported dtype %s", c10::toString(t));
  throw python_error();
}

at::ScalarType dtype_of(PyObject* o) {
  if (!THPDtype_Check(o)) fail(PyExc_TypeError, "out_dtype must be a torch.dtype");
  return reinterpret_cast<THPDtype*>(o)->scalar_type;
}

// The object behind an address that the binding's Outliers / Packed hold (0 once freed).
template <class T>
T* object(PyObject* o) {
  void* p = PyLong_AsVoidPtr(o);
  if (!p) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_AttributeError, "the object has been freed");
    throw python_error();
  }
  return static_cast<T*>(p);
}

long device_index(PyObject* o) {
  const long index = PyLong_AsLong(o);
  if (index < 0) throw python_error();
  return index;
}

at::Tensor empty(at::IntArrayRef size, at::ScalarType type, at::Device device) {
  return at::detail::empty_cuda(size, type, device, std::nullopt);
}

size_t bytes_of(const at::Tensor& t) { return (size_t)t.numel() * t.element_size(); }

void need_args(Py_ssize_t n, Py_ssize_t want) {
  if (n != want) fail(PyExc_TypeError, "wrong number of arguments");
}

// The workspace of a call that needs `need` bytes: the caller's where it is large enough, else a new tensor; undefined
// where none is needed and none was given.
at::Tensor workspace_for(PyObject* given, size_t need, at::Device device) {
  at::Tensor ws;
  if (given != Py_None) ws = tensor(given, "workspace");
  if (need > 0 && (!ws.defined() || bytes_of(ws) < need)) ws = empty({(int64_t)need}, at::kByte, device);
  return ws;
}

void run_linear(const gwq_packed* P, const at::Tensor& x, gwq_dtype xd, const at::Tensor& out, const at::Tensor& ws,
                cudaStream_t stream) {
  const gwq_dtype yd = dtype_code(out.scalar_type());
  const int32_t M = (int32_t)x.size(0);
  const void* px = x.data_ptr();
  void *py = out.data_ptr(), *pw = ws.defined() ? ws.data_ptr() : nullptr;
  const size_t wb = ws.defined() ? bytes_of(ws) : 0;
  gwq_status st;
  {
    no_gil released;
    st = gwq_linear_ws(P, px, xd, M, py, yd, pw, wb, stream);
  }
  check(st, "gwq_linear");
}

// linear(P, x, out_dtype, out, workspace)
PyObject* py_linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 5);
    const at::Tensor& x = cuda_tensor(a[1], "x");
    const gwq_packed* P = object<const gwq_packed>(a[0]);
    if (x.dim() != 2 || x.size(1) != P->K) fail(PyExc_ValueError, "x must be [M, K]");
    const bool make = a[3] == Py_None;
    at::Tensor out = make ? empty({x.size(0), P->N}, a[2] == Py_None ? x.scalar_type() : dtype_of(a[2]), x.device())
                          : cuda_tensor(a[3], "out");
    const gwq_dtype xd = dtype_code(x.scalar_type());
    const size_t need = xd == GWQ_F32 ? 0 : gwq_linear_workspace_bytes(P, xd, (int32_t)x.size(0));
    run_linear(P, x, xd, out, workspace_for(a[4], need, x.device()), at::cuda::getCurrentCUDAStream());
    if (!make) {
      Py_INCREF(a[3]);
      return a[3];
    }
    return THPVariable_Wrap(std::move(out));
  });
}

// linear_multi([P, ...], x, out_dtype, outs, workspace) -> outs
PyObject* py_linear_multi(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 5);
    const at::Tensor& x = cuda_tensor(a[1], "x");
    if (!PyList_Check(a[0]) || (a[3] != Py_None && !PyList_Check(a[3]))) fail(PyExc_TypeError, "lists are expected");
    const Py_ssize_t count = PyList_GET_SIZE(a[0]);
    std::vector<const gwq_packed*> P(count);
    bool same = x.dim() == 2;
    for (Py_ssize_t i = 0; i < count; ++i) {
      P[i] = object<const gwq_packed>(PyList_GET_ITEM(a[0], i));
      same = same && P[i]->K == x.size(1);
    }
    if (!same) fail(PyExc_ValueError, "x must be [M, K] with the K of every layer");
    const bool make = a[3] == Py_None;
    std::vector<at::Tensor> outs;
    outs.reserve(count);
    if (make) {
      const at::ScalarType type = a[2] == Py_None ? x.scalar_type() : dtype_of(a[2]);
      for (Py_ssize_t i = 0; i < count; ++i) outs.push_back(empty({x.size(0), P[i]->N}, type, x.device()));
    } else {
      for (Py_ssize_t i = 0; i < PyList_GET_SIZE(a[3]); ++i) outs.push_back(cuda_tensor(PyList_GET_ITEM(a[3], i), "out"));
    }
    bool fits = (Py_ssize_t)outs.size() == count;
    for (const at::Tensor& o : outs) fits = fits && o.scalar_type() == outs[0].scalar_type();
    if (!fits) fail(PyExc_ValueError, "one output per layer, all of one dtype");
    const gwq_dtype xd = dtype_code(x.scalar_type());
    const int32_t M = (int32_t)x.size(0);
    const cudaStream_t stream = at::cuda::getCurrentCUDAStream();
    // more layers than one call takes: one by one, on one workspace (stream order), where it is the tensor-core kernels that want it
    size_t alone = 0;
    for (Py_ssize_t i = 0; i < count && count > GWQ_MULTI_MAX && xd != GWQ_F32; ++i)
      if (!gwq_takes_decode(P[i], xd, M)) alone = std::max(alone, gwq_linear_workspace_bytes(P[i], xd, M));
    if (alone > 0) {
      for (Py_ssize_t i = 0; i < count; ++i) alone = std::max(alone, gwq_linear_workspace_bytes(P[i], xd, M));
      const at::Tensor ws = workspace_for(a[4], alone, x.device());
      for (Py_ssize_t i = 0; i < count; ++i) run_linear(P[i], x, xd, outs[i], ws, stream);
    } else {
      std::vector<void*> y(std::max<Py_ssize_t>(count, 1), nullptr);
      for (Py_ssize_t i = 0; i < count; ++i) y[i] = outs[i].data_ptr();
      const gwq_dtype yd = count ? dtype_code(outs[0].scalar_type()) : GWQ_F16;
      const void* px = x.data_ptr();
      P.resize(std::max<Py_ssize_t>(count, 1), nullptr);
      const at::Tensor ws = workspace_for(a[4], gwq_linear_multi_workspace_bytes(P.data(), (int32_t)count, xd, M), x.device());
      void* pw = ws.defined() ? ws.data_ptr() : nullptr;
      const size_t wb = ws.defined() ? bytes_of(ws) : 0;
      gwq_status st;
      {
        no_gil released;
        st = gwq_linear_multi_ws(P.data(), (int32_t)count, px, xd, M, y.data(), yd, pw, wb, stream);
      }
      check(st, "gwq_linear_multi");
    }
    if (!make) {
      Py_INCREF(a[3]);
      return a[3];
    }
    PyObject* list = PyList_New(count);
    if (!list) throw python_error();
    for (Py_ssize_t i = 0; i < count; ++i) PyList_SET_ITEM(list, i, THPVariable_Wrap(std::move(outs[i])));
    return list;
  });
}

// linear_host(P, device index, x, y, asynchronous)
PyObject* py_linear_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 5);
    const bool async = a[4] == Py_True;
    const char* where = async ? "gwq_linear_host_async" : "gwq_linear_host";
    const at::Tensor &x = tensor(a[2], "x_host"), &y = tensor(a[3], "y_host");
    if (x.is_cuda() || y.is_cuda()) {
      PyErr_Format(PyExc_ValueError, "%s takes host tensors", where);
      throw python_error();
    }
    gwq_packed* P = object<gwq_packed>(a[0]);
    const c10::cuda::CUDAGuard on((c10::DeviceIndex)device_index(a[1]));
    const gwq_dtype xd = dtype_code(x.scalar_type()), yd = dtype_code(y.scalar_type());
    const int32_t M = (int32_t)x.size(0);
    const void* px = x.data_ptr();
    void* py = y.data_ptr();
    const cudaStream_t stream = at::cuda::getCurrentCUDAStream();
    gwq_status st;
    {
      no_gil released;
      st = (async ? gwq_linear_host_async : gwq_linear_host)(P, px, xd, M, py, yd, stream);
    }
    check(st, where);
    Py_INCREF(a[3]);
    return a[3];
  });
}

// Encoding -----------------------------------------------------------------------------------------------------------

// select(W, G, frac) -> address of the outlier object
PyObject* py_select(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 3);
    const at::Tensor &W = cuda_tensor(a[0], "W"), &G = cuda_tensor(a[1], "G");
    if (W.scalar_type() != at::kHalf || G.scalar_type() != at::kFloat || W.dim() != 2 || W.sizes() != G.sizes())
      fail(PyExc_ValueError, "W must be fp16 [N,K] and G fp32 [N,K]");
    const double frac = PyFloat_AsDouble(a[2]);
    if (frac == -1.0 && PyErr_Occurred()) throw python_error();
    const c10::cuda::CUDAGuard on(W.device());
    const uint16_t* w = static_cast<const uint16_t*>(W.data_ptr());
    const float* g = static_cast<const float*>(G.data_ptr());
    const int32_t N = (int32_t)W.size(0), K = (int32_t)W.size(1);
    const cudaStream_t stream = at::cuda::getCurrentCUDAStream();
    gwq_outliers* S = nullptr;
    gwq_status st;
    {
      no_gil released;
      st = gwq_select_outliers(w, g, N, K, frac, &S, stream);
    }
    check(st, "gwq_select_outliers");
    return PyLong_FromVoidPtr(S);
  });
}

// pack(W, S, bits, group) -> address of the packed layer (which owns S from then on)
PyObject* py_pack(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 4);
    const at::Tensor& W = cuda_tensor(a[0], "W");
    if (W.scalar_type() != at::kHalf || W.dim() != 2) fail(PyExc_ValueError, "W must be fp16 [N,K]");
    gwq_outliers* S = static_cast<gwq_outliers*>(PyLong_AsVoidPtr(a[1]));
    const long bits = PyLong_AsLong(a[2]), group = PyLong_AsLong(a[3]);
    if (PyErr_Occurred()) throw python_error();
    const c10::cuda::CUDAGuard on(W.device());
    const uint16_t* w = static_cast<const uint16_t*>(W.data_ptr());
    const int32_t N = (int32_t)W.size(0), K = (int32_t)W.size(1);
    const cudaStream_t stream = at::cuda::getCurrentCUDAStream();
    gwq_packed* P = nullptr;
    gwq_status st;
    {
      no_gil released;
      st = gwq_pack(w, S, N, K, (int32_t)bits, (int32_t)group, &P, stream);
    }
    check(st, "gwq_pack");
    return PyLong_FromVoidPtr(P);
  });
}

// gradient_mean([G, ...], out) -> out
PyObject* py_gradient_mean(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 2);
    if (!PyList_Check(a[0])) fail(PyExc_TypeError, "a list of gradients is expected");
    const Py_ssize_t count = PyList_GET_SIZE(a[0]);
    if (count < 1) fail(PyExc_ValueError, "at least one gradient");
    std::vector<const float*> g(count);
    const at::Tensor& first = cuda_tensor(PyList_GET_ITEM(a[0], 0), "G");
    for (Py_ssize_t i = 0; i < count; ++i) {
      const at::Tensor& t = cuda_tensor(PyList_GET_ITEM(a[0], i), "G");
      if (t.scalar_type() != at::kFloat || t.sizes() != first.sizes())
        fail(PyExc_ValueError, "gradients must be contiguous fp32 tensors of one shape");
      g[i] = static_cast<const float*>(t.data_ptr());
    }
    const bool make = a[1] == Py_None;
    at::Tensor out = make ? empty(first.sizes(), at::kFloat, first.device()) : tensor(a[1], "out");
    const c10::cuda::CUDAGuard on(first.device());
    float* p = static_cast<float*>(out.data_ptr());
    const int64_t numel = first.numel();
    const cudaStream_t stream = at::cuda::getCurrentCUDAStream();
    gwq_status st;
    {
      no_gil released;
      st = gwq_gradient_mean(g.data(), (int32_t)count, numel, p, stream);
    }
    check(st, "gwq_gradient_mean");
    if (!make) {
      Py_INCREF(a[1]);
      return a[1];
    }
    return THPVariable_Wrap(std::move(out));
  });
}

// quality(W, G, P, device index) -> (squared error, first-order change)
PyObject* py_quality(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 4);
    const at::Tensor &W = cuda_tensor(a[0], "W"), &G = cuda_tensor(a[1], "G");
    const gwq_packed* P = object<const gwq_packed>(a[2]);
    if (W.scalar_type() != at::kHalf || G.scalar_type() != at::kFloat || W.dim() != 2 || W.size(0) != P->N ||
        W.size(1) != P->K || W.sizes() != G.sizes())
      fail(PyExc_ValueError, "W must be fp16 [N,K] and G fp32 [N,K] of the layer's shape");
    const c10::cuda::CUDAGuard on((c10::DeviceIndex)device_index(a[3]));
    const uint16_t* w = static_cast<const uint16_t*>(W.data_ptr());
    const float* g = static_cast<const float*>(G.data_ptr());
    const cudaStream_t stream = at::cuda::getCurrentCUDAStream();
    double sq = 0.0, fo = 0.0;
    gwq_status st;
    {
      no_gil released;
      st = gwq_quality(w, g, P, &sq, &fo, stream);
    }
    check(st, "gwq_quality");
    return Py_BuildValue("dd", sq, fo);
  });
}

// Copies of library arrays in new tensors, in order on the current stream.  The library's objects are complete when the
// call that made them returns and are not released before the device is idle: nothing to wait for.
struct copies {
  at::Device device;
  c10::cuda::CUDAGuard on;
  std::vector<at::Tensor> made;
  std::vector<const void*> from;
  std::vector<void*> to;
  std::vector<size_t> bytes;
  explicit copies(long index) : device(at::kCUDA, (c10::DeviceIndex)index), on(device) {}
  void add(const void* p, at::IntArrayRef size, at::ScalarType type) {
    made.push_back(empty(size, type, device));
    from.push_back(p);
    to.push_back(made.back().data_ptr());
    bytes.push_back(bytes_of(made.back()));
  }
  void run() {
    const cudaError_t e = gwq_copy_arrays((int)made.size(), from.data(), to.data(), bytes.data(), at::cuda::getCurrentCUDAStream());
    if (e != cudaSuccess) {
      PyErr_Format(PyExc_RuntimeError, "copying an object's arrays failed: %d", (int)e);
      throw python_error();
    }
  }
  PyObject* wrapped(int i) { return THPVariable_Wrap(std::move(made[i])); }
};

// outlier_arrays(S, device index) -> (row_ptr, col_idx, val)
PyObject* py_outlier_arrays(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 2);
    const gwq_outliers* S = object<const gwq_outliers>(a[0]);
    copies c(device_index(a[1]));
    c.add(S->row_ptr, {(int64_t)S->N + 1}, at::kInt);
    c.add(S->col_idx, {S->nnz}, at::kInt);
    c.add(S->val, {S->nnz}, at::kShort);
    c.run();
    return Py_BuildValue("NNN", c.wrapped(0), c.wrapped(1), c.wrapped(2));
  });
}

// packed_arrays(P, device index) -> dict
PyObject* py_packed_arrays(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    need_args(n, 2);
    const gwq_packed* P = object<const gwq_packed>(a[0]);
    const gwq_outliers* S = P->S;
    const int64_t N = P->N, words = P->K / 32 * P->bits, groups = P->K / P->group;
    copies c(device_index(a[1]));
    c.add(P->codes, {N, words}, at::kInt);
    c.add(P->scales, {N, groups}, at::kShort);
    c.add(P->zeros, {N, groups}, at::kByte);
    c.add(S->row_ptr, {N + 1}, at::kInt);
    c.add(S->col_idx, {S->nnz}, at::kInt);
    c.add(S->val, {S->nnz}, at::kShort);
    c.run();
    return Py_BuildValue("{sNsNsNsNsNsN}", "words", c.wrapped(0), "scales", c.wrapped(1), "zeros", c.wrapped(2),
                         "row_ptr", c.wrapped(3), "col_idx", c.wrapped(4), "val", c.wrapped(5));
  });
}

// set_error(type): the exception raised for a status of the library
PyObject* py_set_error(PyObject*, PyObject* type) {
  Py_INCREF(type);
  Py_XDECREF(g_error);
  g_error = type;
  Py_RETURN_NONE;
}

#define GWQ_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {GWQ_METHOD(linear), GWQ_METHOD(linear_multi), GWQ_METHOD(linear_host), GWQ_METHOD(select),
                         GWQ_METHOD(pack), GWQ_METHOD(gradient_mean), GWQ_METHOD(quality), GWQ_METHOD(outlier_arrays),
                         GWQ_METHOD(packed_arrays), {"set_error", py_set_error, METH_O, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_gwq_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__gwq_torch() { return PyModule_Create(&module); }
