// The calls of the Python binding whose device work takes microseconds, marshalled in C++: device
// pointers, shapes and leading dimensions are read from the tensor objects directly and the C entry
// point is called with the interpreter lock released.  The same marshalling in Python with ctypes costs
// 8 to 12 us of host time a call, more than most of these kernels run for on a small matrix; here it is
// 0.2 us, and a call with one launch 2.4 to 3.1.  Every function takes its arguments by position and returns the
// library's status code;
// names, defaults and documentation are those of binding.py.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <algorithm>

#include "bsp.h"

namespace {

struct Matrix {
  void* p;
  int rows, cols, ld;
};

// Positional arguments of one call; a failed conversion throws and ends as a Python exception.
class Args {
 public:
  Args(const char* name, PyObject* const* a, Py_ssize_t n, Py_ssize_t want) : a_(a) {
    TORCH_CHECK_TYPE(n == want, name, " takes ", want, " arguments, got ", n);
  }
  const at::Tensor& tensor(int i) const {
    TORCH_CHECK_TYPE(THPVariable_Check(a_[i]), "expected a tensor");
    const at::Tensor& t = THPVariable_Unpack(a_[i]);
    TORCH_CHECK_VALUE(t.is_cuda(), "expected a CUDA tensor");
    return t;
  }
  // Device pointer of a tensor, null for None.
  template <class T = void>
  T* ptr(int i) const {
    return a_[i] == Py_None ? nullptr : static_cast<T*>(tensor(i).data_ptr());
  }
  size_t bytes(int i) const { return a_[i] == Py_None ? 0 : tensor(i).nbytes(); }
  Matrix matrix(int i) const {
    const at::Tensor& t = tensor(i);
    TORCH_CHECK_VALUE(t.dim() == 2 && t.stride(1) == 1, "expected a 2-D tensor with unit inner stride");
    const int64_t ld = t.size(0) > 1 ? t.stride(0) : std::max(t.stride(0), t.size(1));
    return Matrix{t.data_ptr(), static_cast<int>(t.size(0)), static_cast<int>(t.size(1)), static_cast<int>(ld)};
  }
  long long integer(int i) const {
    const long long v = PyLong_AsLongLong(a_[i]);
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
  }
  int i32(int i) const { return static_cast<int>(integer(i)); }
  double real(int i) const {
    const double v = PyFloat_AsDouble(a_[i]);
    if (v == -1.0 && PyErr_Occurred()) throw python_error();
    return v;
  }
  float f32(int i) const { return static_cast<float>(real(i)); }
  // None = torch's current stream; otherwise a stream object, a raw handle, or a ctypes object that holds one.
  void* stream(int i) const {
    if (a_[i] == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    if (PyLong_Check(a_[i])) return handle(a_[i]);
    PyObject* h = PyObject_GetAttrString(a_[i], "cuda_stream");
    if (h == nullptr && PyErr_ExceptionMatches(PyExc_AttributeError)) {
      PyErr_Clear();
      h = PyObject_GetAttrString(a_[i], "value");
    }
    if (h == nullptr) throw python_error();
    const THPObjectPtr owner(h);
    return h == Py_None ? nullptr : handle(h);              // (the value of a null pointer is None)
  }
  void* address(int i) const { return handle(a_[i]); }

 private:
  static void* handle(PyObject* number) {
    void* p = PyLong_AsVoidPtr(number);
    if (p == nullptr && PyErr_Occurred()) throw python_error();
    return p;
  }
  PyObject* const* a_;
};

template <class F>
PyObject* status_of(F call) {
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

#define NATIVE(name) PyObject* name(PyObject*, PyObject* const* argv, Py_ssize_t argc)
#define NATIVE_ARGS(name, want) HANDLE_TH_ERRORS const Args A(#name, argv, argc, want)
#define NATIVE_END END_HANDLE_TH_ERRORS

// (W, block, orient, eps, pen, norms, gamma_in, gamma_out, penalty, stream)
NATIVE(group_norms) {
  NATIVE_ARGS(group_norms, 10);
  const Matrix W = A.matrix(0);
  const int block = A.i32(1), orient = A.i32(2), pen = A.i32(4);
  const float eps = A.f32(3);
  float *norms = A.ptr<float>(5), *gin = A.ptr<float>(6), *gout = A.ptr<float>(7);
  double* penalty = A.ptr<double>(8);
  void* s = A.stream(9);
  return status_of([&] { return bsp_group_norms(W.p, W.rows, W.cols, W.ld, block, orient, eps, pen, norms, gin, gout, penalty, s); });
  NATIVE_END
}

// (W, block, orient, pen, gamma, scale, grad, accumulate, stream)
NATIVE(penalty_grad) {
  NATIVE_ARGS(penalty_grad, 9);
  const Matrix W = A.matrix(0), G = A.matrix(6);
  const int block = A.i32(1), orient = A.i32(2), pen = A.i32(3), acc = A.i32(7);
  const float* gamma = A.ptr<float>(4);
  const float scale = A.f32(5);
  void* s = A.stream(8);
  return status_of([&] {
    return bsp_penalty_grad(W.p, W.rows, W.cols, W.ld, block, orient, pen, gamma, scale, static_cast<float*>(G.p), G.ld, acc, s);
  });
  NATIVE_END
}

// (W, block, orient, threshold, threshold_dev, keep_per_block, keep, blk_ptr, idx, vals, kept_weights, ws, stream)
NATIVE(prune_pack) {
  NATIVE_ARGS(prune_pack, 13);
  const Matrix W = A.matrix(0);
  const int block = A.i32(1), orient = A.i32(2), keep_n = A.i32(5);
  const float t = A.f32(3);
  const float* td = A.ptr<float>(4);
  uint8_t* keep = A.ptr<uint8_t>(6);
  int32_t *bp = A.ptr<int32_t>(7), *idx = A.ptr<int32_t>(8);
  void* vals = A.ptr(9);
  int64_t* kw = A.ptr<int64_t>(10);
  void* ws = A.ptr(11);
  const size_t wsb = A.bytes(11);
  void* s = A.stream(12);
  return status_of([&] {
    return bsp_prune_pack(W.p, W.rows, W.cols, W.ld, block, orient, t, td, keep_n, keep, bp, idx, vals, kw, ws, wsb, s);
  });
  NATIVE_END
}

// (W, block, orient, rate, threshold_out, ws, stream)
NATIVE(percentile_threshold) {
  NATIVE_ARGS(percentile_threshold, 7);
  const Matrix W = A.matrix(0);
  const int block = A.i32(1), orient = A.i32(2);
  const double rate = A.real(3);
  float* out = A.ptr<float>(4);
  void* ws = A.ptr(5);
  const size_t wsb = A.bytes(5);
  void* s = A.stream(6);
  return status_of([&] { return bsp_percentile_threshold(W.p, W.rows, W.cols, W.ld, block, orient, rate, out, ws, wsb, s); });
  NATIVE_END
}

// (W, block, orient, keep, stream)
NATIVE(apply_mask) {
  NATIVE_ARGS(apply_mask, 5);
  const Matrix W = A.matrix(0);
  const int block = A.i32(1), orient = A.i32(2);
  const uint8_t* keep = A.ptr<uint8_t>(3);
  void* s = A.stream(4);
  return status_of([&] { return bsp_apply_mask(W.p, W.rows, W.cols, W.ld, block, orient, keep, s); });
  NATIVE_END
}

// (address of the job array, number of jobs, block, eps, pen, stream)
NATIVE(prepare_batched) {
  NATIVE_ARGS(prepare_batched, 6);
  const bsp_layer_job* jobs = static_cast<const bsp_layer_job*>(A.address(0));
  const int n = A.i32(1), block = A.i32(2), pen = A.i32(4);
  const float eps = A.f32(3);
  void* s = A.stream(5);
  return status_of([&] { return bsp_prepare_batched(jobs, n, block, eps, pen, s); });
  NATIVE_END
}

// (address of the job array, number of jobs, block, address of the rates, stream)
NATIVE(percentile_threshold_batched) {
  NATIVE_ARGS(percentile_threshold_batched, 5);
  const bsp_layer_job* jobs = static_cast<const bsp_layer_job*>(A.address(0));
  const int n = A.i32(1), block = A.i32(2);
  const double* rates = static_cast<const double*>(A.address(3));
  void* s = A.stream(4);
  return status_of([&] { return bsp_percentile_threshold_batched(jobs, n, block, rates, s); });
  NATIVE_END
}

// (which: 0 = C form, 1 = R form, 2 = transposed; blk_ptr, idx, vals, rows, cols, block, plan, stream)
NATIVE(linear_plan) {
  NATIVE_ARGS(linear_plan, 9);
  const int which = A.i32(0);
  const int32_t *bp = A.ptr<int32_t>(1), *idx = A.ptr<int32_t>(2);
  const void* vals = A.ptr(3);
  const int n = A.i32(4), k = A.i32(5), block = A.i32(6);
  void* plan = A.ptr(7);
  const size_t bytes = A.bytes(7);
  void* s = A.stream(8);
  return status_of([&] {
    return which == 0   ? bsp_linear_plan(bp, idx, vals, n, k, block, plan, bytes, s)
           : which == 1 ? bsp_linear_plan_r(bp, idx, vals, n, k, block, plan, bytes, s)
                        : bsp_linear_plan_t(bp, idx, vals, n, k, block, plan, bytes, s);
  });
  NATIVE_END
}

// (dY, X, block, keep, dW, stream)
NATIVE(linear_backward_weight) {
  NATIVE_ARGS(linear_backward_weight, 6);
  const Matrix dY = A.matrix(0), X = A.matrix(1), dW = A.matrix(4);
  const int block = A.i32(2);
  const uint8_t* keep = A.ptr<uint8_t>(3);
  void* s = A.stream(5);
  return status_of([&] {
    return bsp_linear_backward_weight(dY.p, dY.ld, X.p, X.ld, dY.rows, dY.cols, X.cols, block, keep, dW.p, dW.ld, s);
  });
  NATIVE_END
}

// (plan, n_out, k_in, block, X, bias, act, Y, algo, stream)
NATIVE(linear_planned) {
  NATIVE_ARGS(linear_planned, 10);
  const void* plan = A.ptr(0);
  const int n = A.i32(1), k = A.i32(2), block = A.i32(3), act = A.i32(6), algo = A.i32(8);
  const Matrix X = A.matrix(4), Y = A.matrix(7);
  const void* bias = A.ptr(5);
  void* s = A.stream(9);
  return status_of([&] { return bsp_linear_planned_ex(plan, n, k, block, X.p, X.rows, X.ld, bias, act, Y.p, Y.ld, algo, s); });
  NATIVE_END
}

// (blk_ptr, idx, vals, rows, cols, block, X, bias, act, Y, ws, stream)
NATIVE(linear_packed) {
  NATIVE_ARGS(linear_packed, 12);
  const int32_t *bp = A.ptr<int32_t>(0), *idx = A.ptr<int32_t>(1);
  const void* vals = A.ptr(2);
  const int n = A.i32(3), k = A.i32(4), block = A.i32(5), act = A.i32(8);
  const Matrix X = A.matrix(6), Y = A.matrix(9);
  const void* bias = A.ptr(7);
  void* ws = A.ptr(10);
  const size_t wsb = A.bytes(10);
  void* s = A.stream(11);
  return status_of([&] { return bsp_linear(bp, idx, vals, n, k, block, X.p, X.rows, X.ld, bias, act, Y.p, Y.ld, ws, wsb, s); });
  NATIVE_END
}

// (W, grad, m, v, keep, block, orient, lr, beta1, beta2, eps, weight_decay, step, W_bf16, stream)
NATIVE(masked_adam_step) {
  NATIVE_ARGS(masked_adam_step, 15);
  const Matrix W = A.matrix(0), G = A.matrix(1);
  float *m = A.ptr<float>(2), *v = A.ptr<float>(3);
  const uint8_t* keep = A.ptr<uint8_t>(4);
  const int block = A.i32(5), orient = A.i32(6), step = A.i32(12);
  const float lr = A.f32(7), b1 = A.f32(8), b2 = A.f32(9), eps = A.f32(10), wd = A.f32(11);
  Matrix Wb{nullptr, 0, 0, 0};
  if (argv[13] != Py_None) Wb = A.matrix(13);
  void* s = A.stream(14);
  return status_of([&] {
    return bsp_masked_adam_step(static_cast<float*>(W.p), static_cast<const float*>(G.p), m, v, W.rows, W.cols, W.ld, G.ld, keep,
                                block, orient, lr, b1, b2, eps, wd, step, Wb.p, Wb.ld, s);
  });
  NATIVE_END
}

// (W, block, blk_ptr, idx, vals, stream)
NATIVE(repack_values) {
  NATIVE_ARGS(repack_values, 6);
  const Matrix W = A.matrix(0);
  const int block = A.i32(1);
  const int32_t *bp = A.ptr<int32_t>(2), *idx = A.ptr<int32_t>(3);
  void* vals = A.ptr(4);
  void* s = A.stream(5);
  return status_of([&] { return bsp_repack_values(W.p, W.rows, W.cols, W.ld, block, bp, idx, vals, s); });
  NATIVE_END
}

// (X, XT, stream)
NATIVE(transpose) {
  NATIVE_ARGS(transpose, 3);
  const Matrix X = A.matrix(0), XT = A.matrix(1);
  void* s = A.stream(2);
  return status_of([&] { return bsp_transpose(X.p, X.rows, X.cols, X.ld, XT.p, XT.ld, s); });
  NATIVE_END
}

// (gplan, n_out, k_in, block, XT, bias, act, Y, out_transposed, stream)
NATIVE(linear_gathered) {
  NATIVE_ARGS(linear_gathered, 10);
  const void* gplan = A.ptr(0);
  const int n = A.i32(1), k = A.i32(2), block = A.i32(3), act = A.i32(6), tr = A.i32(8);
  const Matrix XT = A.matrix(4), Y = A.matrix(7);
  const void* bias = A.ptr(5);
  void* s = A.stream(9);
  return status_of([&] { return bsp_linear_gathered_ex(gplan, n, k, block, XT.p, XT.cols, XT.ld, bias, act, Y.p, Y.ld, tr, s); });
  NATIVE_END
}

// (address of the call descriptor, route, stream) -> status if it is not zero, else the route taken (positive)
NATIVE(linear_run) {
  NATIVE_ARGS(linear_run, 3);
  const bsp_linear_call* call = static_cast<const bsp_linear_call*>(A.address(0));
  const int route = A.i32(1);
  void* s = A.stream(2);
  return status_of([&] {
    int taken = 0;
    const int st = bsp_linear_run(call, route, &taken, s);
    return st != BSP_OK ? st : taken;
  });
  NATIVE_END
}

#define ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    ENTRY(group_norms), ENTRY(penalty_grad), ENTRY(prune_pack), ENTRY(percentile_threshold), ENTRY(apply_mask),
    ENTRY(prepare_batched), ENTRY(percentile_threshold_batched), ENTRY(linear_plan), ENTRY(linear_backward_weight),
    ENTRY(linear_planned), ENTRY(linear_packed), ENTRY(masked_adam_step), ENTRY(repack_values), ENTRY(transpose),
    ENTRY(linear_gathered), ENTRY(linear_run), {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_bsp_native", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__bsp_native() { return PyModule_Create(&kModule); }
