// The Python side of the calls that take microseconds (draft sampling, verification, one projection): argument checks,
// output tensors and the call into the C ABI in one native function each.
//
// What it is for: on the host such a call used to take longer than its kernels on the GPU.  Two torch.empty() of a few bytes
// 4.3 us, attribute look-ups 2, ctypes 1.2, the launches 2.1 each: a verification of one sequence 12.4 us, a draw 7.2, a small projection
// 9.1; this way 7.1, 4.5 and 4.4.  No arithmetic of the method is here.
#include <Python.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/hsd.h"

namespace {

decltype(&hsd_draft_sample) draft_sample_fn = nullptr;
decltype(&hsd_verify_workspace_bytes) verify_bytes_fn = nullptr;
decltype(&hsd_verify_level) verify_level_fn = nullptr;
decltype(&hsd_gemm_workspace_bytes) gemm_bytes_fn = nullptr;
decltype(&hsd_gemm_bf16) gemm_fn = nullptr;
decltype(&hsd_gemm_status) gemm_status_fn = nullptr;
decltype(&hsd_strerror) strerror_fn = nullptr;
PyObject *error_class = nullptr;

struct Failed {};                                          // a Python exception is set

const at::Tensor &tensor(PyObject *o) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a tensor, got %.80s", Py_TYPE(o)->tp_name);
    throw Failed();
  }
  return THPVariable_Unpack(o);
}
void *device_data(const at::Tensor &t) {
  if (!t.is_cuda() || !t.is_contiguous()) {
    PyErr_SetString(error_class, "expected a contiguous CUDA tensor");
    throw Failed();
  }
  return t.data_ptr();
}
const at::Tensor &shaped(PyObject *o, int64_t dims) {
  const at::Tensor &t = tensor(o);
  if (t.dim() != dims) {
    PyErr_Format(PyExc_ValueError, "expected %d dimensions, got %d", (int)dims, (int)t.dim());
    throw Failed();
  }
  return t;
}
int dtype_code(const at::Tensor &t) {
  if (t.scalar_type() == at::kFloat) return HSD_F32;
  if (t.scalar_type() == at::kBFloat16) return HSD_BF16;
  PyErr_Format(error_class, "unsupported logits dtype %s", c10::toString(t.scalar_type()));
  throw Failed();
}
uint64_t word(PyObject *o) {                               // modulo 2^64, as a C prototype takes a Python integer
  const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
  if (v == (unsigned long long)-1 && PyErr_Occurred()) throw Failed();
  return v;
}
void check(int status) {
  if (!status) return;
  PyErr_Format(error_class, "hsd call failed: %s (%d)", strerror_fn(status), status);
  throw Failed();
}
void arguments(Py_ssize_t got, Py_ssize_t want) {
  if (got == want) return;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
  throw Failed();
}
template <class F> int released(F &&f) {                   // other threads run while the call is made, as with ctypes
  PyThreadState *state = PyEval_SaveThread();
  const int status = f();
  PyEval_RestoreThread(state);
  return status;
}
void *current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// init(addresses of the C functions, in the order below; error class)
PyObject *init(PyObject *, PyObject *const *args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  try {
    arguments(n, 8);
    draft_sample_fn = reinterpret_cast<decltype(draft_sample_fn)>(word(args[0]));
    verify_bytes_fn = reinterpret_cast<decltype(verify_bytes_fn)>(word(args[1]));
    verify_level_fn = reinterpret_cast<decltype(verify_level_fn)>(word(args[2]));
    gemm_bytes_fn = reinterpret_cast<decltype(gemm_bytes_fn)>(word(args[3]));
    gemm_fn = reinterpret_cast<decltype(gemm_fn)>(word(args[4]));
    gemm_status_fn = reinterpret_cast<decltype(gemm_status_fn)>(word(args[5]));
    strerror_fn = reinterpret_cast<decltype(strerror_fn)>(word(args[6]));
    Py_INCREF(args[7]);
    error_class = args[7];
    Py_RETURN_NONE;
  } catch (const Failed &) { return nullptr; }
  END_HANDLE_TH_ERRORS
}

// draft_sample(logits [batch, rows, vocab], seed, call_serial, out_tokens or None)
PyObject *draft_sample(PyObject *, PyObject *const *args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  try {
    arguments(n, 4);
    const at::Tensor &logits = shaped(args[0], 3);
    void *data = device_data(logits);
    const int dtype = dtype_code(logits);
    const int batch = (int)logits.size(0), rows = (int)logits.size(1), vocab = (int)logits.size(2);
    const uint64_t seed = word(args[1]), serial = word(args[2]);
    at::Tensor out = args[3] == Py_None ? at::empty({batch, rows}, logits.options().dtype(at::kInt).requires_grad(false)) : tensor(args[3]);
    int32_t *to = static_cast<int32_t *>(device_data(out));
    void *stream = current_stream();
    check(released([&] { return draft_sample_fn(data, batch, rows, vocab, dtype, seed, serial, stream, to); }));
    return THPVariable_Wrap(std::move(out));
  } catch (const Failed &) { return nullptr; }
  END_HANDLE_TH_ERRORS
}

// verify_level(level, target [batch, t + 1, vocab], draft [batch, t, vocab], tokens [batch, t], seed, call_serial, workspace, out_tokens,
// out_n_accepted), the last three or None
PyObject *verify_level(PyObject *, PyObject *const *args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  try {
    arguments(n, 9);
    const int level = (int)word(args[0]);
    const at::Tensor &target = shaped(args[1], 3);
    void *p = device_data(target);
    const int batch = (int)target.size(0), t = (int)target.size(1) - 1, vocab = (int)target.size(2);
    void *q = t > 0 ? device_data(tensor(args[2])) : nullptr;
    int32_t *tokens = t > 0 ? static_cast<int32_t *>(device_data(tensor(args[3]))) : nullptr;
    const int dtype = dtype_code(target);
    const uint64_t seed = word(args[4]), serial = word(args[5]);
    const auto options = target.options().requires_grad(false);
    at::Tensor ws = args[6] == Py_None ? at::empty({std::max<int64_t>(16, (int64_t)verify_bytes_fn(batch, t))}, options.dtype(at::kByte)) : tensor(args[6]);
    at::Tensor out = args[7] == Py_None ? at::empty({batch, t + 1}, options.dtype(at::kInt)) : tensor(args[7]);
    at::Tensor accepted = args[8] == Py_None ? at::empty({batch}, options.dtype(at::kInt)) : tensor(args[8]);
    void *scratch = device_data(ws), *to = device_data(out), *count = device_data(accepted), *stream = current_stream();
    check(released([&] {
      return verify_level_fn(level, p, q, tokens, batch, t, vocab, dtype, seed, serial, scratch, (size_t)ws.numel(), stream,
                             static_cast<int32_t *>(to), static_cast<int32_t *>(count));
    }));
    PyObject *first = THPVariable_Wrap(std::move(out)), *second = THPVariable_Wrap(std::move(accepted)), *both = nullptr;
    if (first && second) both = PyTuple_Pack(2, first, second);
    Py_XDECREF(first);
    Py_XDECREF(second);
    return both;
  } catch (const Failed &) { return nullptr; }
  END_HANDLE_TH_ERRORS
}

// gemm_bf16(A [R, K], W [N, K], out or None, workspace or None, check)
PyObject *gemm_bf16(PyObject *, PyObject *const *args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  try {
    arguments(n, 5);
    const at::Tensor &a = shaped(args[0], 2), &w = tensor(args[1]);
    const int R = (int)a.size(0), K = (int)a.size(1), N = (int)w.size(0);
    const size_t need = gemm_bytes_fn(R, N, K);
    if (need == 0) {
      PyErr_Format(error_class, "hsd_gemm_bf16: unsupported shape R=%d N=%d K=%d", R, N, K);
      throw Failed();
    }
    void *pa = device_data(a), *pw = device_data(w);
    const auto options = a.options().requires_grad(false);
    at::Tensor ws = args[3] == Py_None ? at::empty({(int64_t)need + 256}, options.dtype(at::kByte)) : tensor(args[3]);
    at::Tensor out = args[2] == Py_None ? at::empty({R, N}, options.dtype(at::kFloat)) : tensor(args[2]);
    float *to = static_cast<float *>(device_data(out));
    const uintptr_t start = reinterpret_cast<uintptr_t>(ws.data_ptr()), base = (start + 255) / 256 * 256;
    void *scratch = reinterpret_cast<void *>(base), *stream = current_stream();
    const int64_t left = ws.numel() - (int64_t)(base - start);
    check(released([&] { return gemm_fn(pa, R, K, pw, N, to, scratch, left < 0 ? 0 : (size_t)left, stream); }));
    const int wanted = PyObject_IsTrue(args[4]);
    if (wanted < 0) throw Failed();
    if (wanted) check(released([&] { return gemm_status_fn(scratch, stream); }));
    return THPVariable_Wrap(std::move(out));
  } catch (const Failed &) { return nullptr; }
  END_HANDLE_TH_ERRORS
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr
PyMethodDef methods[] = {{"init", FAST(init)}, {"draft_sample", FAST(draft_sample)}, {"verify_level", FAST(verify_level)},
                         {"gemm_bf16", FAST(gemm_bf16)}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_calls(void) { return PyModule_Create(&module); }
