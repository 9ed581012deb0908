// Argument marshalling of the binding's tensor calls in native code: the ordinary call (plain contiguous CUDA tensors, torch's
// current stream, the binding's own scratch) without the Python statements and the ctypes conversion around the C entry point.
// It does what binding.py does for the same call, in the same order, and returns NotImplemented, with nothing done, for every
// call that it does not know in full: binding.py then takes it, with its checks and errors.
//
// Why: a decode step of one sequence is 10 us on the GPU and was 12.3 us on the host, 5 of them the two launches (a small fp32
// call 8.9 and 10.0).  The tensors' attributes alone are some twenty Python calls.
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime_api.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>

#include "../../include/kata.h"

namespace {

PyObject* not_implemented() { Py_RETURN_NOTIMPLEMENTED; }

struct Held {                    // a reference until the end of the call (or null)
  PyObject* o;
  ~Held() { Py_XDECREF(o); }
};

// A tensor whose attributes are what they seem: no subclass, in memory of its own, on a CUDA device.
const at::Tensor* plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  return t.defined() && t.is_cuda() && t.layout() == at::kStrided && t.has_storage() ? &t : nullptr;
}
const at::Tensor* plain_contiguous(PyObject* o) {
  const at::Tensor* t = plain(o);
  return t != nullptr && t->is_contiguous() ? t : nullptr;
}

bool dtype_code(const at::Tensor& t, int32_t& code) {
  if (t.scalar_type() == at::kFloat) code = KATA_F32;
  else if (t.scalar_type() == at::kBFloat16) code = KATA_BF16;
  else return false;
  return true;
}

// The keyword options of a call; false: one that is not an int of 32 bits, or not known here.
bool read_options(PyObject* kw, kata_opts& o) {
  o = kata_opts{};
  o.struct_size = sizeof(kata_opts);
  o.feature_order = 2;
  if (!PyDict_CheckExact(kw)) return false;
  PyObject *key, *value;
  Py_ssize_t pos = 0;
  while (PyDict_Next(kw, &pos, &key, &value)) {
    static const struct { const char* name; int32_t kata_opts::* field; } kFields[] = {
        {"feature_groups", &kata_opts::feature_groups}, {"state_layout", &kata_opts::state_layout},
        {"inter_chunk", &kata_opts::inter_chunk},       {"feature_order", &kata_opts::feature_order},
        {"impl", &kata_opts::impl},                     {"scan_group", &kata_opts::scan_group}};
    if (!PyUnicode_Check(key) || !PyLong_CheckExact(value)) return false;
    int overflow = 0;
    const long long x = PyLong_AsLongLongAndOverflow(value, &overflow);
    if (overflow != 0 || x < INT_MIN || x > INT_MAX) return false;
    bool known = false;
    for (const auto& f : kFields)
      if (PyUnicode_CompareWithASCIIString(key, f.name) == 0) {
        o.*(f.field) = (int32_t)x;
        known = true;
        break;
      }
    if (!known) return false;
  }
  return true;
}

bool int_size(int64_t x, int& out) {
  out = (int)x;
  return x >= 0 && x <= INT_MAX;
}

// The stream of the call and, where it needs scratch, the buffer that binding.py keeps for this thread, device and stream.
// `held` is a new reference to hold until the call is made (or null).  false: binding.py has to make a buffer first.
bool stream_and_scratch(PyObject* owner, const at::Tensor& q, int fn, int B, int H, int T, int d_k, int d_v, int C, kata_opts& o,
                        PyObject*& held) {
  held = nullptr;
  const c10::DeviceIndex dev = q.device().index();
  cudaStream_t stream = c10::cuda::getCurrentCUDAStream(dev).stream();
  o.stream = stream;
  const size_t need = kata_workspace_bytes(fn, B, H, T, d_k, d_v, C, &o);
  if (need == 0) return true;
  if (stream != nullptr) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &status) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (status != cudaStreamCaptureStatusNone) return false;
  }
  static PyObject* const name = PyUnicode_InternFromString("bufs");
  PyObject* bufs = PyObject_GetAttr(owner, name);
  PyObject* key = stream != nullptr ? Py_BuildValue("(iN)", (int)dev, PyLong_FromVoidPtr(stream)) : Py_BuildValue("(iO)", (int)dev, Py_None);
  PyObject* entry = bufs != nullptr && key != nullptr && PyDict_Check(bufs) ? PyDict_GetItemWithError(bufs, key) : nullptr;
  Py_XINCREF(entry);
  Py_XDECREF(key);
  Py_XDECREF(bufs);
  if (entry != nullptr && PyTuple_CheckExact(entry) && PyTuple_GET_SIZE(entry) == 3) {
    const size_t size = PyLong_AsSize_t(PyTuple_GET_ITEM(entry, 2));
    void* ptr = PyLong_AsVoidPtr(PyTuple_GET_ITEM(entry, 1));
    if (!PyErr_Occurred() && size >= need) {
      o.workspace = ptr;
      o.workspace_bytes = size;
      held = entry;
      return true;
    }
  }
  Py_XDECREF(entry);
  PyErr_Clear();
  return false;
}

// Room for what the kernels read or write behind a pointer, which take sizes, type and device from q (binding.py _check_room).
bool has_room(const at::Tensor& t, const at::Tensor& q, at::ScalarType type, int64_t n) {
  return t.numel() >= n && t.scalar_type() == type && t.device() == q.device() && t.is_contiguous();
}
bool input_fits(const at::Tensor& t, const at::Tensor& q, int64_t heads, int64_t n) {
  return has_room(t, q, q.scalar_type(), n) && (t.numel() == n || heads == 1);
}

// The result of a call: the tensors, or the status as an int.
PyObject* result(int status, std::initializer_list<const at::Tensor*> out) {
  if (status != KATA_OK) return PyLong_FromLong(status);
  if (out.size() == 1) return THPVariable_Wrap(**out.begin());
  PyObject* tuple = PyTuple_New((Py_ssize_t)out.size());
  Py_ssize_t i = 0;
  for (const at::Tensor* t : out) {
    PyObject* x = tuple != nullptr ? THPVariable_Wrap(*t) : nullptr;
    if (x == nullptr) {
      Py_XDECREF(tuple);
      return nullptr;
    }
    PyTuple_SET_ITEM(tuple, i++, x);
  }
  return tuple;
}

// The tensor that was passed for an output of n elements, or a new one like `like`; false: one that is not plain, or too small.
bool output_ok(PyObject* o, const at::Tensor& q, int64_t n) {
  if (o == Py_None) return true;
  const at::Tensor* p = plain(o);
  return p != nullptr && has_room(*p, q, q.scalar_type(), n);
}
at::Tensor output(PyObject* o, const at::Tensor& like) { return o == Py_None ? at::empty_like(like) : THPVariable_Unpack(o); }

bool pointer(PyObject* o, const at::Tensor& q, at::ScalarType type, int64_t n, void*& p) {
  p = nullptr;
  if (o == Py_None) return true;
  const at::Tensor* t = plain(o);
  if (t == nullptr || !has_room(*t, q, type, n)) return false;
  p = t->data_ptr();
  return true;
}

// Feature rows of a state (binding.py decode_n_psi).
int64_t state_rows(const kata_opts& o, int d_k) {
  const int g = o.feature_groups > 1 ? o.feature_groups : 1, m = d_k / g;
  return o.feature_order == 1 ? d_k : (int64_t)g * (o.state_layout == KATA_LAYOUT_PACKED ? (int64_t)m * (m + 1) / 2 : (int64_t)m * m);
}

// The three calls.  With None for the scratch owner they only look the tensors over: True, they are plain and have room.

// forward(fn, scratch owner, q, k, v, out, C, s_pre, z_pre, s_init, z_init, device_status, options)
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 13 || !PyLong_CheckExact(a[0]) || !PyLong_CheckExact(a[6]) || at::impl::torch_function_mode_enabled()) return not_implemented();
  const int fn = (int)PyLong_AsLong(a[0]);
  int overflow = 0;
  const long c_arg = PyLong_AsLongAndOverflow(a[6], &overflow);
  kata_opts o;
  if (overflow != 0 || c_arg < INT_MIN || c_arg > INT_MAX || !read_options(a[12], o)) return not_implemented();
  const at::Tensor *q = plain_contiguous(a[2]), *k = plain_contiguous(a[3]), *v = plain_contiguous(a[4]);
  if (q == nullptr || k == nullptr || v == nullptr || q->dim() != 4 || v->dim() < 1 || !dtype_code(*q, o.dtype)) return not_implemented();
  int B, H, T, d_k, d_v;
  if (!int_size(q->size(0), B) || !int_size(q->size(1), H) || !int_size(q->size(2), T) || !int_size(q->size(3), d_k) ||
      !int_size(v->size(-1), d_v))
    return not_implemented();
  const int64_t heads = (int64_t)B * H, nv = heads * T * d_v;
  if (!input_fits(*k, *q, heads, q->numel()) || !input_fits(*v, *q, heads, nv) || !output_ok(a[5], *q, nv)) return not_implemented();
  void *s_pre, *z_pre, *s_init, *z_init, *device_status;
  const int64_t rows = heads * state_rows(o, d_k);
  const int64_t rows_pre = fn == KATA_FN_CHUNK_STATE_SCAN && c_arg > 0 ? rows * ((T + c_arg - 1) / c_arg) : rows;
  if (!pointer(a[7], *q, at::kFloat, rows_pre * d_v, s_pre) || !pointer(a[8], *q, at::kFloat, rows_pre, z_pre) ||
      !pointer(a[9], *q, at::kFloat, rows * d_v, s_init) || !pointer(a[10], *q, at::kFloat, rows, z_init) ||
      !pointer(a[11], *q, at::kInt, 1, device_status))
    return not_implemented();
  o.s_pre = static_cast<float*>(s_pre);
  o.z_pre = static_cast<float*>(z_pre);
  o.s_init = static_cast<const float*>(s_init);
  o.z_init = static_cast<const float*>(z_init);
  o.device_status = static_cast<int*>(device_status);
  if (a[1] == Py_None) Py_RETURN_TRUE;
  PyObject* held;
  if (!stream_and_scratch(a[1], *q, fn, B, H, T, d_k, d_v, (int)c_arg, o, held)) return not_implemented();
  const Held hold{held};
  const at::Tensor out = output(a[5], *v);
  const auto call = fn == KATA_FN_QUADRATIC ? kata_fwd_quadratic : fn == KATA_FN_CHUNKED ? kata_fwd_chunked : kata_chunk_state_scan;
  const void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr();
  void* op = out.data_ptr();
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = call(qp, kp, vp, op, B, H, T, d_k, d_v, (int)c_arg, &o);
  Py_END_ALLOW_THREADS
  return result(st, {&out});
  END_HANDLE_TH_ERRORS
}

// decode(scratch owner, q, k, v, S, Z, out, options)
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  kata_opts o;
  if (n != 8 || !read_options(a[7], o) || at::impl::torch_function_mode_enabled()) return not_implemented();
  const at::Tensor *q = plain_contiguous(a[1]), *k = plain_contiguous(a[2]), *v = plain_contiguous(a[3]), *S = plain_contiguous(a[4]),
                   *Z = plain_contiguous(a[5]);
  if (q == nullptr || k == nullptr || v == nullptr || S == nullptr || Z == nullptr || q->dim() != 3 || v->dim() < 1 ||
      !dtype_code(*q, o.dtype) || S->scalar_type() != at::kFloat || Z->scalar_type() != at::kFloat || S->dim() != 4 || Z->dim() != 3)
    return not_implemented();
  int B, H, d_k, d_v;
  if (!int_size(q->size(0), B) || !int_size(q->size(1), H) || !int_size(q->size(2), d_k) || !int_size(v->size(-1), d_v)) return not_implemented();
  const int64_t heads = (int64_t)B * H, rows = state_rows(o, d_k);
  if (!input_fits(*k, *q, heads, q->numel()) || !input_fits(*v, *q, heads, heads * d_v) || !output_ok(a[6], *q, heads * d_v) ||
      S->device() != q->device() || Z->device() != q->device())
    return not_implemented();
  if (S->size(0) != B || S->size(1) != H || S->size(2) != rows || S->size(3) != d_v || Z->size(0) != B || Z->size(1) != H || Z->size(2) != rows)
    return not_implemented();
  if (a[0] == Py_None) Py_RETURN_TRUE;
  PyObject* held;
  if (!stream_and_scratch(a[0], *q, KATA_FN_DECODE_STEP, B, H, 1, d_k, d_v, 0, o, held)) return not_implemented();
  const Held hold{held};
  const at::Tensor out = output(a[6], *v);
  const void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr();
  void *op = out.data_ptr(), *sp = S->data_ptr(), *zp = Z->data_ptr();
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = kata_decode_step(qp, kp, vp, op, static_cast<float*>(sp), static_cast<float*>(zp), B, H, d_k, d_v, &o);
  Py_END_ALLOW_THREADS
  return result(st, {&out});
  END_HANDLE_TH_ERRORS
}

// backward(fn, scratch owner, q, k, v, dout, dq, dk, dv, C, options)
PyObject* backward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  kata_opts o;
  if (n != 11 || !PyLong_CheckExact(a[0]) || !PyLong_CheckExact(a[9]) || !read_options(a[10], o) || at::impl::torch_function_mode_enabled())
    return not_implemented();
  const int fn = (int)PyLong_AsLong(a[0]);
  int overflow = 0;
  const long c_arg = PyLong_AsLongAndOverflow(a[9], &overflow);
  if (overflow != 0 || c_arg < INT_MIN || c_arg > INT_MAX) return not_implemented();
  const at::Tensor *q = plain_contiguous(a[2]), *k = plain_contiguous(a[3]), *v = plain_contiguous(a[4]), *dout = plain_contiguous(a[5]);
  if (q == nullptr || k == nullptr || v == nullptr || dout == nullptr || q->dim() != 4 || v->dim() < 1 || !dtype_code(*q, o.dtype))
    return not_implemented();
  int B, H, T, d_k, d_v;
  if (!int_size(q->size(0), B) || !int_size(q->size(1), H) || !int_size(q->size(2), T) || !int_size(q->size(3), d_k) ||
      !int_size(v->size(-1), d_v))
    return not_implemented();
  const int64_t heads = (int64_t)B * H, nk = q->numel(), nv = heads * T * d_v;
  if (!input_fits(*k, *q, heads, nk) || !input_fits(*v, *q, heads, nv) || !input_fits(*dout, *q, heads, nv) || !output_ok(a[6], *q, nk) ||
      !output_ok(a[7], *q, nk) || !output_ok(a[8], *q, nv))
    return not_implemented();
  if (a[1] == Py_None) Py_RETURN_TRUE;
  PyObject* held;
  if (!stream_and_scratch(a[1], *q, fn, B, H, T, d_k, d_v, (int)c_arg, o, held)) return not_implemented();
  const Held hold{held};
  const at::Tensor dq = output(a[6], *q), dk = output(a[7], *k), dv = output(a[8], *v);
  const void *qp = q->data_ptr(), *kp = k->data_ptr(), *vp = v->data_ptr(), *gp = dout->data_ptr();
  void *dqp = dq.data_ptr(), *dkp = dk.data_ptr(), *dvp = dv.data_ptr();
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = fn == KATA_FN_BWD_QUADRATIC ? kata_bwd_quadratic(qp, kp, vp, gp, dqp, dkp, dvp, B, H, T, d_k, d_v, &o)
                                   : kata_bwd_chunked(qp, kp, vp, gp, dqp, dkp, dvp, B, H, T, d_k, d_v, (int)c_arg, &o);
  Py_END_ALLOW_THREADS
  return result(st, {&dq, &dk, &dv});
  END_HANDLE_TH_ERRORS
}

PyMethodDef kMethods[] = {{"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(forward)), METH_FASTCALL, nullptr},
                          {"decode", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(decode)), METH_FASTCALL, nullptr},
                          {"backward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(backward)), METH_FASTCALL, nullptr},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_kata_torch", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// The torch and the Python that this was compiled against; the binding looks for it in the file and loads no other.
extern "C" __attribute__((visibility("default"), used)) const char kata_host_tag[] = KATA_HOST_TAG;

PyMODINIT_FUNC PyInit__kata_torch(void) { return PyModule_Create(&kModule); }
