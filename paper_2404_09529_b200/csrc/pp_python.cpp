// CPython side of the binding for the calls that a program makes once per step: takes numpy arrays and
// torch tensors apart and calls the C ABI. Through ctypes a step of a few small prompts spent 60 us on
// the host, most of it on one pointer object per argument (1.4 us each) and stream and event look-ups, for
// 15 us of kernels; here an argument costs tens of nanoseconds. No arithmetic of the method lives here.
// Functions return the C ABI's status; binding.py turns it into exceptions.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#define NPY_NO_DEPRECATED_API NPY_1_7_API_VERSION
#include <numpy/arrayobject.h>

#include <cuda_runtime.h>

#include "../../include/pp.h"

namespace {

// Arguments of one call: converted arrays are kept until the call is over. The first failed conversion
// leaves a Python exception and makes every later one a no-op.
class Args {
 public:
  Args(PyObject* const* args, Py_ssize_t n) : args_(args), n_(n) {}
  ~Args() {
    for (int i = 0; i < n_kept_; ++i) Py_DECREF(kept_[i]);
    if (have_params_) PyBuffer_Release(&params_);
  }
  bool count(Py_ssize_t want, const char* name) {
    if (n_ == want) return true;
    PyErr_Format(PyExc_TypeError, "%s takes %zd arguments (%zd given)", name, want, n_);
    return false;
  }
  bool failed() const { return failed_; }

  // pp_attn_params from a ctypes structure
  const pp_attn_params* params() {
    PyObject* x = next();
    if (failed_) return nullptr;
    if (PyObject_GetBuffer(x, &params_, PyBUF_SIMPLE) != 0) return fail<pp_attn_params>();
    have_params_ = true;
    if (params_.len < (Py_ssize_t)sizeof(pp_attn_params)) {
      PyErr_SetString(PyExc_TypeError, "AttnParams expected");
      return fail<pp_attn_params>();
    }
    return static_cast<const pp_attn_params*>(params_.buf);
  }
  // anything that numpy makes an int32 / int64 array of; `length` receives its first dimension
  const int32_t* i32(Py_ssize_t* length = nullptr) { return static_cast<const int32_t*>(array(NPY_INT32, length)); }
  const int64_t* i64() { return static_cast<const int64_t*>(array(NPY_INT64, nullptr)); }
  // address of a torch tensor / numpy array / raw integer / None
  void* address() {
    PyObject* x = next();
    if (failed_ || x == Py_None) return nullptr;
    if (PyLong_Check(x)) return as_pointer(x);
    if (PyArray_Check(x)) return PyArray_DATA(reinterpret_cast<PyArrayObject*>(x));
    static PyObject* const name = PyUnicode_InternFromString("data_ptr");
    PyObject* r = PyObject_CallMethodNoArgs(x, name);
    if (!r) {
      if (PyErr_ExceptionMatches(PyExc_AttributeError)) PyErr_SetObject(PyExc_TypeError, reinterpret_cast<PyObject*>(Py_TYPE(x)));
      return fail<void>();
    }
    void* p = as_pointer(r);
    Py_DECREF(r);
    return p;
  }
  size_t size() {
    PyObject* x = next();
    if (failed_) return 0;
    const size_t v = PyLong_AsSize_t(x);
    if (v == (size_t)-1 && PyErr_Occurred()) failed_ = true;
    return v;
  }
  int32_t integer() {
    PyObject* x = next();
    if (failed_) return 0;
    const long v = PyLong_AsLong(x);
    if (v == -1 && PyErr_Occurred()) failed_ = true;
    return static_cast<int32_t>(v);
  }

 private:
  PyObject* next() { return args_[at_++]; }
  template <typename T> T* fail() { failed_ = true; return nullptr; }
  void* as_pointer(PyObject* x) {
    void* p = PyLong_AsVoidPtr(x);
    if (!p && PyErr_Occurred()) failed_ = true;
    return p;
  }
  void* array(int type, Py_ssize_t* length) {
    PyObject* x = next();
    if (failed_) return nullptr;
    PyArrayObject* a;
    if (PyArray_Check(x) && PyArray_TYPE(reinterpret_cast<PyArrayObject*>(x)) == type &&
        PyArray_ISCARRAY_RO(reinterpret_cast<PyArrayObject*>(x))) {
      a = reinterpret_cast<PyArrayObject*>(x);
    } else {
      a = reinterpret_cast<PyArrayObject*>(PyArray_FROMANY(x, type, 0, 0, NPY_ARRAY_CARRAY_RO | NPY_ARRAY_FORCECAST));
      if (!a) return fail<void>();
      kept_[n_kept_++] = reinterpret_cast<PyObject*>(a);
    }
    if (length) *length = PyArray_NDIM(a) ? PyArray_DIM(a, 0) : 1;
    return PyArray_DATA(a);
  }

  PyObject* const* args_;
  Py_ssize_t n_, at_ = 0;
  PyObject* kept_[8];          // a call has at most seven arrays
  int n_kept_ = 0;
  bool failed_ = false, have_params_ = false;
  Py_buffer params_;
};

#define PP_CALL(expr)            \
  int status;                    \
  Py_BEGIN_ALLOW_THREADS         \
  status = (expr);               \
  Py_END_ALLOW_THREADS           \
  return PyLong_FromLong(status)

// pack(lengths, capacity) -> (status, n_bins, capacity, bin_seg_ptr, seg_prompt, seg_start, seg_len, bin_of, off_of)
PyObject* pack(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  if (!a.count(2, "pack")) return nullptr;
  Py_ssize_t k = 0;
  const int32_t* lengths = a.i32(&k);
  const int32_t capacity = a.integer();
  if (a.failed()) return nullptr;
  npy_intp dim = k > 0 ? k : 0, dim_ptr = dim + 1;
  PyObject* out[6];
  int32_t* data[6];
  for (int i = 0; i < 6; ++i) {
    out[i] = PyArray_SimpleNew(1, i ? &dim : &dim_ptr, NPY_INT32);
    if (!out[i]) {
      while (i > 0) Py_DECREF(out[--i]);
      return nullptr;
    }
    data[i] = static_cast<int32_t*>(PyArray_DATA(reinterpret_cast<PyArrayObject*>(out[i])));
  }
  int32_t n_bins = 0, cap = 0;
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = pp_pack(lengths, static_cast<int32_t>(k), capacity, &n_bins, &cap, data[0], data[1], data[2], data[3], data[4], data[5]);
  Py_END_ALLOW_THREADS
  if (status == PP_OK) {           // entries 0 .. n_bins are written
    npy_intp used = n_bins + 1;
    PyObject* ptr = PyArray_SimpleNew(1, &used, NPY_INT32);
    if (!ptr) {
      for (PyObject* o : out) Py_DECREF(o);
      return nullptr;
    }
    memcpy(PyArray_DATA(reinterpret_cast<PyArrayObject*>(ptr)), data[0], sizeof(int32_t) * (size_t)used);
    Py_DECREF(out[0]);
    out[0] = ptr;
  }
  return Py_BuildValue("iiiNNNNNN", status, (int)n_bins, (int)cap, out[0], out[1], out[2], out[3], out[4], out[5]);
}

// prefill_fused(params, bin_seg_ptr, seg_start, seg_len, seg_prompt, lengths, q, k, v, o, k_cache, v_cache, cache_off,
//               cache_cap, workspace, host_workspace, workspace_bytes, device_status, stream); k = len(seg_start)
PyObject* prefill_fused(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  if (!a.count(19, "prefill_fused")) return nullptr;
  Py_ssize_t k = 0;
  const pp_attn_params* p = a.params();
  const int32_t *ptr = a.i32(), *start = a.i32(&k), *len = a.i32(), *prompt = a.i32(), *lengths = a.i32();
  void *q = a.address(), *kk = a.address(), *v = a.address(), *o = a.address(), *kc = a.address(), *vc = a.address();
  const int64_t* off = a.i64();
  const int32_t* cap = a.i32();
  void *ws = a.address(), *host = a.address();
  const size_t bytes = a.size();
  void *st = a.address(), *stream = a.address();
  if (a.failed()) return nullptr;
  PP_CALL(pp_prefill_fused(p, ptr, start, len, prompt, static_cast<int32_t>(k), lengths, q, kk, v, o, kc, vc, off, cap, ws, host,
                           bytes, static_cast<int32_t*>(st), stream));
}

// prefill_attention(params, bin_seg_ptr, seg_start, seg_len, q, k, v, o, workspace, host_workspace, workspace_bytes,
//                   device_status, stream); k = len(seg_start)
PyObject* prefill_attention(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  if (!a.count(13, "prefill_attention")) return nullptr;
  Py_ssize_t k = 0;
  const pp_attn_params* p = a.params();
  const int32_t *ptr = a.i32(), *start = a.i32(&k), *len = a.i32();
  void *q = a.address(), *kk = a.address(), *v = a.address(), *o = a.address(), *ws = a.address(), *host = a.address();
  const size_t bytes = a.size();
  void *st = a.address(), *stream = a.address();
  if (a.failed()) return nullptr;
  PP_CALL(pp_prefill_attention(p, ptr, start, len, static_cast<int32_t>(k), q, kk, v, o, ws, host, bytes,
                               static_cast<int32_t*>(st), stream));
}

// unpack_kv(params, bin_of, off_of, lengths, k_rot, v, k_cache, v_cache, cache_off, cache_cap, workspace, host_workspace,
//           workspace_bytes, stream); k = len(lengths)
PyObject* unpack_kv(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  if (!a.count(14, "unpack_kv")) return nullptr;
  Py_ssize_t k = 0;
  const pp_attn_params* p = a.params();
  const int32_t *bin = a.i32(), *row = a.i32(), *lengths = a.i32(&k);
  void *kr = a.address(), *v = a.address(), *kc = a.address(), *vc = a.address();
  const int64_t* off = a.i64();
  const int32_t* cap = a.i32();
  void *ws = a.address(), *host = a.address();
  const size_t bytes = a.size();
  void* stream = a.address();
  if (a.failed()) return nullptr;
  PP_CALL(pp_unpack_kv(p, bin, row, lengths, static_cast<int32_t>(k), kr, v, kc, vc, off, cap, ws, host, bytes, stream));
}

// decode_workspace_bytes(params, lengths)
PyObject* decode_workspace_bytes(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  if (!a.count(2, "decode_workspace_bytes")) return nullptr;
  Py_ssize_t k = 0;
  const pp_attn_params* p = a.params();
  const int32_t* lengths = a.i32(&k);
  if (a.failed()) return nullptr;
  return PyLong_FromSize_t(pp_decode_workspace_bytes(p, lengths, static_cast<int32_t>(k)));
}

// decode_step(params, lengths, q_new, k_new, v_new, o, k_cache, v_cache, cache_off, cache_cap, workspace,
//             host_workspace, workspace_bytes, stream); k = len(lengths)
PyObject* decode_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n);
  if (!a.count(14, "decode_step")) return nullptr;
  Py_ssize_t k = 0;
  const pp_attn_params* p = a.params();
  const int32_t* lengths = a.i32(&k);
  void *q = a.address(), *kn = a.address(), *vn = a.address(), *o = a.address(), *kc = a.address(), *vc = a.address();
  const int64_t* off = a.i64();
  const int32_t* cap = a.i32();
  void *ws = a.address(), *host = a.address();
  const size_t bytes = a.size();
  void* stream = a.address();
  if (a.failed()) return nullptr;
  PP_CALL(pp_decode_step(p, lengths, static_cast<int32_t>(k), q, kn, vn, o, kc, vc, off, cap, ws, host, bytes, stream));
}

// ------------------------------------------------------------------------------------------
// Fence: a CUDA event without timing, made on its first record (on the device that is current then).
// ------------------------------------------------------------------------------------------
struct Fence {
  PyObject_HEAD
  cudaEvent_t event;
};
PyObject* cuda_failed(cudaError_t e) {
  PyErr_Format(PyExc_RuntimeError, "CUDA: %s", cudaGetErrorString(e));
  return nullptr;
}
PyObject* fence_record(PyObject* self, PyObject* stream) {
  Fence* f = reinterpret_cast<Fence*>(self);
  void* s = PyLong_AsVoidPtr(stream);
  if (!s && PyErr_Occurred()) return nullptr;
  cudaError_t e = f->event ? cudaSuccess : cudaEventCreateWithFlags(&f->event, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventRecord(f->event, static_cast<cudaStream_t>(s));
  if (e != cudaSuccess) return cuda_failed(e);
  Py_RETURN_NONE;
}
// Waits until what the last record stands for has happened; returns at once if there was none.
PyObject* fence_synchronize(PyObject* self, PyObject*) {
  Fence* f = reinterpret_cast<Fence*>(self);
  if (!f->event) Py_RETURN_NONE;
  cudaError_t e = cudaEventQuery(f->event);
  if (e == cudaErrorNotReady) {
    (void)cudaGetLastError();
    Py_BEGIN_ALLOW_THREADS
    e = cudaEventSynchronize(f->event);
    Py_END_ALLOW_THREADS
  }
  if (e != cudaSuccess) return cuda_failed(e);
  Py_RETURN_NONE;
}
void fence_dealloc(PyObject* self) {
  Fence* f = reinterpret_cast<Fence*>(self);
  if (f->event) cudaEventDestroy(f->event);
  PyTypeObject* type = Py_TYPE(self);
  type->tp_free(self);
  Py_DECREF(type);
}
PyMethodDef fence_methods[] = {
    {"record", fence_record, METH_O, "record(stream): the fence stands for the work enqueued on the stream so far"},
    {"synchronize", fence_synchronize, METH_NOARGS, "wait until that work is done"},
    {nullptr, nullptr, 0, nullptr}};
PyType_Slot fence_slots[] = {{Py_tp_methods, fence_methods},
                             {Py_tp_dealloc, reinterpret_cast<void*>(fence_dealloc)},
                             {Py_tp_new, reinterpret_cast<void*>(PyType_GenericNew)},
                             {0, nullptr}};
PyType_Spec fence_spec = {"paper_2404_09529_b200._native.Fence", sizeof(Fence), 0, Py_TPFLAGS_DEFAULT, fence_slots};

#define PP_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PP_METHOD(pack), PP_METHOD(prefill_fused), PP_METHOD(prefill_attention), PP_METHOD(unpack_kv),
                         PP_METHOD(decode_workspace_bytes), PP_METHOD(decode_step), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  import_array();
  PyObject* m = PyModule_Create(&module);
  if (!m) return nullptr;
  PyObject* type = PyType_FromSpec(&fence_spec);
  if (!type || PyModule_AddObject(m, "Fence", type) != 0) {
    Py_XDECREF(type);
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
