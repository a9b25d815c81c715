// Argument marshalling of the calls of a layer step for Python: tensors, integers and streams to the C ABI's pointers.
// Through ctypes, with a Python-level check of every tensor, a call of this kind cost about 10 us of host time, more than its
// kernels take for a few short requests.  Nothing is computed, allocated or remembered here.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include <stdint.h>
#include "fastpool.h"

namespace {

struct Bad {};      // a Python error is set

// Device address of a contiguous CUDA tensor; an integer is taken as it is, None is null.
void* address(PyObject* o, size_t* bytes = nullptr) {
  if (o == Py_None) return nullptr;
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) {
      PyErr_SetString(PyExc_AssertionError, "a contiguous CUDA tensor is needed");
      throw Bad();
    }
    if (bytes) *bytes = t.nbytes();
    return t.data_ptr();
  }
  void* p = PyLong_AsVoidPtr(o);
  if (!p && PyErr_Occurred()) throw Bad();
  return p;
}

// A handle: an integer, or an object (of ctypes) whose `value` is one.
template <typename T>
T* handle(PyObject* o) {
  if (o == Py_None) return nullptr;
  if (PyLong_Check(o)) return static_cast<T*>(PyLong_AsVoidPtr(o));
  PyObject* v = PyObject_GetAttrString(o, "value");
  if (!v) throw Bad();
  void* p = v == Py_None ? nullptr : PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  if (!p && PyErr_Occurred()) throw Bad();
  return static_cast<T*>(p);
}

// None: torch's current stream; else a raw stream or an object with `cuda_stream`.
fl_stream stream(PyObject* o) {
  if (o == Py_None) return (fl_stream)c10::cuda::getCurrentCUDAStream().stream();
  if (PyLong_Check(o)) return (fl_stream)PyLong_AsVoidPtr(o);
  PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
  if (!v) throw Bad();
  void* p = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  if (!p && PyErr_Occurred()) throw Bad();
  return (fl_stream)p;
}

int integer(PyObject* o) {
  const long v = PyLong_Check(o) ? PyLong_AsLong(o) : -1;
  if (!PyLong_Check(o)) {      // numpy integers and the like
    PyObject* i = PyNumber_Index(o);
    if (!i) throw Bad();
    const long w = PyLong_AsLong(i);
    Py_DECREF(i);
    if (w == -1 && PyErr_Occurred()) throw Bad();
    return (int)w;
  }
  if (v == -1 && PyErr_Occurred()) throw Bad();
  return (int)v;
}

float real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Bad();
  return (float)v;
}

const fl_bf16* bf16(PyObject* o) { return static_cast<const fl_bf16*>(address(o)); }
fl_bf16* bf16_out(PyObject* o) { return static_cast<fl_bf16*>(address(o)); }
const int32_t* i32(PyObject* o) { return static_cast<const int32_t*>(address(o)); }
const uint32_t* u32(PyObject* o) { return static_cast<const uint32_t*>(address(o)); }

// Up to FL_MAX_MATS entries of a sequence; a longer one leaves the rest to the library's own check of the count.
struct Items {
  PyObject* fast;
  Py_ssize_t n;
  explicit Items(PyObject* o) : fast(PySequence_Fast(o, "a sequence is needed")) {
    if (!fast) throw Bad();
    n = PySequence_Fast_GET_SIZE(fast);
  }
  ~Items() { Py_XDECREF(fast); }
  PyObject* operator[](Py_ssize_t i) const { return PySequence_Fast_GET_ITEM(fast, i); }
};
struct Ptrs {
  fl_bf16* p[FL_MAX_MATS] = {};
  Py_ssize_t n;
  explicit Ptrs(PyObject* o) {
    Items v(o);
    n = v.n;
    for (Py_ssize_t i = 0; i < n && i < FL_MAX_MATS; ++i) p[i] = bf16_out(v[i]);
  }
};
struct Ints {
  int p[FL_MAX_MATS] = {};
  Py_ssize_t n;
  explicit Ints(PyObject* o) {
    Items v(o);
    n = v.n;
    for (Py_ssize_t i = 0; i < n && i < FL_MAX_MATS; ++i) p[i] = integer(v[i]);
  }
};
// The library takes one count for all of them: an entry too few would be read as null or as projection 0.
void same_length(Py_ssize_t ys, Py_ssize_t others) {
  if (ys == others) return;
  PyErr_Format(PyExc_ValueError, "%zd outputs, but %zd entries in a list that goes with them", ys, others);
  throw Bad();
}

// Runs a library call, whose arguments have been read, without the interpreter's lock, as ctypes does: a launch may block (a full
// launch queue, a module that is loaded on its first use), and other threads go on meanwhile.
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};
template <typename F, typename... A>
int unlocked(F* call, A... args) {
  Unlocked u;
  return call(args...);
}

template <typename F>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F f) {
  if (n != want) {
    PyErr_Format(PyExc_TypeError, "%zd arguments given, %zd needed", n, want);
    return nullptr;
  }
  try {
    const int rc = f();
    return PyErr_Occurred() ? nullptr : PyLong_FromLong(rc);
  } catch (const Bad&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

#define CALL(name) PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n)

// pool, y, x, mat_index, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, stream
CALL(lora_sgmv) {
  return guarded(n, 11, [&] {
    size_t wb = 0;
    void* ws = address(a[9], &wb);
    return unlocked(fl_lora_sgmv, handle<fl_pool>(a[0]), bf16_out(a[1]), bf16(a[2]), integer(a[3]), i32(a[4]), i32(a[5]), integer(a[6]), integer(a[7]),
                        real(a[8]), ws, wb, stream(a[10]));
  });
}
// pool, y, x, mat_index, seg_indptr, lora_ids, n_seg, n_tokens, scale, stream
CALL(lora_sgmv_static) {
  return guarded(n, 10, [&] {
    return unlocked(fl_lora_sgmv_static, handle<fl_pool>(a[0]), bf16_out(a[1]), bf16(a[2]), integer(a[3]), i32(a[4]), i32(a[5]), integer(a[6]),
                               integer(a[7]), real(a[8]), stream(a[9]));
  });
}
// pool, ys, x, mat_indices, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, stream
CALL(lora_sgmv_multi) {
  return guarded(n, 11, [&] {
    const Ptrs ys(a[1]);
    const Ints mats(a[3]);
    same_length(ys.n, mats.n);
    size_t wb = 0;
    void* ws = address(a[9], &wb);
    return unlocked(fl_lora_sgmv_multi, handle<fl_pool>(a[0]), ys.p, bf16(a[2]), mats.p, (int)ys.n, i32(a[4]), i32(a[5]), integer(a[6]), integer(a[7]),
                              real(a[8]), ws, wb, stream(a[10]));
  });
}
// pool, y_q, y_k, y_v, x, mat_q, mat_k, mat_v, seg_indptr, lora_ids, n_seg, n_tokens, scale, req_indptr, kv_tbl_indptr, kv_tbl,
// prefix_lens, n_req, n_kv_heads, workspace, stream
CALL(lora_sgmv_qkv_append) {
  return guarded(n, 21, [&] {
    size_t wb = 0;
    void* ws = address(a[19], &wb);
    return unlocked(fl_lora_sgmv_qkv_append, handle<fl_pool>(a[0]), bf16_out(a[1]), bf16(a[2]), bf16(a[3]), bf16(a[4]), integer(a[5]), integer(a[6]),
                                   integer(a[7]), i32(a[8]), i32(a[9]), integer(a[10]), integer(a[11]), real(a[12]), i32(a[13]), i32(a[14]),
                                   u32(a[15]), i32(a[16]), integer(a[17]), integer(a[18]), ws, wb, stream(a[20]));
  });
}
// pool, y, x, w, mat_index, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, stream
CALL(lora_linear) {
  return guarded(n, 12, [&] {
    size_t wb = 0;
    void* ws = address(a[10], &wb);
    return unlocked(fl_lora_linear, handle<fl_pool>(a[0]), bf16_out(a[1]), bf16(a[2]), bf16(a[3]), integer(a[4]), i32(a[5]), i32(a[6]), integer(a[7]),
                          integer(a[8]), real(a[9]), ws, wb, stream(a[11]));
  });
}
// pool, ys, x, ws, mat_indices, seg_indptr, lora_ids, n_seg, n_tokens, scale, workspace, stream
CALL(lora_linear_multi) {
  return guarded(n, 12, [&] {
    const Ptrs ys(a[1]), w(a[3]);
    const Ints mats(a[4]);
    same_length(ys.n, w.n);
    same_length(ys.n, mats.n);
    size_t wb = 0;
    void* ws = address(a[10], &wb);
    return unlocked(fl_lora_linear_multi, handle<fl_pool>(a[0]), ys.p, bf16(a[2]), w.p, mats.p, (int)ys.n, i32(a[5]), i32(a[6]), integer(a[7]),
                                integer(a[8]), real(a[9]), ws, wb, stream(a[11]));
  });
}
// pool, y_q, x, w_q, w_k, w_v, mat_q, mat_k, mat_v, seg_indptr, lora_ids, n_seg, n_tokens, scale, req_indptr, kv_tbl_indptr, kv_tbl,
// prefix_lens, n_req, n_kv_heads, scratch_k, scratch_v, workspace, stream
CALL(lora_linear_qkv_append) {
  return guarded(n, 24, [&] {
    size_t wb = 0;
    void* ws = address(a[22], &wb);
    return unlocked(fl_lora_linear_qkv_append, handle<fl_pool>(a[0]), bf16_out(a[1]), bf16(a[2]), bf16(a[3]), bf16(a[4]), bf16(a[5]), integer(a[6]),
                                     integer(a[7]), integer(a[8]), i32(a[9]), i32(a[10]), integer(a[11]), integer(a[12]), real(a[13]),
                                     i32(a[14]), i32(a[15]), u32(a[16]), i32(a[17]), integer(a[18]), integer(a[19]), bf16_out(a[20]),
                                     bf16_out(a[21]), ws, wb, stream(a[23]));
  });
}
// pool, k_new, v_new, req_indptr, kv_tbl_indptr, kv_tbl, prefix_lens, n_req, n_tokens, n_kv_heads, stream
CALL(kv_append) {
  return guarded(n, 11, [&] {
    return unlocked(fl_kv_append, handle<fl_pool>(a[0]), bf16(a[1]), bf16(a[2]), i32(a[3]), i32(a[4]), u32(a[5]), i32(a[6]), integer(a[7]), integer(a[8]),
                        integer(a[9]), stream(a[10]));
  });
}
// pool, out, q, req_indptr, kv_tbl_indptr, kv_tbl, prefix_lens, new_lens, n_req, n_tokens, n_tbl, n_q_heads, n_kv_heads, sm_scale,
// workspace, stream
CALL(paged_attention) {
  return guarded(n, 16, [&] {
    size_t wb = 0;
    void* ws = address(a[14], &wb);
    return unlocked(fl_paged_attention, handle<fl_pool>(a[0]), bf16_out(a[1]), bf16(a[2]), i32(a[3]), i32(a[4]), u32(a[5]), i32(a[6]), i32(a[7]),
                              integer(a[8]), integer(a[9]), integer(a[10]), integer(a[11]), integer(a[12]), real(a[13]), ws, wb, stream(a[15]));
  });
}

#define ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY(lora_sgmv), ENTRY(lora_sgmv_static), ENTRY(lora_sgmv_multi), ENTRY(lora_sgmv_qkv_append), ENTRY(lora_linear),
                         ENTRY(lora_linear_multi), ENTRY(lora_linear_qkv_append), ENTRY(kv_append), ENTRY(paged_attention),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// What the module was built against, for build.py, which finds it in the file.
PyMODINIT_FUNC PyInit__native() {
  PyObject* m = PyModule_Create(&module);
  if (m && PyModule_AddStringConstant(m, "built_against", FL_NATIVE_TAG) < 0) {
    Py_DECREF(m);
    return nullptr;
  }
  return m;
}
