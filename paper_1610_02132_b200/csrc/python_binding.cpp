// Python binding of the entry points that a training loop calls every step (include/qsgd.h): argument
// marshalling only. A call hands over up to two dozen tensors; taking their addresses, the current
// stream and the scalars here instead of through ctypes is what keeps the host ahead of the GPU on
// small gradients (one fixed-width encode of 4096 coordinates: 10.7 us of host time through ctypes,
// of which the launch itself is about 3; sixteen-message decode: 18.5 us).
//
// Every function takes positional arguments in the order of the C call, with tensors for pointers and a
// stream object or None last, and returns the C call's status. Arguments that must be contiguous CUDA
// tensors and are not raise the package's own exception, handed over once by set_error.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/qsgd.h"

namespace {

PyObject* g_error = nullptr;      // QsgdError

struct Fail {};                   // a Python exception is set

const at::Tensor& cuda_tensor(PyObject* o, const char* name) {
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.is_cuda() && t.is_contiguous()) return t;
  }
  PyErr_Format(g_error ? g_error : PyExc_RuntimeError, "%s must be a contiguous CUDA tensor", name);
  throw Fail{};
}

PyObject* g_ctypes_number = nullptr;   // ctypes' c_uint64, c_float and the like

// A number, also one of ctypes' own.
struct Number {
  PyObject* o;
  explicit Number(PyObject* v) : o(Py_NewRef(v)) {
    if (PyIndex_Check(v) || PyFloat_Check(v)) return;
    const int mine = g_ctypes_number ? PyObject_IsInstance(v, g_ctypes_number) : 0;
    if (mine) Py_SETREF(o, mine > 0 ? PyObject_GetAttrString(v, "value") : nullptr);
    if (!o) throw Fail{};
  }
  Number(const Number&) = delete;
  ~Number() { Py_XDECREF(o); }
};

uint64_t u64(PyObject* v) {
  const Number n(v);
  const unsigned long long u = PyLong_AsUnsignedLongLongMask(n.o);
  if (u == ~0ull && PyErr_Occurred()) throw Fail{};
  return u;
}
uint32_t u32(PyObject* o) { return static_cast<uint32_t>(u64(o)); }
int i32(PyObject* o) { return static_cast<int>(u64(o)); }

float f32(PyObject* o) {
  const Number n(o);
  const double v = PyFloat_AsDouble(n.o);
  if (v == -1.0 && PyErr_Occurred()) throw Fail{};
  return static_cast<float>(v);
}

// Where a tensor, or whatever else has a data_ptr(), lies.
void* data_of(PyObject* o) {
  if (THPVariable_Check(o)) return THPVariable_Unpack(o).data_ptr();
  PyObject* p = PyObject_CallMethod(o, "data_ptr", nullptr);
  if (!p) throw Fail{};
  const unsigned long long v = PyLong_AsUnsignedLongLongMask(p);
  Py_DECREF(p);
  if (v == ~0ull && PyErr_Occurred()) throw Fail{};
  return reinterpret_cast<void*>(v);
}
void* data_or_null(PyObject* o) { return o == Py_None ? nullptr : data_of(o); }

// The same, or a raw device address given as an integer.
void* address(PyObject* o) {
  return !THPVariable_Check(o) && PyIndex_Check(o) ? reinterpret_cast<void*>(u64(o)) : data_of(o);
}

qsgd_stream_t stream_of(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
  if (!v) throw Fail{};
  if (v == Py_None) { Py_DECREF(v); return nullptr; }
  const unsigned long long s = PyLong_AsUnsignedLongLongMask(v);
  Py_DECREF(v);
  if (s == ~0ull && PyErr_Occurred()) throw Fail{};
  return reinterpret_cast<qsgd_stream_t>(s);
}

// The K addresses of a sequence. More than the library takes are counted but not stored: the C call
// refuses them by their number before it looks at any.
struct Peers {
  void* p[QSGD_MAX_PEERS] = {};
  uint32_t K = 0;
  bool given = false;
  template <typename T> const T* const* as() const { return given ? reinterpret_cast<const T* const*>(p) : nullptr; }
};

struct Sequence {                 // borrowed items of a list or tuple (or of a copy of any other sequence)
  PyObject* fast = nullptr;
  explicit Sequence(PyObject* o) {
    // what has no length (a generator) could be gone through only once
    if (PyObject_Size(o) >= 0) fast = PySequence_Fast(o, "a sequence is required");
    if (!fast) throw Fail{};
  }
  ~Sequence() { Py_DECREF(fast); }
  uint32_t size() const { return static_cast<uint32_t>(PySequence_Fast_GET_SIZE(fast)); }
  PyObject* operator[](uint32_t i) const { return PySequence_Fast_GET_ITEM(fast, i); }
};

void peers(PyObject* o, Peers* out) {
  if (o == Py_None) return;                       // the library says where that is allowed
  const Sequence s(o);
  out->given = true;
  out->K = s.size();
  for (uint32_t k = 0; k < out->K && k < QSGD_MAX_PEERS; ++k) out->p[k] = address(s[k]);
}

// Fewer tables or byte counts than messages: what is missing would read as "none given", and the payload's bound
// would be gone. (Fixed-width messages have neither: nothing is looked at.)
void at_least(uint32_t have, const Peers& msgs, int code, const char* name) {
  if (have >= msgs.K || (code != QSGD_CODE_ELIAS && code != QSGD_CODE_ELIAS_DENSE)) return;
  PyErr_Format(g_error ? g_error : PyExc_RuntimeError, "%u %s given for %u messages", have, name, msgs.K);
  throw Fail{};
}

// Byte counts of the messages: the given list, or (sizes_of_msgs) the sizes of the message tensors.
const uint64_t* byte_counts(PyObject* o, PyObject* msgs, const Peers& read, int code, bool sizes_of_msgs, uint64_t* out) {
  if (o == Py_None && !sizes_of_msgs) return nullptr;
  const Sequence s(o == Py_None ? msgs : o);
  at_least(s.size(), read, code, "byte counts");
  for (uint32_t k = 0; k < s.size() && k < QSGD_MAX_PEERS; ++k) {
    if (o != Py_None) {
      PyObject* v = PyNumber_Long(s[k]);
      if (!v) throw Fail{};
      out[k] = PyLong_AsUnsignedLongLongMask(v);
      Py_DECREF(v);
    } else if (THPVariable_Check(s[k])) {
      out[k] = THPVariable_Unpack(s[k]).nbytes();
    } else {
      PyErr_SetString(g_error ? g_error : PyExc_RuntimeError, "msg_bytes is required for messages given by address");
      throw Fail{};
    }
  }
  return out;
}

// Runs a C call with the interpreter lock released: a launch may block when the stream's queue is full.
template <typename F>
PyObject* unlocked(F&& call) {
  PyThreadState* save = PyEval_SaveThread();
  const int st = call();
  PyEval_RestoreThread(save);
  return PyLong_FromLong(st);
}

#define QSGD_ARGS(count)                                                                     \
  if (nargs != (count)) {                                                                    \
    PyErr_Format(PyExc_TypeError, "%s takes %d arguments, %zd given", __func__, (count), nargs); \
    return nullptr;                                                                          \
  }
#define QSGD_TRY try {
#define QSGD_CATCH                                                            \
  } catch (const Fail&) {                                                     \
    return nullptr;                                                           \
  } catch (const std::exception& e) {                                         \
    PyErr_SetString(PyExc_RuntimeError, e.what());                            \
    return nullptr;                                                           \
  }

// encode(g, n or None, bucket, s, norm, code, seed, step, worker, out, out_bits, workspace, status, stream)
PyObject* encode(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  QSGD_ARGS(14)
  QSGD_TRY
  void* ws = data_or_null(a[11]);
  const at::Tensor& g = cuda_tensor(a[0], "g");
  const at::Tensor& out = cuda_tensor(a[9], "out");
  const at::Tensor& info = cuda_tensor(a[10], "out_bits");
  const at::Tensor& status = cuda_tensor(a[12], "status_dev");
  const uint64_t n = a[1] == Py_None ? static_cast<uint64_t>(g.numel()) : u64(a[1]);
  const uint32_t bucket = u32(a[2]), s = u32(a[3]), step = u32(a[7]), worker = u32(a[8]);
  const int norm = i32(a[4]), code = i32(a[5]);
  const uint64_t seed = u64(a[6]);
  const qsgd_stream_t stream = stream_of(a[13]);
  return unlocked([&] {
    return qsgd_encode(static_cast<const float*>(g.data_ptr()), n, bucket, s, norm, code, seed, step, worker,
                       out.data_ptr(), out.nbytes(), static_cast<uint64_t*>(info.data_ptr()), ws,
                       static_cast<uint32_t*>(status.data_ptr()), stream);
  });
  QSGD_CATCH
}

// encode_static(g, bucket, s, norm, code, seed, step, worker, out, out_bits, status, stream)
PyObject* encode_static(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  QSGD_ARGS(12)
  QSGD_TRY
  const at::Tensor& g = cuda_tensor(a[0], "g");
  const at::Tensor& out = cuda_tensor(a[8], "out");
  const at::Tensor& info = cuda_tensor(a[9], "out_bits");
  const at::Tensor& status = cuda_tensor(a[10], "status_dev");
  const uint32_t bucket = u32(a[1]), s = u32(a[2]), step = u32(a[6]), worker = u32(a[7]);
  const int norm = i32(a[3]), code = i32(a[4]);
  const uint64_t seed = u64(a[5]);
  const qsgd_stream_t stream = stream_of(a[11]);
  return unlocked([&] {
    return qsgd_encode_elias_static(static_cast<const float*>(g.data_ptr()), static_cast<uint64_t>(g.numel()), bucket,
                                    s, norm, code, seed, step, worker, out.data_ptr(), out.nbytes(),
                                    static_cast<uint64_t*>(info.data_ptr()),
                                    static_cast<uint32_t*>(status.data_ptr()), stream);
  });
  QSGD_CATCH
}

// policy_encode(g, address of a qsgd_policy, bucket, s, norm, code, seed, step, worker, out, out_bits,
//               workspace, status, stream)
PyObject* policy_encode(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  QSGD_ARGS(14)
  QSGD_TRY
  void* ws = data_or_null(a[11]);
  const at::Tensor& g = cuda_tensor(a[0], "g");
  const at::Tensor& out = cuda_tensor(a[9], "out");
  const at::Tensor& info = cuda_tensor(a[10], "out_bits");
  const at::Tensor& status = cuda_tensor(a[12], "status_dev");
  const qsgd_policy* plan = static_cast<const qsgd_policy*>(address(a[1]));
  const uint32_t bucket = u32(a[2]), s = u32(a[3]), step = u32(a[7]), worker = u32(a[8]);
  const int norm = i32(a[4]), code = i32(a[5]);
  const uint64_t seed = u64(a[6]);
  const qsgd_stream_t stream = stream_of(a[13]);
  return unlocked([&] {
    return qsgd_policy_encode(static_cast<const float*>(g.data_ptr()), plan, bucket, s, norm, code, seed, step, worker,
                              out.data_ptr(), out.nbytes(), static_cast<uint64_t*>(info.data_ptr()), ws,
                              static_cast<uint32_t*>(status.data_ptr()), stream);
  });
  QSGD_CATCH
}

// decode(packed, msgs, tables or infos, bytes, n, bucket, s, code, out, eta or None, status, stream):
// eta None: the sum into `out`; else the step on `out`
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  QSGD_ARGS(12)
  QSGD_TRY
  const bool packed = a[0] == Py_True, fused = a[9] != Py_None;
  uint32_t* status = static_cast<uint32_t*>(data_of(a[10]));
  Peers msgs, tables;
  uint64_t count[QSGD_MAX_PEERS] = {};
  peers(a[1], &msgs);
  peers(a[2], &tables);
  const int code = i32(a[7]);
  if (tables.given) at_least(tables.K, msgs, code, packed ? "info words" : "tables");
  const uint64_t* bytes = byte_counts(a[3], a[1], msgs, code, packed, count);
  const uint64_t n = u64(a[4]);
  const uint32_t bucket = u32(a[5]), s = u32(a[6]);
  const float eta = fused ? f32(a[9]) : 0.f;
  float* out = static_cast<float*>(cuda_tensor(a[8], fused ? "x" : "acc").data_ptr());
  const qsgd_stream_t stream = stream_of(a[11]);
  const void* const* mp = msgs.as<void>();
  const uint64_t* const* tp = tables.as<uint64_t>();
  return unlocked([&] {
    if (fused)
      return (packed ? qsgd_decode_sgd_step_packed : qsgd_decode_sgd_step)(mp, tp, bytes, msgs.K, n, bucket, s, code,
                                                                             out, eta, status, stream);
    return (packed ? qsgd_decode_accumulate_packed : qsgd_decode_accumulate)(mp, tp, bytes, msgs.K, n, bucket, s, code,
                                                                               out, status, stream);
  });
  QSGD_CATCH
}

// policy_decode(msgs, tables, bytes, address of a qsgd_policy, bucket, s, code, out, eta or None, status, stream)
PyObject* policy_decode(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  QSGD_ARGS(11)
  QSGD_TRY
  const bool fused = a[8] != Py_None;
  uint32_t* status = static_cast<uint32_t*>(data_of(a[9]));
  Peers msgs, tables;
  uint64_t count[QSGD_MAX_PEERS] = {};
  peers(a[0], &msgs);
  peers(a[1], &tables);
  const qsgd_policy* plan = static_cast<const qsgd_policy*>(address(a[3]));
  const uint32_t bucket = u32(a[4]), s = u32(a[5]);
  const int code = i32(a[6]), lists = plan && !plan->n_buckets ? QSGD_CODE_FIXED : code;      // raw tensors alone: no tables
  if (tables.given) at_least(tables.K, msgs, lists, "tables");
  const uint64_t* bytes = byte_counts(a[2], a[0], msgs, lists, false, count);
  const float eta = fused ? f32(a[8]) : 0.f;
  float* out = static_cast<float*>(cuda_tensor(a[7], fused ? "x" : "acc").data_ptr());
  const qsgd_stream_t stream = stream_of(a[10]);
  const void* const* mp = msgs.as<void>();
  const uint64_t* const* tp = tables.as<uint64_t>();
  return unlocked([&] {
    return fused ? qsgd_policy_decode_sgd_step(mp, tp, bytes, msgs.K, plan, bucket, s, code, out, eta, status, stream)
                 : qsgd_policy_decode_accumulate(mp, tp, bytes, msgs.K, plan, bucket, s, code, out, status, stream);
  });
  QSGD_CATCH
}

// sgd_step(x, acc, eta, K, stream)
PyObject* sgd_step(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  QSGD_ARGS(5)
  QSGD_TRY
  const at::Tensor& x = cuda_tensor(a[0], "x");
  const at::Tensor& acc = cuda_tensor(a[1], "acc");
  const float eta = f32(a[2]);
  const uint32_t K = u32(a[3]);
  const qsgd_stream_t stream = stream_of(a[4]);
  return unlocked([&] {
    return qsgd_sgd_step(static_cast<float*>(x.data_ptr()), static_cast<const float*>(acc.data_ptr()), eta, K,
                         static_cast<uint64_t>(x.numel()), stream);
  });
  QSGD_CATCH
}

PyObject* set_error(PyObject*, PyObject* cls) {
  Py_XINCREF(cls);
  Py_XSETREF(g_error, cls);
  Py_RETURN_NONE;
}

#define QSGD_FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {QSGD_FAST(encode),        QSGD_FAST(encode_static), QSGD_FAST(policy_encode),
                          QSGD_FAST(decode),        QSGD_FAST(policy_decode), QSGD_FAST(sgd_step),
                          {"set_error", set_error, METH_O, nullptr},          {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_qsgd_native", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__qsgd_native(void) {
  PyObject* ctypes = PyImport_ImportModule("_ctypes");
  if (!ctypes) return nullptr;
  g_ctypes_number = PyObject_GetAttrString(ctypes, "_SimpleCData");
  Py_DECREF(ctypes);
  return g_ctypes_number ? PyModule_Create(&kModule) : nullptr;
}
