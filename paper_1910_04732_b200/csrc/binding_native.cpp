// The single calls of the Python binding in native code: arguments are read from the tensors directly and handed to the C
// ABI.  A few-token forward keeps the GPU busy for 4 us; reading its arguments in Python and marshalling them through ctypes
// took about 10 us, so the host was what such a call waited for.
//
// Checks and conversions are those of a plain ctypes call: matrices are 2-d with unit column stride (AssertionError), storage is
// bf16 or fp32 (TypeError), integers wrap to 64 bits, None is a null pointer.  Every function returns the status of
// the call; the interpreter lock is released while the library runs.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/flop.h"

namespace {

struct Stop {};   // a Python exception is set

const at::Tensor* tensor(PyObject* o) {   // nullptr for None
  if (o == Py_None) return nullptr;
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a torch.Tensor, got %s", Py_TYPE(o)->tp_name);
    throw Stop{};
  }
  return &THPVariable_Unpack(o);
}
const at::Tensor& required(PyObject* o) {
  const at::Tensor* t = tensor(o);
  if (!t) { PyErr_SetString(PyExc_AttributeError, "'NoneType' object has no attribute 'shape'"); throw Stop{}; }
  return *t;
}
template <typename T = void> T* ptr(PyObject* o) {
  const at::Tensor* t = tensor(o);
  return t ? static_cast<T*>(t->data_ptr()) : nullptr;
}

struct Mat { void* p = nullptr; int64_t ld = 0, rows = 0, cols = 0; };
int storage(const at::Tensor& t) {
  if (t.scalar_type() == at::kBFloat16) return FLOP_BF16;
  if (t.scalar_type() == at::kFloat) return FLOP_F32;
  PyErr_Format(PyExc_TypeError, "unsupported dtype %s", at::toString(t.scalar_type()));
  throw Stop{};
}
Mat matrix(PyObject* o) {
  const at::Tensor& t = required(o);
  if (t.dim() != 2 || t.stride(1) != 1) {
    PyErr_SetString(PyExc_AssertionError, "matrices must be row-major with unit column stride");
    throw Stop{};
  }
  Mat m;
  m.p = t.data_ptr();
  m.rows = t.size(0); m.cols = t.size(1);
  m.ld = m.rows > 1 ? t.stride(0) : std::max(t.stride(0), m.cols);
  return m;
}
Mat optional_matrix(PyObject* o) { return o == Py_None ? Mat{} : matrix(o); }

int64_t integer(PyObject* o) {
  const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
  if (v == (unsigned long long)-1 && PyErr_Occurred()) throw Stop{};
  return (int64_t)v;
}
int flag(PyObject* o) {   // int(o)
  PyObject* v = PyNumber_Long(o);
  if (!v) throw Stop{};
  const unsigned long m = PyLong_AsUnsignedLongMask(v);
  Py_DECREF(v);
  return (int)m;
}
flop_hc_params_t hard_concrete(PyObject* o) {
  float v[3];
  for (int i = 0; i < 3; ++i) {
    PyObject* at = PyLong_FromLong(i);
    PyObject* e = at ? PyObject_GetItem(o, at) : nullptr;   // float(o[i]), whatever o is
    Py_XDECREF(at);
    PyObject* d = e ? PyNumber_Float(e) : nullptr;
    Py_XDECREF(e);
    if (!d) throw Stop{};
    v[i] = (float)PyFloat_AS_DOUBLE(d);
    Py_DECREF(d);
  }
  return flop_hc_params_t{v[0], v[1], v[2]};
}
void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }
size_t numel(PyObject* o) { const at::Tensor* t = tensor(o); return t ? (size_t)t->numel() : 0; }

// Runs the library call without the interpreter lock and returns its status as a Python integer.  The lock is back before an
// exception (the library's planners allocate on the host) leaves the call and becomes a Python one.
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};
template <typename F> PyObject* call(F&& f) {
  int status;
  {
    Unlocked u;
    status = f();
  }
  return PyLong_FromLong(status);
}

#define FLOP_METHOD(name, count)                                                        \
  PyObject* name##_body(PyObject* const* a);                                            \
  PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n) {                         \
    HANDLE_TH_ERRORS                                                                    \
    if (n != (count)) {                                                                 \
      PyErr_Format(PyExc_TypeError, #name ": %d arguments expected", (int)(count));     \
      return nullptr;                                                                   \
    }                                                                                   \
    try { return name##_body(a); } catch (const Stop&) { return nullptr; }              \
    END_HANDLE_TH_ERRORS                                                                \
  }                                                                                     \
  PyObject* name##_body(PyObject* const* a)

FLOP_METHOD(gate_sample, 7) {   // log_alpha, hc, seed, offset, z, mask, dz_dla
  const float* la = static_cast<const float*>(required(a[0]).data_ptr());
  const int64_t n = (int64_t)numel(a[0]);
  const flop_hc_params_t hc = hard_concrete(a[1]);
  const uint64_t seed = (uint64_t)integer(a[2]), offset = (uint64_t)integer(a[3]);
  float* z = ptr<float>(a[4]); uint8_t* mask = ptr<uint8_t>(a[5]); float* dz = ptr<float>(a[6]);
  void* st = stream();
  return call([&] { return flop_gate_sample(la, n, hc, seed, offset, z, mask, dz, st); });
}

FLOP_METHOD(gated_lowrank_fwd, 7) {   // X, Q, P, z, Y, H_save, ws
  const Mat X = matrix(a[0]), Q = matrix(a[1]), P = matrix(a[2]), Y = matrix(a[4]), H = optional_matrix(a[5]);
  const int dt = storage(required(a[0]));
  const float* z = ptr<float>(a[3]); void* ws = ptr(a[6]); const size_t wb = numel(a[6]);
  void* st = stream();
  return call([&] { return flop_gated_lowrank_fwd(X.p, X.ld, Q.p, Q.ld, P.p, P.ld, z, Y.p, Y.ld, H.p, H.ld, X.rows, X.cols, P.rows, P.cols, dt, ws, wb, st); });
}

FLOP_METHOD(gated_lowrank_bwd, 13) {   // dY, X, Q, P, z, dz_dla, H_save, dX, dP, dQ, dlog_alpha, ws, accumulate
  const Mat dY = matrix(a[0]), X = matrix(a[1]), Q = matrix(a[2]), P = matrix(a[3]), H = matrix(a[6]);
  const Mat dX = optional_matrix(a[7]), dP = optional_matrix(a[8]), dQ = optional_matrix(a[9]);
  const int dt = storage(required(a[1]));
  const int wdt = a[8] != Py_None ? storage(required(a[8])) : a[9] != Py_None ? storage(required(a[9])) : dt;
  const float *z = ptr<float>(a[4]), *dz = ptr<float>(a[5]); float* dla = ptr<float>(a[10]);
  void* ws = ptr(a[11]); const size_t wb = numel(a[11]); const int acc = flag(a[12]);
  void* st = stream();
  return call([&] {
    return flop_gated_lowrank_bwd(dY.p, dY.ld, X.p, X.ld, Q.p, Q.ld, P.p, P.ld, z, dz, H.p, H.ld, dX.p, dX.ld, dP.p, dP.ld, dQ.p, dQ.ld, dla, acc,
                                  X.rows, X.cols, P.rows, P.cols, dt, wdt, ws, wb, st);
  });
}

FLOP_METHOD(expected_l0_lagrangian, 10) {   // log_alpha, seg_off, seg_size, hc, target, lam, out4, seg_expected, dlog_alpha, ws
  const float* la = static_cast<const float*>(required(a[0]).data_ptr());
  const int64_t n = (int64_t)numel(a[0]);
  const int32_t n_seg = (int32_t)required(a[2]).numel();
  const int64_t* off = ptr<int64_t>(a[1]); const float* size = ptr<float>(a[2]);
  const flop_hc_params_t hc = hard_concrete(a[3]);
  const float *target = ptr<float>(a[4]), *lam = ptr<float>(a[5]);
  float *out4 = ptr<float>(a[6]), *seg = ptr<float>(a[7]), *dla = ptr<float>(a[8]);
  void* ws = ptr(a[9]); const size_t wb = numel(a[9]);
  void* st = stream();
  return call([&] { return flop_expected_l0_lagrangian(la, n, off, size, n_seg, hc, target, lam, out4, seg, dla, ws, wb, st); });
}

FLOP_METHOD(gated_embedding_fwd, 6) {   // ids, E, O, z, Y, H_save
  const Mat E = matrix(a[1]), O = matrix(a[2]), Y = matrix(a[4]), H = matrix(a[5]);
  const int dt = storage(required(a[1]));
  const int64_t T = required(a[0]).numel();
  const int32_t* ids = ptr<int32_t>(a[0]); const float* z = ptr<float>(a[3]);
  void* st = stream();
  return call([&] { return flop_gated_embedding_fwd(ids, T, E.p, E.ld, E.rows, O.p, O.ld, z, Y.p, Y.ld, H.p, H.ld, E.cols, O.cols, dt, st); });
}

FLOP_METHOD(gated_embedding_bwd, 12) {   // dY, ids, E, O, z, dz_dla, H_save, dE, dO, dlog_alpha, ws, accumulate
  const Mat dY = matrix(a[0]), E = matrix(a[2]), O = matrix(a[3]), H = matrix(a[6]), dE = optional_matrix(a[7]), dO = optional_matrix(a[8]);
  const int dt = storage(required(a[2])), wdt = a[8] != Py_None ? storage(required(a[8])) : (int)FLOP_BF16;
  const int64_t T = required(a[1]).numel();
  const int32_t* ids = ptr<int32_t>(a[1]); const float *z = ptr<float>(a[4]), *dz = ptr<float>(a[5]); float* dla = ptr<float>(a[9]);
  void* ws = ptr(a[10]); const size_t wb = numel(a[10]); const int acc = flag(a[11]);
  void* st = stream();
  return call([&] {
    return flop_gated_embedding_bwd(dY.p, dY.ld, ids, T, E.p, E.ld, E.rows, O.p, O.ld, z, dz, H.p, H.ld, (float*)dE.p, dE.ld, dO.p, dO.ld, dla, acc,
                                    E.cols, O.cols, dt, wdt, ws, wb, st);
  });
}

FLOP_METHOD(compact_ranks, 10) {   // log_alpha_or_z, mode, hc, idx, k_dev, z_det, P, Q, Pc, Qc
  const float* in = static_cast<const float*>(required(a[0]).data_ptr());
  const int64_t r = (int64_t)numel(a[0]);
  const int mode = (int)integer(a[1]);
  const flop_hc_params_t hc = hard_concrete(a[2]);
  int32_t *idx = ptr<int32_t>(a[3]), *k = ptr<int32_t>(a[4]); float* z = ptr<float>(a[5]);
  const Mat P = optional_matrix(a[6]), Q = optional_matrix(a[7]), Pc = optional_matrix(a[8]), Qc = optional_matrix(a[9]);
  const int dt = a[6] != Py_None ? storage(required(a[6])) : (int)FLOP_F32;
  void* st = stream();
  return call([&] {
    return flop_compact_ranks(in, mode, hc, r, P.p, P.ld, Q.p, Q.ld, Q.cols, P.rows, dt, idx, k, z, Pc.p, Pc.ld, Qc.p, Qc.ld, nullptr, 0, st);
  });
}

FLOP_METHOD(compact_fwd, 6) {   // X, Qc, Pc, Y, k, ws
  const Mat X = matrix(a[0]), Qc = matrix(a[1]), Pc = matrix(a[2]), Y = matrix(a[3]);
  const int dt = storage(required(a[0]));
  const int64_t k = integer(a[4]);
  void* ws = ptr(a[5]); const size_t wb = numel(a[5]);
  void* st = stream();
  return call([&] { return flop_compact_fwd(X.p, X.ld, Qc.p, Qc.ld, Pc.p, Pc.ld, Y.p, Y.ld, X.rows, X.cols, Pc.rows, k, dt, ws, wb, st); });
}

#define FLOP_ENTRY(name) {#name, (PyCFunction)(void*)name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FLOP_ENTRY(gate_sample), FLOP_ENTRY(gated_lowrank_fwd), FLOP_ENTRY(gated_lowrank_bwd), FLOP_ENTRY(expected_l0_lagrangian),
                         FLOP_ENTRY(gated_embedding_fwd), FLOP_ENTRY(gated_embedding_bwd), FLOP_ENTRY(compact_ranks), FLOP_ENTRY(compact_fwd),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding_native(void) { return PyModule_Create(&module); }
