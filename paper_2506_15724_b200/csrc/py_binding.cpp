// Python entry points of the library's asynchronous calls: pointers, strides and sizes are read from the tensors here, the
// status comes back as an int. What bounds a call on one layer is the host: with the arguments gathered in Python and handed
// over by ctypes a decode call took 5.4 us, here 3.1, nearly all of it the launch.
#define PY_SSIZE_T_CLEAN
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "madakv.h"

namespace {

// The arguments of one call, in order. A failed conversion throws; the Python error is set.
struct Args {
  PyObject* const* at;
  Py_ssize_t left;
  Py_buffer cfg_buf;
  bool has_cfg = false;

  Args(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) : at(args), left(n) {
    if (n != want) fail(PyExc_TypeError, "wrong number of arguments");
  }
  ~Args() {
    if (has_cfg) PyBuffer_Release(&cfg_buf);
  }
  [[noreturn]] static void fail(PyObject* type, const char* what) {
    PyErr_SetString(type, what);
    throw python_error();
  }
  PyObject* next() {
    --left;
    return *at++;
  }
  const madakv_config* config() {
    PyObject* o = next();
    PyObject* inner = PyObject_CheckBuffer(o) ? nullptr : PyObject_GetAttrString(o, "_obj");  // (what ctypes.byref gives)
    if (!inner && PyErr_Occurred()) throw python_error();
    const int rc = PyObject_GetBuffer(inner ? inner : o, &cfg_buf, PyBUF_SIMPLE);
    Py_XDECREF(inner);
    if (rc) throw python_error();
    has_cfg = true;
    if (cfg_buf.len < (Py_ssize_t)sizeof(madakv_config)) fail(PyExc_TypeError, "expected a MadakvConfig");
    return static_cast<const madakv_config*>(cfg_buf.buf);
  }
  const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a tensor");
    return THPVariable_Unpack(o);
  }
  template <typename T = void>
  T* ptr() {
    PyObject* o = next();
    return o == Py_None ? nullptr : static_cast<T*>(tensor(o).data_ptr());
  }
  const at::Tensor& tensor() { return tensor(next()); }
  int32_t integer() {
    const long v = PyLong_AsLong(next());
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return (int32_t)v;
  }
};

madakv_strides strides(const at::Tensor& t) {
  const auto st = t.strides();
  if (st.size() != 5 || st[4] != 1) Args::fail(PyExc_AssertionError, "expected [B, L, H, tokens, d] with contiguous d");
  return {st[0], st[1], st[2], st[3]};
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The call itself runs without the interpreter's lock, as it does through ctypes: a launch may wait for room in the queue.
template <typename F>
PyObject* without_lock(F call) {
  int rc;
  Py_BEGIN_ALLOW_THREADS;
  rc = call();
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(rc);
}

template <bool kGiven>
PyObject* score(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(args, n, 7);
  const madakv_config* cfg = a.config();
  const at::Tensor &q = a.tensor(), &k = a.tensor();
  const madakv_strides sq = strides(q), sk = strides(k);
  const int32_t* seq_len = a.ptr<int32_t>();
  float *lse = a.ptr<float>(), *psi = a.ptr<float>();
  const at::Tensor& ws = a.tensor();
  void *qp = q.data_ptr(), *kp = k.data_ptr(), *wp = ws.data_ptr(), *st = stream();
  const size_t bytes = (size_t)ws.numel();
  return without_lock([&] {
    return kGiven ? madakv_score_lse(cfg, qp, sq, kp, sk, seq_len, lse, psi, wp, bytes, st)
                  : madakv_score(cfg, qp, sq, kp, sk, seq_len, lse, psi, wp, bytes, st);
  });
  END_HANDLE_TH_ERRORS
}

PyObject* allocate(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(args, n, 11);
  const madakv_config* cfg = a.config();
  const float* psi = a.ptr<float>();
  const uint8_t* mask = a.ptr<uint8_t>();
  const int32_t *seq_len = a.ptr<int32_t>(), *budget = a.ptr<int32_t>();
  double *mass = a.ptr<double>(), *pref = a.ptr<double>();
  int32_t* demand = a.ptr<int32_t>();
  double* phi = a.ptr<double>();
  int32_t* budgets = a.ptr<int32_t>();
  const at::Tensor& ws = a.tensor();
  void *wp = ws.data_ptr(), *st = stream();
  const size_t bytes = (size_t)ws.numel();
  return without_lock(
      [&] { return madakv_allocate(cfg, psi, mask, seq_len, budget, mass, pref, demand, phi, budgets, wp, bytes, st); });
  END_HANDLE_TH_ERRORS
}

PyObject* allocate_layer(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(args, n, 12);
  const madakv_config* cfg = a.config();
  const int32_t layer = a.integer();
  const float* psi = a.ptr<float>();
  const uint8_t* mask = a.ptr<uint8_t>();
  const int32_t *seq_len = a.ptr<int32_t>(), *budget = a.ptr<int32_t>();
  double *mass = a.ptr<double>(), *pref = a.ptr<double>();
  int32_t* demand = a.ptr<int32_t>();
  double* phi = a.ptr<double>();
  int32_t* budgets = a.ptr<int32_t>();
  const at::Tensor& ws = a.tensor();
  void *wp = ws.data_ptr(), *st = stream();
  const size_t bytes = (size_t)ws.numel();
  return without_lock([&] {
    return madakv_allocate_layer(cfg, layer, psi, mask, seq_len, budget, mass, pref, demand, phi, budgets, wp, bytes, st);
  });
  END_HANDLE_TH_ERRORS
}

PyObject* demand_layer(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(args, n, 8);
  const madakv_config* cfg = a.config();
  const float* psi = a.ptr<float>();
  const uint8_t* mask = a.ptr<uint8_t>();
  const int32_t* seq_len = a.ptr<int32_t>();
  double *mass = a.ptr<double>(), *pref = a.ptr<double>();
  int32_t* demand = a.ptr<int32_t>();
  const at::Tensor& ws = a.tensor();
  void *wp = ws.data_ptr(), *st = stream();
  const size_t bytes = (size_t)ws.numel();
  return without_lock([&] { return madakv_demand_layer(cfg, psi, mask, seq_len, mass, pref, demand, wp, bytes, st); });
  END_HANDLE_TH_ERRORS
}

PyObject* select(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(args, n, 9);
  const madakv_config* cfg = a.config();
  const float* psi = a.ptr<float>();
  const uint8_t* mask = a.ptr<uint8_t>();
  const int32_t *seq_len = a.ptr<int32_t>(), *budgets = a.ptr<int32_t>();
  int32_t* kept_len = a.ptr<int32_t>();
  int64_t* seg_off = a.ptr<int64_t>();
  const at::Tensor &kept_idx = a.tensor(), &ws = a.tensor();
  int32_t* ip = static_cast<int32_t*>(kept_idx.data_ptr());
  const int64_t capacity = kept_idx.numel();
  void *wp = ws.data_ptr(), *st = stream();
  const size_t bytes = (size_t)ws.numel();
  return without_lock(
      [&] { return madakv_select(cfg, psi, mask, seq_len, budgets, kept_len, seg_off, ip, capacity, wp, bytes, st); });
  END_HANDLE_TH_ERRORS
}

PyObject* compact(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(args, n, 9);
  const madakv_config* cfg = a.config();
  const at::Tensor &k = a.tensor(), &v = a.tensor();
  if (k.strides() != v.strides()) Args::fail(PyExc_AssertionError, "k and v must have the same strides");
  const madakv_strides skv = strides(k);
  const int32_t* kept_idx = a.ptr<int32_t>();
  const int64_t* seg_off = a.ptr<int64_t>();
  const int32_t* kept_len = a.ptr<int32_t>();
  const at::Tensor& k_c = a.tensor();
  void* v_c = a.ptr();
  const at::Tensor& ws = a.tensor();
  void *kp = k.data_ptr(), *vp = v.data_ptr(), *kc = k_c.data_ptr(), *wp = ws.data_ptr(), *st = stream();
  const int64_t capacity = k_c.size(0);
  const size_t bytes = (size_t)ws.numel();
  return without_lock(
      [&] { return madakv_compact(cfg, kp, vp, skv, kept_idx, seg_off, kept_len, kc, v_c, capacity, wp, bytes, st); });
  END_HANDLE_TH_ERRORS
}

PyObject* decode_attn(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args a(args, n, 12);
  const madakv_config* cfg = a.config();
  const int32_t layer = a.integer();
  const void *q = a.ptr(), *k_new = a.ptr(), *v_new = a.ptr();
  const at::Tensor& k_c = a.tensor();
  void* v_c = a.ptr();
  const int64_t* seg_off = a.ptr<int64_t>();
  int32_t* kept_len = a.ptr<int32_t>();
  void* out = a.ptr();
  float* lse = a.ptr<float>();
  const at::Tensor& ws = a.tensor();
  void *kc = k_c.data_ptr(), *wp = ws.data_ptr(), *st = stream();
  const int64_t capacity = k_c.size(0);
  const size_t bytes = (size_t)ws.numel();
  return without_lock([&] {
    return madakv_decode_attn(cfg, layer, q, k_new, v_new, kc, v_c, seg_off, kept_len, capacity, out, lse, wp, bytes, st);
  });
  END_HANDLE_TH_ERRORS
}

template <typename F>
PyCFunction as_method(F f) {
  return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f));
}
PyMethodDef methods[] = {
    {"score", as_method(score<false>), METH_FASTCALL, nullptr},
    {"score_lse", as_method(score<true>), METH_FASTCALL, nullptr},
    {"allocate", as_method(allocate), METH_FASTCALL, nullptr},
    {"allocate_layer", as_method(allocate_layer), METH_FASTCALL, nullptr},
    {"demand_layer", as_method(demand_layer), METH_FASTCALL, nullptr},
    {"select", as_method(select), METH_FASTCALL, nullptr},
    {"compact", as_method(compact), METH_FASTCALL, nullptr},
    {"decode_attn", as_method(decode_attn), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
