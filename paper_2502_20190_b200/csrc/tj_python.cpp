// CPython entry points for the calls a training loop makes every iteration (binding.py holds the rest in ctypes): plain integers and
// floats in, the C ABI's status out.  A ctypes call costs 1.5-3 us of marshalling, as much as a kernel launch; these cost 0.1-0.3.
// The functions of libtj.so are handed over by address (init), so this file links against nothing.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/tj.h"

namespace {

decltype(&tj_actor_step) f_actor_step;
decltype(&tj_replay_sample) f_replay_sample;
decltype(&tj_td_error) f_td_error;
decltype(&tj_publish_weights) f_publish_weights;
decltype(&tj_sgd_step) f_sgd_step;
decltype(&tj_adam_step) f_adam_step;
decltype(&tj_ppo_step) f_ppo_step;
decltype(&tj_gae) f_gae;
decltype(&tj_normalize) f_normalize;
decltype(&tj_segment_minibatch) f_segment_minibatch;

bool ready = false;   // init() has handed over every function

// arguments in order, converted as they are asked for; `bad` stays set after the first failure
struct Args {
  PyObject* const* a;
  Py_ssize_t n, i = 0;
  bool bad = false;
  Args(PyObject* const* args, Py_ssize_t count, Py_ssize_t want, bool needs_init = true) : a(args), n(count) {
    if (needs_init && !ready) {
      PyErr_SetString(PyExc_RuntimeError, "init() has not been called with the library's functions");
      bad = true;
    } else if (n != want) {
      PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
      bad = true;
    }
  }
  unsigned long long word() {                 // an integer modulo 2^64, as ctypes takes it; the caller narrows it
    if (bad) return 0;
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(a[i++]);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) bad = true;
    return v;
  }
  long long integer() { return (long long)word(); }
  double real() {
    if (bad) return 0.0;
    const double v = PyFloat_AsDouble(a[i++]);
    if (v == -1.0 && PyErr_Occurred()) bad = true;
    return v;
  }
  // an address: None is null
  template <typename T>
  T* pointer() {
    if (bad) return nullptr;
    PyObject* o = a[i++];
    if (o == Py_None) return nullptr;
    const unsigned long long v = PyLong_AsUnsignedLongLong(o);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) bad = true;
    return reinterpret_cast<T*>(static_cast<uintptr_t>(v));
  }
  // a ctypes structure, by its buffer
  template <typename T>
  const T* structure() {
    if (bad) return nullptr;
    Py_buffer b;
    if (PyObject_GetBuffer(a[i++], &b, PyBUF_SIMPLE) != 0) { bad = true; return nullptr; }
    const T* p = b.len == (Py_ssize_t)sizeof(T) ? static_cast<const T*>(b.buf) : nullptr;
    PyBuffer_Release(&b);                     // the caller's argument keeps the structure alive during the call
    if (!p) {
      PyErr_SetString(PyExc_TypeError, "a structure of another size");
      bad = true;
    }
    return p;
  }
};

PyObject* init(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 10, false);
  ready = false;
  f_actor_step = reinterpret_cast<decltype(f_actor_step)>(a.pointer<void>());
  f_replay_sample = reinterpret_cast<decltype(f_replay_sample)>(a.pointer<void>());
  f_td_error = reinterpret_cast<decltype(f_td_error)>(a.pointer<void>());
  f_publish_weights = reinterpret_cast<decltype(f_publish_weights)>(a.pointer<void>());
  f_sgd_step = reinterpret_cast<decltype(f_sgd_step)>(a.pointer<void>());
  f_adam_step = reinterpret_cast<decltype(f_adam_step)>(a.pointer<void>());
  f_ppo_step = reinterpret_cast<decltype(f_ppo_step)>(a.pointer<void>());
  f_gae = reinterpret_cast<decltype(f_gae)>(a.pointer<void>());
  f_normalize = reinterpret_cast<decltype(f_normalize)>(a.pointer<void>());
  f_segment_minibatch = reinterpret_cast<decltype(f_segment_minibatch)>(a.pointer<void>());
  if (a.bad) return nullptr;
  if (!f_actor_step || !f_replay_sample || !f_td_error || !f_publish_weights || !f_sgd_step || !f_adam_step || !f_ppo_step || !f_gae ||
      !f_normalize || !f_segment_minibatch) {
    PyErr_SetString(PyExc_ValueError, "a null function");
    return nullptr;
  }
  ready = true;
  Py_RETURN_NONE;
}

PyObject* status(int st) { return PyLong_FromLong(st); }

// the library's calls may wait for the GPU's queue: other threads run meanwhile, as under ctypes
#define TJ_CALL(expr) Py_BEGIN_ALLOW_THREADS st = (expr); Py_END_ALLOW_THREADS

PyObject* actor_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 3);
  tj_ctx* h = a.pointer<tj_ctx>();
  const int steps = (int)a.integer();
  float* dbg = a.pointer<float>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_actor_step(h, steps, dbg))
  return status(st);
}

PyObject* replay_sample(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 4);
  tj_ctx* h = a.pointer<tj_ctx>();
  const int bound = (int)a.integer();
  int32_t* idx = a.pointer<int32_t>();
  const tj_batch* b = a.structure<tj_batch>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_replay_sample(h, bound, idx, b))
  return status(st);
}

PyObject* td_error(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 5);
  tj_ctx* h = a.pointer<tj_ctx>();
  const tj_batch* b = a.structure<tj_batch>();
  float *td = a.pointer<float>(), *hub = a.pointer<float>(), *loss = a.pointer<float>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_td_error(h, b, td, hub, loss))
  return status(st);
}

// -> (status, version)
PyObject* publish_weights(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 4);
  tj_ctx* h = a.pointer<tj_ctx>();
  const void* blob = a.pointer<void>();
  const size_t bytes = (size_t)a.integer();
  const int on_device = (int)a.integer();
  if (a.bad) return nullptr;
  int st;
  int64_t version = 0;
  TJ_CALL(f_publish_weights(h, blob, bytes, on_device, &version))
  PyObject* t = PyTuple_New(2);
  if (!t) return nullptr;
  PyTuple_SET_ITEM(t, 0, PyLong_FromLong(st));
  PyTuple_SET_ITEM(t, 1, PyLong_FromLongLong(version));
  return t;
}

PyObject* sgd_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 6);
  tj_ctx* h = a.pointer<tj_ctx>();
  const tj_batch* b = a.structure<tj_batch>();
  const float lr = (float)a.real();
  float* theta = a.pointer<float>();
  const float* target = a.pointer<float>();
  float* loss = a.pointer<float>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_sgd_step(h, b, lr, theta, target, loss))
  return status(st);
}

PyObject* adam_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 12);
  tj_ctx* h = a.pointer<tj_ctx>();
  const tj_batch* b = a.structure<tj_batch>();
  const float lr = (float)a.real(), b1 = (float)a.real(), b2 = (float)a.real(), eps = (float)a.real();
  const int64_t t = a.integer();
  float* theta = a.pointer<float>();
  const float* target = a.pointer<float>();
  float *m = a.pointer<float>(), *v = a.pointer<float>(), *loss = a.pointer<float>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_adam_step(h, b, lr, b1, b2, eps, t, theta, target, m, v, loss))
  return status(st);
}

// the batch's six fields, then the hyperparameters
PyObject* ppo_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 19);
  tj_ctx* h = a.pointer<tj_ctx>();
  tj_ppo_batch b;
  b.n = (int32_t)a.integer();
  b.obs = a.pointer<float>(); b.act = a.pointer<int32_t>(); b.logp_old = a.pointer<float>(); b.adv = a.pointer<float>(); b.ret = a.pointer<float>();
  const float lr = (float)a.real(), b1 = (float)a.real(), b2 = (float)a.real(), eps = (float)a.real();
  const int64_t t = a.integer();
  const float clip = (float)a.real(), cv = (float)a.real(), ce = (float)a.real();
  float *theta = a.pointer<float>(), *m = a.pointer<float>(), *v = a.pointer<float>(), *stats = a.pointer<float>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_ppo_step(h, &b, lr, b1, b2, eps, t, clip, cv, ce, theta, m, v, stats))
  return status(st);
}

PyObject* gae(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 10);
  tj_ctx* h = a.pointer<tj_ctx>();
  const float *rew = a.pointer<float>(), *val = a.pointer<float>();
  const uint8_t* done = a.pointer<uint8_t>();
  const int T = (int)a.integer(), N = (int)a.integer();
  const float gamma = (float)a.real(), lambda = (float)a.real();
  float *adv = a.pointer<float>(), *ret = a.pointer<float>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_gae(h, rew, val, done, T, N, gamma, lambda, adv, ret))
  return status(st);
}

PyObject* normalize(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 5);
  tj_ctx* h = a.pointer<tj_ctx>();
  const float* x = a.pointer<float>();
  const int64_t count = a.integer();
  const float eps = (float)a.real();
  float* out = a.pointer<float>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_normalize(h, x, count, eps, out))
  return status(st);
}

PyObject* segment_minibatch(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Args a(args, n, 7);
  tj_ctx* h = a.pointer<tj_ctx>();
  const tj_segment* seg = a.structure<tj_segment>();
  const float *adv = a.pointer<float>(), *ret = a.pointer<float>();
  const uint64_t id = a.word();
  const int64_t first = a.integer();
  const tj_ppo_minibatch* mb = a.structure<tj_ppo_minibatch>();
  if (a.bad) return nullptr;
  int st;
  TJ_CALL(f_segment_minibatch(h, seg, adv, ret, id, first, mb))
  return status(st);
}

#define TJ_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {TJ_METHOD(init), TJ_METHOD(actor_step), TJ_METHOD(replay_sample), TJ_METHOD(td_error), TJ_METHOD(publish_weights),
                         TJ_METHOD(sgd_step), TJ_METHOD(adam_step), TJ_METHOD(ppo_step), TJ_METHOD(gae), TJ_METHOD(normalize),
                         TJ_METHOD(segment_minibatch), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tjcall", "libtj's per-iteration calls", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tjcall() { return PyModule_Create(&module); }
