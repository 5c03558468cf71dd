// Argument marshalling of the calls a training loop makes: torch tensors -> device pointers -> the C entry points.
//
// One function per entry point, same argument order as include/shadowsync.h; each returns the ss_status as an int
// (binding.py turns a negative one into SsError).  Unpacking a tensor here costs a few nanoseconds where the ctypes
// route pays a Python call per attribute: the host side of a small call is mostly this.  Nothing is computed here.
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>
#include <string.h>
#include "../../include/shadowsync.h"

namespace {

struct Bad {};   // a Python error is set

struct Args {
  PyObject* const* v;
  Py_ssize_t n, i = 0;
  PyObject* next() {
    if (i >= n) { PyErr_SetString(PyExc_TypeError, "too few arguments"); throw Bad(); }
    return v[i++];
  }
  const at::Tensor* tensor() {
    PyObject* o = next();
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a tensor or None"); throw Bad(); }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda()) { PyErr_SetString(PyExc_ValueError, "expected a CUDA tensor"); throw Bad(); }
    if (!t.is_contiguous()) { PyErr_SetString(PyExc_ValueError, "expected a contiguous tensor"); throw Bad(); }
    return &t;
  }
  template <typename T> T* ptr() {
    const at::Tensor* t = tensor();
    return t ? static_cast<T*>(t->data_ptr()) : nullptr;
  }
  void* buffer(size_t* bytes) {     // a workspace: pointer and size
    const at::Tensor* t = tensor();
    *bytes = t ? (size_t)t->nbytes() : 0;
    return t ? t->data_ptr() : nullptr;
  }
  int64_t i64() {
    const long long x = PyLong_AsLongLong(next());
    if (x == -1 && PyErr_Occurred()) throw Bad();
    return x;
  }
  int i32() {
    const int64_t x = i64();
    if (x != (int)x) { PyErr_SetString(PyExc_OverflowError, "argument does not fit a C int"); throw Bad(); }
    return (int)x;
  }
  float f32() {
    const double x = PyFloat_AsDouble(next());
    if (x == -1.0 && PyErr_Occurred()) throw Bad();
    return (float)x;
  }
  const ss_mlp_desc* desc() {       // address of the ctypes struct an MlpSpec holds
    void* p = PyLong_AsVoidPtr(next());
    if (!p && PyErr_Occurred()) throw Bad();
    return static_cast<const ss_mlp_desc*>(p);
  }
  ss_step_plan plan() {             // None, or the handle as an int
    PyObject* o = next();
    if (o == Py_None) return nullptr;
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) throw Bad();
    return static_cast<ss_step_plan>(p);
  }
  // None: torch's current stream; an object with .cuda_stream; or the handle as an int
  ss_stream stream() {
    PyObject* o = next();
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    if (PyLong_Check(o)) return PyLong_AsVoidPtr(o);
    static PyObject* name = PyUnicode_InternFromString("cuda_stream");
    PyObject* h = PyObject_GetAttr(o, name);
    if (!h) throw Bad();
    void* p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!p && PyErr_Occurred()) throw Bad();
    return p;
  }
  // a list or tuple of tensors -> array of pointers; returns the length, -1 for None
  int tensors(void** out, int cap) {
    PyObject* o = next();
    if (o == Py_None) return -1;
    PyObject* seq = PySequence_Fast(o, "expected a sequence of tensors");
    if (!seq) throw Bad();
    const Py_ssize_t m = PySequence_Fast_GET_SIZE(seq);
    Args e{PySequence_Fast_ITEMS(seq), m};
    try {
      for (Py_ssize_t k = 0; k < m; ++k) {
        void* p = e.ptr<void>();
        if (k < cap) out[k] = p;
      }
    } catch (Bad&) { Py_DECREF(seq); throw; }
    Py_DECREF(seq);
    return (int)m;
  }
};

struct NoGil {     // the interpreter lock is released while the call enqueues (a launch may wait for room in the queue)
  PyThreadState* s = PyEval_SaveThread();
  ~NoGil() { PyEval_RestoreThread(s); }
};

template <typename F>
PyObject* guarded(PyObject* const* args, Py_ssize_t n, F f) {
  try {
    Args a{args, n};
    const int status = f(a);
    return PyLong_FromLong(status);
  } catch (Bad&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

#define SS_PY(NAME) PyObject* NAME(PyObject*, PyObject* const* args, Py_ssize_t nargs)

SS_PY(embbag_fwd) {
  return guarded(args, nargs, [](Args& a) {
    const float* tables = a.ptr<float>();
    const int T = a.i32(); const int64_t N = a.i64(); const int D = a.i32();
    const int32_t* indices = a.ptr<int32_t>(); const int32_t* offsets = a.ptr<int32_t>();
    const int B = a.i32();
    float* f = a.ptr<float>(); const int64_t ldf = a.i64();
    void* h = a.ptr<void>(); const int64_t ldh = a.i64();
    const int col0 = a.i32();
    int32_t* st = a.ptr<int32_t>();
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_embbag_fwd(tables, T, N, D, indices, offsets, B, f, ldf, h, ldh, col0, st, stream);
  });
}

SS_PY(embbag_bwd_adagrad) {
  return guarded(args, nargs, [](Args& a) {
    float* tables = a.ptr<float>(); float* row_state = a.ptr<float>();
    const int T = a.i32(); const int64_t N = a.i64(); const int D = a.i32();
    const int32_t* indices = a.ptr<int32_t>(); const int32_t* offsets = a.ptr<int32_t>();
    const int B = a.i32(); const int64_t L = a.i64();
    const float* grad = a.ptr<float>(); const int64_t ld = a.i64(); const int col0 = a.i32();
    const float lr = a.f32(), eps = a.f32();
    size_t bytes; void* ws = a.buffer(&bytes);
    int32_t* uniq = a.ptr<int32_t>(); int32_t* seg = a.ptr<int32_t>(); int32_t* perm = a.ptr<int32_t>();
    int32_t* num = a.ptr<int32_t>(); int32_t* st = a.ptr<int32_t>();
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_embbag_bwd_adagrad(tables, row_state, T, N, D, indices, offsets, B, L, grad, ld, col0, lr, eps, ws, bytes,
                                 uniq, seg, perm, num, st, stream);
  });
}

SS_PY(embbag_bwd_sort) {
  return guarded(args, nargs, [](Args& a) {
    const int T = a.i32(); const int64_t N = a.i64(); const int D = a.i32();
    const int32_t* indices = a.ptr<int32_t>(); const int32_t* offsets = a.ptr<int32_t>();
    const int B = a.i32(); const int64_t L = a.i64();
    size_t bytes; void* ws = a.buffer(&bytes);
    int32_t* uniq = a.ptr<int32_t>(); int32_t* seg = a.ptr<int32_t>(); int32_t* perm = a.ptr<int32_t>();
    int32_t* num = a.ptr<int32_t>(); int32_t* st = a.ptr<int32_t>();
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_embbag_bwd_sort(T, N, D, indices, offsets, B, L, ws, bytes, uniq, seg, perm, num, st, stream);
  });
}

SS_PY(embbag_bwd_apply) {
  return guarded(args, nargs, [](Args& a) {
    float* tables = a.ptr<float>(); float* row_state = a.ptr<float>();
    const int T = a.i32(); const int64_t N = a.i64(); const int D = a.i32();
    const int B = a.i32(); const int64_t L = a.i64();
    const float* grad = a.ptr<float>(); const int64_t ld = a.i64(); const int col0 = a.i32();
    const float lr = a.f32(), eps = a.f32();
    size_t bytes; void* ws = a.buffer(&bytes);
    int32_t* st = a.ptr<int32_t>();
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_embbag_bwd_apply(tables, row_state, T, N, D, B, L, grad, ld, col0, lr, eps, ws, bytes, st, stream);
  });
}

SS_PY(mlp_fwd) {
  return guarded(args, nargs, [](Args& a) {
    const ss_mlp_desc* d = a.desc();
    const float* w = a.ptr<float>(); const void* wb = a.ptr<void>(); const float* dense = a.ptr<float>();
    float* cf = a.ptr<float>(); void* cb = a.ptr<void>();
    const int B = a.i32();
    const float* labels = a.ptr<float>(); float* logit = a.ptr<float>(); float* prob = a.ptr<float>();
    float* loss = a.ptr<float>();
    size_t bytes; void* ws = a.buffer(&bytes);
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_mlp_fwd(d, w, wb, dense, cf, cb, B, labels, logit, prob, loss, ws, bytes, stream);
  });
}

SS_PY(mlp_bwd) {
  return guarded(args, nargs, [](Args& a) {
    const ss_mlp_desc* d = a.desc();
    float* w = a.ptr<float>(); void* wb = a.ptr<void>(); float* acc = a.ptr<float>(); float* grads = a.ptr<float>();
    const float* dense = a.ptr<float>(); const float* cf = a.ptr<float>(); const void* cb = a.ptr<void>();
    const float* labels = a.ptr<float>(); const float* prob = a.ptr<float>();
    const int B = a.i32(); const float lr = a.f32(), eps = a.f32(); const int apply = a.i32();
    float* gp = a.ptr<float>(); const int64_t ld = a.i64();
    size_t bytes; void* ws = a.buffer(&bytes);
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_mlp_bwd(d, w, wb, acc, grads, dense, cf, cb, labels, prob, B, lr, eps, apply, gp, ld, ws, bytes, stream);
  });
}

SS_PY(ne_accumulate) {
  return guarded(args, nargs, [](Args& a) {
    const float* logit = a.ptr<float>(); const float* labels = a.ptr<float>();
    const int B = a.i32();
    double* acc = a.ptr<double>();
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_ne_accumulate(logit, labels, B, acc, stream);
  });
}

// The replica pointers of a synchronisation call and its optional mirrors.
struct Replicas {
  static constexpr int kCap = 64;                    // the library refuses more than 16 with SS_ERR_SHAPE
  void *w[kCap], *m[kCap];
  float* const* weights() { return reinterpret_cast<float* const*>(w); }
};
int replica_count(Args& a, Replicas& r) {
  const int R = a.tensors(r.w, Replicas::kCap);
  if (R < 0) { PyErr_SetString(PyExc_TypeError, "expected a sequence of tensors"); throw Bad(); }
  return R > Replicas::kCap ? Replicas::kCap : R;
}
void* const* mirrors(Args& a, Replicas& r, int R) {
  const int m = a.tensors(r.m, Replicas::kCap);
  if (m >= 0 && m < R) { PyErr_SetString(PyExc_ValueError, "fewer mirrors than replicas"); throw Bad(); }
  return m < 0 ? nullptr : r.m;
}

SS_PY(sync_easgd) {
  return guarded(args, nargs, [](Args& a) {
    Replicas r;
    const int R = replica_count(a, r);
    float* c = a.ptr<float>(); const int64_t n = a.i64(); const float alpha = a.f32(); const int flags = a.i32();
    void* const* m = mirrors(a, r, R);
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_sync_easgd(r.weights(), R, c, n, alpha, flags, m, stream);
  });
}

SS_PY(sync_ma) {
  return guarded(args, nargs, [](Args& a) {
    Replicas r;
    const int R = replica_count(a, r);
    float* g = a.ptr<float>(); const int64_t n = a.i64(); const float alpha = a.f32(); const int flags = a.i32();
    void* const* m = mirrors(a, r, R);
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_sync_ma(r.weights(), R, g, n, alpha, flags, m, stream);
  });
}

SS_PY(sync_bmuf) {
  return guarded(args, nargs, [](Args& a) {
    Replicas r;
    const int R = replica_count(a, r);
    float* g = a.ptr<float>(); float* d = a.ptr<float>(); const int64_t n = a.i64();
    const float alpha = a.f32(), eta = a.f32(), mu = a.f32(); const int flags = a.i32();
    void* const* m = mirrors(a, r, R);
    const ss_stream stream = a.stream();
    NoGil released;
    return ss_sync_bmuf(r.weights(), R, g, d, n, alpha, eta, mu, flags, m, stream);
  });
}

SS_PY(train_step) {
  return guarded(args, nargs, [](Args& a) {
    ss_step_args s;
    memset(&s, 0, sizeof(s));       // padding too: a plan compares steps byte by byte
    s.desc = a.desc();
    s.tables = a.ptr<float>(); s.row_state = a.ptr<float>();
    s.T = a.i32(); s.N = a.i64(); s.D = a.i32(); s.B = a.i32();
    s.indices = a.ptr<int32_t>(); s.offsets = a.ptr<int32_t>(); s.L = a.i64();
    s.dense = a.ptr<float>(); s.labels = a.ptr<float>();
    s.w = a.ptr<float>(); s.w_bf16 = a.ptr<void>(); s.adagrad_acc = a.ptr<float>();
    s.concat_f32 = a.ptr<float>(); s.concat_bf16 = a.ptr<void>();
    s.logit = a.ptr<float>(); s.prob = a.ptr<float>(); s.loss = a.ptr<float>(); s.grad_pooled = a.ptr<float>();
    s.mlp_ws = a.buffer(&s.mlp_ws_bytes); s.emb_ws = a.buffer(&s.emb_ws_bytes);
    s.uniq_keys = a.ptr<int32_t>(); s.seg_off = a.ptr<int32_t>(); s.perm = a.ptr<int32_t>();
    s.d_num_unique = a.ptr<int32_t>(); s.d_status = a.ptr<int32_t>();
    s.lr = a.f32(); s.eps = a.f32();
    s.replicas = a.i32();
    s.stream = a.stream(); s.sort_stream = a.stream(); s.mlp_stream = a.stream();
    s.plan = a.plan();
    NoGil released;
    return ss_train_step(&s);
  });
}

#define SS_ENTRY(NAME) {"ss_" #NAME, (PyCFunction)(void (*)(void))NAME, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {SS_ENTRY(embbag_fwd), SS_ENTRY(embbag_bwd_adagrad), SS_ENTRY(embbag_bwd_sort),
                         SS_ENTRY(embbag_bwd_apply), SS_ENTRY(mlp_fwd), SS_ENTRY(mlp_bwd), SS_ENTRY(ne_accumulate),
                         SS_ENTRY(sync_easgd), SS_ENTRY(sync_ma), SS_ENTRY(sync_bmuf), SS_ENTRY(train_step),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "argument marshalling of the ss_* calls", -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
