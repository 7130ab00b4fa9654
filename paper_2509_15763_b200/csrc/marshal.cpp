// Argument marshalling of the Python binding: takes torch tensors, checks that they are contiguous CUDA tensors, and
// calls the C entry point of the same name (include/unigist.h).  Nothing is kept between calls.  Every tensor is read
// under the interpreter lock; what runs without it sees plain pointers and numbers.
// A generation loop makes two of these calls per token and is bound by them: through ctypes, with a Python-level
// check and a pointer object per tensor, a decode call took 14 us of host time against 6 this way.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <c10/cuda/CUDAStream.h>

#include <vector>

#include "unigist.h"

namespace {

[[noreturn]] void raise(PyObject* type, const char* msg) {
  PyErr_SetString(type, msg);
  throw python_error();  // "a Python exception is set"
}

// A tensor argument as the C call takes it: its address (null for None), and what is needed of its sizes.
struct Arg {
  const at::Tensor* t;
  void* p;
  size_t bytes;
  operator void*() const { return p; }
  operator float*() const { return static_cast<float*>(p); }
  operator int32_t*() const { return static_cast<int32_t*>(p); }
};

// A problem's fields by name.  The names are made once, when the module is loaded (ten strings a call took 0.75 us).
enum { kBatch, kRawLen, kNumSinks, kRatio, kWindow, kNumQHeads, kNumKvHeads, kHeadDim, kSoftmaxScale, kFlags, kFields };
constexpr const char* kFieldName[kFields] = {"batch",        "raw_len",  "num_sinks",     "ratio", "window", "num_q_heads",
                                             "num_kv_heads", "head_dim", "softmax_scale", "flags"};
PyObject* g_field[kFields];

// The arguments of one call, read left to right (the caller holds a reference to each for the length of the call).
struct Args {
  PyObject* const* a;
  Py_ssize_t n, at = 0;

  PyObject* next() {
    if (at >= n) raise(PyExc_TypeError, "too few arguments");
    return a[at++];
  }
  Arg tensor() {  // (data_ptr() throws for a tensor without storage: a transform's or a tracer's)
    PyObject* o = next();
    if (o == Py_None) return {nullptr, nullptr, 0};
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch.Tensor");
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) raise(PyExc_ValueError, "tensors must be contiguous CUDA tensors");
    return {&t, t.data_ptr(), (size_t)t.numel() * t.element_size()};
  }
  long long integer() {
    const long long v = PyLong_AsLongLong(next());
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
  }
  double real() {
    const double v = PyFloat_AsDouble(next());
    if (v == -1.0 && PyErr_Occurred()) throw python_error();
    return v;
  }
  void* stream() {  // None: torch's current stream
    PyObject* o = next();
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw python_error();
    void* p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!p && PyErr_Occurred()) throw python_error();
    return p;
  }
  unigist_problem problem() {
    PyObject* o = next();
    auto field = [&](int name) {
      PyObject* v = PyObject_GetAttr(o, g_field[name]);
      if (!v) throw python_error();
      if (!PyLong_CheckExact(v)) {
        PyObject* i = PyNumber_Index(v);  // whatever counts as an integer (numpy's too), as ctypes takes it; no float
        Py_DECREF(v);
        if (!i) throw python_error();
        v = i;
      }
      const unsigned long long x = PyLong_AsUnsignedLongLongMask(v);
      Py_DECREF(v);
      if (PyErr_Occurred()) throw python_error();
      return x;
    };
    unigist_problem p;
    p.batch = (int32_t)field(kBatch);
    p.raw_len = (int32_t)field(kRawLen);
    p.num_sinks = (int32_t)field(kNumSinks);
    p.ratio = (int32_t)field(kRatio);
    p.window = (int32_t)field(kWindow);
    p.num_q_heads = (int32_t)field(kNumQHeads);
    p.num_kv_heads = (int32_t)field(kNumKvHeads);
    p.head_dim = (int32_t)field(kHeadDim);
    PyObject* s = PyObject_GetAttr(o, g_field[kSoftmaxScale]);
    if (!s) throw python_error();
    p.softmax_scale = (float)PyFloat_AsDouble(s);
    Py_DECREF(s);
    if (PyErr_Occurred()) throw python_error();
    p.flags = (uint32_t)field(kFlags);
    return p;
  }
  std::vector<int32_t> int_list() {
    PyObject* seq = PySequence_Fast(next(), "expected a sequence of document lengths");
    if (!seq) throw python_error();
    std::vector<int32_t> v;
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(seq); ++i) {
      PyObject* x = PyNumber_Long(PySequence_Fast_GET_ITEM(seq, i));
      v.push_back(x ? (int32_t)PyLong_AsUnsignedLongLongMask(x) : 0);
      Py_XDECREF(x);
      if (PyErr_Occurred()) {
        Py_DECREF(seq);
        throw python_error();
      }
    }
    Py_DECREF(seq);
    return v;
  }
};

int32_t dim(const Arg& a, int64_t i) {
  if (!a.t) raise(PyExc_TypeError, "a tensor is missing");
  if (i >= a.t->dim()) raise(PyExc_IndexError, "a tensor has too few dimensions");
  return (int32_t)a.t->size(i);
}

// Runs a call with the interpreter lock released and hands its status back.
template <typename Fn>
int32_t unlocked(Fn fn) {
  struct Released {
    PyThreadState* state = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(state); }  // also when the call throws (out of memory)
  } released;
  return fn();
}

// A METH_FASTCALL function around `body(Args&) -> status`.
template <int32_t (*kBody)(Args&)>
PyObject* call(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  Args args{a, n};
  return PyLong_FromLong(kBody(args));
  END_HANDLE_TH_ERRORS
}

template <decltype(unigist_gist_shift)* kFn>
int32_t shift(Args& a) {
  const unigist_problem p = a.problem();
  const Arg src = a.tensor(), dst = a.tensor();
  void* st = a.stream();
  const int32_t heads = dim(src, 2), eb = (int32_t)src.t->element_size();
  return unlocked([&] { return kFn(&p, src, dst, heads, eb, st); });
}

int32_t rope(Args& a) {
  const unigist_problem p = a.problem();
  const Arg src = a.tensor(), dst = a.tensor();
  const float base = (float)a.real();
  const uint32_t flags = (uint32_t)a.integer();
  void* st = a.stream();
  const int32_t heads = dim(src, 2);
  return unlocked([&] { return unigist_rope(&p, src, dst, heads, base, flags, st); });
}

int32_t attn_fwd(Args& a) {
  const unigist_problem p = a.problem();
  const Arg q = a.tensor(), k = a.tensor(), v = a.tensor(), o = a.tensor(), lse = a.tensor(), ws = a.tensor();
  void* st = a.stream();
  return unlocked([&] { return unigist_attn_fwd(&p, q, k, v, o, lse, ws, ws.bytes, st); });
}

int32_t attn_bwd(Args& a) {
  const unigist_problem p = a.problem();
  const Arg q = a.tensor(), k = a.tensor(), v = a.tensor(), o = a.tensor(), lse = a.tensor(), d_o = a.tensor(),
            dq = a.tensor(), dk = a.tensor(), dv = a.tensor(), ws = a.tensor();
  void* st = a.stream();
  return unlocked([&] { return unigist_attn_bwd(&p, q, k, v, o, lse, d_o, dq, dk, dv, ws, ws.bytes, st); });
}

int32_t attn_fwd_docs(Args& a) {
  const unigist_problem p = a.problem();
  const std::vector<int32_t> docs = a.int_list();
  const Arg q = a.tensor(), k = a.tensor(), v = a.tensor(), o = a.tensor(), lse = a.tensor(), ws = a.tensor();
  void* st = a.stream();
  return unlocked([&] {
    return unigist_attn_fwd_docs(&p, (int32_t)docs.size(), docs.data(), q, k, v, o, lse, ws, ws.bytes, st);
  });
}

int32_t attn_bwd_docs(Args& a) {
  const unigist_problem p = a.problem();
  const std::vector<int32_t> docs = a.int_list();
  const Arg q = a.tensor(), k = a.tensor(), v = a.tensor(), o = a.tensor(), lse = a.tensor(), d_o = a.tensor(),
            dq = a.tensor(), dk = a.tensor(), dv = a.tensor(), ws = a.tensor();
  void* st = a.stream();
  return unlocked([&] {
    return unigist_attn_bwd_docs(&p, (int32_t)docs.size(), docs.data(), q, k, v, o, lse, d_o, dq, dk, dv, ws,
                                 ws.bytes, st);
  });
}

int32_t kv_compact(Args& a) {
  const unigist_problem p = a.problem();
  const Arg k = a.tensor(), v = a.tensor(), kc = a.tensor(), vc = a.tensor(), table = a.tensor(), lens = a.tensor(),
            kept = a.tensor(), ws = a.tensor();
  void* st = a.stream();
  const int32_t blocks = dim(kc, 0), width = dim(table, 1);
  return unlocked([&] {
    return unigist_kv_compact(&p, k, v, kc, vc, blocks, table, width, lens, kept, ws, ws.bytes, st);
  });
}

int32_t prefill_chunk(Args& a) {
  const unigist_problem p = a.problem();
  const int32_t u0 = (int32_t)a.integer(), c = (int32_t)a.integer();
  const Arg q = a.tensor(), k = a.tensor(), v = a.tensor(), kc = a.tensor(), vc = a.tensor(), table = a.tensor(),
            lens = a.tensor(), o = a.tensor(), lse = a.tensor(), ws = a.tensor();
  void* st = a.stream();
  const int32_t blocks = dim(kc, 0), width = dim(table, 1);
  return unlocked([&] {
    return unigist_prefill_chunk(&p, u0, c, q, k, v, kc, vc, blocks, table, width, lens, o, lse, ws, ws.bytes, st);
  });
}

int32_t cache_state_init(Args& a) {
  const unigist_problem p = a.problem();
  const int32_t units = (int32_t)a.integer();
  const Arg state = a.tensor();
  void* st = a.stream();
  return unlocked([&] { return unigist_cache_state_init(&p, units, state, st); });
}

int32_t cache_append(Args& a) {
  const unigist_problem p = a.problem();
  const Arg k = a.tensor(), v = a.tensor();
  const int32_t is_gist = (int32_t)a.integer();
  const Arg kc = a.tensor(), vc = a.tensor(), table = a.tensor(), lens = a.tensor(), state = a.tensor();
  void* st = a.stream();
  const int32_t blocks = dim(kc, 0), width = dim(table, 1);
  return unlocked([&] {
    return unigist_cache_append(&p, k, v, is_gist, kc, vc, blocks, table, width, lens, state, st);
  });
}

int32_t decode_step(Args& a) {
  const unigist_problem p = a.problem();
  const Arg q = a.tensor(), kc = a.tensor(), vc = a.tensor(), table = a.tensor(), lens = a.tensor(),
            state = a.tensor(), o = a.tensor(), lse = a.tensor(), ws = a.tensor();
  void* st = a.stream();
  const int32_t blocks = dim(kc, 0), width = dim(table, 1);
  return unlocked([&] {
    return unigist_decode_step(&p, q, kc, vc, blocks, table, width, lens, state, o, lse, ws, ws.bytes, st);
  });
}

template <bool kStatic>
int32_t decode(Args& a) {
  const Arg q = a.tensor(), kc = a.tensor(), vc = a.tensor(), table = a.tensor(), lens = a.tensor(), o = a.tensor(),
            lse = a.tensor(), ws = kStatic ? Arg{} : a.tensor();
  const float scale = (float)a.real();
  void* st = a.stream();
  if (!q.t || q.t->dim() != 3) raise(PyExc_ValueError, "q must be [num_seqs, num_q_heads, head_dim]");
  const int32_t S = dim(q, 0), Hq = dim(q, 1), D = dim(q, 2), Hkv = dim(kc, 1), blocks = dim(kc, 0), width = dim(table, 1);
  return unlocked([&] {
    return kStatic
               ? unigist_decode_static(S, Hq, Hkv, D, scale, q, kc, vc, blocks, table, width, lens, o, lse, st)
               : unigist_decode(S, Hq, Hkv, D, scale, q, kc, vc, blocks, table, width, lens, o, lse, ws, ws.bytes, st);
  });
}

#define FN(name, ...) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&call<__VA_ARGS__>)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {FN("gist_shift", shift<unigist_gist_shift>),
                          FN("gist_unshift", shift<unigist_gist_unshift>),
                          FN("rope", rope),
                          FN("attn_fwd", attn_fwd),
                          FN("attn_bwd", attn_bwd),
                          FN("attn_fwd_docs", attn_fwd_docs),
                          FN("attn_bwd_docs", attn_bwd_docs),
                          FN("kv_compact", kv_compact),
                          FN("prefill_chunk", prefill_chunk),
                          FN("cache_state_init", cache_state_init),
                          FN("cache_append", cache_append),
                          FN("decode_step", decode_step),
                          FN("decode", decode<false>),
                          FN("decode_static", decode<true>),
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
  for (int i = 0; i < kFields; ++i)
    if (!g_field[i] && !(g_field[i] = PyUnicode_InternFromString(kFieldName[i]))) return nullptr;
  return PyModule_Create(&kModule);
}
