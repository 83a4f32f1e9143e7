// Native side of the Python binding: turns the arguments of one compute call (torch tensors, integers, a stream) into
// the arguments of its C entry point and makes the call. Nothing of the method happens here.
//
// A decoding step is some forty calls of 5 to 15 us of device time each, so what a call costs the host decides
// whether the device waits for it. Through ctypes, with a Python-level pointer extraction per tensor and
// torch.cuda.current_stream(), a call of cast_tree_attention took 15 to 18 us (19 arguments) and one of
// cast_tree_expand 11 to 13 us; here the tensors are unpacked through torch's own C++ interface.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "cast.h"

namespace {

// Arguments are taken in order; the first one that does not fit sets a Python exception and ends the call.
struct Args {
  PyObject* const* a;
  Py_ssize_t n;
  Py_ssize_t at = 0;
  bool ok = true;
  bool known_dtype = true;

  PyObject* next() {
    if (!ok) return nullptr;
    if (at >= n) {
      PyErr_SetString(PyExc_TypeError, "too few arguments");
      ok = false;
      return nullptr;
    }
    return a[at++];
  }
  int integer() {
    PyObject* o = next();
    if (!o) return 0;
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) ok = false;
    return (int)v;
  }
  size_t size() {
    PyObject* o = next();
    if (!o) return 0;
    const size_t v = PyLong_AsSize_t(o);
    if (v == (size_t)-1 && PyErr_Occurred()) ok = false;
    return v;
  }
  double real() {
    PyObject* o = next();
    if (!o) return 0.0;
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) ok = false;
    return v;
  }
  cast_ctx* context() {
    PyObject* o = next();
    if (!o) return nullptr;
    void* p = PyLong_AsVoidPtr(o);
    if (p == nullptr && PyErr_Occurred()) ok = false;
    return static_cast<cast_ctx*>(p);
  }
  // device address of a tensor argument, null for None; `dtype`, where given, receives the logits / cache type
  template <typename T = void>
  T* tensor(cast_dtype* dtype = nullptr) {
    PyObject* o = next();
    if (!o || (o == Py_None && dtype == nullptr)) return nullptr;
    if (!THPVariable_Check(o)) {
      PyErr_SetString(PyExc_TypeError, "torch tensor expected");
      ok = false;
      return nullptr;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) {
      PyErr_SetString(PyExc_AssertionError, "device-resident contiguous tensor expected");
      ok = false;
      return nullptr;
    }
    if (dtype != nullptr) {
      if (t.scalar_type() == at::kFloat) *dtype = CAST_F32;
      else if (t.scalar_type() == at::kBFloat16) *dtype = CAST_BF16;
      else known_dtype = false;
    }
    return static_cast<T*>(t.data_ptr());
  }
  // the last argument: a torch stream, or None for the current one
  void* stream() {
    PyObject* o = next();
    if (!o) return nullptr;
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (h == nullptr) {
      ok = false;
      return nullptr;
    }
    void* s = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (s == nullptr && PyErr_Occurred()) ok = false;
    return s;
  }
  bool ready() {
    if (ok && at != n) {
      PyErr_SetString(PyExc_TypeError, "too many arguments");
      ok = false;
    }
    return ok;
  }
};

// Every wrapper returns the entry point's status as a Python integer. The call itself runs without the interpreter
// lock: a launch can block while the device's queue is full.
#define CALL(expr)                                            \
  if (!g.ready()) return nullptr;                             \
  if (!g.known_dtype) return PyLong_FromLong(CAST_ERR_DTYPE); \
  cast_status status;                                         \
  Py_BEGIN_ALLOW_THREADS                                      \
  status = (expr);                                            \
  Py_END_ALLOW_THREADS                                        \
  return PyLong_FromLong((long)status)

PyObject* step_begin(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g{a, n};
  cast_ctx* c = g.context();
  const int B = g.integer();
  auto* root = g.tensor<int32_t>();
  auto* kv_len = g.tensor<int32_t>();
  void* s = g.stream();
  CALL(cast_step_begin(c, B, root, kv_len, s));
}

PyObject* tree_expand(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g{a, n};
  cast_dtype dt = CAST_F32;
  cast_ctx* c = g.context();
  const int layer = g.integer();
  auto* logits = g.tensor(&dt);
  auto* tokens = g.tensor<int32_t>();
  auto* rows = g.tensor<int32_t>();
  auto* count = g.tensor<int32_t>();
  void* s = g.stream();
  CALL(cast_tree_expand(c, layer, logits, dt, tokens, rows, count, s));
}

PyObject* select_nodes(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g{a, n};
  cast_ctx* c = g.context();
  auto* tokens = g.tensor<int32_t>();
  auto* parent = g.tensor<int32_t>();
  auto* depth = g.tensor<int32_t>();
  auto* anc = g.tensor<uint32_t>();
  auto* pool = g.tensor<int32_t>();
  auto* scores = g.tensor<double>();
  auto* n_tree = g.tensor<int32_t>();
  void* s = g.stream();
  CALL(cast_select_nodes(c, tokens, parent, depth, anc, pool, scores, n_tree, s));
}

// cast_tree_attention and, with `rows`, cast_tree_attention_rows
template <bool kRows>
PyObject* tree_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g{a, n};
  cast_dtype dt = CAST_F32;
  cast_ctx* c = g.context();
  auto* q = g.tensor(&dt);
  auto* k = g.tensor();
  auto* v = g.tensor();
  const int B = g.integer(), Hq = g.integer(), Hkv = g.integer(), D = g.integer(), page = g.integer();
  auto* table = g.tensor<int32_t>();
  const int cap = g.integer(), pages = g.integer();
  auto* kv_len = g.tensor<int32_t>();
  auto* anc = g.tensor<uint32_t>();
  auto* n_tree = g.tensor<int32_t>();
  int32_t* first = kRows ? g.tensor<int32_t>() : nullptr;
  const float scale = (float)g.real();
  auto* out = g.tensor();
  void* s = g.stream();
  CALL(cast_tree_attention_rows(c, q, k, v, dt, B, Hq, Hkv, D, page, table, cap, pages, kv_len, anc, n_tree, first, scale,
                                out, s));
}

PyObject* accept(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g{a, n};
  cast_dtype dt = CAST_F32;
  cast_ctx* c = g.context();
  auto* logits = g.tensor(&dt);
  const int B = g.integer();
  auto* tokens = g.tensor<int32_t>();
  auto* parent = g.tensor<int32_t>();
  auto* depth = g.tensor<int32_t>();
  auto* anc = g.tensor<uint32_t>();
  auto* n_tree = g.tensor<int32_t>();
  auto* len = g.tensor<int32_t>();
  auto* path = g.tensor<int32_t>();
  auto* bonus = g.tensor<int32_t>();
  void* s = g.stream();
  CALL(cast_accept(c, logits, dt, B, tokens, parent, depth, anc, n_tree, len, path, bonus, s));
}

PyObject* accept_stochastic(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g{a, n};
  cast_dtype dt = CAST_F32;
  cast_ctx* c = g.context();
  auto* target = g.tensor(&dt);
  auto* draft = g.tensor();
  const int B = g.integer();
  const double temperature = g.real();
  auto* tokens = g.tensor<int32_t>();
  auto* parent = g.tensor<int32_t>();
  auto* n_tree = g.tensor<int32_t>();
  auto* u_accept = g.tensor<double>();
  auto* u_bonus = g.tensor<double>();
  auto* len = g.tensor<int32_t>();
  auto* path = g.tensor<int32_t>();
  auto* bonus = g.tensor<int32_t>();
  void* s = g.stream();
  CALL(cast_accept_stochastic(c, target, draft, dt, B, temperature, tokens, parent, n_tree, u_accept, u_bonus, len, path,
                              bonus, s));
}

PyObject* accept_static(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g{a, n};
  cast_dtype dt = CAST_F32;
  auto* logits = g.tensor(&dt);
  const int B = g.integer(), n_cap = g.integer(), vocab = g.integer(), max_depth = g.integer();
  auto* tokens = g.tensor<int32_t>();
  auto* parent = g.tensor<int32_t>();
  auto* n_tree = g.tensor<int32_t>();
  auto* len = g.tensor<int32_t>();
  auto* path = g.tensor<int32_t>();
  auto* bonus = g.tensor<int32_t>();
  void* s = g.stream();
  CALL(cast_accept_static(logits, dt, B, n_cap, vocab, max_depth, tokens, parent, n_tree, len, path, bonus, s));
}

PyObject* compact_kv(PyObject*, PyObject* const* a, Py_ssize_t n) {
  Args g{a, n};
  cast_dtype dt = CAST_F32;
  cast_ctx* c = g.context();
  auto* k = g.tensor(&dt);
  auto* v = g.tensor();
  const int B = g.integer(), layers = g.integer();
  const size_t stride = g.size();
  const int Hkv = g.integer(), D = g.integer(), page = g.integer();
  auto* table = g.tensor<int32_t>();
  const int cap = g.integer(), pages = g.integer();
  auto* path = g.tensor<int32_t>();
  auto* len = g.tensor<int32_t>();
  auto* kv_len = g.tensor<int32_t>();
  void* s = g.stream();
  CALL(cast_compact_kv(c, k, v, dt, B, layers, stride, Hkv, D, page, table, cap, pages, path, len, kv_len, s));
}

#define METHOD(name, fn) {name, (PyCFunction)(void (*)())(fn), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    METHOD("step_begin", step_begin),
    METHOD("tree_expand", tree_expand),
    METHOD("select_nodes", select_nodes),
    METHOD("tree_attention", tree_attention<false>),
    METHOD("tree_attention_rows", tree_attention<true>),
    METHOD("accept", accept),
    METHOD("accept_stochastic", accept_stochastic),
    METHOD("accept_static", accept_static),
    METHOD("compact_kv", compact_kv),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_cast_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__cast_calls() { return PyModule_Create(&module); }
