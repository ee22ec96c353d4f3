// CPython side of twig.py: reads sizes, strides and device pointers out of torch tensors and calls
// the C ABI.  Nothing of the path is computed here.
//
// Why native: a decoding step is 30 and more short calls, and through ctypes a call cost the host
// 10 us (18 converted arguments, a dozen tensor attribute look-ups, torch's stream object) while the
// kernel behind it runs 5.5 us, so the host was what bounded a single user's verification step
// (338 us for 34 calls).  Here a call is 1.0 us plus the launch itself.
//
// Every function takes the arguments of the Python function of the same name, positionally and
// complete, and returns the twig_status.  The C functions are looked up by twig.py in the library
// that it has loaded (bind), so there is one copy of the library in the process.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>
#include <stdexcept>

#include "twig.h"

namespace {

struct PyError {};      // a Python exception is set

// ---- the library's functions ------------------------------------------------------------------
#define TWIG_FUNCTIONS(X)                                                                                          \
  X(ttp_score) X(ttp_score_gated) X(ttp_score_multiquery) X(ttp_score_noalloc) X(ttp_topk) X(ttp_compact)          \
  X(ttp_compact_rows) X(ttp_score_topk_compact) X(tree_verify_attention_ex) X(tree_reset) X(tree_expand_level)     \
  X(tree_select_expansion) X(tree_finalize) X(tree_grow_level) X(tree_base_argmax) X(chain_draft_reset)            \
  X(chain_draft_step) X(tree_accept_compact)

struct Library {
#define X(name) decltype(&::name) name = nullptr;
  TWIG_FUNCTIONS(X)
#undef X
} lib;

// ---- arguments ----------------------------------------------------------------------------------
const at::Tensor &tensor(PyObject *o) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "expected a torch tensor, got %s", Py_TYPE(o)->tp_name);
    throw PyError();
  }
  return THPVariable_Unpack(o);
}
const at::Tensor &tensor(PyObject *o, int64_t dims) {
  const at::Tensor &t = tensor(o);
  if (t.dim() != dims) {
    PyErr_Format(PyExc_ValueError, "expected a tensor of %lld dimensions, got %lld", (long long)dims, (long long)t.dim());
    throw PyError();
  }
  return t;
}
void require(bool ok) {
  if (ok) return;
  PyErr_SetString(PyExc_AssertionError, "shapes or strides do not fit each other");
  throw PyError();
}
int32_t dim32(const at::Tensor &t, int64_t d) { return (int32_t)t.size(d); }

template <class T = void>
T *ptr(PyObject *o) {
  return o == Py_None ? nullptr : static_cast<T *>(tensor(o).data_ptr());
}
int32_t i32(PyObject *o) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) throw PyError();
  return (int32_t)v;
}
float f32(PyObject *o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw PyError();
  return (float)v;
}
size_t bytes_of(const at::Tensor &t) { return (size_t)t.numel() * t.element_size(); }
int32_t is_f32(const at::Tensor &t) { return t.scalar_type() == at::kFloat ? 1 : 0; }

// rows of logits of all requests at one stride
void require_rows(const at::Tensor &logits) {
  require(logits.stride(2) == 1 && logits.stride(0) == logits.size(1) * logits.stride(1));
}

void *stream_of(PyObject *o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw PyError();
  void *s = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (!s && PyErr_Occurred()) throw PyError();
  return s;
}

// a KV structure (ctypes.Structure with the layout of twig_kv)
class KvArg {
 public:
  explicit KvArg(PyObject *o) {
    if (PyObject_GetBuffer(o, &view_, PyBUF_SIMPLE) != 0) throw PyError();
    if (view_.len != (Py_ssize_t)sizeof(twig_kv)) {
      PyBuffer_Release(&view_);
      PyErr_SetString(PyExc_TypeError, "expected a KV");
      throw PyError();
    }
  }
  ~KvArg() { PyBuffer_Release(&view_); }
  KvArg(const KvArg &) = delete;
  const twig_kv *get() const { return static_cast<const twig_kv *>(view_.buf); }

 private:
  Py_buffer view_;
};

// the call itself, without the interpreter's lock (a launch waits when the stream's queue is full)
template <class F, class... A>
twig_status call(F fn, A... args) {
  if (!fn) {
    PyErr_SetString(PyExc_RuntimeError, "bind() has not been called");
    throw PyError();
  }
  twig_status s;
  Py_BEGIN_ALLOW_THREADS
  s = fn(args...);
  Py_END_ALLOW_THREADS
  return s;
}

// ---- one function per entry point -------------------------------------------------------------
twig_status do_ttp_score(PyObject *const *a) {
  const at::Tensor &q = tensor(a[0], 3), &k = tensor(a[1], 4), &scores = tensor(a[5], 2), &ws = tensor(a[6]);
  return call(lib.ttp_score, q.data_ptr(), k.data_ptr(), k.stride(0), k.stride(1), k.stride(2), dim32(k, 2),
              ptr<int32_t>(a[2]), ptr<int32_t>(a[3]), ptr<int32_t>(a[4]), dim32(q, 0), dim32(q, 1), dim32(k, 1),
              dim32(q, 2), i32(a[7]), f32(a[8]), ptr<float>(a[5]), dim32(scores, 1), ptr<int32_t>(a[9]), ws.data_ptr(),
              bytes_of(ws), stream_of(a[10]));
}

twig_status do_ttp_score_gated(PyObject *const *a) {
  const at::Tensor &q = tensor(a[0], 3), &qg = tensor(a[1]), &k = tensor(a[2], 4), &kg = tensor(a[3]),
                   &scores = tensor(a[7], 2), &ws = tensor(a[8]);
  require(qg.sizes() == q.sizes() && qg.is_contiguous());
  require(kg.sizes() == k.sizes() && kg.strides() == k.strides());
  return call(lib.ttp_score_gated, q.data_ptr(), qg.data_ptr(), k.data_ptr(), kg.data_ptr(), k.stride(0), k.stride(1),
              k.stride(2), dim32(k, 2), ptr<int32_t>(a[4]), ptr<int32_t>(a[5]), ptr<int32_t>(a[6]), dim32(q, 0),
              dim32(q, 1), dim32(k, 1), dim32(q, 2), i32(a[9]), f32(a[10]), ptr<float>(a[7]), dim32(scores, 1),
              ptr<int32_t>(a[11]), ws.data_ptr(), bytes_of(ws), stream_of(a[12]));
}

twig_status do_ttp_score_multiquery(PyObject *const *a) {
  const at::Tensor &q = tensor(a[0], 4), &k = tensor(a[1], 4), &scores = tensor(a[5], 2), &ws = tensor(a[6]);
  require(q.is_contiguous());
  return call(lib.ttp_score_multiquery, q.data_ptr(), dim32(q, 2), k.data_ptr(), k.stride(0), k.stride(1), k.stride(2),
              dim32(k, 2), ptr<int32_t>(a[2]), ptr<int32_t>(a[3]), ptr<int32_t>(a[4]), dim32(q, 0), dim32(q, 1),
              dim32(k, 1), dim32(q, 3), f32(a[7]), ptr<float>(a[5]), dim32(scores, 1), ptr<int32_t>(a[8]), ws.data_ptr(),
              bytes_of(ws), stream_of(a[9]));
}

twig_status do_ttp_score_noalloc(PyObject *const *a) {
  const at::Tensor &q = tensor(a[0], 3), &k = tensor(a[1], 4), &scores = tensor(a[5], 2);
  return call(lib.ttp_score_noalloc, q.data_ptr(), k.data_ptr(), k.stride(0), k.stride(1), k.stride(2), dim32(k, 2),
              ptr<int32_t>(a[2]), ptr<int32_t>(a[3]), ptr<int32_t>(a[4]), dim32(q, 0), dim32(q, 1), dim32(k, 1),
              dim32(q, 2), i32(a[6]), f32(a[7]), ptr<float>(a[5]), dim32(scores, 1), ptr<int32_t>(a[8]),
              stream_of(a[9]));
}

twig_status do_ttp_topk(PyObject *const *a) {
  const at::Tensor &scores = tensor(a[0], 2), &kept = tensor(a[3], 2);
  return call(lib.ttp_topk, ptr<float>(a[0]), ptr<int32_t>(a[1]), ptr<int32_t>(a[2]), dim32(scores, 0), dim32(scores, 1),
              dim32(kept, 1), ptr<int32_t>(a[3]), ptr<int32_t>(a[4]), stream_of(a[5]));
}

twig_status do_ttp_compact(PyObject *const *a) {
  KvArg src(a[0]), dst(a[1]);
  const at::Tensor &kept = tensor(a[2], 2);
  const int32_t pos_stride = a[7] == Py_None ? 0 : dim32(tensor(a[7], 2), 1);
  return call(lib.ttp_compact, src.get(), dst.get(), ptr<int32_t>(a[2]), dim32(kept, 1), ptr<int32_t>(a[3]),
              ptr<int32_t>(a[4]), ptr<int32_t>(a[5]), ptr<int32_t>(a[6]), ptr<int32_t>(a[7]), ptr<int32_t>(a[8]),
              pos_stride, ptr<int32_t>(a[9]), ptr<int32_t>(a[10]), stream_of(a[11]));
}

twig_status do_ttp_compact_rows(PyObject *const *a) {
  const at::Tensor &src = tensor(a[0]), &dst = tensor(a[1]), &kept = tensor(a[2], 2);
  require(src.dim() == 3 && dst.dim() == 3 && src.stride(2) == 1 && dst.stride(2) == 1);
  const int64_t es = src.element_size();
  return call(lib.ttp_compact_rows, src.data_ptr(), dst.data_ptr(), src.size(2) * es, src.stride(1) * es,
              src.stride(0) * es, dim32(src, 1), dst.stride(1) * es, dst.stride(0) * es, dim32(dst, 1), dim32(src, 0),
              ptr<int32_t>(a[2]), dim32(kept, 1), ptr<int32_t>(a[3]), ptr<int32_t>(a[4]), ptr<int32_t>(a[5]),
              ptr<int32_t>(a[6]), ptr<int32_t>(a[7]), ptr<int32_t>(a[8]), stream_of(a[9]));
}

twig_status do_ttp_score_topk_compact(PyObject *const *a) {
  const at::Tensor &q = tensor(a[0]), &k = tensor(a[1], 4), &scores = tensor(a[6], 2), &kept = tensor(a[7], 2),
                   &ws = tensor(a[10]);
  KvArg src(a[8]), dst(a[9]);
  const int32_t pos_stride = a[11] == Py_None ? 0 : dim32(tensor(a[11], 2), 1);
  return call(lib.ttp_score_topk_compact, q.data_ptr(), k.data_ptr(), k.stride(0), k.stride(1), k.stride(2), dim32(k, 2),
              ptr<int32_t>(a[2]), ptr<int32_t>(a[3]), ptr<int32_t>(a[4]), ptr<int32_t>(a[5]), dim32(q, 1), i32(a[14]),
              f32(a[15]), ptr<float>(a[6]), dim32(scores, 1), ptr<int32_t>(a[7]), dim32(kept, 1), src.get(), dst.get(),
              ptr<int32_t>(a[11]), ptr<int32_t>(a[12]), pos_stride, ptr<int32_t>(a[13]), ptr<int32_t>(a[16]),
              ws.data_ptr(), bytes_of(ws), stream_of(a[17]));
}

twig_status do_tree_verify_attention(PyObject *const *a) {
  const at::Tensor &q = tensor(a[0], 4);
  KvArg cache(a[3]);
  const size_t ws_bytes = a[12] == Py_None ? 0 : bytes_of(tensor(a[12]));
  uint32_t flags = 0;
  if (a[14] != Py_None) {
    const unsigned long v = PyLong_AsUnsignedLongMask(a[14]);
    if (v == (unsigned long)-1 && PyErr_Occurred()) throw PyError();
    flags = (uint32_t)v;
  }
  return call(lib.tree_verify_attention_ex, q.data_ptr(), ptr(a[1]), ptr(a[2]), cache.get(), i32(a[4]),
              ptr<int32_t>(a[5]), ptr<int32_t>(a[6]), ptr<int32_t>(a[7]), dim32(q, 1), dim32(q, 2), f32(a[10]), ptr(a[8]),
              ptr<float>(a[9]), ptr<int32_t>(a[11]), ptr(a[12]), ws_bytes, stream_of(a[13]), flags);
}

// (the tree state arrives as its tensors tok, parent, score and its sizes cap, batch)
twig_status do_tree_reset(PyObject *const *a) {
  return call(lib.tree_reset, ptr<int32_t>(a[0]), ptr<int32_t>(a[1]), ptr<float>(a[2]), i32(a[3]), i32(a[4]),
              stream_of(a[5]));
}

twig_status do_tree_expand_level(PyObject *const *a) {
  const at::Tensor &logits = tensor(a[0], 3);
  require_rows(logits);
  return call(lib.tree_expand_level, logits.data_ptr(), is_f32(logits), logits.stride(1), dim32(logits, 2),
              dim32(logits, 1), ptr<int32_t>(a[1]), i32(a[2]), i32(a[3]), ptr<int32_t>(a[4]), ptr<int32_t>(a[5]),
              ptr<float>(a[6]), i32(a[7]), dim32(logits, 0), ptr<int32_t>(a[8]), stream_of(a[9]));
}

twig_status do_tree_select_expansion(PyObject *const *a) {
  return call(lib.tree_select_expansion, ptr<float>(a[0]), i32(a[1]), i32(a[3]), i32(a[4]), dim32(tensor(a[5], 2), 1),
              ptr<int32_t>(a[5]), i32(a[2]), ptr<int32_t>(a[6]), stream_of(a[7]));
}

twig_status do_tree_finalize(PyObject *const *a) {
  return call(lib.tree_finalize, ptr<int32_t>(a[0]), ptr<int32_t>(a[1]), ptr<float>(a[2]), i32(a[3]), i32(a[5]),
              i32(a[6]), ptr<int32_t>(a[7]), ptr<int32_t>(a[8]), ptr<int32_t>(a[9]), ptr<int32_t>(a[10]),
              dim32(tensor(a[7], 2), 1), i32(a[4]), ptr<int32_t>(a[11]), stream_of(a[12]));
}

twig_status do_tree_grow_level(PyObject *const *a) {
  const at::Tensor &logits = tensor(a[0], 3);
  require_rows(logits);
  const int32_t n_select = a[9] == Py_None ? 0 : dim32(tensor(a[9], 2), 1);
  const int32_t t_max = a[11] == Py_None ? 0 : dim32(tensor(a[11], 2), 1);
  return call(lib.tree_grow_level, logits.data_ptr(), is_f32(logits), logits.stride(1), dim32(logits, 2), dim32(logits, 1),
              ptr<int32_t>(a[1]), i32(a[2]), i32(a[3]), ptr<int32_t>(a[4]), ptr<int32_t>(a[5]), ptr<float>(a[6]),
              i32(a[7]), dim32(logits, 0), n_select, ptr<int32_t>(a[9]), i32(a[10]), ptr<int32_t>(a[11]),
              ptr<int32_t>(a[12]), ptr<int32_t>(a[13]), ptr<int32_t>(a[14]), t_max, ptr<int32_t>(a[8]),
              ptr<int32_t>(a[15]), stream_of(a[16]));
}

twig_status do_tree_base_argmax(PyObject *const *a) {
  const at::Tensor &logits = tensor(a[0], 3);
  require_rows(logits);
  return call(lib.tree_base_argmax, logits.data_ptr(), is_f32(logits), logits.stride(1), dim32(logits, 2),
              ptr<int32_t>(a[1]), dim32(logits, 0), dim32(logits, 1), ptr<int32_t>(a[2]), ptr<int32_t>(a[3]),
              stream_of(a[4]));
}

twig_status do_chain_draft_reset(PyObject *const *a) {
  const at::Tensor &parent = tensor(a[0], 2);
  return call(lib.chain_draft_reset, ptr<int32_t>(a[0]), ptr<int32_t>(a[1]), ptr<float>(a[4]), ptr<int32_t>(a[2]),
              ptr<int32_t>(a[3]), dim32(parent, 1), dim32(parent, 0), stream_of(a[5]));
}

twig_status do_chain_draft_step(PyObject *const *a) {
  const at::Tensor &logits = tensor(a[0], 2);
  require(logits.stride(1) == 1);
  return call(lib.chain_draft_step, logits.data_ptr(), is_f32(logits), logits.stride(0), dim32(logits, 1), i32(a[1]),
              f32(a[2]), ptr<int32_t>(a[3]), ptr<int32_t>(a[4]), ptr<float>(a[7]), ptr<int32_t>(a[5]), ptr<int32_t>(a[6]),
              dim32(tensor(a[3], 2), 1), dim32(logits, 0), ptr<int32_t>(a[8]), stream_of(a[9]));
}

twig_status do_tree_accept_compact(PyObject *const *a) {
  KvArg cache(a[6]);
  return call(lib.tree_accept_compact, ptr<int32_t>(a[0]), ptr<int32_t>(a[1]), ptr<int32_t>(a[2]), ptr<int32_t>(a[3]),
              dim32(tensor(a[0], 2), 1), dim32(tensor(a[9], 2), 1), ptr(a[4]), ptr(a[5]), cache.get(), ptr<int32_t>(a[7]),
              ptr<int32_t>(a[8]), ptr<int32_t>(a[9]), ptr<int32_t>(a[10]), ptr<int32_t>(a[11]), stream_of(a[12]));
}

template <twig_status (*FN)(PyObject *const *), int N_ARGS>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n) {
  if (n != N_ARGS) {
    PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N_ARGS, n);
    return nullptr;
  }
  try {
    return PyLong_FromLong((long)FN(args));
  } catch (const PyError &) {
  } catch (const std::exception &e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
  }
  return nullptr;
}

// bind(name, address): the C function of that name
PyObject *bind(PyObject *, PyObject *args) {
  const char *name = nullptr;
  PyObject *address = nullptr;
  if (!PyArg_ParseTuple(args, "sO", &name, &address)) return nullptr;
  void *p = PyLong_AsVoidPtr(address);
  if (!p) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null address");
    return nullptr;
  }
  const std::string want(name);
#define X(fn) if (want == #fn) lib.fn = reinterpret_cast<decltype(lib.fn)>(p);
  TWIG_FUNCTIONS(X)
#undef X
  Py_RETURN_NONE;
}

#define TWIG_ENTRY(name, n_args) \
  {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(&entry<do_##name, n_args>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    TWIG_ENTRY(ttp_score, 11), TWIG_ENTRY(ttp_score_gated, 13), TWIG_ENTRY(ttp_score_multiquery, 10),
    TWIG_ENTRY(ttp_score_noalloc, 10), TWIG_ENTRY(ttp_topk, 6), TWIG_ENTRY(ttp_compact, 12),
    TWIG_ENTRY(ttp_compact_rows, 10), TWIG_ENTRY(ttp_score_topk_compact, 18), TWIG_ENTRY(tree_verify_attention, 15),
    TWIG_ENTRY(tree_reset, 6), TWIG_ENTRY(tree_expand_level, 10), TWIG_ENTRY(tree_select_expansion, 8),
    TWIG_ENTRY(tree_finalize, 13), TWIG_ENTRY(tree_grow_level, 17), TWIG_ENTRY(tree_base_argmax, 5),
    TWIG_ENTRY(chain_draft_reset, 6), TWIG_ENTRY(chain_draft_step, 10), TWIG_ENTRY(tree_accept_compact, 13),
    {"bind", bind, METH_VARARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&module); }
