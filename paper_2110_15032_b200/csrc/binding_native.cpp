// Native side of the Python binding: fills sbp_tensor descriptors from SbpTensor objects and makes the
// library call, for the entry points that run on every step of a program.
//
// What bounds a small call is the host.  Filling three descriptors through ctypes, asking torch's Python
// layer for the current stream and converting the arguments took 8-10 us of a call whose launch takes
// 4-5 us; here the same work, made anew for every call from the tensors as they are at that moment (no
// descriptor, pointer or check is kept), takes about one.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <exception>

#include "sbp.h"

namespace {

PyObject *s_shape, *s_dtype, *s_sigs, *s_pshape, *s_locals, *s_kind, *s_axis, *s_cuda_stream;

struct Ref {      // owned reference
  PyObject* p;
  explicit Ref(PyObject* o) : p(o) {}
  ~Ref() { Py_XDECREF(p); }
  Ref(const Ref&) = delete;
  Ref& operator=(const Ref&) = delete;
};

bool as_i64(PyObject* o, int64_t* out) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) return false;
  *out = v;
  return true;
}

// An attribute that is a list or a tuple.
PyObject* field(PyObject* obj, PyObject* name) {
  Ref v(PyObject_GetAttr(obj, name));
  return v.p ? PySequence_Fast(v.p, "a sequence is needed here") : nullptr;
}

// Leading dimension of a local tensor: 0 when it is contiguous, its row pitch when it is a row-strided
// window, -1 when it is neither.
int64_t row_pitch(const at::Tensor& t) {
  if (t.is_contiguous()) return 0;
  const int64_t nd = t.dim();
  if (nd < 2 || t.stride(nd - 1) != 1) return -1;
  const int64_t pitch = t.stride(nd - 2);
  if (pitch < t.size(nd - 1)) return -1;
  for (int64_t i = 0; i < nd - 2; ++i)      // every axis before the last two is dense over the pitch
    if (t.size(i) != 1 && t.stride(i) != t.stride(i + 1) * t.size(i + 1)) return -1;
  return pitch;
}

// obj is an SbpTensor; false with a Python error set when it cannot be described.
bool fill(PyObject* obj, sbp_tensor* d) {
  memset(d, 0, sizeof(*d));
  Ref shape(field(obj, s_shape)), dtype(PyObject_GetAttr(obj, s_dtype)), sigs(field(obj, s_sigs));
  if (!shape.p || !dtype.p || !sigs.p) return false;
  Ref pshape(field(obj, s_pshape)), locals(field(obj, s_locals));
  if (!pshape.p || !locals.p) return false;
  const Py_ssize_t nd = PySequence_Fast_GET_SIZE(shape.p), np = PySequence_Fast_GET_SIZE(pshape.p), nl = PySequence_Fast_GET_SIZE(locals.p);
  if (nd > SBP_MAX_DIMS || np > SBP_MAX_PDIMS || nl > SBP_MAX_K || PySequence_Fast_GET_SIZE(sigs.p) < np) {
    PyErr_SetString(PyExc_IndexError, "more axes or local tensors than a descriptor holds");
    return false;
  }
  d->ndim = (int32_t)nd;
  for (Py_ssize_t i = 0; i < nd; ++i)
    if (!as_i64(PySequence_Fast_GET_ITEM(shape.p, i), &d->shape[i])) return false;
  if (!THPDtype_Check(dtype.p)) {
    PyErr_SetString(PyExc_TypeError, "an SbpTensor's dtype is a torch dtype");
    return false;
  }
  switch (reinterpret_cast<THPDtype*>(dtype.p)->scalar_type) {
    case at::kFloat: d->dtype = SBP_F32; break;
    case at::kBFloat16: d->dtype = SBP_BF16; break;
    case at::kLong: d->dtype = SBP_I64; break;
    default: PyErr_SetObject(PyExc_KeyError, dtype.p); return false;
  }
  d->pdims = (int32_t)np;
  d->pshape[1] = 1;
  for (Py_ssize_t i = 0; i < np; ++i) {
    int64_t v, kind, axis;
    if (!as_i64(PySequence_Fast_GET_ITEM(pshape.p, i), &v)) return false;
    PyObject* sig = PySequence_Fast_GET_ITEM(sigs.p, i);
    Ref k(PyObject_GetAttr(sig, s_kind)), a(PyObject_GetAttr(sig, s_axis));
    if (!k.p || !a.p || !as_i64(k.p, &kind) || !as_i64(a.p, &axis)) return false;
    d->pshape[i] = (int32_t)v;
    d->sbp[i].kind = (int32_t)kind;
    d->sbp[i].axis = (int32_t)axis;
  }
  for (Py_ssize_t r = 0; r < nl; ++r) {
    PyObject* o = PySequence_Fast_GET_ITEM(locals.p, r);
    if (o == Py_None) continue;              // a local tensor another device holds
    if (!THPVariable_Check(o)) {
      PyErr_SetString(PyExc_TypeError, "local tensors must be torch tensors");
      return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    const int64_t pitch = row_pitch(t);
    if (pitch < 0) {
      PyErr_SetString(PyExc_ValueError, "local tensors must be contiguous, or row-strided windows of a row-major buffer");
      return false;
    }
    d->local[r] = t.data_ptr();
    d->local_ld[r] = pitch;
  }
  return true;
}

bool stream_of(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  Ref v(PyObject_GetAttr(o, s_cuda_stream));
  if (!v.p) return false;
  *out = PyLong_AsVoidPtr(v.p);
  return !PyErr_Occurred();
}

// A plain tensor used as memory (a workspace, a counter).
bool memory_of(PyObject* o, bool optional, void** ptr, size_t* bytes) {
  *ptr = nullptr;
  *bytes = 0;
  if (o == Py_None && optional) return true;
  if (!THPVariable_Check(o)) {
    PyErr_SetString(PyExc_AttributeError, "a torch tensor is needed here");
    return false;
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  *ptr = t.data_ptr();
  *bytes = (size_t)t.numel() * t.element_size();
  return true;
}

typedef sbp_tensor T;
struct {
  sbp_status (*boxing)(const T*, T*, void*);
  sbp_status (*boxing_shard)(const T*, T*, int32_t, void*);
  sbp_status (*matmul)(const T*, const T*, T*, uint32_t, void*, size_t, void*);
  sbp_status (*softmax_xent)(const T*, const T*, T*, T*, T*, void*, size_t, void*);
  sbp_status (*softmax_xent_static)(const T*, const T*, T*, T*, T*, void*);
  sbp_status (*softmax_xent_backward)(const T*, const T*, const T*, const T*, T*, void*);
  sbp_status (*matmul_softmax_xent)(const T*, const T*, const T*, T*, T*, T*, void*, size_t, void*);
  sbp_status (*matmul_softmax_xent_backward)(const T*, const T*, const T*, const T*, const T*, T*, void*);
  sbp_status (*embedding)(const T*, const T*, T*, int32_t*, void*);
  sbp_status (*embedding_backward)(const T*, const T*, T*, int32_t*, void*);
} lib;

// Arguments: the first n_desc are SbpTensors (those of the bits in `optional` may be None), the last is the
// stream or None; what lies between is the caller's.
struct Call {
  T d[6];
  T* at[6];
  void* stream;
  bool ok;
  Call(const char* name, PyObject* const* args, Py_ssize_t n, Py_ssize_t want, int n_desc, unsigned optional) : ok(false) {
    if (n != want) {
      PyErr_Format(PyExc_TypeError, "%s takes %zd arguments", name, want);
      return;
    }
    for (int i = 0; i < n_desc; ++i) {
      if (args[i] == Py_None && (optional >> i & 1)) {
        at[i] = nullptr;
        continue;
      }
      if (!fill(args[i], &d[i])) return;
      at[i] = &d[i];
    }
    ok = stream_of(args[n - 1], &stream);
  }
};

#define ENTRY(name) PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t n)
// Other Python threads run during a library call; the lock is held again however the call ends.
struct Unlocked {
  PyThreadState* state = PyEval_SaveThread();
  ~Unlocked() { PyEval_RestoreThread(state); }
};
#define RUN(expr)           \
  sbp_status st;            \
  {                         \
    Unlocked other_threads; \
    st = (expr);            \
  }                         \
  return PyLong_FromLong((long)st)
#define GUARDED(body)                                \
  try {                                              \
    body                                             \
  } catch (const std::exception& e) {                \
    PyErr_SetString(PyExc_RuntimeError, e.what());   \
    return nullptr;                                  \
  }

ENTRY(boxing) {
  GUARDED(Call c("boxing", args, n, 3, 2, 0); if (!c.ok) return nullptr;
          RUN(lib.boxing(c.at[0], c.at[1], c.stream));)
}
ENTRY(boxing_shard) {
  GUARDED(Call c("boxing_shard", args, n, 4, 2, 0); int64_t shard; if (!c.ok || !as_i64(args[2], &shard)) return nullptr;
          RUN(lib.boxing_shard(c.at[0], c.at[1], (int32_t)shard, c.stream));)
}
ENTRY(matmul) {
  GUARDED(Call c("matmul", args, n, 6, 3, 0); int64_t flags; void* ws; size_t bytes;
          if (!c.ok || !as_i64(args[3], &flags) || !memory_of(args[4], true, &ws, &bytes)) return nullptr;
          RUN(lib.matmul(c.at[0], c.at[1], c.at[2], (uint32_t)flags, ws, bytes, c.stream));)
}
ENTRY(softmax_xent) {
  GUARDED(Call c("softmax_xent", args, n, 7, 5, 0x18); void* ws; size_t bytes;
          if (!c.ok || !memory_of(args[5], false, &ws, &bytes)) return nullptr;
          RUN(lib.softmax_xent(c.at[0], c.at[1], c.at[2], c.at[3], c.at[4], ws, bytes, c.stream));)
}
ENTRY(softmax_xent_static) {
  GUARDED(Call c("softmax_xent_static", args, n, 6, 5, 0x18); if (!c.ok) return nullptr;
          RUN(lib.softmax_xent_static(c.at[0], c.at[1], c.at[2], c.at[3], c.at[4], c.stream));)
}
ENTRY(softmax_xent_backward) {
  GUARDED(Call c("softmax_xent_backward", args, n, 6, 5, 0); if (!c.ok) return nullptr;
          RUN(lib.softmax_xent_backward(c.at[0], c.at[1], c.at[2], c.at[3], c.at[4], c.stream));)
}
ENTRY(matmul_softmax_xent) {
  GUARDED(Call c("matmul_softmax_xent", args, n, 8, 6, 0x30); void* ws; size_t bytes;
          if (!c.ok || !memory_of(args[6], false, &ws, &bytes)) return nullptr;
          RUN(lib.matmul_softmax_xent(c.at[0], c.at[1], c.at[2], c.at[3], c.at[4], c.at[5], ws, bytes, c.stream));)
}
ENTRY(matmul_softmax_xent_backward) {
  GUARDED(Call c("matmul_softmax_xent_backward", args, n, 7, 6, 0); if (!c.ok) return nullptr;
          RUN(lib.matmul_softmax_xent_backward(c.at[0], c.at[1], c.at[2], c.at[3], c.at[4], c.at[5], c.stream));)
}
ENTRY(embedding) {
  GUARDED(Call c("embedding", args, n, 5, 3, 0); void* oob; size_t bytes;
          if (!c.ok || !memory_of(args[3], true, &oob, &bytes)) return nullptr;
          RUN(lib.embedding(c.at[0], c.at[1], c.at[2], static_cast<int32_t*>(oob), c.stream));)
}
ENTRY(embedding_backward) {
  GUARDED(Call c("embedding_backward", args, n, 5, 3, 0); void* oob; size_t bytes;
          if (!c.ok || !memory_of(args[3], true, &oob, &bytes)) return nullptr;
          RUN(lib.embedding_backward(c.at[0], c.at[1], c.at[2], static_cast<int32_t*>(oob), c.stream));)
}

// bind(addresses): the library's entry points, in the order of `lib`, from the library the process loaded.
PyObject* py_bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
  constexpr Py_ssize_t kEntries = sizeof(lib) / sizeof(void*);
  if (n != kEntries) {
    PyErr_Format(PyExc_TypeError, "bind takes %zd addresses", kEntries);
    return nullptr;
  }
  void* v[kEntries];
  for (Py_ssize_t i = 0; i < n; ++i) {
    v[i] = PyLong_AsVoidPtr(args[i]);
    if (!v[i]) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null entry point");
      return nullptr;
    }
  }
  memcpy(&lib, v, sizeof(lib));
  Py_RETURN_NONE;
}

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(bind),
                         METHOD(boxing),
                         METHOD(boxing_shard),
                         METHOD(matmul),
                         METHOD(softmax_xent),
                         METHOD(softmax_xent_static),
                         METHOD(softmax_xent_backward),
                         METHOD(matmul_softmax_xent),
                         METHOD(matmul_softmax_xent_backward),
                         METHOD(embedding),
                         METHOD(embedding_backward),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  s_shape = PyUnicode_InternFromString("shape");
  s_dtype = PyUnicode_InternFromString("dtype");
  s_sigs = PyUnicode_InternFromString("sigs");
  s_pshape = PyUnicode_InternFromString("pshape");
  s_locals = PyUnicode_InternFromString("locals");
  s_kind = PyUnicode_InternFromString("kind");
  s_axis = PyUnicode_InternFromString("axis");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  return PyModule_Create(&module);
}
