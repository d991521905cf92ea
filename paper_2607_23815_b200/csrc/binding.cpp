// Native half of the Python binding: unpacks torch tensors and calls the C ABI.
//
// A call of the library is worth 3-7 us of host time (one to two kernel launches).  Marshalling the arguments of such a
// call through ctypes cost as much again and more (attn_decode 11.1 us, of which 4.2 in the library; attn_extend_append
// 15.6 and 7.2), which bounded every small call: the kernel behind a decode of one sequence takes 4.2 us.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/kvattn.h"

namespace {

// Thrown with a Python exception set.
struct Raised {};

[[noreturn]] void raise(PyObject* type, const char* what) {
  PyErr_SetString(type, what);
  throw Raised{};
}

const at::Tensor& tensor(PyObject* o) {
  if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch tensor");
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_contiguous()) raise(PyExc_AssertionError, "tensors passed to the library must be contiguous");
  if (!t.is_cuda()) raise(PyExc_AssertionError, "expected a CUDA tensor");
  return t;
}

// Addresses are taken before the interpreter lock is let go: a tensor without storage of its own (a fake one) throws here.
// read: for what the library only reads; written: the tensor's own memory, brought about if it still shares another's.
template <typename T = void>
const T* read(const at::Tensor& t) { return static_cast<const T*>(t.const_data_ptr()); }
template <typename T = void>
T* written(const at::Tensor& t) { return static_cast<T*>(t.mutable_data_ptr()); }
template <typename T = void>
const T* read(PyObject* o) { return o == Py_None ? nullptr : read<T>(tensor(o)); }
template <typename T = void>
T* written(PyObject* o) { return o == Py_None ? nullptr : written<T>(tensor(o)); }
int size(const at::Tensor& t, int dim) {
  if (dim >= t.dim()) raise(PyExc_IndexError, "tensor has too few dimensions");
  return (int)t.size(dim);
}

int integer(PyObject* o) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) throw Raised{};
  return (int)v;
}
float real(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Raised{};
  return (float)v;
}
kv_pool_t* pool(PyObject* o) {
  if (o == Py_None) return nullptr;
  void* p = PyLong_AsVoidPtr(o);
  if (p == nullptr && PyErr_Occurred()) throw Raised{};
  return static_cast<kv_pool_t*>(p);
}
// None: torch's current stream; else a stream object or its handle (anything that int() takes).
void* stream(PyObject* o) {
  if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
  PyObject* h = PyObject_HasAttrString(o, "cuda_stream") ? PyObject_GetAttrString(o, "cuda_stream") : PyNumber_Long(o);
  if (h == nullptr) throw Raised{};
  void* p = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (p == nullptr && PyErr_Occurred()) throw Raised{};
  return p;
}
struct Workspace {
  void* p = nullptr;
  size_t bytes = 0;
  explicit Workspace(PyObject* o) {
    if (o == Py_None) return;
    const at::Tensor& t = tensor(o);
    p = written(t);
    bytes = t.nbytes();
  }
};
// A ctypes structure (or None).
struct Struct {
  Py_buffer view{};
  explicit Struct(PyObject* o) {
    if (o != Py_None && PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Raised{};
  }
  ~Struct() {
    if (view.obj != nullptr) PyBuffer_Release(&view);
  }
  template <typename T>
  const T* as() const {
    if (view.buf == nullptr) return nullptr;
    if (view.len != (Py_ssize_t)sizeof(T)) raise(PyExc_TypeError, "argument structure of the wrong size");
    return static_cast<const T*>(view.buf);
  }
};

// Runs body(args), which returns a function to be called without the interpreter lock, and returns its status.
template <typename Body>
PyObject* call(Py_ssize_t got, Py_ssize_t want, Body body) {
  if (got != want) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  try {
    return PyLong_FromLong(body());
  } catch (const Raised&) {
    return nullptr;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}
// Calls f without the interpreter lock, which is held again however f is left.
template <typename F>
long unlocked(F f) {
  struct Unlock {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlock() { PyEval_RestoreThread(state); }
  } unlock;
  return f();
}

PyObject* append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 8, [&] {
    kv_pool_t* p = pool(a[0]);
    const at::Tensor &k = tensor(a[1]), &start = tensor(a[4]), &bt = tensor(a[6]);
    const void *kp = read(k), *vp = read(a[2]);
    const int *cu = read<int>(a[3]), *startp = read<int>(start), *row = read<int>(a[5]), *btp = read<int>(bt);
    void* st = stream(a[7]);
    const int pages = size(bt, 1), segs = (int)start.numel(), total = size(k, 0);
    return unlocked([&] { return kv_append(p, kp, vp, cu, startp, row, btp, pages, segs, total, st); });
  });
}

PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 10, [&] {
    kv_pool_t* p = pool(a[0]);
    const at::Tensor &q = tensor(a[1]), &bt = tensor(a[2]);
    const void* qp = read(q);
    const int *btp = read<int>(bt), *ctx = read<int>(a[3]);
    const int max_ctx = integer(a[4]), hq = size(q, 1), pages = size(bt, 1), batch = size(q, 0);
    const float scale = real(a[5]);
    void *out = written(a[6]), *st = stream(a[9]);
    float* lse = written<float>(a[7]);
    const Workspace ws(a[8]);
    return unlocked([&] { return attn_decode(p, qp, hq, btp, pages, ctx, batch, max_ctx, scale, out, lse, ws.p, ws.bytes, st); });
  });
}

// what attn_extend, attn_extend_planned and attn_extend_append share
template <typename F>
PyObject* extend_like(PyObject* const* a, Py_ssize_t n, int lead, F f) {  // lead: arguments before cu_q
  return call(n, lead + 11, [&] {
    kv_pool_t* p = pool(a[0]);
    const at::Tensor& q = tensor(a[1]);
    PyObject* const* b = a + lead;
    const at::Tensor &bt = tensor(b[1]), &pl = tensor(b[2]);
    const void* qp = read(q);
    const int *cu = read<int>(b[0]), *btp = read<int>(bt), *plp = read<int>(pl), *el = read<int>(b[3]);
    const int batch = (int)pl.numel(), max_e = integer(b[4]), max_l = integer(b[5]), hq = size(q, 1), total = size(q, 0), pages = size(bt, 1);
    const float scale = real(b[6]);
    void *out = written(b[7]), *st = stream(b[10]);
    float* lse = written<float>(b[8]);
    const Workspace ws(b[9]);
    const void *k = lead == 4 ? read(a[2]) : nullptr, *v = lead == 4 ? read(a[3]) : nullptr;
    return unlocked([&] {
      return f(p, qp, k, v, hq, cu, btp, pages, plp, el, batch, total, max_e, max_l, scale, out, lse, ws.p, ws.bytes, st);
    });
  });
}
PyObject* extend(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return extend_like(a, n, 2, [](kv_pool_t* p, const void* q, const void*, const void*, auto... rest) { return attn_extend(p, q, rest...); });
}
PyObject* extend_planned(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return extend_like(a, n, 2, [](kv_pool_t* p, const void* q, const void*, const void*, auto... rest) { return attn_extend_planned(p, q, rest...); });
}
PyObject* extend_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return extend_like(a, n, 4, [](auto... all) { return attn_extend_append(all...); });
}

PyObject* extend_plan(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 11, [&] {
    kv_pool_t* p = pool(a[0]);
    const int hq = integer(a[1]), total = integer(a[6]), max_e = integer(a[7]), max_l = integer(a[8]);
    const at::Tensor &bt = tensor(a[3]), &pl = tensor(a[4]);
    const int *cu = read<int>(a[2]), *btp = read<int>(bt), *plp = read<int>(pl), *el = read<int>(a[5]);
    const int pages = size(bt, 1), batch = (int)pl.numel();
    const Workspace ws(a[9]);
    void* st = stream(a[10]);
    return unlocked([&] { return attn_extend_plan(p, hq, cu, btp, pages, plp, el, batch, total, max_e, max_l, ws.p, ws.bytes, st); });
  });
}

PyObject* extend_shared(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 16, [&] {
    kv_pool_t* p = pool(a[0]);
    const at::Tensor &q = tensor(a[1]), &pt = tensor(a[4]), &pl = tensor(a[5]), &ct = tensor(a[6]), &cl = tensor(a[7]);
    const void* qp = read(q);
    const int *cu = read<int>(a[2]), *cc = read<int>(a[3]), *ptp = read<int>(pt), *plp = read<int>(pl), *ctp = read<int>(ct), *clp = read<int>(cl);
    const int max_c = integer(a[8]), max_rows = integer(a[9]), max_p = integer(a[10]), parents = (int)pl.numel(), children = (int)cl.numel();
    const int hq = size(q, 1), total = size(q, 0), pages_p = size(pt, 1), pages_c = size(ct, 1);
    const float scale = real(a[11]);
    void *out = written(a[12]), *st = stream(a[15]);
    float* lse = written<float>(a[13]);
    const Workspace ws(a[14]);
    return unlocked([&] {
      return attn_extend_shared(p, qp, hq, cu, cc, ptp, pages_p, plp, ctp, pages_c, clp, parents, children, total, max_c, max_rows, max_p,
                                scale, out, lse, ws.p, ws.bytes, st);
    });
  });
}

PyObject* mixed(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 7, [&] {
    kv_pool_t* p = pool(a[0]);
    const int hq = integer(a[1]);
    const float scale = real(a[2]);
    const Struct ext(a[3]), dec(a[4]);
    const auto* e = ext.as<attn_extend_args_t>();
    const auto* d = dec.as<attn_decode_args_t>();
    const Workspace ws(a[5]);
    void* st = stream(a[6]);
    return unlocked([&] { return attn_mixed(p, hq, scale, e, d, ws.p, ws.bytes, st); });
  });
}

const at::Tensor& host_tensor(PyObject* o) {
  if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch tensor");
  const at::Tensor& t = THPVariable_Unpack(o);
  if (t.is_cuda() || !t.is_contiguous()) raise(PyExc_ValueError, "attn_extend_host takes contiguous host tensors");
  return t;
}
PyObject* extend_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
  return call(n, 15, [&] {
    kv_pool_t* p = pool(a[0]);
    const at::Tensor &q = host_tensor(a[1]), &k = host_tensor(a[2]), &v = host_tensor(a[3]), &cu = host_tensor(a[4]), &bt = host_tensor(a[5]),
                     &pl = host_tensor(a[6]), &el = host_tensor(a[7]), &out = host_tensor(a[11]), &lse = host_tensor(a[12]);
    const void *qp = read(q), *kp = read(k), *vp = read(v);
    const int *cup = read<int>(cu), *btp = read<int>(bt), *plp = read<int>(pl), *elp = read<int>(el);
    const int max_e = integer(a[8]), max_l = integer(a[9]), hq = size(q, 1), total = size(q, 0), pages = size(bt, 1), batch = (int)pl.numel();
    const float scale = real(a[10]);
    void* outp = written(out);
    float* lsep = written<float>(lse);
    const Workspace staging(a[13]);
    void* st = stream(a[14]);
    return unlocked([&] {
      return attn_extend_host(p, qp, kp, vp, hq, cup, btp, pages, plp, elp, batch, total, max_e, max_l, scale, outp, lsep, staging.p,
                              staging.bytes, st);
    });
  });
}

#define ENTRY(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY("kv_append", append),
                         ENTRY("attn_decode", decode),
                         ENTRY("attn_extend", extend),
                         ENTRY("attn_extend_append", extend_append),
                         ENTRY("attn_extend_plan", extend_plan),
                         ENTRY("attn_extend_planned", extend_planned),
                         ENTRY("attn_extend_shared", extend_shared),
                         ENTRY("attn_mixed", mixed),
                         ENTRY("attn_extend_host", extend_host),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_kvattn_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__kvattn_native(void) { return PyModule_Create(&module); }
