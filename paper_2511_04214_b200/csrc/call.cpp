// Argument marshalling of the Python binding for the calls that a program makes per layer or per tensor: tensors in, pointers, sizes
// and strides out, one call into libbro.  Through ctypes that took 3.1 us of a call (reading the tensors' fields from Python 1.9,
// converting a dozen arguments 1.2), half of a small launch and as much as the launch itself; here it is a few tenths.
//
// Every function returns the library's status, or -1 where the arguments are not plainly what it is made for (a tensor subclass, another
// type or rank, a shape that the binding would reject, a tensor without storage): the binding then goes the general way, with its
// own checks and errors.  The lock of the interpreter is released around the library call, as ctypes does.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/bro.h"

namespace {

#define BRO_CALLS(X)                                                                                                        \
  X(bro_rotate_quantize_mxfp4) X(bro_rotate_quantize_mxfp4_ex) X(bro_pack_weights) X(bro_pack_weights_rs) X(bro_gemm_mxfp4) \
  X(bro_linear) X(bro_linear_rs) X(bro_swiglu_linear) X(bro_swiglu_rotate_quantize_mxfp4) X(bro_group_quant_error_fmt)      \
  X(bro_rotate_fake_quantize_ws) X(bro_group_scale_bytes) X(bro_outlier_groups) X(bro_scale_histogram) X(bro_scale_inflation)

// The library's functions, from the addresses that the binding hands over (it has loaded the library).
struct Library {
#define BRO_MEMBER(f) decltype(&f) f = nullptr;
  BRO_CALLS(BRO_MEMBER)
#undef BRO_MEMBER
} lib;
bool bound = false;

// The arguments of one call, read in order; `ok` turns false at the first that is not what was asked for.
struct Args {
  PyObject* const* a;
  Py_ssize_t n, i = 0;
  bool ok;
  Args(PyObject* const* a_, Py_ssize_t n_, Py_ssize_t want) : a(a_), n(n_), ok(bound && n_ == want) {}

  const at::Tensor* any(bool optional = false) {
    if (!ok) return nullptr;
    PyObject* o = a[i++];
    if (optional && o == Py_None) return nullptr;
    if (!THPVariable_CheckExact(o)) { ok = false; return nullptr; }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined()) { ok = false; return nullptr; }
    return &t;
  }
  const at::Tensor* typed(at::ScalarType type, bool optional = false) {
    const at::Tensor* t = any(optional);
    if (t && t->scalar_type() != type) ok = false;
    return ok ? t : nullptr;
  }
  // rows and columns, rows of one memory run (`unit`: asked for)
  const at::Tensor* matrix(at::ScalarType type, bool unit) {
    const at::Tensor* t = typed(type);
    if (t && (t->dim() != 2 || (unit && t->stride(1) != 1))) ok = false;
    return ok ? t : nullptr;
  }
  int64_t integer() {
    if (!ok) return 0;
    PyObject* o = a[i++];
    if (!PyLong_CheckExact(o)) { ok = false; return 0; }
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    if (over) ok = false;
    return v;
  }
  int int32() {
    const int64_t v = integer();
    if (v != (int64_t)(int)v) ok = false;
    return (int)v;
  }
  void* stream() {
    if (!ok) return nullptr;
    PyObject* o = a[i++];
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) { PyErr_Clear(); ok = false; return nullptr; }
    const bool is_int = PyLong_CheckExact(h);
    void* s = is_int ? PyLong_AsVoidPtr(h) : nullptr;
    Py_DECREF(h);
    if (!is_int || (!s && PyErr_Occurred())) { PyErr_Clear(); ok = false; }
    return s;
  }
};

inline void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
inline int64_t ld(const at::Tensor& t, int64_t rows, int64_t cols) { return rows > 1 || t.stride(0) > cols ? t.stride(0) : cols; }
inline size_t bytes(const at::Tensor* t) { return t ? (size_t)t->numel() * t->element_size() : 0; }
inline bool dense(const at::Tensor* t, int64_t rows, int64_t cols) {
  return t->dim() == 2 && t->size(0) == rows && t->size(1) == cols && t->is_contiguous();
}

constexpr at::ScalarType kBf16 = at::kBFloat16, kF32 = at::kFloat, kU8 = at::kByte, kI64 = at::kLong;

// Runs `body(args)`, which returns the call to make as a function without arguments, or leaves args.ok false.
template <typename Body>
PyObject* call(PyObject* const* a, Py_ssize_t n, Py_ssize_t want, Body&& body) {
  long status = -1;
  try {
    Args args(a, n, want);
    status = body(args);
  } catch (...) {                 // a tensor without storage and the like: the general way reports it
    status = -1;
  }
  return PyLong_FromLong(status);
}
template <typename Call>
long unlocked(Call&& f) {
  long status;
  Py_BEGIN_ALLOW_THREADS
  status = (long)f();
  Py_END_ALLOW_THREADS
  return status;
}

#define ENTRY(name) PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n)

// x, block, codes, scales, layout, signs, stream
ENTRY(rotate_quantize) {
  return call(a, n, 7, [](Args& g) -> long {
    const at::Tensor* x = g.matrix(kBf16, true);
    const int block = g.int32();
    const at::Tensor *codes = g.any(), *scales = g.any();
    const int layout = g.int32();
    const at::Tensor* signs = g.any(true);
    void* st = g.stream();
    if (!g.ok) return -1;
    const int64_t M = x->size(0), K = x->size(1), ldx = ld(*x, M, K);
    void *px = ptr(x), *pc = ptr(codes), *ps = ptr(scales), *pn = ptr(signs);
    return unlocked([&] {
      return signs ? lib.bro_rotate_quantize_mxfp4_ex(px, M, K, ldx, block, pn, pc, ps, (bro_layout)layout, 0u, st)
                   : lib.bro_rotate_quantize_mxfp4(px, M, K, ldx, block, pc, ps, (bro_layout)layout, st);
    });
  });
}

// w, block, wcodes, wscales, signs, stream
ENTRY(pack_weights) {
  return call(a, n, 6, [](Args& g) -> long {
    const at::Tensor* w = g.matrix(kBf16, false);
    const int block = g.int32();
    const at::Tensor *codes = g.any(), *scales = g.any(), *signs = g.typed(kBf16, true);
    void* st = g.stream();
    if (!g.ok || (signs ? signs->numel() != w->size(1) : w->stride(1) != 1)) return -1;
    const int64_t N = w->size(0), K = w->size(1), ldw = ld(*w, N, K);
    void *pw = ptr(w), *pc = ptr(codes), *ps = ptr(scales), *pn = ptr(signs);
    return unlocked([&] {
      return signs ? lib.bro_pack_weights_rs(pw, N, K, ldw, block, pn, pc, ps, st) : lib.bro_pack_weights(pw, N, K, ldw, block, pc, ps, st);
    });
  });
}

// acodes, ascales, wcodes, wscales, M, N, K, y, workspace, stream
ENTRY(gemm) {
  return call(a, n, 10, [](Args& g) -> long {
    const at::Tensor *ac = g.any(), *as = g.any(), *wc = g.any(), *ws = g.any();
    const int64_t M = g.integer(), N = g.integer(), K = g.integer();
    const at::Tensor *y = g.any(), *work = g.any(true);
    void* st = g.stream();
    if (!g.ok || y->dim() != 2 || y->stride(1) != 1) return -1;
    const bool bf16 = y->scalar_type() == kBf16;
    if (!bf16 && y->scalar_type() != kF32) return -1;
    const int64_t ldy = ld(*y, M, N);
    const size_t wbytes = work ? (size_t)work->numel() : 0;
    void *pac = ptr(ac), *pas = ptr(as), *pwc = ptr(wc), *pws = ptr(ws), *py = ptr(y), *pk = ptr(work);
    return unlocked([&] {
      return lib.bro_gemm_mxfp4(pac, pas, pwc, pws, M, N, K, py, ldy, bf16 ? BRO_OUT_BF16 : BRO_OUT_F32, pk, wbytes, st);
    });
  });
}

// x, block, wcodes, wscales, N, y, workspace, signs, stream
ENTRY(linear) {
  return call(a, n, 9, [](Args& g) -> long {
    const at::Tensor* x = g.matrix(kBf16, false);
    const int block = g.int32();
    const at::Tensor *wc = g.any(), *ws = g.any();
    const int64_t N = g.integer();
    const at::Tensor *y = g.matrix(kBf16, false), *work = g.any(), *signs = g.typed(kBf16, true);
    void* st = g.stream();
    if (!g.ok) return -1;
    // (the plain layer takes the rows of y from x, the one with signs from y)
    const int64_t M = x->size(0), K = x->size(1), ldx = ld(*x, M, K), ldy = ld(*y, signs ? y->size(0) : M, N);
    const size_t wbytes = (size_t)work->numel();
    void *px = ptr(x), *pwc = ptr(wc), *pws = ptr(ws), *py = ptr(y), *pk = ptr(work), *pn = ptr(signs);
    return unlocked([&] {
      return signs ? lib.bro_linear_rs(px, M, K, ldx, block, pn, pwc, pws, N, py, ldy, pk, wbytes, st)
                   : lib.bro_linear(px, M, K, ldx, block, pwc, pws, N, py, ldy, pk, wbytes, st);
    });
  });
}

// gate, up, block, wcodes, wscales, N, y, workspace, signs, stream
ENTRY(swiglu_linear) {
  return call(a, n, 10, [](Args& g) -> long {
    const at::Tensor *gate = g.matrix(kBf16, false), *up = g.matrix(kBf16, false);
    const int block = g.int32();
    const at::Tensor *wc = g.any(), *ws = g.any();
    const int64_t N = g.integer();
    const at::Tensor *y = g.matrix(kBf16, false), *work = g.any(), *signs = g.any(true);
    void* st = g.stream();
    if (!g.ok || gate->sizes() != up->sizes()) return -1;
    const int64_t M = gate->size(0), K = gate->size(1), ldg = ld(*gate, M, K), ldu = ld(*up, M, K), ldy = ld(*y, y->size(0), N);
    const size_t wbytes = (size_t)work->numel();
    void *pg = ptr(gate), *pu = ptr(up), *pwc = ptr(wc), *pws = ptr(ws), *py = ptr(y), *pk = ptr(work), *pn = ptr(signs);
    return unlocked([&] { return lib.bro_swiglu_linear(pg, pu, M, K, ldg, ldu, block, pn, pwc, pws, N, py, ldy, pk, wbytes, st); });
  });
}

// gate, up, block, codes, scales, layout, signs, stream
ENTRY(swiglu_rotate_quantize) {
  return call(a, n, 8, [](Args& g) -> long {
    const at::Tensor *gate = g.matrix(kBf16, true), *up = g.matrix(kBf16, true);
    const int block = g.int32();
    const at::Tensor *codes = g.any(), *scales = g.any();
    const int layout = g.int32();
    const at::Tensor* signs = g.any(true);
    void* st = g.stream();
    if (!g.ok || gate->sizes() != up->sizes()) return -1;
    const int64_t M = gate->size(0), K = gate->size(1), ldg = ld(*gate, M, K), ldu = ld(*up, M, K);
    void *pg = ptr(gate), *pu = ptr(up), *pc = ptr(codes), *ps = ptr(scales), *pn = ptr(signs);
    return unlocked(
        [&] { return lib.bro_swiglu_rotate_quantize_mxfp4(pg, pu, M, K, ldg, ldu, block, pn, pc, ps, (bro_layout)layout, st); });
  });
}

// x, block, mse, signs, format, stream
ENTRY(group_quant_error) {
  return call(a, n, 6, [](Args& g) -> long {
    const at::Tensor* x = g.matrix(kBf16, false);
    const int block = g.int32();
    const at::Tensor *mse = g.typed(kF32), *signs = g.any(true);
    const int format = g.int32();
    void* st = g.stream();
    if (!g.ok || !dense(mse, x->size(0), x->size(1) / 32)) return -1;
    const int64_t M = x->size(0), K = x->size(1), ldx = ld(*x, M, K);
    void *px = ptr(x), *pn = ptr(signs);
    float* pm = static_cast<float*>(ptr(mse));
    return unlocked([&] { return lib.bro_group_quant_error_fmt(px, M, K, ldx, block, pn, (bro_format)format, pm, st); });
  });
}

// x, block, deq, format, signs, workspace, stream
ENTRY(rotate_fake_quantize) {
  return call(a, n, 7, [](Args& g) -> long {
    const at::Tensor* x = g.matrix(kBf16, false);
    const int block = g.int32();
    const at::Tensor* deq = g.matrix(kF32, false);
    const int format = g.int32();
    const at::Tensor *signs = g.any(true), *work = g.any(true);
    void* st = g.stream();
    if (!g.ok || deq->sizes() != x->sizes()) return -1;
    const int64_t M = x->size(0), K = x->size(1), ldx = ld(*x, M, K), ldd = ld(*deq, M, K);
    const size_t wbytes = bytes(work);
    void *px = ptr(x), *pn = ptr(signs), *pk = ptr(work);
    float* pd = static_cast<float*>(ptr(deq));
    return unlocked([&] { return lib.bro_rotate_fake_quantize_ws(px, M, K, ldx, block, pn, (bro_format)format, pd, ldd, pk, wbytes, st); });
  });
}

// x, block, scales, signs, stream
ENTRY(group_scale_bytes) {
  return call(a, n, 5, [](Args& g) -> long {
    const at::Tensor* x = g.matrix(kBf16, false);
    const int block = g.int32();
    const at::Tensor *scales = g.typed(kU8), *signs = g.any(true);
    void* st = g.stream();
    if (!g.ok || !dense(scales, x->size(0), x->size(1) / 32)) return -1;
    const int64_t M = x->size(0), K = x->size(1), ldx = ld(*x, M, K);
    void *px = ptr(x), *pn = ptr(signs);
    uint8_t* ps = static_cast<uint8_t*>(ptr(scales));
    return unlocked([&] { return lib.bro_group_scale_bytes(px, M, K, ldx, block, pn, ps, st); });
  });
}

// x, mask, info, workspace, top_ppm, stream
ENTRY(outlier_groups) {
  return call(a, n, 6, [](Args& g) -> long {
    const at::Tensor *x = g.matrix(kBf16, false), *mask = g.typed(kU8), *info = g.any(), *work = g.any();
    const int64_t ppm = g.integer();
    void* st = g.stream();
    if (!g.ok || !dense(mask, x->size(0), x->size(1) / 32) || info->numel() < 4 || info->element_size() != 4) return -1;
    const int64_t M = x->size(0), K = x->size(1), ldx = ld(*x, M, K);
    const size_t wbytes = bytes(work);
    void *px = ptr(x), *pk = ptr(work);
    uint8_t* pm = static_cast<uint8_t*>(ptr(mask));
    uint32_t* pi = static_cast<uint32_t*>(ptr(info));
    return unlocked([&] { return lib.bro_outlier_groups(px, M, K, ldx, ppm, pm, pi, pk, wbytes, st); });
  });
}

// scales, mask, hist, stream
ENTRY(scale_histogram) {
  return call(a, n, 4, [](Args& g) -> long {
    const at::Tensor *scales = g.typed(kU8), *mask = g.typed(kU8), *hist = g.typed(kI64);
    void* st = g.stream();
    if (!g.ok || !scales->is_contiguous() || !mask->is_contiguous() || !hist->is_contiguous() || hist->numel() != 512 ||
        scales->numel() != mask->numel())
      return -1;
    const int64_t groups = scales->numel();
    const uint8_t *ps = static_cast<uint8_t*>(ptr(scales)), *pm = static_cast<uint8_t*>(ptr(mask));
    uint64_t* ph = static_cast<uint64_t*>(ptr(hist));
    return unlocked([&] { return lib.bro_scale_histogram(ps, pm, groups, ph, st); });
  });
}

// before, after, mask, counts, stream
ENTRY(scale_inflation) {
  return call(a, n, 5, [](Args& g) -> long {
    const at::Tensor *before = g.typed(kU8), *after = g.typed(kU8), *mask = g.typed(kU8), *counts = g.typed(kI64);
    void* st = g.stream();
    if (!g.ok || !before->is_contiguous() || !after->is_contiguous() || !mask->is_contiguous() || counts->numel() != 6 ||
        before->numel() != after->numel() || after->numel() != mask->numel())
      return -1;
    const int64_t groups = before->numel();
    const uint8_t *pb = static_cast<uint8_t*>(ptr(before)), *pa = static_cast<uint8_t*>(ptr(after)), *pm = static_cast<uint8_t*>(ptr(mask));
    uint64_t* pc = static_cast<uint64_t*>(ptr(counts));
    return unlocked([&] { return lib.bro_scale_inflation(pb, pa, pm, groups, pc, st); });
  });
}

// {name: address} of the library's functions
PyObject* bind(PyObject*, PyObject* addresses) {
  if (!PyDict_Check(addresses)) {
    PyErr_SetString(PyExc_TypeError, "a dict of addresses");
    return nullptr;
  }
#define BRO_BIND(f)                                                                                    \
  {                                                                                                    \
    PyObject* v = PyDict_GetItemString(addresses, #f);                                                 \
    if (!v) return PyErr_Format(PyExc_KeyError, "%s", #f);                                             \
    lib.f = reinterpret_cast<decltype(&f)>(PyLong_AsVoidPtr(v));                                       \
    if (!lib.f) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_ValueError, "%s is null", #f);  \
  }
  BRO_CALLS(BRO_BIND)
#undef BRO_BIND
  bound = true;
  Py_RETURN_NONE;
}

#define METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(rotate_quantize), METHOD(pack_weights), METHOD(gemm), METHOD(linear), METHOD(swiglu_linear),
                         METHOD(swiglu_rotate_quantize), METHOD(group_quant_error), METHOD(rotate_fake_quantize),
                         METHOD(group_scale_bytes), METHOD(outlier_groups), METHOD(scale_histogram), METHOD(scale_inflation),
                         {"bind", bind, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call() {
  PyObject* m = PyModule_Create(&module);
  if (!m) return nullptr;
  PyObject* names = PyList_New(0);
#define BRO_NAME(f)                                    \
  {                                                    \
    PyObject* s = PyUnicode_FromString(#f);            \
    PyList_Append(names, s);                           \
    Py_DECREF(s);                                      \
  }
  BRO_CALLS(BRO_NAME)
#undef BRO_NAME
  PyModule_AddObject(m, "NAMES", names);
  PyModule_AddStringConstant(m, "TAG", BRO_CALL_TAG);      // the torch, the ABI and the Python of the build, which the binding compares
  return m;
}
