// Argument marshalling of the Python binding: torch tensors -> device pointers -> C entry points.
// Nothing is computed here.  A call through ctypes costs 8 to 12 us of interpreter time (four
// attribute look-ups and a conversion per tensor), as long as a small layer takes on the GPU;
// through this module 1.3 us.  The entry points are called by address (bind()), so the module
// works with whichever build of the library the Python side has loaded.
#define PY_SSIZE_T_CLEAN
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>

#include <algorithm>
#include <cstring>
#include <string>

#include "xnor.h"

namespace {

// The entry points this module calls, in the order bind() takes their addresses.
struct Entry {
  decltype(&xnor_binarize_weights) binarize_weights;
  decltype(&xnor_binactiv) binactiv;
  decltype(&xnor_conv2d_forward) conv2d_forward;
  decltype(&xnor_shortcut_conv1x1) shortcut_conv1x1;
  decltype(&xnor_conv2d_forward_binactiv) conv2d_forward_binactiv;
  decltype(&xnor_binactiv_finish) binactiv_finish;
  decltype(&xnor_maxpool2d) maxpool2d;
  decltype(&xnor_binactiv_kbit) binactiv_kbit;
  decltype(&xnor_conv2d_forward_kbit) conv2d_forward_kbit;
  decltype(&xnor_bwn_prepare_input) bwn_prepare_input;
  decltype(&xnor_bwn_conv2d_forward) bwn_conv2d_forward;
  decltype(&xnor_binarize_weights_transposed) binarize_weights_transposed;
  decltype(&xnor_binary_gradient_backward) binary_gradient_backward;
} E;
constexpr Py_ssize_t kEntries = sizeof(Entry) / sizeof(void *);
PyObject *desc_type = nullptr;         // the ctypes structure xnor_conv_desc
PyObject *py_address = nullptr;        // (object, type name) -> its checked address through Python attributes

// Arguments of one call, converted in order; the first failure sets a Python error and sticks.
struct Args {
  PyObject *const *a;
  Py_ssize_t n;
  bool ok;
  Py_ssize_t i = 0;

  Args(PyObject *const *args, Py_ssize_t nargs, Py_ssize_t want) : a(args), n(nargs), ok(nargs == want) {
    if (!ok) PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs);
  }
  void fail_attr(const char *fmt, PyObject *t, const char *attr) {
    if (PyObject *v = PyObject_GetAttrString(t, attr)) {
      PyErr_Format(PyExc_ValueError, fmt, v);
      Py_DECREF(v);
    }
    ok = false;
  }
  // Tensors and parameters are read here.  Subclasses and other objects with a tensor's attributes may
  // define these in Python, so they are asked there.
  void *ptr(at::ScalarType type, const char *name) {
    PyObject *o = a[i++];
    if (!ok || o == Py_None) return nullptr;
    if (!THPVariable_CheckExact(o)) {
      PyObject *v = PyObject_CallFunction(py_address, "Os", o, name);
      void *p = v != nullptr ? PyLong_AsVoidPtr(v) : nullptr;
      Py_XDECREF(v);
      ok = !PyErr_Occurred();
      return p;
    }
    const at::Tensor &t = THPVariable_Unpack(o);
    if (!t.is_cuda()) {
      fail_attr("libxnor takes device pointers: tensor is on %S", o, "device");
    } else if (!t.is_contiguous()) {
      PyErr_SetString(PyExc_ValueError, "tensor must be contiguous");
      ok = false;
    } else if (t.scalar_type() != type) {
      const std::string fmt = std::string("expected torch.") + name + ", got %S";
      fail_attr(fmt.c_str(), o, "dtype");
    } else {
      return t.data_ptr();
    }
    return nullptr;
  }
  float *f32() { return (float *)ptr(at::kFloat, "float32"); }
  uint32_t *u32() { return (uint32_t *)ptr(at::kInt, "int32"); }
  int32_t *i32() { return (int32_t *)ptr(at::kInt, "int32"); }
  uint16_t *bf16() { return (uint16_t *)ptr(at::kBFloat16, "bfloat16"); }
  int num() {
    PyObject *o = a[i++];
    if (!ok) return 0;
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) ok = false;
    else if (v != (long)(int)v) { PyErr_SetString(PyExc_OverflowError, "argument out of int range"); ok = false; }
    return (int)v;
  }
  // an xnor_conv_desc and nothing else of its size, read through the buffer protocol
  xnor_conv_desc desc() {
    xnor_conv_desc d = {};
    PyObject *o = a[i++];
    if (!ok) return d;
    Py_buffer b;
    const int is = PyObject_IsInstance(o, desc_type);
    if (is == 0) PyErr_Format(PyExc_TypeError, "expected an xnor_conv_desc, got %S", (PyObject *)Py_TYPE(o));
    if (is != 1 || PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) { ok = false; return d; }
    memcpy(&d, b.buf, std::min((size_t)b.len, sizeof(d)));
    PyBuffer_Release(&b);
    return d;
  }
  // None: torch's current stream; else a torch stream, or a raw cudaStream_t as anything int() takes
  void *stream() {
    PyObject *o = a[i++];
    if (!ok) return nullptr;
    if (o == Py_None) return (void *)c10::cuda::getCurrentCUDAStream().stream();
    PyObject *v = PyObject_GetAttrString(o, "cuda_stream");
    if (v == nullptr && PyErr_ExceptionMatches(PyExc_AttributeError)) {
      PyErr_Clear();
      v = PyNumber_Long(o);
    }
    ok = v != nullptr;
    if (!ok) return nullptr;
    void *s = nullptr;
    if (PyLong_Check(v)) s = PyLong_AsVoidPtr(v);
    else PyErr_Format(PyExc_TypeError, "expected a stream, got %S", (PyObject *)Py_TYPE(o));
    Py_DECREF(v);
    if (s == nullptr && PyErr_Occurred()) ok = false;
    return s;
  }
};

// Runs the call without the GIL and returns its status.
template <class F>
PyObject *finish(const Args &A, F &&call) {
  if (!A.ok) return nullptr;
  xnor_status s;
  Py_BEGIN_ALLOW_THREADS
  s = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)s);
}

// Sizes of a tensor argument of `dims` dimensions (0: any number, the first size); anything else is an error.
void sizes_of(Args &A, PyObject *o, int dims, int *out) {
  if (!A.ok) return;
  const int want = dims > 0 ? dims : 1;
  if (THPVariable_CheckExact(o)) {
    const at::Tensor &t = THPVariable_Unpack(o);
    A.ok = dims > 0 ? t.dim() == dims : t.dim() > 0;
    for (int i = 0; A.ok && i < want; ++i) out[i] = (int)t.size(i);
  } else {
    PyObject *shape = PyObject_GetAttrString(o, "shape"), *s = shape != nullptr ? PySequence_Tuple(shape) : nullptr;
    Py_XDECREF(shape);
    if (s != nullptr) A.ok = dims > 0 ? PyTuple_GET_SIZE(s) == dims : PyTuple_GET_SIZE(s) > 0;
    for (int i = 0; s != nullptr && A.ok && i < want; ++i) out[i] = (int)PyLong_AsLong(PyTuple_GET_ITEM(s, i));
    Py_XDECREF(s);
    if (PyErr_Occurred()) { A.ok = false; return; }
  }
  if (!A.ok) PyErr_Format(PyExc_ValueError, "expected a tensor of %d dimensions", want);
}

// Torch's accessors throw (a tensor under vmap has no data pointer, one with symbolic sizes no size): an
// exception must become a Python error before it reaches the interpreter, which is C.
template <PyObject *(*kCall)(PyObject *const *, Py_ssize_t)>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t nargs) {
  HANDLE_TH_ERRORS
  return kCall(args, nargs);
  END_HANDLE_TH_ERRORS
}

#define XNOR_PY(name) PyObject *name(PyObject *const *args, Py_ssize_t nargs)

XNOR_PY(binarize_weights) {          // w, w_packed, alpha, stream
  Args A(args, nargs, 4);
  int z[4] = {};
  if (A.ok) sizes_of(A, args[0], 4, z);
  if (!A.ok) return nullptr;
  const float *w = A.f32(); uint32_t *wp = A.u32(); float *alpha = A.f32(); void *st = A.stream();
  return finish(A, [&] { return E.binarize_weights(w, z[0], z[1], z[2], z[3], wp, alpha, st); });
}

XNOR_PY(binarize_weights_transposed) {   // w, wT_packed, stream
  Args A(args, nargs, 3);
  int z[4] = {};
  if (A.ok) sizes_of(A, args[0], 4, z);
  if (!A.ok) return nullptr;
  const float *w = A.f32(); uint32_t *wp = A.u32(); void *st = A.stream();
  return finish(A, [&] { return E.binarize_weights_transposed(w, z[0], z[1], z[2], z[3], wp, st); });
}

XNOR_PY(binactiv) {                  // x, bn_scale, bn_shift, d, x_packed, A, K, stream
  Args A(args, nargs, 8);
  if (!A.ok) return nullptr;
  const float *x = A.f32(), *sc = A.f32(), *sh = A.f32(); const xnor_conv_desc d = A.desc();
  uint32_t *xp = A.u32(); float *a = A.f32(), *k = A.f32(); void *st = A.stream();
  return finish(A, [&] { return E.binactiv(x, sc, sh, &d, xp, a, k, st); });
}

XNOR_PY(binactiv_kbit) {             // x, bn_scale, bn_shift, d, kbits, x_planes, A, K, stream
  Args A(args, nargs, 9);
  if (!A.ok) return nullptr;
  const float *x = A.f32(), *sc = A.f32(), *sh = A.f32(); const xnor_conv_desc d = A.desc();
  const int kb = A.num(); uint32_t *xp = A.u32(); float *a = A.f32(), *k = A.f32(); void *st = A.stream();
  return finish(A, [&] { return E.binactiv_kbit(x, sc, sh, &d, kb, xp, a, k, st); });
}

XNOR_PY(conv2d_forward) {            // x_packed, w_packed, alpha, K, residual, d, out, acc_out, stream
  Args A(args, nargs, 9);
  if (!A.ok) return nullptr;
  const uint32_t *xp = A.u32(), *wp = A.u32(); const float *al = A.f32(), *k = A.f32(), *res = A.f32();
  const xnor_conv_desc d = A.desc(); float *out = A.f32(); int32_t *acc = A.i32(); void *st = A.stream();
  return finish(A, [&] { return E.conv2d_forward(xp, wp, al, k, res, &d, out, acc, st); });
}

XNOR_PY(conv2d_forward_kbit) {       // x_planes, kbits, w_packed, alpha, K, residual, d, out, acc_out, stream
  Args A(args, nargs, 10);
  if (!A.ok) return nullptr;
  const uint32_t *xp = A.u32(); const int kb = A.num(); const uint32_t *wp = A.u32();
  const float *al = A.f32(), *k = A.f32(), *res = A.f32(); const xnor_conv_desc d = A.desc();
  float *out = A.f32(); int32_t *acc = A.i32(); void *st = A.stream();
  return finish(A, [&] { return E.conv2d_forward_kbit(xp, kb, wp, al, k, res, &d, out, acc, st); });
}

XNOR_PY(conv2d_forward_binactiv) {   // x_packed, w_packed, alpha, K, residual, d, out, next_scale, next_shift,
  Args A(args, nargs, 12);           // x_packed_next, A_parts, stream
  if (!A.ok) return nullptr;
  const uint32_t *xp = A.u32(), *wp = A.u32(); const float *al = A.f32(), *k = A.f32(), *res = A.f32();
  const xnor_conv_desc d = A.desc(); float *out = A.f32(); const float *ns = A.f32(), *nh = A.f32();
  uint32_t *xn = A.u32(); float *ap = A.f32(); void *st = A.stream();
  return finish(A, [&] { return E.conv2d_forward_binactiv(xp, wp, al, k, res, &d, out, ns, nh, xn, ap, st); });
}

XNOR_PY(binactiv_finish) {           // A_parts, parts, d_next, A, K, stream
  Args A(args, nargs, 6);
  if (!A.ok) return nullptr;
  const float *ap = A.f32(); const int parts = A.num(); const xnor_conv_desc d = A.desc();
  float *a = A.f32(), *k = A.f32(); void *st = A.stream();
  return finish(A, [&] { return E.binactiv_finish(ap, parts, &d, a, k, st); });
}

XNOR_PY(shortcut_conv1x1) {          // x, w, stride, out, stream
  Args A(args, nargs, 5);
  int z[4] = {};
  if (A.ok) sizes_of(A, args[0], 4, z);
  if (!A.ok) return nullptr;
  const float *x = A.f32(), *w = A.f32(); const int s = A.num(); float *out = A.f32(); void *st = A.stream();
  int co = 0;                        // filters are [C_out][C_in] or [C_out][C_in][1][1]
  if (args[1] != Py_None) sizes_of(A, args[1], 0, &co);
  return finish(A, [&] { return E.shortcut_conv1x1(x, w, z[0], z[1], z[2], z[3], co, s, out, st); });
}

XNOR_PY(maxpool2d) {                 // x, k, stride, pad, relu, out, stream
  Args A(args, nargs, 7);
  int z[4] = {};
  if (A.ok) sizes_of(A, args[0], 4, z);
  if (!A.ok) return nullptr;
  const float *x = A.f32(); const int k = A.num(), s = A.num(), p = A.num(), r = A.num();
  float *out = A.f32(); void *st = A.stream();
  return finish(A, [&] { return E.maxpool2d(x, z[0], z[1], z[2], z[3], k, s, p, r, out, st); });
}

XNOR_PY(bwn_prepare_input) {         // x, bn_scale, bn_shift, d, x_stream, stream
  Args A(args, nargs, 6);
  if (!A.ok) return nullptr;
  const float *x = A.f32(), *sc = A.f32(), *sh = A.f32(); const xnor_conv_desc d = A.desc();
  uint16_t *xs = A.bf16(); void *st = A.stream();
  return finish(A, [&] { return E.bwn_prepare_input(x, sc, sh, &d, xs, st); });
}

XNOR_PY(bwn_conv2d_forward) {        // x_stream, w_packed, alpha, residual, d, out, stream
  Args A(args, nargs, 7);
  if (!A.ok) return nullptr;
  const uint16_t *xs = A.bf16(); const uint32_t *wp = A.u32(); const float *al = A.f32(), *res = A.f32();
  const xnor_conv_desc d = A.desc(); float *out = A.f32(); void *st = A.stream();
  return finish(A, [&] { return E.bwn_conv2d_forward(xs, wp, al, res, &d, out, st); });
}

XNOR_PY(binary_gradient_backward) {  // g, wT_packed, alpha, d, gmax, g_stream, grad_in, stream
  Args A(args, nargs, 8);
  if (!A.ok) return nullptr;
  const float *g = A.f32(); const uint32_t *wT = A.u32(); const float *al = A.f32();
  const xnor_conv_desc d = A.desc(); float *gm = A.f32(); uint16_t *gs = A.bf16(); float *gi = A.f32();
  void *st = A.stream();
  return finish(A, [&] { return E.binary_gradient_backward(g, wT, al, &d, gm, gs, gi, st); });
}

// bind(addresses, descriptor, address): the entry points' addresses, in the order of struct Entry, the
// descriptor's class, and the Python conversion of what is not exactly a tensor
PyObject *bind(PyObject *, PyObject *const *args, Py_ssize_t nargs) {
  if (nargs != 3) return PyErr_Format(PyExc_TypeError, "expected 3 arguments, got %zd", nargs);
  PyObject *t = PySequence_Tuple(args[0]);
  if (t == nullptr) return nullptr;
  void *p[kEntries];
  bool ok = PyTuple_GET_SIZE(t) == kEntries;
  if (!ok) PyErr_Format(PyExc_ValueError, "expected %zd addresses", kEntries);
  for (Py_ssize_t i = 0; ok && i < kEntries; ++i) {
    p[i] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(t, i));
    if (p[i] == nullptr) { ok = false; if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null address"); }
  }
  Py_DECREF(t);
  if (!ok) return nullptr;
  memcpy((void *)&E, p, sizeof(E));
  Py_XSETREF(desc_type, Py_NewRef(args[1]));
  Py_XSETREF(py_address, Py_NewRef(args[2]));
  Py_RETURN_NONE;
}

#define XNOR_FAST(name) {#name, (PyCFunction)(void (*)(void))entry<name>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, nullptr},
    XNOR_FAST(binarize_weights), XNOR_FAST(binactiv), XNOR_FAST(conv2d_forward), XNOR_FAST(shortcut_conv1x1),
    XNOR_FAST(conv2d_forward_binactiv), XNOR_FAST(binactiv_finish), XNOR_FAST(maxpool2d), XNOR_FAST(binactiv_kbit),
    XNOR_FAST(conv2d_forward_kbit), XNOR_FAST(bwn_prepare_input), XNOR_FAST(bwn_conv2d_forward),
    XNOR_FAST(binarize_weights_transposed), XNOR_FAST(binary_gradient_backward),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pymarshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pymarshal(void) { return PyModule_Create(&module); }
