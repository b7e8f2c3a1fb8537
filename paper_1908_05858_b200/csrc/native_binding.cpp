// The calls that a program makes per layer, without Python between the tensors and the C ABI: argument checks, the output from
// torch's allocator, the current stream and the call itself.  A small layer's two kernels take about 6 us; through ctypes its two
// calls took 18.1 us of host time, most of it attribute look-ups, struct marshalling and torch.empty's argument parser; 8.4 like this.
//
// Only the ordinary case is handled here -- plain contiguous CUDA tensors of the right types on the current device, outputs made
// by torch.  Everything else, refused arguments included, returns None: binding.py then takes its general path, which converts,
// allocates through the caller's hook, or raises.  A launch that failed is not made again: its status is raised from here.  Nothing
// is kept from one call for the next.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>

#include "dabnn.h"

namespace {

// Entry points of the loaded library, in the order binding.py passes their addresses.
struct Entries {
  decltype(&dabnn_pack) pack;
  decltype(&dabnn_bconv2d) bconv2d;
  decltype(&dabnn_bconv2d_bn_sign_pack) bn_sign_pack;
  decltype(&dabnn_bconv2d_bn_add_sign_pack) bn_add_sign_pack;
  decltype(&dabnn_tc_bconv2d) tc_bconv2d;
  decltype(&dabnn_tc_bconv2d_bn_sign_pack) tc_bn_sign_pack;
  decltype(&dabnn_tc_bconv2d_bn_add_sign_pack) tc_bn_add_sign_pack;
};
Entries g_entries;
PyObject* g_check;  // binding.py's: raises what a status stands for

PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
  static_assert(sizeof(Entries) == 7 * sizeof(void*), "one address per entry");
  if (n != 8 || !PyCallable_Check(args[7])) {
    PyErr_SetString(PyExc_TypeError, "bind takes seven addresses and what raises a status");
    return nullptr;
  }
  void* address[7];
  for (int i = 0; i < 7; i++) {
    address[i] = PyLong_AsVoidPtr(args[i]);
    if (PyErr_Occurred()) return nullptr;
  }
  memcpy(&g_entries, address, sizeof(g_entries));
  Py_XSETREF(g_check, Py_NewRef(args[7]));
  Py_RETURN_NONE;
}

// The tensor behind `o` if it is a plain contiguous CUDA tensor of this type, else nullptr.
const at::Tensor* plain(PyObject* o, at::ScalarType type) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || !t.is_cuda() || t.scalar_type() != type || t.layout() != at::kStrided || !t.is_contiguous()) return nullptr;
  return &t;
}

bool fits(int64_t v) { return v >= 0 && v <= INT_MAX; }

// A Python int of C's range (bool and other types: no).
bool integer(PyObject* o, int& v) {
  if (!PyLong_CheckExact(o)) return false;
  int overflow = 0;
  const long l = PyLong_AsLongAndOverflow(o, &overflow);
  if (overflow != 0 || l < INT_MIN || l > INT_MAX) return false;
  v = (int)l;
  return true;
}
bool pair(PyObject* o, int& a, int& b) {
  return PyTuple_CheckExact(o) && PyTuple_GET_SIZE(o) == 2 && integer(PyTuple_GET_ITEM(o, 0), a) && integer(PyTuple_GET_ITEM(o, 1), b);
}

// dabnn_out_dim; -1 for a padded size that no int holds.
int out_dim(int in, int k, int stride, int pad) {
  const long long padded = (long long)in + 2LL * pad, span = padded - k;
  if (padded > INT_MAX) return -1;
  return span >= 0 && stride > 0 ? (int)(span / stride + 1) : 0;
}

at::Tensor make(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like) {
  return at::empty(sizes, at::TensorOptions().dtype(type).device(like.device()));
}

// The call itself, with the interpreter released as ctypes does.
template <typename F>
dabnn_status status_of(F f) {
  dabnn_status s;
  Py_BEGIN_ALLOW_THREADS
  s = f();
  Py_END_ALLOW_THREADS
  return s;
}

// What a call with a status other than OK returns.  Arguments are refused before anything is launched: the general path meets the
// same refusal and reports it.  After any other status the launch may have gone out, and the library has read (and so cleared) the
// runtime's error: a second call could succeed in silence.
PyObject* not_made(dabnn_status s) {
  switch (s) {
    case DABNN_ERR_NULL:
    case DABNN_ERR_SHAPE:
    case DABNN_ERR_UNSUPPORTED:
    case DABNN_ERR_ALIGNMENT:
    case DABNN_ERR_WORKSPACE:
    case DABNN_ERR_STATIC_LIMIT: Py_RETURN_NONE;
    default: break;
  }
  PyObject* returned = PyObject_CallFunction(g_check, "i", (int)s);
  if (returned != nullptr) {
    Py_DECREF(returned);
    PyErr_Format(PyExc_RuntimeError, "dabnn status %d", (int)s);
  }
  return nullptr;
}

template <typename F>
PyObject* guarded(F f) {
  try {
    return f();
  } catch (...) {  // (a tensor without storage, an allocation that failed: the general path meets it again and raises)
    PyErr_Clear();
    Py_RETURN_NONE;
  }
}

// What the convolutions share: activations, filter geometry (from the packed weights, or given beside a prepared buffer), output size.
struct Geometry {
  const at::Tensor* a;
  const void* w;
  dabnn_shape in;
  dabnn_conv cv;
  int O, OH, OW;
  void* stream;
};
bool geometry(Geometry& g, PyObject* a, PyObject* stride, PyObject* pad, PyObject* pad_value, int words) {
  g.a = plain(a, at::kLong);
  if (g.a == nullptr || g.a->dim() != 4) return false;
  for (int d = 0; d < 4; d++)
    if (!fits(g.a->size(d))) return false;
  if (g.a->size(3) != words || g.in.C <= 0 || words != (g.in.C + 63LL) / 64) return false;
  g.in.N = (int)g.a->size(0);
  g.in.H = (int)g.a->size(1);
  g.in.W = (int)g.a->size(2);
  if (!pair(stride, g.cv.stride_h, g.cv.stride_w) || !pair(pad, g.cv.pad_h, g.cv.pad_w) || !integer(pad_value, g.cv.pad_value)) return false;
  if (g.cv.stride_h <= 0 || g.cv.stride_w <= 0 || !fits(g.cv.pad_h) || !fits(g.cv.pad_w)) return false;
  g.OH = out_dim(g.in.H, g.cv.kh, g.cv.stride_h, g.cv.pad_h);
  g.OW = out_dim(g.in.W, g.cv.kw, g.cv.stride_w, g.cv.pad_w);
  if (g.OH < 0 || g.OW < 0) return false;
  const auto stream = c10::cuda::getCurrentCUDAStream();
  g.stream = stream.stream();
  return g.a->device() == stream.device();
}
// packed weights [O][kh][kw][Cw]
bool from_packed(Geometry& g, PyObject* w_obj, PyObject* C, int& words) {
  const at::Tensor* w = plain(w_obj, at::kLong);
  if (w == nullptr || w->dim() != 4 || !integer(C, g.in.C)) return false;
  for (int d = 0; d < 4; d++)
    if (!fits(w->size(d))) return false;
  g.O = (int)w->size(0);
  g.cv.kh = (int)w->size(1);
  g.cv.kw = (int)w->size(2);
  words = (int)w->size(3);
  g.w = w->data_ptr();
  return true;
}
// a prepared buffer and (C, O, kh, kw)
bool from_prepared(Geometry& g, PyObject* buf, PyObject* C, PyObject* O, PyObject* kh, PyObject* kw, int& words) {
  const at::Tensor* w = plain(buf, at::kByte);
  if (w == nullptr || !integer(C, g.in.C) || !integer(O, g.O) || !integer(kh, g.cv.kh) || !integer(kw, g.cv.kw)) return false;
  words = (int)((g.in.C + 63LL) / 64);
  g.w = w->data_ptr();
  return true;
}

at::Tensor sums_like(const Geometry& g, int layout) {
  return layout == DABNN_NHWC ? make({g.in.N, g.OH, g.OW, g.O}, at::kInt, *g.a) : make({g.in.N, g.O, g.OH, g.OW}, at::kInt, *g.a);
}
at::Tensor words_like(const Geometry& g) { return make({g.in.N, g.OH, g.OW, (g.O + 63LL) / 64}, at::kLong, *g.a); }

// pack(x, layout)
PyObject* pack(PyObject*, PyObject* const* args, Py_ssize_t n) {
  return guarded([&]() -> PyObject* {
    int layout;
    const at::Tensor* x = n == 2 && integer(args[1], layout) && (layout == DABNN_NCHW || layout == DABNN_NHWC) ? plain(args[0], at::kFloat) : nullptr;
    if (x == nullptr || x->dim() != 4) Py_RETURN_NONE;
    for (int d = 0; d < 4; d++)
      if (!fits(x->size(d))) Py_RETURN_NONE;
    const bool nchw = layout == DABNN_NCHW;
    const dabnn_shape in = {(int)x->size(0), (int)x->size(nchw ? 1 : 3), (int)x->size(nchw ? 2 : 1), (int)x->size(nchw ? 3 : 2)};
    const auto stream = c10::cuda::getCurrentCUDAStream();
    if (x->device() != stream.device()) Py_RETURN_NONE;
    at::Tensor out = make({in.N, in.H, in.W, (in.C + 63LL) / 64}, at::kLong, *x);
    const float* src = static_cast<const float*>(x->data_ptr());
    uint64_t* dst = static_cast<uint64_t*>(out.data_ptr());
    const dabnn_status s = status_of([&] { return g_entries.pack(src, (dabnn_layout)layout, in, dst, stream.stream()); });
    if (s != DABNN_OK) return not_made(s);
    return THPVariable_Wrap(std::move(out));
  });
}

template <typename W>
PyObject* conv_int32(decltype(&dabnn_tc_bconv2d) entry, decltype(&dabnn_bconv2d) packed_entry, PyObject* a, PyObject* const* tail, W weights) {
  return guarded([&]() -> PyObject* {  // tail: stride, pad, pad_value, out_layout
    Geometry g;
    int words, layout;
    if (!weights(g, words) || !geometry(g, a, tail[0], tail[1], tail[2], words)) Py_RETURN_NONE;
    if (!integer(tail[3], layout) || (layout != DABNN_NCHW && layout != DABNN_NHWC)) Py_RETURN_NONE;
    at::Tensor out = sums_like(g, layout);
    const uint64_t* ap = static_cast<const uint64_t*>(g.a->data_ptr());
    int32_t* dst = static_cast<int32_t*>(out.data_ptr());
    const dabnn_status s = status_of([&] {
      return entry != nullptr ? entry(ap, g.in, g.w, g.O, g.cv, dst, (dabnn_layout)layout, g.stream)
                              : packed_entry(ap, g.in, static_cast<const uint64_t*>(g.w), g.O, g.cv, dst, (dabnn_layout)layout, g.stream);
    });
    if (s != DABNN_OK) return not_made(s);
    return THPVariable_Wrap(std::move(out));
  });
}

// (the library reads O values from each; the general path checks no more than this)
const float* vector(PyObject* o) {
  const at::Tensor* t = plain(o, at::kFloat);
  return t != nullptr ? static_cast<const float*>(t->data_ptr()) : nullptr;
}

template <typename W>
PyObject* conv_signs(decltype(&dabnn_tc_bconv2d_bn_sign_pack) entry, decltype(&dabnn_bconv2d_bn_sign_pack) packed_entry, PyObject* a,
                     PyObject* const* tail, W weights) {
  return guarded([&]() -> PyObject* {  // tail: scale, shift, stride, pad, pad_value
    Geometry g;
    int words;
    if (!weights(g, words) || !geometry(g, a, tail[2], tail[3], tail[4], words)) Py_RETURN_NONE;
    const float *scale = vector(tail[0]), *shift = vector(tail[1]);
    if (scale == nullptr || shift == nullptr) Py_RETURN_NONE;
    at::Tensor out = words_like(g);
    const uint64_t* ap = static_cast<const uint64_t*>(g.a->data_ptr());
    uint64_t* dst = static_cast<uint64_t*>(out.data_ptr());
    const dabnn_status s = status_of([&] {
      return entry != nullptr ? entry(ap, g.in, g.w, g.O, g.cv, scale, shift, dst, g.stream)
                              : packed_entry(ap, g.in, static_cast<const uint64_t*>(g.w), g.O, g.cv, scale, shift, dst, g.stream);
    });
    if (s != DABNN_OK) return not_made(s);
    return THPVariable_Wrap(std::move(out));
  });
}

template <typename W>
PyObject* conv_block(decltype(&dabnn_tc_bconv2d_bn_add_sign_pack) entry, decltype(&dabnn_bconv2d_bn_add_sign_pack) packed_entry, PyObject* a,
                     PyObject* const* tail, W weights) {
  return guarded([&]() -> PyObject* {  // tail: scale, shift, residual, stride, pad, pad_value, want_bits
    Geometry g;
    int words;
    if (!weights(g, words) || !geometry(g, a, tail[3], tail[4], tail[5], words)) Py_RETURN_NONE;
    const float *scale = vector(tail[0]), *shift = vector(tail[1]);
    const at::Tensor* residual = plain(tail[2], at::kFloat);
    if (scale == nullptr || shift == nullptr || residual == nullptr || residual->dim() != 4 || residual->size(0) != g.in.N ||
        residual->size(1) != g.OH || residual->size(2) != g.OW || residual->size(3) != g.O || !PyBool_Check(tail[6]))
      Py_RETURN_NONE;
    at::Tensor y = make(residual->sizes(), at::kFloat, *g.a), bits;
    if (tail[6] == Py_True) bits = words_like(g);
    const uint64_t* ap = static_cast<const uint64_t*>(g.a->data_ptr());
    const float* rp = static_cast<const float*>(residual->data_ptr());
    float* yp = static_cast<float*>(y.data_ptr());
    uint64_t* bp = bits.defined() ? static_cast<uint64_t*>(bits.data_ptr()) : nullptr;
    const dabnn_status s = status_of([&] {
      return entry != nullptr ? entry(ap, g.in, g.w, g.O, g.cv, scale, shift, rp, yp, bp, g.stream)
                              : packed_entry(ap, g.in, static_cast<const uint64_t*>(g.w), g.O, g.cv, scale, shift, rp, yp, bp, g.stream);
    });
    if (s != DABNN_OK) return not_made(s);
    PyObject* py = THPVariable_Wrap(std::move(y));
    if (py == nullptr) return nullptr;
    PyObject* pb = bits.defined() ? THPVariable_Wrap(std::move(bits)) : Py_NewRef(Py_None);
    if (pb == nullptr) {
      Py_DECREF(py);
      return nullptr;
    }
    PyObject* both = PyTuple_New(2);
    if (both == nullptr) {
      Py_DECREF(py);
      Py_DECREF(pb);
      return nullptr;
    }
    PyTuple_SET_ITEM(both, 0, py);
    PyTuple_SET_ITEM(both, 1, pb);
    return both;
  });
}

// On packed weights: (a, C, w, ...); on prepared ones: (a, buf, C, O, kh, kw, ...); the rest as in each function above.
#define DABNN_CALL(name, function, entry, packed_entry, head, rest, weights)                \
  PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t n) {                          \
    if (n != (head) + (rest)) Py_RETURN_NONE;                                               \
    return function(entry, packed_entry, args[0], args + (head), [&](Geometry& g, int& words) { return weights; }); \
  }
#define DABNN_PACKED from_packed(g, args[2], args[1], words)
#define DABNN_PREPARED from_prepared(g, args[1], args[2], args[3], args[4], args[5], words)
DABNN_CALL(bconv2d, conv_int32, nullptr, g_entries.bconv2d, 3, 4, DABNN_PACKED)
DABNN_CALL(bn_sign_pack, conv_signs, nullptr, g_entries.bn_sign_pack, 3, 5, DABNN_PACKED)
DABNN_CALL(bn_add_sign_pack, conv_block, nullptr, g_entries.bn_add_sign_pack, 3, 7, DABNN_PACKED)
DABNN_CALL(tc_bconv2d, conv_int32, g_entries.tc_bconv2d, nullptr, 6, 4, DABNN_PREPARED)
DABNN_CALL(tc_bn_sign_pack, conv_signs, g_entries.tc_bn_sign_pack, nullptr, 6, 5, DABNN_PREPARED)
DABNN_CALL(tc_bn_add_sign_pack, conv_block, g_entries.tc_bn_add_sign_pack, nullptr, 6, 7, DABNN_PREPARED)

#define DABNN_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {DABNN_METHOD(bind), DABNN_METHOD(pack), DABNN_METHOD(bconv2d), DABNN_METHOD(bn_sign_pack),
                         DABNN_METHOD(bn_add_sign_pack), DABNN_METHOD(tc_bconv2d), DABNN_METHOD(tc_bn_sign_pack),
                         DABNN_METHOD(tc_bn_add_sign_pack), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
