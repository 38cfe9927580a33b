// Marshalling of the entry points that a program calls per layer or per batch: torch tensors to raw pointers, the current
// stream, one call of the C ABI without the interpreter lock.  The same checks, errors and results as the ctypes layer in
// binding.py, which holds the declarations and everything that is called rarely; a call through ctypes costs its eleven
// conversions (q8_conv2d of the smallest layer 7.0 us of host time, detection output with six sources 52 us).
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <cstdint>
#include <vector>

#include "q8.h"

namespace {

// C ABI entry points, by the addresses the ctypes layer has loaded (one copy of the library, one set of error strings).
struct Entry {
  decltype(&q8_conv2d) conv2d;
  decltype(&q8_conv2d_then_1x1) then_1x1;
  decltype(&q8_calibrate_maxabs) maxabs;
  decltype(&q8_quantize) quantize;
  decltype(&q8_dequantize) dequantize;
  decltype(&q8_detection_output_workspace_bytes) det_bytes;
  decltype(&q8_detection_output) detect;
} g_q8;

void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Address of a contiguous CUDA tensor or of nothing (None); on anything else a TypeError is set and false returned.
bool dev(PyObject* o, const char* what, void** p) {
  *p = nullptr;
  if (o == Py_None) return true;
  if (THPVariable_Check(o)) {
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.is_cuda() && t.is_contiguous()) {
      *p = t.numel() ? t.data_ptr() : nullptr;
      return true;
    }
  }
  PyErr_Format(PyExc_TypeError, "%s: expected a contiguous CUDA tensor", what);
  return false;
}

PyObject* g_desc_type = nullptr;  // the binding's ctypes structure

// The bytes of a descriptor, an instance of that structure or of a class derived from it.
struct Bytes {
  Py_buffer b{};
  bool ok = false;
  explicit Bytes(PyObject* o) { ok = PyObject_IsInstance(o, g_desc_type) == 1 && PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) == 0; }
  ~Bytes() { if (ok) PyBuffer_Release(&b); }
  const q8_conv_desc* desc() const {
    if (ok && (size_t)b.len >= sizeof(q8_conv_desc)) return static_cast<const q8_conv_desc*>(b.buf);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "expected a q8_conv_desc");
    return nullptr;
  }
};

template <typename F>
PyObject* call(F f) {
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

bool number(PyObject* o, float* v) {
  const double d = PyFloat_AsDouble(o);
  if (d == -1.0 && PyErr_Occurred()) return false;
  *v = (float)d;
  return true;
}
bool number(PyObject* o, int* v) {
  const long l = PyLong_AsLong(o);
  if (l == -1 && PyErr_Occurred()) return false;
  *v = (int)l;
  return true;
}

bool count(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return true;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments", want);
  return false;
}

// (desc, x, w, bias, scale, residual, residual_scale, y, workspace) -> status
PyObject* py_conv2d(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!count(n, 9)) return nullptr;
  HANDLE_TH_ERRORS
  Bytes d(a[0]);
  const q8_conv_desc* desc = d.desc();
  void *x, *w, *bias, *scale, *res, *y, *ws;
  float rs;
  if (!desc || !dev(a[1], "x", &x) || !dev(a[2], "w", &w) || !dev(a[3], "bias", &bias) || !dev(a[4], "scale", &scale) ||
      !dev(a[5], "residual", &res) || !number(a[6], &rs) || !dev(a[7], "y", &y) || !dev(a[8], "workspace", &ws))
    return nullptr;
  const size_t bytes = a[8] == Py_None ? 0 : THPVariable_Unpack(a[8]).nbytes();
  void* s = current_stream();
  return call([&] {
    return g_q8.conv2d(desc, x, static_cast<const int8_t*>(w), static_cast<const int32_t*>(bias), static_cast<const float*>(scale), res, rs,
                       y, ws, bytes, s);
  });
  END_HANDLE_TH_ERRORS
}

// (d1, d2, x, w1, bias1, scale1, w2, bias2, scale2, residual, residual_scale, y) -> status
PyObject* py_then_1x1(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!count(n, 12)) return nullptr;
  HANDLE_TH_ERRORS
  Bytes b1(a[0]), b2(a[1]);
  const q8_conv_desc* d1 = b1.desc();
  const q8_conv_desc* d2 = d1 ? b2.desc() : nullptr;
  void *x, *w1, *bias1, *scale1, *w2, *bias2, *scale2, *res, *y;
  float rs;
  if (!d1 || !d2 || !dev(a[2], "x", &x) || !dev(a[3], "w1", &w1) || !dev(a[4], "bias1", &bias1) || !dev(a[5], "scale1", &scale1) ||
      !dev(a[6], "w2", &w2) || !dev(a[7], "bias2", &bias2) || !dev(a[8], "scale2", &scale2) || !dev(a[9], "residual", &res) ||
      !number(a[10], &rs) || !dev(a[11], "y", &y))
    return nullptr;
  void* s = current_stream();
  return call([&] {
    return g_q8.then_1x1(d1, d2, x, static_cast<const int8_t*>(w1), static_cast<const int32_t*>(bias1), static_cast<const float*>(scale1),
                         static_cast<const int8_t*>(w2), static_cast<const int32_t*>(bias2), static_cast<const float*>(scale2), res, rs, y, s);
  });
  END_HANDLE_TH_ERRORS
}

// The elements of a tensor; anything else has the error of its attribute (dev() has let nothing but None through).
bool numel(PyObject* o, size_t* n) {
  if (THPVariable_Check(o)) {
    *n = (size_t)THPVariable_Unpack(o).numel();
    return true;
  }
  THPObjectPtr attr(PyObject_GetAttrString(o, "numel"));
  if (attr) PyErr_SetString(PyExc_TypeError, "expected a tensor");
  return false;
}

// (x, running_max) -> status
PyObject* py_maxabs(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!count(n, 2)) return nullptr;
  HANDLE_TH_ERRORS
  void *x, *m;
  size_t k;
  if (!dev(a[0], "x", &x) || !dev(a[1], "running_max", &m) || !numel(a[0], &k)) return nullptr;
  void* s = current_stream();
  return call([&] { return g_q8.maxabs(static_cast<const float*>(x), k, static_cast<float*>(m), s); });
  END_HANDLE_TH_ERRORS
}

// (x, q, type, out) -> status
PyObject* py_quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!count(n, 4)) return nullptr;
  HANDLE_TH_ERRORS
  void *x, *out;
  float q;
  int type;
  size_t k;
  if (!dev(a[0], "x", &x) || !number(a[1], &q) || !number(a[2], &type) || !dev(a[3], "out", &out) || !numel(a[0], &k)) return nullptr;
  void* s = current_stream();
  return call([&] { return g_q8.quantize(static_cast<const float*>(x), k, q, type, out, s); });
  END_HANDLE_TH_ERRORS
}

// (z, type, q, out) -> status
PyObject* py_dequantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!count(n, 4)) return nullptr;
  HANDLE_TH_ERRORS
  void *z, *out;
  float q;
  int type;
  size_t k;
  if (!dev(a[0], "z", &z) || !number(a[1], &type) || !number(a[2], &q) || !dev(a[3], "out", &out) || !numel(a[0], &k)) return nullptr;
  void* s = current_stream();
  return call([&] { return g_q8.dequantize(z, type, k, q, static_cast<float*>(out), s); });
  END_HANDLE_TH_ERRORS
}

// Address, cell stride in floats and cells per image of a CUDA fp32 tensor [N, cells..., values] whose cells lie a fixed
// stride apart (a contiguous tensor, or a slice of the last dimension of one).
bool cell_view(PyObject* o, const char* what, const float** p, int* stride, int* cells, int64_t* images) {
  const at::Tensor* t = THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr;
  if (!t || !t->is_cuda() || t->scalar_type() != at::kFloat || t->dim() < 2 || t->stride(-1) != 1) {
    PyErr_Format(PyExc_TypeError, "%s: expected a CUDA fp32 tensor with unit stride in its last dimension", what);
    return false;
  }
  *p = static_cast<const float*>(t->numel() ? t->data_ptr() : nullptr);
  *images = t->size(0);
  const int64_t d = t->dim();
  if (d == 2) {
    *stride = (int)t->stride(0);
    *cells = 1;
    return true;
  }
  *stride = (int)t->stride(-2);
  int64_t c = 1;
  for (int64_t i = 0; i < d - 2; ++i)
    if (t->size(i) > 1 && t->stride(i) != t->stride(i + 1) * t->size(i + 1)) {
      PyErr_Format(PyExc_TypeError, "%s: cells are not a fixed stride apart", what);
      return false;
    }
  for (int64_t i = 1; i < d - 1; ++i) c *= t->size(i);
  *cells = (int)c;
  return true;
}

// The sources of a detection output, a sequence of (loc, conf, boxes per cell); what int() takes counts boxes.
struct Sources {
  std::vector<const float*> loc, conf;
  std::vector<int> ls, cs, cells, boxes;
  int64_t images = 0;
  long long P = 0;   // boxes per image

  bool parse(PyObject* sources) {
    THPObjectPtr seq(PySequence_Fast(sources, "sources: expected a sequence"));
    if (!seq) return false;
    const Py_ssize_t k = PySequence_Fast_GET_SIZE(seq.get());
    loc.resize(k); conf.resize(k);
    ls.resize(k); cs.resize(k); cells.resize(k); boxes.resize(k);
    for (Py_ssize_t i = 0; i < k; ++i) {
      THPObjectPtr item(PySequence_Fast(PySequence_Fast_GET_ITEM(seq.get(), i), "sources: expected (loc, conf, boxes per cell)"));
      if (!item) return false;
      if (PySequence_Fast_GET_SIZE(item.get()) != 3) { PyErr_SetString(PyExc_ValueError, "sources: expected (loc, conf, boxes per cell)"); return false; }
      PyObject** e = PySequence_Fast_ITEMS(item.get());
      int ccells;
      int64_t ni, nc;
      if (!cell_view(e[0], "loc", &loc[i], &ls[i], &cells[i], &ni) || !cell_view(e[1], "conf", &conf[i], &cs[i], &ccells, &nc)) return false;
      if (i == 0) images = ni;
      if (ccells != cells[i] || nc != images || ni != images) {
        PyErr_SetString(PyExc_ValueError, "loc and conf of a source must cover the same cells of the same images");
        return false;
      }
      THPObjectPtr count(PyNumber_Long(e[2]));
      if (!count || !number(count.get(), &boxes[i])) return false;
      P += (long long)cells[i] * boxes[i];
    }
    return true;
  }
  int boxes_per_image() const { return (int)(P > 0x7fffffff ? 0x7fffffff : P); }
};

// (sources) -> (images, boxes per image)
PyObject* py_detect_size(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!count(n, 1)) return nullptr;
  HANDLE_TH_ERRORS
  Sources src;
  if (!src.parse(a[0])) return nullptr;
  return Py_BuildValue("Li", (long long)src.images, src.boxes_per_image());
  END_HANDLE_TH_ERRORS
}

// Up to four numbers, what float() takes; those not given are zero.
bool variances(PyObject* o, float (&var)[4]) {
  THPObjectPtr vars(PySequence_Fast(o, "variances: expected a sequence"));
  if (!vars) return false;
  const Py_ssize_t k = PySequence_Fast_GET_SIZE(vars.get());
  if (k > 4) { PyErr_SetString(PyExc_IndexError, "variances: more than four values"); return false; }
  for (Py_ssize_t i = 0; i < 4; ++i) {
    var[i] = 0.0f;
    if (i >= k) continue;
    THPObjectPtr v(PyNumber_Float(PySequence_Fast_GET_ITEM(vars.get(), i)));
    if (!v || !number(v.get(), &var[i])) return false;
  }
  return true;
}

// (sources, priors, variances, classes, background, conf_thresh, nms_thresh, nms_top_k, keep_top_k, workspace, out, counts)
// -> status.  workspace, out and counts are given.
PyObject* py_detect(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!count(n, 12)) return nullptr;
  HANDLE_TH_ERRORS
  Sources src;
  float var[4];
  if (!src.parse(a[0]) || !variances(a[2], var)) return nullptr;
  void *priors, *ws, *out, *counts;
  int classes, background, top, keep;
  float ct, nt;
  if (!dev(a[1], "priors", &priors) || !number(a[3], &classes) || !number(a[4], &background) || !number(a[5], &ct) || !number(a[6], &nt) ||
      !number(a[7], &top) || !number(a[8], &keep) || !dev(a[9], "workspace", &ws) || !dev(a[10], "out", &out) || !dev(a[11], "counts", &counts))
    return nullptr;
  size_t ws_bytes;
  if (!numel(a[9], &ws_bytes)) return nullptr;
  void* s = current_stream();
  return call([&] {
    size_t need;
    const int rc = g_q8.det_bytes((int)src.images, src.boxes_per_image(), classes, background, top, keep, &need);
    if (rc != Q8_OK) return rc;
    return g_q8.detect((int)src.loc.size(), src.loc.data(), src.ls.data(), src.conf.data(), src.cs.data(), src.cells.data(), src.boxes.data(),
                       static_cast<const float*>(priors), var, (int)src.images, classes, background, ct, nt, top, keep, ws, ws_bytes,
                       static_cast<float*>(out), static_cast<int32_t*>(counts), s);
  });
  END_HANDLE_TH_ERRORS
}

// (addresses of the entry points, in the order of Entry, the descriptors' class)
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!count(n, 8)) return nullptr;
  void* p[7];
  for (int i = 0; i < 7; ++i) {
    p[i] = PyLong_AsVoidPtr(a[i]);
    if (!p[i]) return nullptr;
  }
  PyObject* old = g_desc_type;
  Py_INCREF(a[7]);
  g_desc_type = a[7];
  Py_XDECREF(old);
  g_q8.conv2d = reinterpret_cast<decltype(g_q8.conv2d)>(p[0]);
  g_q8.then_1x1 = reinterpret_cast<decltype(g_q8.then_1x1)>(p[1]);
  g_q8.maxabs = reinterpret_cast<decltype(g_q8.maxabs)>(p[2]);
  g_q8.quantize = reinterpret_cast<decltype(g_q8.quantize)>(p[3]);
  g_q8.dequantize = reinterpret_cast<decltype(g_q8.dequantize)>(p[4]);
  g_q8.det_bytes = reinterpret_cast<decltype(g_q8.det_bytes)>(p[5]);
  g_q8.detect = reinterpret_cast<decltype(g_q8.detect)>(p[6]);
  Py_RETURN_NONE;
}

#define Q8_METHOD(name, f) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {Q8_METHOD("bind", py_bind),         Q8_METHOD("conv2d", py_conv2d),     Q8_METHOD("then_1x1", py_then_1x1),
                         Q8_METHOD("maxabs", py_maxabs),     Q8_METHOD("quantize", py_quantize), Q8_METHOD("dequantize", py_dequantize),
                         Q8_METHOD("detect", py_detect),     Q8_METHOD("detect_size", py_detect_size),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_q8native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__q8native(void) { return PyModule_Create(&module); }
