// The calls of binding.py that a running program repeats, as a CPython module: arguments checked, outputs allocated and the
// C ABI called without going through ctypes and a Python-level tensor method per argument.  The kernels of one 4096 x 4096
// projection at one token take 8 us; the two calls it needs took 12.6 us on the host through ctypes (1.4 us a call for the
// argument conversion alone, the rest in tensor methods), which bounded every small case: 12.9 us a projection, 8.1 so (and a
// first pass over new buffers 35 instead of 49).  Failures are reported as the
// C ABI's status, an int, where a call returns tensors otherwise; binding.py turns it into LcdError.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <ATen/ops/zeros.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <vector>

#include "lcd.h"

namespace {

const at::Tensor* tensor_of(PyObject* o, const char* what) {
  if (THPVariable_Check(o)) return &THPVariable_Unpack(o);
  PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor", what);
  return nullptr;
}
// A tensor's address; None: null.
bool address_of(PyObject* o, const char* what, void** out) {
  *out = nullptr;
  if (o == Py_None) return true;
  const at::Tensor* t = tensor_of(o, what);
  if (!t) return false;
  *out = t->data_ptr();
  return true;
}
bool require(bool ok, const char* what) {
  if (!ok) PyErr_SetString(PyExc_AssertionError, what);
  return ok;
}
// The stream of a call: a torch stream object's, or the current one of the current device.  For its life a given stream is the
// current one, so that what the call allocates belongs to the stream that its kernels run on and is cleared there; outputs are
// recorded for the caller's stream as well, whose kernels will read them.
class CallStream {
 public:
  explicit CallStream(PyObject* o) : caller_(c10::cuda::getCurrentCUDAStream()), raw_(caller_.stream()) {
    if (o == Py_None) return;
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    void* given = h ? PyLong_AsVoidPtr(h) : nullptr;
    Py_XDECREF(h);
    failed_ = PyErr_Occurred() != nullptr;
    if (failed_ || given == raw_) return;
    raw_ = static_cast<cudaStream_t>(given);
    c10::cuda::setCurrentCUDAStream(c10::cuda::getStreamFromExternal(raw_, caller_.device_index()));
    other_ = true;
  }
  ~CallStream() {
    if (other_) c10::cuda::setCurrentCUDAStream(caller_);
  }
  CallStream(const CallStream&) = delete;
  CallStream& operator=(const CallStream&) = delete;
  bool ok() const { return !failed_; }
  void* raw() const { return raw_; }
  PyObject* output(const at::Tensor& t) const {
    if (other_) c10::cuda::CUDACachingAllocator::recordStream(t.storage().data_ptr(), caller_);
    return THPVariable_Wrap(t);
  }

 private:
  c10::cuda::CUDAStream caller_;
  cudaStream_t raw_;
  bool failed_ = false, other_ = false;
};
bool count_args(Py_ssize_t have, Py_ssize_t want) {
  if (have != want) PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, have);
  return have == want;
}
template <typename Call>
lcd_status without_gil(Call&& call) {
  lcd_status st;
  Py_BEGIN_ALLOW_THREADS
  st = call();
  Py_END_ALLOW_THREADS
  return st;
}

// (x, inv_smooth, static_scale, act_idx, act_scale, act_bits, stream) -> (act_idx, act_scale) or a status
PyObject* smooth_quantize_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (!count_args(n, 7)) return nullptr;
  const at::Tensor* x = tensor_of(a[0], "x");
  if (!x || !require(x->is_cuda() && x->scalar_type() == at::kHalf && x->dim() == 2 && x->stride(1) == 1,
                     "x: CUDA fp16 [M, K] with unit column stride"))
    return nullptr;
  const int64_t M = x->size(0), K = x->size(1), K_pad = (K + 255) / 256 * 256;
  const long bits = PyLong_AsLong(a[5]);
  if ((bits == -1 && PyErr_Occurred()) || !require(bits == 4 || bits == 8, "act_bits: 4 or 8")) return nullptr;
  const at::ScalarType type = bits == 4 ? at::kByte : at::kChar;
  const CallStream stream(a[6]);
  if (!stream.ok()) return nullptr;
  at::Tensor idx, scale;
  if (a[3] == Py_None) idx = at::empty({M, bits == 4 ? K_pad / 2 : K_pad}, x->options().dtype(type));
  else if (const at::Tensor* t = tensor_of(a[3], "act_idx")) idx = *t;
  else return nullptr;
  if (!require(idx.scalar_type() == type, "act_idx: uint8 for 4-bit levels, int8 for 8-bit levels")) return nullptr;
  if (a[4] == Py_None) scale = at::empty({M}, x->options().dtype(at::kFloat));
  else if (const at::Tensor* t = tensor_of(a[4], "act_scale")) scale = *t;
  else return nullptr;
  void *inv, *fixed;
  if (!address_of(a[1], "inv_smooth", &inv) || !address_of(a[2], "static_scale", &fixed)) return nullptr;
  const lcd_status st = without_gil([&] {
    return lcd_smooth_quantize_act(x->data_ptr(), M, K, x->stride(0), static_cast<float*>(inv), static_cast<float*>(fixed),
                                   (int)bits, static_cast<uint8_t*>(idx.data_ptr()), static_cast<float*>(scale.data_ptr()), stream.raw());
  });
  if (st != LCD_OK) return PyLong_FromLong((long)st);
  PyObject* o0 = a[3] == Py_None ? stream.output(idx) : Py_NewRef(a[3]);
  PyObject* o1 = a[4] == Py_None ? stream.output(scale) : Py_NewRef(a[4]);
  PyObject* out = o0 && o1 ? PyTuple_Pack(2, o0, o1) : nullptr;
  Py_XDECREF(o0);
  Py_XDECREF(o1);
  return out;
  END_HANDLE_TH_ERRORS
}

// (weights, header address, N, {(M, algo): workspace bytes}, act_idx, act_scale, y, algo, workspace, status_word, stream) -> y or a
// status; None: the table does not hold the size yet
PyObject* lut_linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (!count_args(n, 11)) return nullptr;
  const at::Tensor *w = tensor_of(a[0], "weights"), *idx = w ? tensor_of(a[4], "act_idx") : nullptr;
  const at::Tensor* scale = idx ? tensor_of(a[5], "act_scale") : nullptr;
  if (!scale) return nullptr;
  void* header = PyLong_AsVoidPtr(a[1]);
  const int64_t N = PyLong_AsLongLong(a[2]);
  const long algo = PyLong_AsLong(a[7]);
  if (PyErr_Occurred()) return nullptr;
  if (!require(idx->dim() >= 1, "act_idx: [M, levels]")) return nullptr;
  const int64_t M = idx->size(0);
  size_t need = 0;
  {
    PyObject* key = Py_BuildValue("(LO)", (long long)M, a[7]);
    if (!key) return nullptr;
    PyObject* bytes = PyDict_GetItemWithError(a[3], key);
    Py_DECREF(key);
    if (!bytes) {
      if (PyErr_Occurred()) return nullptr;
      Py_RETURN_NONE;
    }
    need = PyLong_AsSize_t(bytes);
    if (PyErr_Occurred()) return nullptr;
  }
  const CallStream stream(a[10]);
  if (!stream.ok()) return nullptr;
  at::Tensor y, ws;
  if (a[6] == Py_None) y = at::empty({M, N}, idx->options().dtype(at::kFloat));
  else if (const at::Tensor* t = tensor_of(a[6], "y")) y = *t;
  else return nullptr;
  if (a[8] != Py_None) {
    const at::Tensor* t = tensor_of(a[8], "workspace");
    if (!t) return nullptr;
    ws = *t;
  }
  size_t have = ws.defined() ? (size_t)ws.numel() * ws.element_size() : 0;
  if (have < need) {
    ws = at::zeros({(int64_t)need}, idx->options().dtype(at::kByte));      // must start zero-filled
    have = need;
  }
  void* word;
  if (!address_of(a[9], "status_word", &word)) return nullptr;
  void* scratch = ws.defined() ? ws.data_ptr() : nullptr;
  const lcd_status st = without_gil([&] {
    const float* s = static_cast<const float*>(scale->data_ptr());
    float* out = static_cast<float*>(y.data_ptr());
    int32_t* flag = static_cast<int32_t*>(word);
    return idx->scalar_type() == at::kChar
               ? lcd_lut_linear_act8(w->data_ptr(), header, static_cast<const int8_t*>(idx->data_ptr()), s, M, out, y.stride(0),
                                     (lcd_algo)algo, scratch, have, flag, stream.raw())
               : lcd_lut_linear(w->data_ptr(), header, static_cast<const uint8_t*>(idx->data_ptr()), s, M, out, y.stride(0),
                                (lcd_algo)algo, scratch, have, flag, stream.raw());
  });
  if (st != LCD_OK) return PyLong_FromLong((long)st);
  return a[6] == Py_None ? stream.output(y) : Py_NewRef(a[6]);
  END_HANDLE_TH_ERRORS
}

// (problem array address, count, act_bits, stream) -> status
PyObject* act_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (!count_args(n, 4)) return nullptr;
  void* arr = PyLong_AsVoidPtr(a[0]);
  const int count = (int)PyLong_AsLong(a[1]), bits = (int)PyLong_AsLong(a[2]);
  if (PyErr_Occurred()) return nullptr;
  const CallStream stream(a[3]);
  if (!stream.ok()) return nullptr;
  return PyLong_FromLong((long)without_gil(
      [&] { return lcd_smooth_quantize_act_batch(static_cast<const lcd_act_problem*>(arr), count, bits, stream.raw()); }));
  END_HANDLE_TH_ERRORS
}

// (form, problem array address, count, algo, workspace, status_word, stream) -> status; form 0: fused, 1: stored 4-bit levels,
// 2: stored 8-bit levels
PyObject* linear_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (!count_args(n, 7)) return nullptr;
  const long form = PyLong_AsLong(a[0]);
  void *arr = PyLong_AsVoidPtr(a[1]), *word;
  const int count = (int)PyLong_AsLong(a[2]);
  const lcd_algo algo = (lcd_algo)PyLong_AsLong(a[3]);
  if (PyErr_Occurred()) return nullptr;
  const at::Tensor* ws = tensor_of(a[4], "workspace");
  if (!ws || !address_of(a[5], "status_word", &word)) return nullptr;
  const CallStream stream(a[6]);
  if (!stream.ok()) return nullptr;
  void* scratch = ws->data_ptr();
  const size_t bytes = (size_t)ws->numel();
  return PyLong_FromLong((long)without_gil([&] {
    int32_t* flag = static_cast<int32_t*>(word);
    if (form == 0) return lcd_linear_fused_batch(static_cast<const lcd_fused_problem*>(arr), count, algo, scratch, bytes, flag, stream.raw());
    const lcd_linear_problem* p = static_cast<const lcd_linear_problem*>(arr);
    return form == 1 ? lcd_lut_linear_batch(p, count, algo, scratch, bytes, flag, stream.raw())
                     : lcd_lut_linear_batch_act8(p, count, algo, scratch, bytes, flag, stream.raw());
  }));
  END_HANDLE_TH_ERRORS
}

// (idx, codebook, delta_w, new_idx, delta_c, counts, stream) -> (new_idx, delta_c, counts) or a status
PyObject* reclassify(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (!count_args(n, 7)) return nullptr;
  const at::Tensor *idx = tensor_of(a[0], "idx"), *cb = idx ? tensor_of(a[1], "codebook") : nullptr;
  const at::Tensor* dw = cb ? tensor_of(a[2], "delta_w") : nullptr;
  if (!dw || !require(idx->scalar_type() == at::kByte && cb->scalar_type() == at::kHalf && dw->scalar_type() == at::kFloat,
                      "idx uint8, codebook fp16, delta_w fp32") ||
      !require(idx->dim() == 2 && cb->dim() == 2 && dw->dim() == 2 && idx->is_contiguous() && cb->is_contiguous() &&
                   dw->stride(1) == 1, "contiguous [N, K], [N, C] and rows of delta_w"))
    return nullptr;
  const int64_t N = idx->size(0), K = idx->size(1), C = cb->size(1);
  const CallStream stream(a[6]);
  if (!stream.ok()) return nullptr;
  at::Tensor out[3];
  if (a[3] == Py_None) {
    out[0] = at::empty_like(*idx);
    out[1] = at::empty({N, C}, idx->options().dtype(at::kDouble));
    out[2] = at::empty({N, C}, idx->options().dtype(at::kInt));
  } else {
    for (int i = 0; i < 3; ++i) {
      const at::Tensor* t = tensor_of(a[3 + i], "out");
      if (!t) return nullptr;
      out[i] = *t;
    }
    if (!require(out[0].scalar_type() == at::kByte && out[1].scalar_type() == at::kDouble && out[2].scalar_type() == at::kInt,
                 "out: uint8, fp64, int32") ||
        !require(out[0].sizes() == idx->sizes() && out[1].sizes() == cb->sizes() && out[2].sizes() == cb->sizes(),
                 "out: [N, K], [N, C], [N, C]"))
      return nullptr;
  }
  const lcd_status st = without_gil([&] {
    return lcd_reclassify(static_cast<const uint8_t*>(idx->data_ptr()), static_cast<const uint16_t*>(cb->data_ptr()),
                          static_cast<const float*>(dw->data_ptr()), N, K, dw->stride(0), (int)C,
                          static_cast<uint8_t*>(out[0].data_ptr()), static_cast<double*>(out[1].data_ptr()),
                          static_cast<int32_t*>(out[2].data_ptr()), stream.raw());
  });
  if (st != LCD_OK) return PyLong_FromLong((long)st);
  if (a[3] != Py_None) return PyTuple_Pack(3, a[3], a[4], a[5]);
  PyObject* r = PyTuple_New(3);
  for (int i = 0; r && i < 3; ++i) {
    PyObject* o = stream.output(out[i]);
    if (!o) Py_CLEAR(r);
    else PyTuple_SET_ITEM(r, i, o);
  }
  return r;
  END_HANDLE_TH_ERRORS
}

// (x, wmax, alphas, stream) -> (best, mse, inv_smooth) or a status
PyObject* smoothing_search(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (!count_args(n, 4)) return nullptr;
  const at::Tensor *x = tensor_of(a[0], "x"), *wmax = x ? tensor_of(a[1], "wmax") : nullptr;
  if (!wmax || !require(x->is_cuda() && x->scalar_type() == at::kHalf && x->dim() == 2 && x->stride(1) == 1,
                        "x: CUDA fp16 [T, K] with unit column stride"))
    return nullptr;
  PyObject* list = PySequence_Fast(a[2], "alphas: a sequence of floats");
  if (!list) return nullptr;
  std::vector<float> alphas((size_t)PySequence_Fast_GET_SIZE(list));
  for (size_t i = 0; i < alphas.size(); ++i) alphas[i] = (float)PyFloat_AsDouble(PySequence_Fast_GET_ITEM(list, (Py_ssize_t)i));
  Py_DECREF(list);
  if (PyErr_Occurred()) return nullptr;
  const int64_t T = x->size(0), K = x->size(1);
  const int G = (int)alphas.size();
  size_t need = 0;
  const lcd_status sized = lcd_smoothing_search_workspace_bytes(T, K, G, &need);
  if (sized != LCD_OK) return PyLong_FromLong((long)sized);
  const CallStream stream(a[3]);
  if (!stream.ok()) return nullptr;
  const at::Tensor ws = at::empty({(int64_t)need}, x->options().dtype(at::kByte));
  const at::Tensor mse = at::empty({G}, x->options().dtype(at::kDouble)), best = at::empty({1}, x->options().dtype(at::kInt)),
                   inv = at::empty({K}, x->options().dtype(at::kFloat));
  const lcd_status st = without_gil([&] {
    return lcd_smoothing_search(x->data_ptr(), T, K, x->stride(0), static_cast<const float*>(wmax->data_ptr()), alphas.data(), G,
                                ws.data_ptr(), need, static_cast<double*>(mse.data_ptr()), static_cast<int32_t*>(best.data_ptr()),
                                static_cast<float*>(inv.data_ptr()), stream.raw());
  });
  if (st != LCD_OK) return PyLong_FromLong((long)st);
  PyObject *o0 = stream.output(best), *o1 = stream.output(mse), *o2 = stream.output(inv);
  PyObject* out = o0 && o1 && o2 ? PyTuple_Pack(3, o0, o1, o2) : nullptr;
  Py_XDECREF(o0);
  Py_XDECREF(o1);
  Py_XDECREF(o2);
  return out;
  END_HANDLE_TH_ERRORS
}

PyMethodDef kMethods[] = {
    {"smooth_quantize_act", reinterpret_cast<PyCFunction>(smooth_quantize_act), METH_FASTCALL, nullptr},
    {"lut_linear", reinterpret_cast<PyCFunction>(lut_linear), METH_FASTCALL, nullptr},
    {"act_batch", reinterpret_cast<PyCFunction>(act_batch), METH_FASTCALL, nullptr},
    {"linear_batch", reinterpret_cast<PyCFunction>(linear_batch), METH_FASTCALL, nullptr},
    {"reclassify", reinterpret_cast<PyCFunction>(reclassify), METH_FASTCALL, nullptr},
    {"smoothing_search", reinterpret_cast<PyCFunction>(smoothing_search), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_host_calls", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host_calls() { return PyModule_Create(&kModule); }
