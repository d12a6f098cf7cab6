// Native marshalling of the calls a program makes once per layer and step (binding.py): reads the
// descriptor, checks the tensors, allocates the output and calls the C entry point with the
// interpreter lock released.  Through ctypes a call of one linear spent more time in Python than its
// kernel on the GPU.  Every function takes its arguments by position, in the order
// binding.py passes them, and keeps nothing from one call for the next.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <vector>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "peqa.h"

namespace {

PyObject* g_error = nullptr;                       // binding.PeqaError
PyObject *s_bits, *s_N, *s_K, *s_group, *s_qweight, *s_zeros, *s_scales;
PyObject *s_w, *s_X, *s_dY, *s_Y, *s_dX, *s_dS, *s_m, *s_v, *s_workspace;

// A Python error is set; unwinds to the function's END_HANDLE_TH_ERRORS.
[[noreturn]] void fail() { throw python_error(); }

struct Ref {                                       // owned reference
  PyObject* p;
  explicit Ref(PyObject* o) : p(o) {
    if (!p) fail();
  }
  Ref(const Ref&) = delete;
  Ref& operator=(const Ref&) = delete;
  ~Ref() { Py_DECREF(p); }
};

const at::Tensor& tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_AttributeError, "%s: expected a tensor, got %.200s", name, Py_TYPE(o)->tp_name);
    fail();
  }
  return THPVariable_Unpack(o);
}

// A contiguous CUDA tensor of this type.
const at::Tensor& dev(PyObject* o, at::ScalarType dtype, const char* name) {
  const at::Tensor& t = tensor(o, name);
  if (!t.is_cuda() || t.scalar_type() != dtype || !t.is_contiguous()) {
    const char* type = dtype == at::kBFloat16 ? "bfloat16" : dtype == at::kFloat ? "float32" : "int32";
    PyErr_Format(PyExc_ValueError, "%s: expected a contiguous CUDA tensor of torch.%s", name, type);
    fail();
  }
  return t;
}

void* ptr_or_null(PyObject* o, const char* name) { return o == Py_None ? nullptr : tensor(o, name).data_ptr(); }

// Whole numbers as ctypes takes them: whatever has __index__, modulo the width.
long long as_long(PyObject* o) {
  const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
  if (v == ~0ull && PyErr_Occurred()) fail();
  return (long long)v;
}
int as_int(PyObject* o) { return (int)as_long(o); }
float as_float(PyObject* o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) fail();
  return (float)v;
}
int attr_int(PyObject* o, PyObject* name) { return as_int(Ref(PyObject_GetAttr(o, name)).p); }
void* attr_ptr(PyObject* o, PyObject* name) {
  Ref t(PyObject_GetAttr(o, name));
  return tensor(t.p, PyUnicode_AsUTF8(name)).data_ptr();
}

peqa_qweight_t weight(PyObject* o) {
  peqa_qweight_t w;
  w.bits = attr_int(o, s_bits);
  w.out_features = attr_int(o, s_N);
  w.in_features = attr_int(o, s_K);
  w.group_size = attr_int(o, s_group);
  w.qweight = static_cast<const uint32_t*>(attr_ptr(o, s_qweight));
  w.zeros = static_cast<const uint8_t*>(attr_ptr(o, s_zeros));
  w.scales = static_cast<const float*>(attr_ptr(o, s_scales));
  return w;
}

struct Workspace {
  void* p = nullptr;
  size_t bytes = 0;
  explicit Workspace(PyObject* o) {
    if (o == Py_None) return;
    const at::Tensor& t = tensor(o, "workspace");
    p = t.data_ptr();
    bytes = (size_t)t.numel() * t.element_size();
  }
};

void* stream() { return static_cast<void*>(c10::cuda::getCurrentCUDAStream().stream()); }

void check(int status, const char* where) {
  if (status == PEQA_OK) return;
  if (!g_error) {
    PyErr_Format(PyExc_RuntimeError, "%s: status %d", where, status);
    fail();
  }
  Ref e(PyObject_CallFunction(g_error, "is", status, where));
  PyErr_SetObject(reinterpret_cast<PyObject*>(Py_TYPE(e.p)), e.p);
  fail();
}

void arity(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return;
  PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  fail();
}

// The output: the caller's, or a new tensor beside `like` (of its class, if that is not torch's own).
PyObject* output(PyObject* given, PyObject* like, int64_t rows, int64_t cols, void** data) {
  if (given != Py_None) {
    *data = tensor(given, "Y").data_ptr();
    Py_INCREF(given);
    return given;
  }
  if (!THPVariable_CheckExact(like)) {
    PyObject* made = PyObject_CallMethod(like, "new_empty", "((LL))", (long long)rows, (long long)cols);
    if (!made) fail();
    if (!THPVariable_Check(made)) {
      Py_DECREF(made);
      PyErr_SetString(PyExc_TypeError, "new_empty did not return a tensor");
      fail();
    }
    *data = THPVariable_Unpack(made).data_ptr();
    return made;
  }
  at::Tensor t = THPVariable_Unpack(like).new_empty({rows, cols});
  *data = t.data_ptr();
  return THPVariable_Wrap(std::move(t));
}

template <typename F>
int unlocked(F&& call) {
  PyThreadState* save = PyEval_SaveThread();
  const int rc = call();
  PyEval_RestoreThread(save);
  return rc;
}

PyObject* bind_error(PyObject*, PyObject* cls) {
  Py_INCREF(cls);
  Py_XSETREF(g_error, cls);
  Py_RETURN_NONE;
}

// (w, X, Y, workspace) -> Y
PyObject* qlinear_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  arity(n, 4);
  const at::Tensor& X = dev(a[1], at::kBFloat16, "X");
  const int64_t T = X.size(0);
  const peqa_qweight_t w = weight(a[0]);
  void* y;
  Ref Y(output(a[2], a[1], T, w.out_features, &y));
  const Workspace ws(a[3]);
  void *x = X.data_ptr(), *st = stream();
  check(unlocked([&] { return peqa_qlinear_fwd(&w, x, (int)T, y, ws.p, ws.bytes, st); }), "peqa_qlinear_fwd");
  Py_INCREF(Y.p);
  return Y.p;
  END_HANDLE_TH_ERRORS
}

// (w, zeros_f, X, Y) -> Y
PyObject* qlinear_fwd_zf(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  arity(n, 4);
  const float* zf = static_cast<const float*>(dev(a[1], at::kFloat, "zeros_f").data_ptr());
  const at::Tensor& X = dev(a[2], at::kBFloat16, "X");
  const int64_t T = X.size(0);
  const peqa_qweight_t w = weight(a[0]);
  void* y;
  Ref Y(output(a[3], a[2], T, w.out_features, &y));
  void *x = X.data_ptr(), *st = stream();
  check(unlocked([&] { return peqa_qlinear_fwd_zf(&w, zf, x, (int)T, y, st); }), "peqa_qlinear_fwd_zf");
  Py_INCREF(Y.p);
  return Y.p;
  END_HANDLE_TH_ERRORS
}

// (w, X, Y, workspace) -> Y
PyObject* qlinear_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  arity(n, 4);
  const at::Tensor& X = dev(a[1], at::kBFloat16, "X");
  const int64_t M = X.size(0);
  const peqa_qweight_t w = weight(a[0]);
  void* y;
  Ref Y(output(a[2], a[1], M, w.out_features, &y));
  void *x = X.data_ptr(), *st = stream();
  const Workspace given(a[3]);
  at::Tensor own;
  void* wp = given.p;
  size_t wb = given.bytes;
  if (a[3] == Py_None) {
    wb = peqa_workspace_bytes(PEQA_OP_DECODE, (int)M, &w);
    if (wb > 0) {
      own = at::empty({(int64_t)wb}, X.options().dtype(at::kByte));
      wp = own.data_ptr();
    }
  }
  check(unlocked([&] { return peqa_qlinear_decode(&w, x, (int)M, y, wp, wb, st); }), "peqa_qlinear_decode");
  Py_INCREF(Y.p);
  return Y.p;
  END_HANDLE_TH_ERRORS
}

// (w, prepared, X, Y, scale_table, task_ids) -> Y
PyObject* qlinear_decode_prepared(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  arity(n, 6);
  const uint32_t* prepared = static_cast<const uint32_t*>(dev(a[1], at::kInt, "prepared").data_ptr());
  const at::Tensor& X = dev(a[2], at::kBFloat16, "X");
  const int64_t M = X.size(0);
  const peqa_qweight_t w = weight(a[0]);
  void* y;
  Ref Y(output(a[3], a[2], M, w.out_features, &y));
  const float* table = nullptr;
  const int32_t* ids = nullptr;
  int n_tasks = 0;
  if (a[5] != Py_None) {
    const at::Tensor& t = dev(a[4], at::kFloat, "scale_table");
    table = static_cast<const float*>(t.data_ptr());
    ids = static_cast<const int32_t*>(dev(a[5], at::kInt, "task_ids").data_ptr());
    n_tasks = (int)t.size(0);
  } else {
    table = static_cast<const float*>(ptr_or_null(a[4], "scale_table"));
  }
  void *x = X.data_ptr(), *st = stream();
  check(unlocked([&] {
          return peqa_qlinear_decode_prepared(&w, prepared, x, (int)M, y, table, n_tasks, ids, st);
        }),
        "peqa_qlinear_decode_prepared");
  Py_INCREF(Y.p);
  return Y.p;
  END_HANDLE_TH_ERRORS
}

// (values, gradient, m, v, lr, beta1, beta2, eps, weight_decay, step), for the scales or the zero-points
template <typename F>
PyObject* adamw(PyObject* const* a, Py_ssize_t n, const char* values, const char* grad, F entry, const char* where) {
  arity(n, 10);
  const at::Tensor& t = dev(a[0], at::kFloat, values);
  float* s = static_cast<float*>(t.data_ptr());
  const int64_t count = t.numel();
  const float* g = static_cast<const float*>(dev(a[1], at::kFloat, grad).data_ptr());
  float* m = static_cast<float*>(dev(a[2], at::kFloat, "m").data_ptr());
  float* v = static_cast<float*>(dev(a[3], at::kFloat, "v").data_ptr());
  float c[5];
  for (int i = 0; i < 5; ++i) c[i] = as_float(a[4 + i]);
  const long long step = as_long(a[9]);
  void* st = stream();
  check(unlocked([&] { return entry(s, g, m, v, count, c[0], c[1], c[2], c[3], c[4], (int64_t)step, st); }), where);
  Py_RETURN_NONE;
}
PyObject* scale_adamw(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  return adamw(a, n, "scales", "dS", peqa_scale_adamw, "peqa_scale_adamw");
  END_HANDLE_TH_ERRORS
}
PyObject* zero_adamw(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  return adamw(a, n, "zeros_f", "dZ", peqa_zero_adamw, "peqa_zero_adamw");
  END_HANDLE_TH_ERRORS
}

// (linears, apply_adamw, lr, beta1, beta2, eps, weight_decay, step)
PyObject* layer_train_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  arity(n, 8);
  if (!PySequence_Check(a[0])) {                   // (an iterator would be used up by one look at it)
    PyErr_SetString(PyExc_TypeError, "linears: expected a sequence of LayerLinear");
    fail();
  }
  Ref seq(PySequence_Fast(a[0], "linears: expected a sequence of LayerLinear"));
  const Py_ssize_t count = PySequence_Fast_GET_SIZE(seq.p);
  if (count == 0) {
    PyErr_SetString(PyExc_IndexError, "linears: at least one linear is needed");
    fail();
  }
  std::vector<peqa_layer_linear_t> L((size_t)count);
  int64_t T = 0;
  for (Py_ssize_t i = 0; i < count; ++i) {
    PyObject* o = PySequence_Fast_GET_ITEM(seq.p, i);
    const Ref X(PyObject_GetAttr(o, s_X)), dY(PyObject_GetAttr(o, s_dY)), Y(PyObject_GetAttr(o, s_Y)),
        dX(PyObject_GetAttr(o, s_dX)), dS(PyObject_GetAttr(o, s_dS)), m(PyObject_GetAttr(o, s_m)),
        v(PyObject_GetAttr(o, s_v)), ws(PyObject_GetAttr(o, s_workspace)), w(PyObject_GetAttr(o, s_w));
    const at::Tensor& tx = dev(X.p, at::kBFloat16, "X");
    const at::Tensor& ty = dev(dY.p, at::kBFloat16, "dY");
    peqa_layer_linear_t& l = L[(size_t)i];
    l.X_bf16 = tx.data_ptr();
    l.dY_bf16 = ty.data_ptr();
    l.Y_bf16 = dev(Y.p, at::kBFloat16, "Y").data_ptr();
    l.dX_bf16 = dev(dX.p, at::kBFloat16, "dX").data_ptr();
    l.dS = static_cast<float*>(dev(dS.p, at::kFloat, "dS").data_ptr());
    if (i == 0) T = ty.size(0);
    if (ty.size(0) != T || tx.size(0) != T) {
      PyErr_SetString(PyExc_ValueError, "all linears of a layer step take the same number of tokens");
      fail();
    }
    l.w = weight(w.p);
    l.m = static_cast<float*>(ptr_or_null(m.p, "m"));
    l.v = static_cast<float*>(ptr_or_null(v.p, "v"));
    const Workspace space(ws.p);
    l.workspace = space.p;
    l.workspace_bytes = space.bytes;
  }
  const int apply = PyObject_IsTrue(a[1]);
  if (apply < 0) fail();
  float c[5];
  for (int i = 0; i < 5; ++i) c[i] = as_float(a[2 + i]);
  const long long step = as_long(a[7]);
  void* st = stream();
  check(unlocked([&] {
          return peqa_layer_train_step(L.data(), (int)count, (int)T, apply, c[0], c[1], c[2], c[3], c[4], (int64_t)step, st);
        }),
        "peqa_layer_train_step");
  Py_RETURN_NONE;
  END_HANDLE_TH_ERRORS
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {FAST(qlinear_fwd),       FAST(qlinear_fwd_zf), FAST(qlinear_decode), FAST(qlinear_decode_prepared),
                          FAST(scale_adamw),       FAST(zero_adamw),     FAST(layer_train_step),
                          {"bind_error", bind_error, METH_O, nullptr},   {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
  const struct {
    PyObject** to;
    const char* text;
  } names[] = {{&s_bits, "bits"}, {&s_N, "N"}, {&s_K, "K"}, {&s_group, "group_size"}, {&s_qweight, "qweight"},
               {&s_zeros, "zeros"}, {&s_scales, "scales"}, {&s_w, "w"}, {&s_X, "X"}, {&s_dY, "dY"}, {&s_Y, "Y"},
               {&s_dX, "dX"}, {&s_dS, "dS"}, {&s_m, "m"}, {&s_v, "v"}, {&s_workspace, "workspace"}};
  for (const auto& e : names)
    if (!(*e.to = PyUnicode_InternFromString(e.text))) return nullptr;
  return PyModule_Create(&kModule);
}
