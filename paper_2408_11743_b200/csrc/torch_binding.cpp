// The per-call part of the Python binding, natively: argument checks, the output tensor, the current stream and the one
// call into libmarlin_b200.  A decode call on a small layer takes 5 us on the GPU; the same steps in Python took 12 us
// (torch.cuda.current_stream() 3.3 us, torch.empty 2.4 us, the ctypes call 1.1 us beside the 2.5 us of the launch
// itself), so that a loop over such layers waited for the host.
//
// A plain CPython extension module: tensors are unpacked with torch's own C++ API, outputs come from its caching
// allocator.  It links to nothing of this library; bind() hands it the addresses of the entry points that the ctypes
// binding has loaded, and what to call to raise MarlinError.
#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>
#include <cstdint>

namespace {

typedef int (*GemmFn)(const void*, const void*, const void*, void*, int, int, int, int, void*, size_t, void*);
typedef int (*GemmExtraFn)(const void*, const void*, const void*, const void*, void*, int, int, int, int, void*, size_t,
                           void*);
typedef int (*MlpFn)(const void*, const void*, const void*, const void*, const void*, void*, void*, int, int, int, int,
                     int, void*, size_t, void*);
typedef size_t (*SizeFn)(int, int, int);
typedef size_t (*SizeFn2)(int, int);

// the kinds of product, in the order of kNames
enum Kind { kDense, kSparse, kZero, kW8, kSwiglu, kKinds };
const char* const kNames[kKinds] = {"marlin_gemm", "marlin_gemm_sparse24", "marlin_gemm_zp", "marlin_gemm_w8",
                                    "marlin_gemm_swiglu"};
void* g_fn[kKinds];
MlpFn g_mlp;
SizeFn g_weight_bytes, g_scale_bytes;
SizeFn2 g_meta_bytes, g_weight_bytes_w8;
PyObject* g_raise;  // raise(status, what)

// an argument as the int that the library takes; false with a Python error set (a size beyond it is no other size)
bool integer(PyObject* o, const char* name, int* out) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) return false;
  if (v < INT_MIN || v > INT_MAX) {
    PyErr_Format(PyExc_ValueError, "%s is out of range", name);
    return false;
  }
  *out = (int)v;
  return true;
}

// nullptr with a Python error set, or the tensor
const at::Tensor* tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s must be a CUDA tensor", name);
    return nullptr;
  }
  return &THPVariable_Unpack(o);
}
const at::Tensor* device_tensor(PyObject* o, at::ScalarType type, const char* name) {
  const at::Tensor* t = tensor(o, name);
  if (!t) return nullptr;
  if (!t->is_cuda()) {
    PyErr_Format(PyExc_TypeError, "%s must be a CUDA tensor", name);
    return nullptr;
  }
  if (t->scalar_type() != type) {
    PyErr_Format(PyExc_TypeError, "%s must have dtype %s", name, type == at::kHalf ? "torch.float16" : "torch.uint8");
    return nullptr;
  }
  if (!t->is_contiguous()) {
    PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
    return nullptr;
  }
  return t;
}
const at::Tensor* activations(PyObject* o, int64_t K) {
  const at::Tensor* t = device_tensor(o, at::kHalf, "A");
  if (t && (t->dim() != 2 || t->size(1) != K)) {
    PyErr_SetString(PyExc_ValueError, "A must be [M, K]");
    return nullptr;
  }
  return t;
}
// `given` (or None: a new tensor from torch's allocator) as fp16 [M][N]; false with a Python error set
bool output(PyObject* given, int64_t M, int64_t N, const at::Device& device, const char* name, at::Tensor* out) {
  if (given == Py_None) {
    *out = at::detail::empty_cuda({M, N}, at::kHalf, device, std::nullopt);
    return true;
  }
  const at::Tensor* t = device_tensor(given, at::kHalf, name);
  if (!t) return false;
  if (t->dim() != 2 || t->size(0) != M || t->size(1) != N) {
    PyErr_Format(PyExc_ValueError, "%s must be [%lld, %lld]", name, (long long)M, (long long)N);
    return false;
  }
  *out = *t;
  return true;
}
// the handle of `stream` (an object with cuda_stream), of the current stream where it is None
bool stream_handle(PyObject* stream, void** handle) {
  if (stream == Py_None) {
    *handle = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  PyObject* h = PyObject_GetAttrString(stream, "cuda_stream");
  if (!h) return false;
  *handle = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  return !PyErr_Occurred();
}
PyObject* finish(int status, const char* what, PyObject* given, at::Tensor&& out) {
  if (status != 0) {
    PyObject* r = PyObject_CallFunction(g_raise, "is", status, what);
    Py_XDECREF(r);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, what);
    return nullptr;
  }
  if (given != Py_None) {
    Py_INCREF(given);
    return given;
  }
  return THPVariable_Wrap(std::move(out));
}

int launch(int kind, const void* A, const void* w, const void* s, const void* x, void* C, int M, int K, int N, int G,
           void* ws, size_t ws_bytes, void* stream) {
  int st;
  Py_BEGIN_ALLOW_THREADS
  if (kind == kSparse)
    st = reinterpret_cast<GemmExtraFn>(g_fn[kind])(A, w, x, s, C, M, K, N, G, ws, ws_bytes, stream);
  else if (kind == kZero)
    st = reinterpret_cast<GemmExtraFn>(g_fn[kind])(A, w, s, x, C, M, K, N, G, ws, ws_bytes, stream);
  else
    st = reinterpret_cast<GemmFn>(g_fn[kind])(A, w, s, C, M, K, N, G, ws, ws_bytes, stream);
  Py_END_ALLOW_THREADS
  return st;
}

bool count_is(Py_ssize_t nargs, Py_ssize_t want) {
  if (nargs == want) return true;
  PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, nargs);
  return false;
}

// C++ exceptions of torch (out of memory, a bad device) become Python errors
#define TRY try {
#define CATCH                                      \
  }                                                \
  catch (const std::exception& e) {                \
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what()); \
    return nullptr;                                \
  }

// ---- one packed layer whose buffers were checked when it was built --------------------------------------------
struct LayerCall {
  PyObject_HEAD
  vectorcallfunc vectorcall;
  int kind, K, N, G, device;
  void *w, *s, *x, *ws;
  size_t ws_bytes;
};

PyObject* layer_call(PyObject* self, PyObject* const* args, size_t nargsf, PyObject* kwnames) {
  TRY
  const LayerCall* L = reinterpret_cast<LayerCall*>(self);
  if (kwnames && PyTuple_GET_SIZE(kwnames) != 0) {
    PyErr_SetString(PyExc_TypeError, "positional arguments only");
    return nullptr;
  }
  if (!count_is(PyVectorcall_NARGS(nargsf), 3)) return nullptr;
  const at::Tensor* A = tensor(args[0], "A");
  if (!A) return nullptr;
  if (A->scalar_type() != at::kHalf || !A->is_cuda() || !A->is_contiguous() || A->dim() != 2 || A->size(1) != L->K) {
    PyErr_SetString(PyExc_ValueError, "A must be a contiguous fp16 CUDA tensor [M, K]");
    return nullptr;
  }
  const int64_t M = A->size(0);
  at::Tensor out;
  if (args[1] == Py_None) {
    out = at::detail::empty_cuda({M, L->N}, at::kHalf, at::Device(at::kCUDA, (c10::DeviceIndex)L->device), std::nullopt);
  } else {
    const at::Tensor* o = tensor(args[1], "out");
    if (!o) return nullptr;
    if (o->scalar_type() != at::kHalf || !o->is_cuda() || !o->is_contiguous() || o->dim() != 2 || o->size(0) != M ||
        o->size(1) != L->N) {
      PyErr_SetString(PyExc_ValueError, "out must be a contiguous fp16 CUDA tensor [M, N]");
      return nullptr;
    }
    out = *o;
  }
  void* stream;
  if (!stream_handle(args[2], &stream)) return nullptr;
  const int st = launch(L->kind, A->data_ptr(), L->w, L->s, L->x, out.data_ptr(), (int)M, L->K, L->N, L->G, L->ws,
                        L->ws_bytes, stream);
  return finish(st, kNames[L->kind], args[1], std::move(out));
  CATCH
}

PyTypeObject LayerCallType = {PyVarObject_HEAD_INIT(nullptr, 0)};

// layer_call(kind, K, N, G, w, s, x, ws, ws_bytes, device): pointers as integers; the caller keeps the tensors alive
PyObject* make_layer_call(PyObject*, PyObject* args) {
  int kind, K, N, G, device;
  unsigned long long w, s, x, ws, ws_bytes;
  if (!PyArg_ParseTuple(args, "iiiiKKKKKi", &kind, &K, &N, &G, &w, &s, &x, &ws, &ws_bytes, &device)) return nullptr;
  if (kind < 0 || kind >= kKinds) {
    PyErr_SetString(PyExc_ValueError, "kind");
    return nullptr;
  }
  LayerCall* L = PyObject_New(LayerCall, &LayerCallType);
  if (!L) return nullptr;
  L->vectorcall = layer_call;
  L->kind = kind; L->K = K; L->N = N; L->G = G; L->device = device;
  L->w = reinterpret_cast<void*>(w); L->s = reinterpret_cast<void*>(s); L->x = reinterpret_cast<void*>(x);
  L->ws = reinterpret_cast<void*>(ws); L->ws_bytes = (size_t)ws_bytes;
  return reinterpret_cast<PyObject*>(L);
}

// ---- the module-level functions ---------------------------------------------------------------------------------
// gemm(kind, A, w_packed, s_packed, metadata, zero points or None, K, N, G, workspace, out or None, stream or None)
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  TRY
  if (!count_is(nargs, 11)) return nullptr;
  int kind, K, N, G;
  if (!integer(a[0], "kind", &kind) || !integer(a[5], "K", &K) || !integer(a[6], "N", &N) || !integer(a[7], "group_size", &G))
    return nullptr;
  const at::Tensor* A = activations(a[1], K);
  if (!A) return nullptr;
  const at::Tensor* w = device_tensor(a[2], at::kByte, "w_packed");
  if (!w) return nullptr;
  const at::Tensor* s = device_tensor(a[3], at::kByte, "s_packed");
  if (!s) return nullptr;
  const at::Tensor* x = nullptr;
  if ((kind == kSparse || kind == kZero) && !(x = device_tensor(a[4], at::kByte, kind == kSparse ? "meta_packed" : "z_packed")))
    return nullptr;
  const at::Tensor* ws = device_tensor(a[8], at::kByte, "workspace");
  if (!ws) return nullptr;
  const size_t wb = kind == kW8 ? g_weight_bytes_w8(K, N) : g_weight_bytes(K, N, kind == kSparse ? 1 : 0);
  const size_t sb = g_scale_bytes(K, N, G);
  const size_t xb = kind == kSparse ? g_meta_bytes(K, N) : sb;
  if ((size_t)w->numel() != wb || (size_t)s->numel() != sb || (x && (size_t)x->numel() != xb)) {
    PyErr_SetString(PyExc_ValueError, "packed buffer sizes do not match K, N, group_size");
    return nullptr;
  }
  const int64_t M = A->size(0);
  at::Tensor out;
  if (!output(a[9], M, kind == kSwiglu ? N / 2 : N, A->device(), "out", &out)) return nullptr;
  void* stream;
  if (!stream_handle(a[10], &stream)) return nullptr;
  const int st = launch(kind, A->data_ptr(), w->data_ptr(), s->data_ptr(), x ? x->data_ptr() : nullptr, out.data_ptr(),
                        (int)M, K, N, G, ws->data_ptr(), (size_t)ws->numel(), stream);
  return finish(st, kNames[kind], a[9], std::move(out));
  CATCH
}

// mlp(A, w_gate_up, s_gate_up, w_down, s_down, K, I, N, G, workspace, H or None, out or None, stream or None)
PyObject* mlp(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  TRY
  if (!count_is(nargs, 13)) return nullptr;
  int K, I, N, G;
  if (!integer(a[5], "K", &K) || !integer(a[6], "I", &I) || !integer(a[7], "N", &N) || !integer(a[8], "group_size", &G))
    return nullptr;
  const at::Tensor* A = activations(a[0], K);
  if (!A) return nullptr;
  const at::Tensor* ws = device_tensor(a[9], at::kByte, "workspace");
  if (!ws) return nullptr;
  static const char* const names[4] = {"w_gate_up", "s_gate_up", "w_down", "s_down"};
  const at::Tensor* t[4];
  for (int i = 0; i < 4; ++i)
    if (!(t[i] = device_tensor(a[1 + i], at::kByte, names[i]))) return nullptr;
  if ((size_t)t[0]->numel() != g_weight_bytes(K, 2 * I, 0) || (size_t)t[1]->numel() != g_scale_bytes(K, 2 * I, G) ||
      (size_t)t[2]->numel() != g_weight_bytes(I, N, 0) || (size_t)t[3]->numel() != g_scale_bytes(I, N, G)) {
    PyErr_SetString(PyExc_ValueError, "packed buffer sizes do not match K, I, N, group_size");
    return nullptr;
  }
  const int64_t M = A->size(0);
  at::Tensor H, out;
  if (!output(a[10], M, I, A->device(), "H", &H) || !output(a[11], M, N, A->device(), "out", &out)) return nullptr;
  void* stream;
  if (!stream_handle(a[12], &stream)) return nullptr;
  int st;
  const void *pa = A->data_ptr(), *p0 = t[0]->data_ptr(), *p1 = t[1]->data_ptr(), *p2 = t[2]->data_ptr(), *p3 = t[3]->data_ptr();
  void *ph = H.data_ptr(), *po = out.data_ptr(), *pw = ws->data_ptr();
  const size_t wsb = (size_t)ws->numel();
  Py_BEGIN_ALLOW_THREADS
  st = g_mlp(pa, p0, p1, p2, p3, ph, po, (int)M, K, I, N, G, pw, wsb, stream);
  Py_END_ALLOW_THREADS
  return finish(st, "marlin_mlp_swiglu", a[11], std::move(out));
  CATCH
}

// bind(addresses, raise): addresses of the library's entry points by name
PyObject* bind(PyObject*, PyObject* args) {
  PyObject *table, *raise;
  if (!PyArg_ParseTuple(args, "O!O", &PyDict_Type, &table, &raise)) return nullptr;
  bool ok = true;
  auto address = [&](const char* name) -> void* {
    PyObject* v = PyDict_GetItemString(table, name);
    void* p = v ? PyLong_AsVoidPtr(v) : nullptr;
    if (!p) ok = false;
    return p;
  };
  for (int k = 0; k < kKinds; ++k) g_fn[k] = address(kNames[k]);
  g_mlp = reinterpret_cast<MlpFn>(address("marlin_mlp_swiglu"));
  g_weight_bytes = reinterpret_cast<SizeFn>(address("marlin_packed_weight_bytes"));
  g_scale_bytes = reinterpret_cast<SizeFn>(address("marlin_packed_scale_bytes"));
  g_meta_bytes = reinterpret_cast<SizeFn2>(address("marlin_packed_meta_bytes"));
  g_weight_bytes_w8 = reinterpret_cast<SizeFn2>(address("marlin_packed_weight_bytes_w8"));
  if (!ok) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_KeyError, "an entry point is missing");
    return nullptr;
  }
  Py_INCREF(raise);
  Py_XDECREF(g_raise);
  g_raise = raise;
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, nullptr},
    {"layer_call", make_layer_call, METH_VARARGS, nullptr},
    {"gemm", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(gemm)), METH_FASTCALL, nullptr},
    {"mlp", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(mlp)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_torch_binding", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__torch_binding(void) {
  LayerCallType.tp_name = "_torch_binding.LayerCall";
  LayerCallType.tp_basicsize = sizeof(LayerCall);
  LayerCallType.tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL;
  LayerCallType.tp_vectorcall_offset = offsetof(LayerCall, vectorcall);
  LayerCallType.tp_call = PyVectorcall_Call;
  if (PyType_Ready(&LayerCallType) < 0) return nullptr;
  return PyModule_Create(&module);
}
