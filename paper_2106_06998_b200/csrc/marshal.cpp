// The binding's calls on ordinary tensors, in native code: what binding.py does for the same call -- checks of layout and shape, the descriptor, the outputs,
// the scratch buffer, the C ABI's call on the current stream -- without the interpreter.  A training step is three calls of 14 to 25 us through the
// interpreter, of 5 to 12 here (57 -> 26 us of host time a step of 16 volumes of 5 x 19 x 19, whose kernels take 54; the launches are two thirds of the rest).
//
// A function returns None for whatever is not the ordinary case (tensors that are not dense CUDA tensors, subclasses, modes that want to see every call, a
// layout or shape that does not fit, an option that is rarely given): binding.py then goes its own way, which is where every error is raised.
#include <torch/csrc/Device.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAGraphsC10Utils.h>
#include <c10/cuda/CUDAStream.h>

#include <cstring>
#include <vector>

#include "../../include/xconv.h"

namespace {

// Entry points of the library that binding.py has loaded, and its functions that raise for a status and hand out scratch buffers.
struct Library {
  decltype(&xconv_workspace_bytes) workspace_bytes;
  decltype(&xconv_forward) forward;
  decltype(&xconv_sketch) sketch;
  decltype(&xconv_wgrad) wgrad;
  decltype(&xconv_dgrad) dgrad;
  decltype(&xconv_sketch_seeded) sketch_seeded;
  decltype(&xconv_wgrad_seeded) wgrad_seeded;
  decltype(&xconv_backprobe) backprobe;
  decltype(&xconv_contract) contract;
} lib{};
PyObject *raise_for_status = nullptr, *workspace = nullptr;

bool watched() {      // modes that are to see the tensor functions of the Python path
  return at::impl::PythonTorchFunctionTLS::stack_len() > 0 || c10::impl::TorchDispatchModeTLS::any_modes_set();
}

// The tensor in `o` if it is an ordinary dense CUDA tensor.
const at::Tensor* plain(PyObject* o) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided) return nullptr;
  using K = c10::DispatchKey;
  const c10::DispatchKeySet keys = t.key_set();
  for (K k : {K::Python, K::PythonTLSSnapshot, K::FuncTorchBatched, K::FuncTorchGradWrapper, K::Functionalize, K::Batched, K::ZeroTensor, K::Conjugate, K::Negative,
              K::Named, K::Fake})
    if (keys.has(k)) return nullptr;
  return &t;
}

int dtype_code(const at::Tensor& t) {
  switch (t.scalar_type()) {
    case at::kFloat: return XCONV_F32;
    case at::kBFloat16: return XCONV_BF16;
    case at::kHalf: return XCONV_F16;
    default: return -1;
  }
}

// A 4-d tensor in channels_last or a 5-d one in channels_last_3d.
struct Image {
  const at::Tensor* t = nullptr;
  int dim = 0, dtype = -1;
  int32_t n = 0, c = 0, D = 1, H = 0, W = 0;
  explicit Image(PyObject* o) {
    const at::Tensor* x = plain(o);
    if (!x) return;
    dim = (int)x->dim();
    if (dim != 4 && dim != 5) return;
    if (!x->is_contiguous(dim == 4 ? at::MemoryFormat::ChannelsLast : at::MemoryFormat::ChannelsLast3d)) return;
    dtype = dtype_code(*x);
    if (dtype < 0) return;
    for (int i = 0; i < dim; ++i)
      if (x->size(i) <= 0 || x->size(i) > INT32_MAX) return;
    n = (int32_t)x->size(0); c = (int32_t)x->size(1);
    D = dim == 5 ? (int32_t)x->size(2) : 1;
    H = (int32_t)x->size(dim - 2); W = (int32_t)x->size(dim - 1);
    t = x;
  }
  explicit operator bool() const { return t != nullptr; }
  bool same_plane(const Image& o) const { return dim == o.dim && D == o.D && H == o.H && W == o.W && dtype == o.dtype; }
};

// The [r, B] sketch: a contiguous float matrix.
const at::Tensor* sketch_of(PyObject* o, int32_t B) {
  const at::Tensor* s = plain(o);
  return s && s->dim() == 2 && s->size(1) == B && s->size(0) > 0 && s->size(0) <= INT32_MAX && s->scalar_type() == at::kFloat && s->is_contiguous() ? s : nullptr;
}

bool small_int(PyObject* o, int32_t* v) {
  if (!PyLong_CheckExact(o)) return false;
  int over = 0;
  const long x = PyLong_AsLongAndOverflow(o, &over);
  if (over || x < 1 || x > 64) return false;
  *v = (int32_t)x;
  return true;
}

// A square kernel, as the descriptor has it (which is made from the last extent alone).
bool square(const Image& W) { return W.H == W.W && W.W <= 64 && W.D <= 64; }
// A kernel over planes, for tensors that have planes: the weights of a planar layer are allocated without them.
bool planes_fit(const Image& g, int32_t KD) { return g.dim == 5 || KD == 1; }

xconv_desc descriptor(int32_t B, int32_t Cin, int32_t Cout, const Image& g, int32_t r, int32_t K, int32_t KD, bool circular) {
  xconv_desc d;
  std::memset(&d, 0, sizeof d);
  d.B = B; d.Cin = Cin; d.Cout = Cout; d.H = g.H; d.W = g.W; d.KH = d.KW = K; d.pad_h = d.pad_w = (K - 1) / 2; d.r = r; d.dtype = g.dtype;
  d.circular = circular ? 1 : 0; d.D = g.D; d.KD = KD; d.pad_d = (KD - 1) / 2;
  return d;
}

// Scratch bytes of a layer, remembered by its sizes (the pointers of a descriptor made here are null).
size_t scratch_bytes(const xconv_desc& d, int op) {
  struct Entry { xconv_desc d; int op = -1; size_t bytes; };
  static thread_local Entry table[64];
  uint32_t h = (uint32_t)op * 2654435761u;
  for (int32_t v : {d.B, d.Cin, d.Cout, d.H, d.W, d.KH, d.r, d.dtype, d.D, d.KD, d.circular}) h = (h ^ (uint32_t)v) * 16777619u;
  Entry& e = table[(h >> 20) & 63];
  if (e.op != op || std::memcmp(&e.d, &d, sizeof d) != 0) {
    e.d = d; e.op = op;
    e.bytes = lib.workspace_bytes(&d, op);
  }
  return e.bytes;
}

// binding.workspace's buffer for this thread and stream.  That pool owns it; what is kept here only finds it again without the interpreter, and holds nothing alive.
struct Found { c10::DeviceIndex device; cudaStream_t stream; c10::weak_intrusive_ptr<c10::TensorImpl> buffer; };
thread_local std::vector<Found> found;

at::Tensor scratch(size_t bytes, const at::Tensor& like, cudaStream_t stream) {
  if (stream && c10::cuda::currentStreamCaptureStatusMayInitCtx() != c10::cuda::CaptureStatus::None)      // (the graph's own, as binding.workspace does)
    return at::empty({(int64_t)std::max<size_t>(bytes, 256)}, like.options().dtype(at::kByte).requires_grad(false));
  const c10::DeviceIndex device = like.device().index();
  for (size_t i = 0; i < found.size(); ++i)
    if (found[i].device == device && found[i].stream == stream) {
      auto impl = found[i].buffer.lock();
      if (impl && (size_t)impl->numel() >= bytes) return at::Tensor(std::move(impl));
      found.erase(found.begin() + (long)i);
      break;
    }
  THPObjectPtr where(THPDevice_New(like.device()));
  THPObjectPtr buffer(where ? PyObject_CallFunction(workspace, "nO", (Py_ssize_t)bytes, where.get()) : nullptr);
  if (!buffer) throw python_error();
  TORCH_CHECK(THPVariable_Check(buffer.get()), "workspace() returns a tensor");
  at::Tensor t = THPVariable_Unpack(buffer.get());
  if (found.size() >= 8) found.erase(found.begin());
  found.push_back({device, stream, c10::weak_intrusive_ptr<c10::TensorImpl>(t.getIntrusivePtr())});
  return t;
}

at::Tensor image_like(const Image& g, int64_t n, int64_t c) {
  const auto opt = g.t->options().requires_grad(false);
  return g.dim == 4 ? at::empty({n, c, g.H, g.W}, opt, at::MemoryFormat::ChannelsLast) : at::empty({n, c, g.D, g.H, g.W}, opt, at::MemoryFormat::ChannelsLast3d);
}
at::Tensor weights_like(const Image& g, int64_t Cout, int64_t Cin, int64_t K, int64_t KD) {
  const auto opt = g.t->options().dtype(at::kFloat).requires_grad(false);
  return g.dim == 4 ? at::empty({Cout, Cin, K, K}, opt, at::MemoryFormat::ChannelsLast) : at::empty({Cout, Cin, KD, K, K}, opt, at::MemoryFormat::ChannelsLast3d);
}
at::Tensor matrix_like(const Image& g, int64_t rows, int64_t cols) { return at::empty({rows, cols}, g.t->options().dtype(at::kFloat).requires_grad(false)); }

// The call itself, with scratch memory, without the interpreter's lock; false with a Python error set.
template <class Call>
bool run(const Image& g, const xconv_desc& d, int op, const char* name, Call&& call) {
  const cudaStream_t stream = c10::cuda::getCurrentCUDAStream().stream();
  const at::Tensor ws = scratch(scratch_bytes(d, op), *g.t, stream);
  void* p = ws.data_ptr();
  const size_t bytes = (size_t)ws.numel();
  xconv_status s;
  Py_BEGIN_ALLOW_THREADS
  s = call(&d, p, bytes, (void*)stream);
  Py_END_ALLOW_THREADS
  if (s == XCONV_OK) return true;
  PyObject* r = PyObject_CallFunction(raise_for_status, "is", (int)s, name);
  Py_XDECREF(r);
  if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, name);
  return false;
}

#define XM_BEGIN(N) HANDLE_TH_ERRORS if (nargs != (N) || !lib.forward || watched()) Py_RETURN_NONE;
#define XM_END END_HANDLE_TH_ERRORS

// forward(X, W, Z, circular) -> (Y, S)
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  XM_BEGIN(4)
  const Image X(a[0]), W(a[1]), Z(a[2]);
  if (!X || !W || !Z || !PyBool_Check(a[3])) Py_RETURN_NONE;
  if (!Z.same_plane(X) || Z.c != X.c || W.c != X.c || W.dim != X.dim || W.dtype != X.dtype || !square(W)) Py_RETURN_NONE;
  const xconv_desc d = descriptor(X.n, X.c, W.n, X, Z.n, W.W, W.D, a[3] == Py_True);
  const at::Tensor Y = image_like(X, X.n, W.n), S = matrix_like(X, Z.n, X.n);
  if (!run(X, d, XCONV_OP_FORWARD, "xconv_forward", [&](const xconv_desc* q, void* ws, size_t n, void* st) {
        return lib.forward(q, X.t->data_ptr(), W.t->data_ptr(), Z.t->data_ptr(), Y.data_ptr(), (float*)S.data_ptr(), ws, n, st); }))
    return nullptr;
  return Py_BuildValue("(NN)", THPVariable_Wrap(Y), THPVariable_Wrap(S));
  XM_END
}

// sketch(X, Z) -> S
PyObject* sketch(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  XM_BEGIN(2)
  const Image X(a[0]), Z(a[1]);
  if (!X || !Z || !Z.same_plane(X) || Z.c != X.c) Py_RETURN_NONE;
  const xconv_desc d = descriptor(X.n, X.c, 1, X, Z.n, 3, 1, false);
  const at::Tensor S = matrix_like(X, Z.n, X.n);
  if (!run(X, d, XCONV_OP_SKETCH, "xconv_sketch", [&](const xconv_desc* q, void* ws, size_t n, void* st) {
        return lib.sketch(q, X.t->data_ptr(), Z.t->data_ptr(), (float*)S.data_ptr(), ws, n, st); }))
    return nullptr;
  return THPVariable_Wrap(S);
  XM_END
}

// sketch_seeded(X, seed, r) -> S
PyObject* sketch_seeded(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  XM_BEGIN(3)
  const Image X(a[0]);
  if (!X || !PyLong_CheckExact(a[1]) || !PyLong_CheckExact(a[2])) Py_RETURN_NONE;
  int over = 0;
  const long r = PyLong_AsLongAndOverflow(a[2], &over);
  if (over || r <= 0 || r > INT32_MAX) Py_RETURN_NONE;
  const unsigned long long seed = PyLong_AsUnsignedLongLongMask(a[1]);
  const xconv_desc d = descriptor(X.n, X.c, 1, X, (int32_t)r, 3, 1, false);
  const at::Tensor S = matrix_like(X, r, X.n);
  if (!run(X, d, XCONV_OP_SKETCH_SEEDED, "xconv_sketch_seeded", [&](const xconv_desc* q, void* ws, size_t n, void* st) {
        return lib.sketch_seeded(q, X.t->data_ptr(), seed, (float*)S.data_ptr(), ws, n, st); }))
    return nullptr;
  return THPVariable_Wrap(S);
  XM_END
}

// wgrad(sketch, dY, Z, kernel_size, kernel_depth, circular) -> dW
PyObject* wgrad(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  XM_BEGIN(6)
  const Image Y(a[1]), Z(a[2]);
  int32_t K, KD;
  if (!Y || !Z || !Z.same_plane(Y) || !small_int(a[3], &K) || !small_int(a[4], &KD) || !planes_fit(Y, KD) || !PyBool_Check(a[5])) Py_RETURN_NONE;
  const at::Tensor* S = sketch_of(a[0], Y.n);
  if (!S || S->size(0) != Z.n) Py_RETURN_NONE;
  const xconv_desc d = descriptor(Y.n, Z.c, Y.c, Y, Z.n, K, KD, a[5] == Py_True);
  const at::Tensor dW = weights_like(Y, Y.c, Z.c, K, KD);
  if (!run(Y, d, XCONV_OP_WGRAD, "xconv_wgrad", [&](const xconv_desc* q, void* ws, size_t n, void* st) {
        return lib.wgrad(q, (const float*)S->data_ptr(), Y.t->data_ptr(), Z.t->data_ptr(), (float*)dW.data_ptr(), ws, n, st); }))
    return nullptr;
  return THPVariable_Wrap(dW);
  XM_END
}

// wgrad_seeded(sketch, dY, seed, Cin, kernel_size, kernel_depth, circular) -> dW
PyObject* wgrad_seeded(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  XM_BEGIN(7)
  const Image Y(a[1]);
  int32_t K, KD;
  if (!Y || !PyLong_CheckExact(a[2]) || !PyLong_CheckExact(a[3]) || !small_int(a[4], &K) || !small_int(a[5], &KD) || !planes_fit(Y, KD) || !PyBool_Check(a[6]))
    Py_RETURN_NONE;
  int over = 0;
  const long Cin = PyLong_AsLongAndOverflow(a[3], &over);
  if (over || Cin <= 0 || Cin > INT32_MAX) Py_RETURN_NONE;
  const at::Tensor* S = sketch_of(a[0], Y.n);
  if (!S) Py_RETURN_NONE;
  const unsigned long long seed = PyLong_AsUnsignedLongLongMask(a[2]);
  const xconv_desc d = descriptor(Y.n, (int32_t)Cin, Y.c, Y, (int32_t)S->size(0), K, KD, a[6] == Py_True);
  const at::Tensor dW = weights_like(Y, Y.c, Cin, K, KD);
  if (!run(Y, d, XCONV_OP_WGRAD_SEEDED, "xconv_wgrad_seeded", [&](const xconv_desc* q, void* ws, size_t n, void* st) {
        return lib.wgrad_seeded(q, (const float*)S->data_ptr(), Y.t->data_ptr(), seed, (float*)dW.data_ptr(), ws, n, st); }))
    return nullptr;
  return THPVariable_Wrap(dW);
  XM_END
}

// dgrad(dY, W, circular) -> dX
PyObject* dgrad(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  XM_BEGIN(3)
  const Image Y(a[0]), W(a[1]);
  if (!Y || !W || !PyBool_Check(a[2]) || W.n != Y.c || W.dtype != Y.dtype || W.dim != Y.dim || !square(W)) Py_RETURN_NONE;
  const xconv_desc d = descriptor(Y.n, W.c, Y.c, Y, 1, W.W, W.D, a[2] == Py_True);
  const at::Tensor dX = image_like(Y, Y.n, W.c);
  if (!run(Y, d, XCONV_OP_DGRAD, "xconv_dgrad", [&](const xconv_desc* q, void* ws, size_t n, void* st) {
        return lib.dgrad(q, Y.t->data_ptr(), W.t->data_ptr(), dX.data_ptr(), ws, n, st); }))
    return nullptr;
  return THPVariable_Wrap(dX);
  XM_END
}

// backprobe(sketch, dY) -> L
PyObject* backprobe(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  XM_BEGIN(2)
  const Image Y(a[1]);
  if (!Y) Py_RETURN_NONE;
  const at::Tensor* S = sketch_of(a[0], Y.n);
  if (!S) Py_RETURN_NONE;
  const xconv_desc d = descriptor(Y.n, 1, Y.c, Y, (int32_t)S->size(0), 3, 1, false);
  const at::Tensor L = image_like(Y, S->size(0), Y.c);
  if (!run(Y, d, XCONV_OP_WGRAD, "xconv_backprobe", [&](const xconv_desc* q, void* ws, size_t n, void* st) {
        return lib.backprobe(q, (const float*)S->data_ptr(), Y.t->data_ptr(), L.data_ptr(), ws, n, st); }))
    return nullptr;
  return THPVariable_Wrap(L);
  XM_END
}

// contract(L, Z, kernel_size, kernel_depth, circular) -> dW
PyObject* contract(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  XM_BEGIN(5)
  const Image L(a[0]), Z(a[1]);
  int32_t K, KD;
  if (!L || !Z || !Z.same_plane(L) || Z.n != L.n || !small_int(a[2], &K) || !small_int(a[3], &KD) || !planes_fit(L, KD) || !PyBool_Check(a[4])) Py_RETURN_NONE;
  const xconv_desc d = descriptor(1, Z.c, L.c, L, L.n, K, KD, a[4] == Py_True);
  const at::Tensor dW = weights_like(L, L.c, Z.c, K, KD);
  if (!run(L, d, XCONV_OP_WGRAD, "xconv_contract", [&](const xconv_desc* q, void* ws, size_t n, void* st) {
        return lib.contract(q, L.t->data_ptr(), Z.t->data_ptr(), (float*)dW.data_ptr(), ws, n, st); }))
    return nullptr;
  return THPVariable_Wrap(dW);
  XM_END
}

// use_library(address of each entry point in the order of Library, raise(status, name), workspace(bytes, device))
PyObject* use_library(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  constexpr Py_ssize_t N = sizeof(Library) / sizeof(void*);
  if (nargs != N + 2) { PyErr_SetString(PyExc_TypeError, "use_library takes the entry points and two functions"); return nullptr; }
  void* at[N];
  for (Py_ssize_t i = 0; i < N; ++i) {
    at[i] = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred()) return nullptr;
  }
  std::memcpy(&lib, at, sizeof lib);
  Py_INCREF(a[N]);
  Py_XSETREF(raise_for_status, a[N]);
  Py_INCREF(a[N + 1]);
  Py_XSETREF(workspace, a[N + 1]);
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
#define XM_FAST(F) {#F, (PyCFunction)(void (*)(void))F, METH_FASTCALL, nullptr}
    XM_FAST(forward), XM_FAST(sketch), XM_FAST(sketch_seeded), XM_FAST(wgrad), XM_FAST(wgrad_seeded), XM_FAST(dgrad), XM_FAST(backprobe), XM_FAST(contract),
    XM_FAST(use_library), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (`key`: what the module was compiled against; binding.py and build.py compare it with what is installed)
PyMODINIT_FUNC PyInit__marshal() {
  PyObject* m = PyModule_Create(&module_def);
  if (m && PyModule_AddStringConstant(m, "key", XM_KEY) != 0) { Py_DECREF(m); return nullptr; }
  return m;
}
