// The binding's short way: the calls a program makes many times per token or per prompt, with torch's tensors checked and
// allocated in C++ instead of Python (a prompt's call spends 12.6 us on the host in Python, its kernel 10).  Each function takes
// only the plain form of its call (every tensor an ordinary contiguous CUDA tensor of the right type and shape on the current
// device, no mode or wrapper in between) and returns None for anything else, errors included: the Python function then goes its
// own way, which decides what such a call means.  A status other than GF_OK comes back as an int.
// The library's entry points are handed over as addresses (bind), so nothing is linked against it.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <atomic>
#include <cstdint>

namespace {

using P = const void*;
typedef int (*PrefillFn)(P, P, P, P, P, P, void*, void*, int, int, int, int, void*);                   // .., u / u2, state_in, state_out, y, B, T, H, N
typedef int (*VarlenFn)(P, P, P, P, P, P, void*, void*, P, int, int, int, int, int, void*);
typedef int (*StepFn)(P, P, P, P, P, P, void*, void*, int, int, int, void*);
typedef int (*LayerNormFn)(P, P, P, float, void*, long long, int, int, void*);
typedef int (*KeyCompressFn)(P, P, void*, long long, int, int, void*);
typedef size_t (*WorkspaceBytesFn)(int, int, int, int);

enum { PREFILL, PREFILL_F32, PREFILL_C2, VARLEN, VARLEN_F32, VARLEN_C2, STEP, STEP_F32, STEP_C2, LAYERNORM, LAYERNORM_F32, KEY_COMPRESS, WORKSPACE_BYTES, N_FNS };
void* fns[N_FNS];
// the scratch that is registered with the library: the device it is on (upper 16 bits), its size in bytes
std::atomic<uint64_t> workspace{0};

// no torch-function or dispatch mode is active: allocations here mean what they mean in Python
bool plain_mode()
{
    return !c10::impl::TorchDispatchModeTLS::any_modes_set() && !at::impl::PythonTorchFunctionTLS::stack_len();
}

const c10::DispatchKeySet odd_keys({c10::DispatchKey::Python, c10::DispatchKey::PythonTLSSnapshot, c10::DispatchKey::FuncTorchBatched,
                                    c10::DispatchKey::FuncTorchGradWrapper, c10::DispatchKey::Functionalize, c10::DispatchKey::Conjugate,
                                    c10::DispatchKey::Negative, c10::DispatchKey::ZeroTensor, c10::DispatchKey::FuncTorchVmapMode,
                                    c10::DispatchKey::Batched});

// the current device if obj is a tensor on it, else -1
int here(PyObject* obj)
{
    if (!THPVariable_CheckExact(obj)) return -1;
    const at::Tensor& t = THPVariable_Unpack(obj);
    if (!t.defined() || !t.is_cuda()) return -1;
    const int dev = c10::cuda::current_device();
    return t.get_device() == dev ? dev : -1;
}
// obj as an ordinary contiguous tensor on device dev, or nullptr
const at::Tensor* plain(PyObject* obj, c10::ScalarType dtype, int dev)
{
    if (!THPVariable_CheckExact(obj)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(obj);
    if (!t.defined() || !t.key_set().has(c10::DispatchKey::CUDA) || t.key_set().has_any(odd_keys)) return nullptr;
    if (t.scalar_type() != dtype || t.layout() != c10::kStrided || t.get_device() != dev || !t.is_contiguous()) return nullptr;
    return &t;
}
const at::Tensor* plain(PyObject* obj, c10::ScalarType dtype, int dev, at::IntArrayRef shape)
{
    const at::Tensor* t = plain(obj, dtype, dev);
    return t && t->sizes() == shape ? t : nullptr;
}
// the same where None is allowed: false if obj is neither
bool optional_plain(PyObject* obj, c10::ScalarType dtype, int dev, at::IntArrayRef shape, P* out)
{
    *out = nullptr;
    if (obj == Py_None) return true;
    const at::Tensor* t = plain(obj, dtype, dev, shape);
    if (!t) return false;
    *out = t->const_data_ptr();
    return true;
}
bool fits_int(int64_t v) { return v >= 0 && v <= INT32_MAX; }

PyObject* pair_or_status(int status, at::Tensor&& a, at::Tensor&& b)
{
    if (status != 0) return PyLong_FromLong(status);
    PyObject *x = THPVariable_Wrap(std::move(a)), *y = x ? THPVariable_Wrap(std::move(b)) : nullptr;
    PyObject* r = y ? PyTuple_New(2) : nullptr;
    if (!r) { Py_XDECREF(x); Py_XDECREF(y); return nullptr; }
    PyTuple_SET_ITEM(r, 0, x);
    PyTuple_SET_ITEM(r, 1, y);
    return r;
}

// No C++ exception (an allocation that fails, say) leaves a function: the Python way meets the same one.
template <typename F> PyObject* guarded(F&& f)
{
    try {
        return f();
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

bool workspace_suffices(int dev, int B, int T, int H)
{
    const size_t need = reinterpret_cast<WorkspaceBytesFn>(fns[WORKSPACE_BYTES])(B, T, H, 64);
    if (need == 0) return true;
    const uint64_t w = workspace.load(std::memory_order_acquire);
    return (int)(w >> 48) == dev && (w & ((1ull << 48) - 1)) >= need;
}

// prefill(r, k, v, x, u or u2 (or None), state_in or None, c2)
PyObject* prefill(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 7 || !plain_mode()) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        const int dev = here(a[0]);
        if (dev < 0) Py_RETURN_NONE;
        const bool c2 = a[6] == Py_True;
        bool f32 = false;
        const at::Tensor* r = plain(a[0], at::kBFloat16, dev);
        if (!r && !c2) { r = plain(a[0], at::kFloat, dev); f32 = r != nullptr; }
        if (!r || r->dim() != 4) Py_RETURN_NONE;
        const at::ScalarType dt = f32 ? at::kFloat : at::kBFloat16;
        const int64_t B = r->size(0), T = r->size(1), H = r->size(2), N = r->size(3);
        if (!fits_int(B) || !fits_int(T) || !fits_int(H) || !fits_int(N)) Py_RETURN_NONE;
        const at::Tensor *k = plain(a[1], dt, dev, r->sizes()), *v = plain(a[2], dt, dev, r->sizes()), *x = plain(a[3], dt, dev, r->sizes());
        P u = nullptr, s = nullptr;
        const int64_t ushape[2] = {H, N}, sshape[4] = {B, H, N, N};
        if (!k || !v || !x || !optional_plain(a[5], at::kFloat, dev, sshape, &s)) Py_RETURN_NONE;
        if (c2 ? !optional_plain(a[4], at::kBFloat16, dev, r->sizes(), &u) : a[4] == Py_None || !optional_plain(a[4], at::kFloat, dev, ushape, &u)) Py_RETURN_NONE;
        if (!f32 && !workspace_suffices(dev, (int)B, (int)T, (int)H)) Py_RETURN_NONE;
        at::Tensor y = at::empty_like(*r), so = at::empty(sshape, r->options().dtype(at::kFloat).requires_grad(false));
        void* st = c10::cuda::getCurrentCUDAStream().stream();
        int status;
        const P pr = r->const_data_ptr(), pk = k->const_data_ptr(), pv = v->const_data_ptr(), px = x->const_data_ptr();
        void *py = y.mutable_data_ptr(), *ps = so.mutable_data_ptr();
        const PrefillFn fn = reinterpret_cast<PrefillFn>(fns[c2 ? PREFILL_C2 : f32 ? PREFILL_F32 : PREFILL]);
        Py_BEGIN_ALLOW_THREADS
        status = fn(pr, pk, pv, px, u, s, ps, py, (int)B, (int)T, (int)H, (int)N, st);
        Py_END_ALLOW_THREADS
        return pair_or_status(status, std::move(y), std::move(so));
    });
}

// prefill_varlen(r, k, v, x, u or u2 (or None), cu_seqlens, max_seqlen, state_in or None, c2)
PyObject* prefill_varlen(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 9 || !plain_mode() || !PyLong_CheckExact(a[6])) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        const int dev = here(a[0]);
        if (dev < 0) Py_RETURN_NONE;
        const bool c2 = a[8] == Py_True;
        bool f32 = false;
        const at::Tensor* r = plain(a[0], at::kBFloat16, dev);
        if (!r && !c2) { r = plain(a[0], at::kFloat, dev); f32 = r != nullptr; }
        const at::Tensor* cu = plain(a[5], at::kInt, dev);
        if (!r || r->dim() != 3 || !cu || cu->numel() < 1) Py_RETURN_NONE;
        const at::ScalarType dt = f32 ? at::kFloat : at::kBFloat16;
        const int64_t T = r->size(0), H = r->size(1), N = r->size(2), S = cu->numel() - 1;
        const long long max_seqlen = PyLong_AsLongLong(a[6]);
        if (max_seqlen == -1 && PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }
        if (!fits_int(T) || !fits_int(H) || !fits_int(N) || !fits_int(S) || !fits_int(max_seqlen)) Py_RETURN_NONE;
        const at::Tensor *k = plain(a[1], dt, dev, r->sizes()), *v = plain(a[2], dt, dev, r->sizes()), *x = plain(a[3], dt, dev, r->sizes());
        P u = nullptr, s = nullptr;
        const int64_t ushape[2] = {H, N}, sshape[4] = {S, H, N, N};
        if (!k || !v || !x || !optional_plain(a[7], at::kFloat, dev, sshape, &s)) Py_RETURN_NONE;
        if (c2 ? !optional_plain(a[4], at::kBFloat16, dev, r->sizes(), &u) : a[4] == Py_None || !optional_plain(a[4], at::kFloat, dev, ushape, &u)) Py_RETURN_NONE;
        if (!f32 && !workspace_suffices(dev, (int)S, (int)max_seqlen, (int)H)) Py_RETURN_NONE;
        at::Tensor y = at::empty_like(*r), so = at::empty(sshape, r->options().dtype(at::kFloat).requires_grad(false));
        void* st = c10::cuda::getCurrentCUDAStream().stream();
        int status;
        const P pr = r->const_data_ptr(), pk = k->const_data_ptr(), pv = v->const_data_ptr(), px = x->const_data_ptr(), pc = cu->const_data_ptr();
        void *py = y.mutable_data_ptr(), *ps = so.mutable_data_ptr();
        const VarlenFn fn = reinterpret_cast<VarlenFn>(fns[c2 ? VARLEN_C2 : f32 ? VARLEN_F32 : VARLEN]);
        Py_BEGIN_ALLOW_THREADS
        status = fn(pr, pk, pv, px, u, s, ps, py, pc, (int)S, (int)T, (int)max_seqlen, (int)H, (int)N, st);
        Py_END_ALLOW_THREADS
        return pair_or_status(status, std::move(y), std::move(so));
    });
}

// step(r, k, v, x, u or u2 (or None), state_in, state_out, y, c2): the outputs are the caller's
PyObject* step(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 9) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        const int dev = here(a[0]);
        if (dev < 0) Py_RETURN_NONE;
        const bool c2 = a[8] == Py_True;
        bool f32 = false;
        const at::Tensor* r = plain(a[0], at::kBFloat16, dev);
        if (!r && !c2) { r = plain(a[0], at::kFloat, dev); f32 = r != nullptr; }
        if (!r || r->dim() != 3) Py_RETURN_NONE;
        const at::ScalarType dt = f32 ? at::kFloat : at::kBFloat16;
        const int64_t B = r->size(0), H = r->size(1), N = r->size(2);
        if (!fits_int(B) || !fits_int(H) || !fits_int(N)) Py_RETURN_NONE;
        const int64_t ushape[2] = {H, N}, sshape[4] = {B, H, N, N};
        const at::Tensor *k = plain(a[1], dt, dev, r->sizes()), *v = plain(a[2], dt, dev, r->sizes()), *x = plain(a[3], dt, dev, r->sizes());
        const at::Tensor *so = plain(a[6], at::kFloat, dev, sshape), *y = plain(a[7], dt, dev, r->sizes());
        P u = nullptr, s = nullptr;
        if (!k || !v || !x || !so || !y || !optional_plain(a[5], at::kFloat, dev, sshape, &s)) Py_RETURN_NONE;
        if (c2 ? !optional_plain(a[4], at::kBFloat16, dev, r->sizes(), &u) : a[4] == Py_None || !optional_plain(a[4], at::kFloat, dev, ushape, &u)) Py_RETURN_NONE;
        void* st = c10::cuda::getCurrentCUDAStream().stream();
        const P pr = r->const_data_ptr(), pk = k->const_data_ptr(), pv = v->const_data_ptr(), px = x->const_data_ptr();
        void *py = y->mutable_data_ptr(), *ps = so->mutable_data_ptr();
        int status;
        const StepFn fn = reinterpret_cast<StepFn>(fns[c2 ? STEP_C2 : f32 ? STEP_F32 : STEP]);
        Py_BEGIN_ALLOW_THREADS
        status = fn(pr, pk, pv, px, u, s, ps, py, (int)B, (int)H, (int)N, st);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(status);
    });
}

// layernorm(y, gamma or None, beta or None, eps): gamma, beta [H*N]
PyObject* layernorm(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 4 || !PyFloat_CheckExact(a[3]) || !plain_mode()) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        const int dev = here(a[0]);
        if (dev < 0) Py_RETURN_NONE;
        bool f32 = false;
        const at::Tensor* y = plain(a[0], at::kBFloat16, dev);
        if (!y) { y = plain(a[0], at::kFloat, dev); f32 = y != nullptr; }
        if (!y || y->dim() < 2) Py_RETURN_NONE;
        const int64_t H = y->size(-2), N = y->size(-1);
        if (!fits_int(H) || !fits_int(N) || H * N == 0) Py_RETURN_NONE;
        const int64_t gshape[1] = {H * N};
        P g = nullptr, b = nullptr;
        if (!optional_plain(a[1], at::kFloat, dev, gshape, &g) || !optional_plain(a[2], at::kFloat, dev, gshape, &b)) Py_RETURN_NONE;
        at::Tensor out = at::empty_like(*y);
        void* st = c10::cuda::getCurrentCUDAStream().stream();
        const P py = y->const_data_ptr();
        void* po = out.mutable_data_ptr();
        const long long rows = y->numel() / (H * N);
        const float eps = (float)PyFloat_AS_DOUBLE(a[3]);
        int status;
        const LayerNormFn fn = reinterpret_cast<LayerNormFn>(fns[f32 ? LAYERNORM_F32 : LAYERNORM]);
        Py_BEGIN_ALLOW_THREADS
        status = fn(py, g, b, eps, po, rows, (int)H, (int)N, st);
        Py_END_ALLOW_THREADS
        return status ? PyLong_FromLong(status) : THPVariable_Wrap(std::move(out));
    });
}

// key_compress(x, w_kd)
PyObject* key_compress(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 2 || !plain_mode()) Py_RETURN_NONE;
    return guarded([&]() -> PyObject* {
        const int dev = here(a[0]);
        if (dev < 0) Py_RETURN_NONE;
        const at::Tensor *x = plain(a[0], at::kBFloat16, dev), *w = plain(a[1], at::kBFloat16, dev);
        if (!x || !w || x->dim() < 1 || w->dim() != 2 || x->size(-1) != w->size(0) || w->size(0) == 0) Py_RETURN_NONE;
        const int64_t D = w->size(0), Dc = w->size(1);
        if (!fits_int(D) || !fits_int(Dc)) Py_RETURN_NONE;
        at::DimVector shape(x->sizes().begin(), x->sizes().end());
        shape.back() = Dc;
        at::Tensor out = at::empty(shape, x->options().requires_grad(false));
        void* st = c10::cuda::getCurrentCUDAStream().stream();
        const P px = x->const_data_ptr(), pw = w->const_data_ptr();
        void* po = out.mutable_data_ptr();
        const long long rows = x->numel() / D;
        int status;
        const KeyCompressFn fn = reinterpret_cast<KeyCompressFn>(fns[KEY_COMPRESS]);
        Py_BEGIN_ALLOW_THREADS
        status = fn(px, pw, po, rows, (int)D, (int)Dc, st);
        Py_END_ALLOW_THREADS
        return status ? PyLong_FromLong(status) : THPVariable_Wrap(std::move(out));
    });
}

// bind(addresses): the entry points, in the order of the enumeration above
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != N_FNS) { PyErr_SetString(PyExc_TypeError, "bind: one address per entry point"); return nullptr; }
    for (Py_ssize_t i = 0; i < n; ++i) {
        void* f = PyLong_AsVoidPtr(a[i]);
        if (!f && PyErr_Occurred()) return nullptr;
        fns[i] = f;
    }
    Py_RETURN_NONE;
}

// set_workspace(device index, bytes): what is registered with the library now (0 bytes: nothing)
PyObject* set_workspace(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 2) { PyErr_SetString(PyExc_TypeError, "set_workspace(device, bytes)"); return nullptr; }
    const unsigned long long dev = PyLong_AsUnsignedLongLong(a[0]), bytes = PyLong_AsUnsignedLongLong(a[1]);
    if (PyErr_Occurred()) return nullptr;
    workspace.store(dev << 48 | (bytes & ((1ull << 48) - 1)), std::memory_order_release);
    Py_RETURN_NONE;
}

#define METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(prefill), METHOD(prefill_varlen), METHOD(step), METHOD(layernorm), METHOD(key_compress), METHOD(bind),
                         METHOD(set_workspace), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() { return PyModule_Create(&module); }
