// Python entry points of the library as a CPython extension: checks the tensors, takes outputs from torch's caching
// allocator and scratch from one workspace kept per (device, stream), and calls the C ABI.
//
// A call on a small shape is bound by the host: the kernels of an MNIST batch take 16 us for a training step, while the
// same two calls through ctypes (argument conversion, four attribute look-ups per tensor, a device context manager and
// a stream look-up in Python) took 34 us, 12 us for the smallest single call.  Here the whole path from the Python
// call to the launch is C++.  The library is not linked: its functions are bound by address (bind), so that the
// binding can be pointed at another build of it.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <string>
#include <unordered_map>

#include "invconv.h"

namespace {

struct Api {
    decltype(&invconv_workspace_bytes) workspace_bytes;
    decltype(&invconv_bf16_workspace_bytes) bf16_workspace_bytes;
    decltype(&invconv_flow_step_workspace_bytes) flow_workspace_bytes;
    decltype(&masked_conv_workspace_bytes) conv_workspace_bytes;
    decltype(&invconv_forward_ws) forward;
    decltype(&invconv_backward_ws) backward;
    decltype(&invconv_forward_logdet_ws) forward_logdet;
    decltype(&invconv_backward_logdet_ws) backward_logdet;
    decltype(&masked_conv_forward_ws) conv;
    decltype(&invconv_logdet) logdet;
    decltype(&invconv_flow_step_forward_ws) flow_forward;
    decltype(&invconv_flow_step_backward_ws) flow_backward;
    decltype(&invconv_forward_bf16) forward_bf16;
    decltype(&invconv_backward_bf16) backward_bf16;
    decltype(&invconv_forward_bf16_ws) forward_bf16_ws;
    decltype(&invconv_backward_bf16_ws) backward_bf16_ws;
} api = {};
constexpr const char* kApiNames[] = {
    "invconv_workspace_bytes", "invconv_bf16_workspace_bytes", "invconv_flow_step_workspace_bytes", "masked_conv_workspace_bytes",
    "invconv_forward_ws", "invconv_backward_ws", "invconv_forward_logdet_ws", "invconv_backward_logdet_ws",
    "masked_conv_forward_ws", "invconv_logdet", "invconv_flow_step_forward_ws", "invconv_flow_step_backward_ws",
    "invconv_forward_bf16", "invconv_backward_bf16", "invconv_forward_bf16_ws", "invconv_backward_bf16_ws"};
constexpr size_t kApiCount = sizeof(kApiNames) / sizeof(kApiNames[0]);
static_assert(sizeof(Api) == kApiCount * sizeof(void*), "one address per name");

PyObject* g_error = nullptr;      // InvConvError(status, what)
bool g_bound = false;

struct Failed {};                 // a Python exception is set

[[noreturn]] void value_error(const std::string& msg)
{
    PyErr_SetString(PyExc_ValueError, msg.c_str());
    throw Failed{};
}

void check(int status, const char* what)
{
    if (status == INVCONV_OK) return;
    PyObject* e = PyObject_CallFunction(g_error, "is", status, what);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Failed{};
}

const at::Tensor& tensor(PyObject* o, const char* name)
{
    if (!THPVariable_Check(o)) value_error(std::string(name) + " must be a tensor");
    return THPVariable_Unpack(o);
}

const at::Tensor& activation(PyObject* o, const char* name, at::ScalarType type = at::kFloat)
{
    const at::Tensor& t = tensor(o, name);
    if (!(t.is_cuda() && t.scalar_type() == type && t.dim() == 4 && t.is_contiguous()))
        value_error(std::string(name) + " must be a contiguous " + (type == at::kFloat ? "fp32" : "bfloat16") + " CUDA tensor [B,C,H,W]");
    return t;
}

struct Shape { int B, C, H, W, k; };

Shape shape_of(const at::Tensor& t) { return {(int)t.size(0), (int)t.size(1), (int)t.size(2), (int)t.size(3), 0}; }

const at::Tensor& kernel(PyObject* o, Shape& s)
{
    const at::Tensor& w = tensor(o, "w");
    if (!(w.is_cuda() && w.scalar_type() == at::kFloat && w.dim() == 4 && w.is_contiguous()))
        value_error("w must be a contiguous fp32 CUDA tensor [C,C,k,k]");
    if (w.size(0) != s.C || w.size(1) != s.C || w.size(2) != w.size(3))
        value_error("w shape (" + std::to_string(w.size(0)) + ", " + std::to_string(w.size(1)) + ", " + std::to_string(w.size(2)) + ", " +
                    std::to_string(w.size(3)) + ") does not match C=" + std::to_string(s.C));
    s.k = (int)w.size(2);
    return w;
}

void* stream_of(PyObject* o, const at::Tensor& t)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream(t.device().index()).stream();
    PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) throw Failed{};
    void* p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (!p && PyErr_Occurred()) throw Failed{};
    return p;
}

// Straight to the caching allocator: the dispatcher adds nothing here and costs about a microsecond per tensor.
at::Tensor new_tensor(at::IntArrayRef sizes, at::ScalarType type, at::Device dev)
{
    return at::Tensor(at::detail::empty_cuda(sizes, type, dev, std::nullopt));
}
at::Tensor new_like(const at::Tensor& t) { return new_tensor(t.sizes(), t.scalar_type(), t.device()); }

// One zero-initialised scratch tensor per (device, stream), grown on demand and kept; every call leaves its control
// words zero, and calls on one stream are ordered, so all of them share it.
struct Workspaces {
    struct Key {
        int dev; void* st;
        bool operator==(const Key& o) const { return dev == o.dev && st == o.st; }
    };
    struct Hash { size_t operator()(const Key& k) const { return std::hash<void*>()(k.st) * 31 + (size_t)k.dev; } };
    std::unordered_map<Key, at::Tensor, Hash> map;      // guarded by the interpreter lock

    void* get(size_t need, const at::Tensor& like, void* st, size_t& bytes)
    {
        bytes = 0;
        if (need == 0) return nullptr;
        at::Tensor& ws = map[Key{(int)like.device().index(), st}];
        if (!ws.defined() || (size_t)ws.numel() < need) ws = at::zeros({(int64_t)need}, like.options().dtype(at::kByte));
        bytes = (size_t)ws.numel();
        return ws.data_ptr();
    }
} g_ws;

float* fp(const at::Tensor& t) { return static_cast<float*>(t.data_ptr()); }
PyObject* wrap(at::Tensor t) { return THPVariable_Wrap(std::move(t)); }
PyObject* given(PyObject* o) { Py_INCREF(o); return o; }

PyObject* pack(std::initializer_list<PyObject*> items)
{
    PyObject* t = PyTuple_New((Py_ssize_t)items.size());
    Py_ssize_t i = 0;
    for (PyObject* o : items) PyTuple_SET_ITEM(t, i++, o);
    return t;
}

PyObject* forward(PyObject* const* a)              // y, w, out, stream
{
    const at::Tensor& y = activation(a[0], "y");
    Shape s = shape_of(y);
    const at::Tensor& w = kernel(a[1], s);
    at::Tensor x = a[2] == Py_None ? new_like(y) : activation(a[2], "out");
    c10::cuda::CUDAGuard guard(y.device());
    void* st = stream_of(a[3], y);
    size_t n;
    void* ws = g_ws.get(api.workspace_bytes(s.B, s.C, s.H, s.W, s.k), y, st, n);
    check(api.forward(fp(y), fp(w), fp(x), s.B, s.C, s.H, s.W, s.k, ws, n, st), "invconv_forward");
    return a[2] == Py_None ? wrap(x) : given(a[2]);
}

PyObject* backward(PyObject* const* a)             // grad_x, x, w, need_grad_w, out_grad_y, out_grad_w, stream
{
    const at::Tensor& gx = activation(a[0], "grad_x");
    const at::Tensor& x = activation(a[1], "x");
    if (gx.sizes() != x.sizes()) value_error("grad_x and x must have the same shape");
    Shape s = shape_of(x);
    const at::Tensor& w = kernel(a[2], s);
    const int need_gw = PyObject_IsTrue(a[3]);
    if (need_gw < 0) throw Failed{};
    at::Tensor gy = a[4] == Py_None ? new_like(gx) : activation(a[4], "out_grad_y");
    at::Tensor gw;
    if (need_gw) gw = a[5] == Py_None ? new_like(w) : tensor(a[5], "out_grad_w");
    c10::cuda::CUDAGuard guard(x.device());
    void* st = stream_of(a[6], x);
    size_t n;
    void* ws = g_ws.get(api.workspace_bytes(s.B, s.C, s.H, s.W, s.k), x, st, n);
    check(api.backward(fp(gx), fp(x), fp(w), fp(gy), need_gw ? fp(gw) : nullptr, s.B, s.C, s.H, s.W, s.k, ws, n, st), "invconv_backward");
    return pack({a[4] == Py_None ? wrap(gy) : given(a[4]), !need_gw ? given(Py_None) : a[5] == Py_None ? wrap(gw) : given(a[5])});
}

PyObject* conv(PyObject* const* a)                 // x, w, out, stream
{
    const at::Tensor& x = activation(a[0], "x");
    Shape s = shape_of(x);
    const at::Tensor& w = kernel(a[1], s);
    at::Tensor y = a[2] == Py_None ? new_like(x) : activation(a[2], "out");
    c10::cuda::CUDAGuard guard(x.device());
    void* st = stream_of(a[3], x);
    size_t n;
    void* ws = g_ws.get(api.conv_workspace_bytes(s.B, s.C, s.H, s.W, s.k), x, st, n);
    check(api.conv(fp(x), fp(w), fp(y), s.B, s.C, s.H, s.W, s.k, ws, n, st), "masked_conv_forward");
    return a[2] == Py_None ? wrap(y) : given(a[2]);
}

PyObject* forward_logdet(PyObject* const* a)       // y, w, stream
{
    const at::Tensor& y = activation(a[0], "y");
    Shape s = shape_of(y);
    const at::Tensor& w = kernel(a[1], s);
    at::Tensor x = new_like(y), ld = new_tensor({1}, at::kFloat, y.device());
    c10::cuda::CUDAGuard guard(y.device());
    void* st = stream_of(a[2], y);
    size_t n;
    void* ws = g_ws.get(api.workspace_bytes(s.B, s.C, s.H, s.W, s.k), y, st, n);
    check(api.forward_logdet(fp(y), fp(w), fp(x), fp(ld), s.B, s.C, s.H, s.W, s.k, ws, n, st), "invconv_forward_logdet");
    return pack({wrap(x), wrap(ld)});
}

PyObject* backward_logdet(PyObject* const* a)      // grad_x, x, w, grad_logdet, stream
{
    const at::Tensor& gx = activation(a[0], "grad_x");
    const at::Tensor& x = activation(a[1], "x");
    if (gx.sizes() != x.sizes()) value_error("grad_x and x must have the same shape");
    const at::Tensor& gld = tensor(a[3], "grad_logdet");
    if (gld.scalar_type() != at::kFloat || gld.numel() != 1 || !gld.is_cuda())
        value_error("grad_logdet must be a one-element fp32 CUDA tensor");
    Shape s = shape_of(x);
    const at::Tensor& w = kernel(a[2], s);
    at::Tensor gy = new_like(gx), gw = new_like(w);
    c10::cuda::CUDAGuard guard(x.device());
    void* st = stream_of(a[4], x);
    size_t n;
    void* ws = g_ws.get(api.workspace_bytes(s.B, s.C, s.H, s.W, s.k), x, st, n);
    check(api.backward_logdet(fp(gx), fp(x), fp(w), fp(gld), fp(gy), fp(gw), s.B, s.C, s.H, s.W, s.k, ws, n, st),
          "invconv_backward_logdet");
    return pack({wrap(gy), wrap(gw)});
}

PyObject* flow_forward(PyObject* const* a)         // y, w, s, b, V, want_logdet, stream
{
    const at::Tensor& y = activation(a[0], "y");
    Shape s = shape_of(y);
    const at::Tensor& w = kernel(a[1], s);
    const at::Tensor &ts = tensor(a[2], "s"), &tb = tensor(a[3], "b"), &tV = tensor(a[4], "V");
    const int want = PyObject_IsTrue(a[5]);
    if (want < 0) throw Failed{};
    at::Tensor x = new_like(y), u = new_like(y), ld;
    if (want) ld = new_tensor({1}, at::kFloat, y.device());
    c10::cuda::CUDAGuard guard(y.device());
    void* st = stream_of(a[6], y);
    size_t n;
    void* ws = g_ws.get(api.flow_workspace_bytes(s.B, s.C, s.H, s.W, s.k), y, st, n);
    check(api.flow_forward(fp(y), fp(w), fp(ts), fp(tb), fp(tV), fp(x), fp(u), want ? fp(ld) : nullptr, s.B, s.C, s.H, s.W, s.k, ws, n, st),
          "invconv_flow_step_forward");
    return pack({wrap(x), wrap(u), want ? wrap(ld) : given(Py_None)});
}

PyObject* flow_backward(PyObject* const* a)        // grad_u, x, w, s, b, V, stream
{
    const at::Tensor& gu = activation(a[0], "grad_u");
    const at::Tensor& x = activation(a[1], "x");
    Shape s = shape_of(x);
    const at::Tensor& w = kernel(a[2], s);
    const at::Tensor &ts = tensor(a[3], "s"), &tb = tensor(a[4], "b"), &tV = tensor(a[5], "V");
    at::Tensor gy = new_like(x), gw = new_like(w), gs = new_like(ts), gb = new_like(tb), gV = new_like(tV);
    c10::cuda::CUDAGuard guard(x.device());
    void* st = stream_of(a[6], x);
    size_t n;
    void* ws = g_ws.get(api.flow_workspace_bytes(s.B, s.C, s.H, s.W, s.k), x, st, n);
    check(api.flow_backward(fp(gu), fp(x), fp(w), fp(ts), fp(tb), fp(tV), fp(gy), fp(gw), fp(gs), fp(gb), fp(gV), s.B, s.C, s.H, s.W, s.k,
                            ws, n, st), "invconv_flow_step_backward");
    return pack({wrap(gy), wrap(gw), wrap(gs), wrap(gb), wrap(gV)});
}

bool off16(const at::Tensor& t) { return (reinterpret_cast<uintptr_t>(t.data_ptr()) & 15) != 0; }

PyObject* forward_bf16(PyObject* const* a)         // y, w, out, stream
{
    const at::Tensor& y = activation(a[0], "y", at::kBFloat16);
    Shape s = shape_of(y);
    const at::Tensor& w = kernel(a[1], s);
    at::Tensor x = a[2] == Py_None ? new_like(y) : activation(a[2], "out", at::kBFloat16);
    c10::cuda::CUDAGuard guard(y.device());
    void* st = stream_of(a[3], y);
    int rc;
    if (s.B == 0 || off16(y) || off16(x)) {
        // buffers off a 16-byte boundary: the library sizes its own scratch for the route it has to take
        rc = api.forward_bf16(y.data_ptr(), fp(w), x.data_ptr(), s.B, s.C, s.H, s.W, s.k, st);
    } else {
        size_t n;
        void* ws = g_ws.get(api.bf16_workspace_bytes(s.B, s.C, s.H, s.W, s.k), y, st, n);
        rc = api.forward_bf16_ws(y.data_ptr(), fp(w), x.data_ptr(), s.B, s.C, s.H, s.W, s.k, ws, n, st);
    }
    check(rc, "invconv_forward_bf16");
    return a[2] == Py_None ? wrap(x) : given(a[2]);
}

PyObject* backward_bf16(PyObject* const* a)        // grad_x, x, w, need_grad_w, out_grad_y, out_grad_w, stream
{
    const at::Tensor& gx = activation(a[0], "grad_x", at::kBFloat16);
    const at::Tensor& x = activation(a[1], "x", at::kBFloat16);
    Shape s = shape_of(x);
    const at::Tensor& w = kernel(a[2], s);
    const int need_gw = PyObject_IsTrue(a[3]);
    if (need_gw < 0) throw Failed{};
    at::Tensor gy = a[4] == Py_None ? new_like(x) : activation(a[4], "out_grad_y", at::kBFloat16);
    at::Tensor gw;
    if (need_gw) gw = a[5] == Py_None ? new_like(w) : tensor(a[5], "out_grad_w");
    c10::cuda::CUDAGuard guard(x.device());
    void* st = stream_of(a[6], x);
    float* gwp = need_gw ? fp(gw) : nullptr;
    int rc;
    if (s.B == 0 || off16(gx) || off16(x) || off16(gy)) {
        rc = api.backward_bf16(gx.data_ptr(), x.data_ptr(), fp(w), gy.data_ptr(), gwp, s.B, s.C, s.H, s.W, s.k, st);
    } else {
        size_t n;
        void* ws = g_ws.get(api.bf16_workspace_bytes(s.B, s.C, s.H, s.W, s.k), x, st, n);
        rc = api.backward_bf16_ws(gx.data_ptr(), x.data_ptr(), fp(w), gy.data_ptr(), gwp, s.B, s.C, s.H, s.W, s.k, ws, n, st);
    }
    check(rc, "invconv_backward_bf16");
    return pack({a[4] == Py_None ? wrap(gy) : given(a[4]), !need_gw ? given(Py_None) : a[5] == Py_None ? wrap(gw) : given(a[5])});
}

template <PyObject* (*F)(PyObject* const*), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n)
{
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
        return nullptr;
    }
    if (!g_bound) {
        PyErr_SetString(PyExc_RuntimeError, "the CUDA library is not loaded");
        return nullptr;
    }
    try {
        return F(args);
    } catch (const Failed&) {
        return nullptr;
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// bind(addresses, error_type): addresses in the order of names().
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n)
{
    if (n != 2 || !PyTuple_Check(args[0]) || (size_t)PyTuple_GET_SIZE(args[0]) != kApiCount) {
        PyErr_SetString(PyExc_TypeError, "bind(addresses, error_type)");
        return nullptr;
    }
    void* addr[kApiCount];
    for (size_t i = 0; i < kApiCount; ++i) {
        addr[i] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(args[0], (Py_ssize_t)i));
        if (!addr[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null address");
            return nullptr;
        }
    }
    memcpy(&api, addr, sizeof(api));
    Py_INCREF(args[1]);
    Py_XSETREF(g_error, args[1]);
    g_bound = true;
    Py_RETURN_NONE;
}

PyObject* names(PyObject*, PyObject*)
{
    PyObject* t = PyTuple_New((Py_ssize_t)kApiCount);
    for (size_t i = 0; i < kApiCount; ++i) PyTuple_SET_ITEM(t, (Py_ssize_t)i, PyUnicode_FromString(kApiNames[i]));
    return t;
}

#define ENTRY(name, n) {#name, (PyCFunction)(void (*)(void))entry<name, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, nullptr},
    {"names", names, METH_NOARGS, nullptr},
    ENTRY(forward, 4), ENTRY(backward, 7), ENTRY(conv, 4), ENTRY(forward_logdet, 3), ENTRY(backward_logdet, 5),
    ENTRY(flow_forward, 7), ENTRY(flow_backward, 7), ENTRY(forward_bf16, 4), ENTRY(backward_bf16, 7),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
