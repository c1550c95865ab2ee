// The per-call host work of the Python binding for the calls a decode loop makes one by one: argument
// checks, the output's allocation, the current stream and the C ABI call, without the interpreter between
// them.  Each function takes only the ordinary case - plain CUDA tensors of the right type on the current
// device, a registered workspace that suffices - and answers None for everything else, where the
// caller's own Python code takes over (and raises what it always raised).
//
// What it is for: 4096 -> 4096 at one token is a 4.4 us kernel, and the Python path took 14.6 us a call.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

typedef size_t (*WorkspaceBytesFn)(int, int, int, int);
typedef int (*LinearPathFn)(const void*, const void*, const void*, const void*, void*, int, int, int, int, int, void*);
typedef int (*LinearInt3Fn)(const void*, const void*, const void*, const void*, void*, void*, int, int, int, int, void*);

WorkspaceBytesFn g_workspace_bytes = nullptr;
LinearPathFn g_linear_path = nullptr;
LinearInt3Fn g_linear_int3 = nullptr;
PyObject* g_workspaces = nullptr;        // the binding's dict: device index -> registered tensor
PyObject* g_check = nullptr;             // the binding's _check(rc, what)

// A plain contiguous CUDA tensor of dtype `t` on device `dev`, or nullptr.
const at::Tensor* plain(PyObject* o, at::ScalarType t, int dev) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& v = THPVariable_Unpack(o);
    if (!v.is_cuda() || v.scalar_type() != t || v.layout() != at::kStrided || !v.is_contiguous() || v.get_device() != dev) return nullptr;
    return &v;
}

bool as_int(PyObject* o, int* out) {
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    const long v = PyLong_AsLongAndOverflow(o, &overflow);
    if (overflow || v < INT_MIN || v > INT_MAX) return false;
    *out = (int)v;
    return true;
}

// true if the device's registered workspace suffices for the call
bool workspace_suffices(int dev, int M, int N, int K, int group) {
    const size_t need = g_workspace_bytes(M, N, K, group);
    if (need == 0) return true;
    PyObject* key = PyLong_FromLong(dev);
    if (!key) { PyErr_Clear(); return false; }
    PyObject* ws = PyDict_GetItemWithError(g_workspaces, key);     // borrowed
    Py_DECREF(key);
    if (!ws) { PyErr_Clear(); return false; }
    return THPVariable_Check(ws) && (size_t)THPVariable_Unpack(ws).numel() >= need;
}

// An uninitialized fp16 tensor [M][N].  Where nothing may take part in the allocation - no dispatch mode or function transform, no
// inference mode, no request to fill new memory - it comes from the allocator without the dispatcher in between (a call
// at one token: 3.96 -> 3.72 us of host time, 4.75 -> 4.35 us from call to call).
at::Tensor new_output(const at::Tensor& x, int M, int N) {
    const auto keys = c10::impl::tls_local_dispatch_key_set();
    if (keys.included_ == c10::default_included_set && keys.excluded_ == c10::default_excluded_set && !at::globalContext().deterministicAlgorithms())
        return at::Tensor(at::detail::empty_cuda({(int64_t)M, (int64_t)N}, at::kHalf, x.device(), std::nullopt));
    return at::empty({(int64_t)M, (int64_t)N}, x.options());
}

// what both layer calls share: x [M][K], packed arrays, N, K, group, out (None: allocated)
struct LayerCall {
    const at::Tensor *x, *qweight, *scales, *zeros;
    at::Tensor y;
    PyObject* out;                       // the caller's tensor (borrowed), or None
    int dev, M, N, K, group;
    bool parse(PyObject* const* a) {     // x, qweight, scales, zeros, N, K, group, out
        if (!THPVariable_CheckExact(a[0]) || !THPVariable_Unpack(a[0]).is_cuda()) return false;
        dev = c10::cuda::current_device();
        if (!(x = plain(a[0], at::kHalf, dev)) || !(qweight = plain(a[1], at::kByte, dev)) ||
            !(scales = plain(a[2], at::kHalf, dev)) || !(zeros = plain(a[3], at::kByte, dev)) ||
            !as_int(a[4], &N) || !as_int(a[5], &K) || !as_int(a[6], &group))
            return false;
        if (x->dim() != 2 || x->size(1) != K || x->size(0) > INT_MAX || N < 1) return false;
        M = (int)x->size(0);
        out = a[7];
        if (out == Py_None) return true;
        const at::Tensor* o = plain(out, at::kHalf, dev);
        if (!o) return false;
        y = *o;
        return true;
    }
    // The output and every address, while the interpreter lock is held: a tensor without memory of its own
    // (the wrapper that a function transform passes) throws here.
    const void *px, *pq, *ps, *pz;
    void* py;
    void resolve() {
        px = x->const_data_ptr(); pq = qweight->const_data_ptr(); ps = scales->const_data_ptr(); pz = zeros->const_data_ptr();
        if (!y.defined()) y = new_output(*x, M, N);
        py = y.mutable_data_ptr();
    }
    PyObject* result(int rc, const char* what) {
        if (rc != 0) return PyObject_CallFunction(g_check, "is", rc, what);          // raises
        if (out != Py_None) { Py_INCREF(out); return out; }
        return THPVariable_Wrap(y);
    }
};

void* current_stream(int dev) { return (void*)c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)dev).stream(); }

// linear(x, qweight, scales, zeros, N, K, group, out, path) -> y, or None
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    LayerCall c;
    int path = 0;
    if (n != 9 || !g_linear_path || !c.parse(a) || !as_int(a[8], &path) || !workspace_suffices(c.dev, c.M, c.N, c.K, c.group))
        Py_RETURN_NONE;
    c.resolve();
    int rc;
    void* stream = current_stream(c.dev);
    Py_BEGIN_ALLOW_THREADS
    rc = g_linear_path(c.px, c.pq, c.ps, c.pz, c.py, c.M, c.N, c.K, c.group, path, stream);
    Py_END_ALLOW_THREADS
    return c.result(rc, "awq_linear");
    END_HANDLE_TH_ERRORS
}

// linear_int3(x, qweight3, scales, zeros, N, K, group, out) -> y, or None; no scratch is offered at first:
// where the kernel reads the 3-bit storage itself none is needed (the library answers 1, null pointer,
// before it launches anything, where it is)
PyObject* linear_int3(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    LayerCall c;
    if (n != 8 || !g_linear_int3 || !c.parse(a) || !workspace_suffices(c.dev, c.M, c.N, c.K, c.group)) Py_RETURN_NONE;
    if (c.K < 1) Py_RETURN_NONE;
    c.resolve();
    at::Tensor scratch;
    int rc = 1;
    void* stream = current_stream(c.dev);
    for (int pass = c.M <= 64 ? 0 : 1; pass < 2 && rc == 1; ++pass) {
        if (pass == 1) scratch = at::empty({(int64_t)c.N * c.K / 2}, c.qweight->options());
        void* s = pass == 1 ? scratch.mutable_data_ptr() : nullptr;
        Py_BEGIN_ALLOW_THREADS
        rc = g_linear_int3(c.px, c.pq, c.ps, c.pz, c.py, s, c.M, c.N, c.K, c.group, stream);
        Py_END_ALLOW_THREADS
    }
    return c.result(rc, "awq_linear_int3");
    END_HANDLE_TH_ERRORS
}

// connect(workspace_bytes, linear_path, linear_int3, workspaces, check): addresses of the C ABI and the binding's objects
PyObject* connect(PyObject*, PyObject* args) {
    unsigned long long wb, lp, l3;
    PyObject *ws, *check;
    if (!PyArg_ParseTuple(args, "KKKO!O", &wb, &lp, &l3, &PyDict_Type, &ws, &check)) return nullptr;
    g_workspace_bytes = (WorkspaceBytesFn)(uintptr_t)wb;
    g_linear_path = (LinearPathFn)(uintptr_t)lp;
    g_linear_int3 = (LinearInt3Fn)(uintptr_t)l3;
    Py_INCREF(ws);
    Py_INCREF(check);
    Py_XSETREF(g_workspaces, ws);
    Py_XSETREF(g_check, check);
    Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"connect", connect, METH_VARARGS, nullptr},
    {"linear", (PyCFunction)(void (*)(void))linear, METH_FASTCALL, nullptr},
    {"linear_int3", (PyCFunction)(void (*)(void))linear_int3, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&g_module); }
