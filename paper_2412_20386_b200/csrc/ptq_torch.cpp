// The forward calls of binding.PtqLinear on torch tensors, without Python in between: checks, allocation of what the
// caller did not pass, the current stream and the C ABI call.  Through Python attribute access and ctypes the same steps
// took 6 to 11 us a call, more than the two kernel launches they lead to (5 us), and bound every layer below that time.
// The offline steps (calibration, step search) go the same way, with host arrays through the buffer protocol: a calibration of
// 8 x 197 x 384 with 192 outputs takes 60 us a call, 78 through ctypes, of which 36 are its copies, launches and the wait for them.
// The C ABI's functions are handed over as addresses by the binding, so this module does not link the library.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/ptq_linear.h"

namespace {

decltype(&ptq_linear_forward) f_forward = nullptr;
decltype(&ptq_linear_forward_static) f_static = nullptr;
decltype(&ptq_linear_forward_dynamic) f_dynamic = nullptr;
decltype(&ptq_linear_workspace_bytes) f_ws = nullptr;
decltype(&ptq_linear_workspace_bytes_dynamic) f_ws_dynamic = nullptr;
decltype(&ptq_calibrate_in) f_calibrate = nullptr;
decltype(&ptq_search_act_step_in) f_search = nullptr;

// Arguments of every call: handle, T, K, N, x, y, workspace (the last two may be None).
struct Call {
    const ptq_linear_t *h;
    int64_t T, K, N, B;
    const at::Tensor *x;
    at::Tensor y, ws;
    bool has_y, has_ws;
};

bool read_call(PyObject *const *args, Py_ssize_t n, Call &c)
{
    if (n != 7) {
        PyErr_SetString(PyExc_TypeError, "seven arguments are wanted");
        return false;
    }
    c.h = static_cast<const ptq_linear_t *>(PyLong_AsVoidPtr(args[0]));
    c.T = PyLong_AsLongLong(args[1]);
    c.K = PyLong_AsLongLong(args[2]);
    c.N = PyLong_AsLongLong(args[3]);
    if (PyErr_Occurred()) return false;
    if (!THPVariable_Check(args[4])) {
        PyErr_SetString(PyExc_TypeError, "x must be a tensor");
        return false;
    }
    c.x = &THPVariable_Unpack(args[4]);
    const at::Tensor &x = *c.x;
    if (x.scalar_type() != at::kHalf || !x.is_cuda() || !x.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "x must be a contiguous CUDA float16 tensor");
        return false;
    }
    if (x.dim() < 1 || x.size(-1) != c.K || x.numel() % (c.T * c.K) != 0) {
        PyErr_Format(PyExc_ValueError, "x must be [B,T,K] with T=%lld K=%lld", static_cast<long long>(c.T), static_cast<long long>(c.K));
        return false;
    }
    c.B = x.numel() / (c.T * c.K);
    if (c.B > 0x7fffffff) {
        PyErr_SetString(PyExc_ValueError, "x is too large");
        return false;
    }
    at::Tensor *dst[2] = {&c.y, &c.ws};
    bool *has[2] = {&c.has_y, &c.has_ws};
    for (int i = 0; i < 2; ++i) {
        *has[i] = args[5 + i] != Py_None;
        if (!*has[i]) continue;
        if (!THPVariable_Check(args[5 + i])) {
            PyErr_SetString(PyExc_TypeError, "y and workspace must be tensors");
            return false;
        }
        *dst[i] = THPVariable_Unpack(args[5 + i]);
    }
    return true;
}

void make_y(Call &c)
{
    if (!c.has_y) c.y = at::Tensor(at::detail::empty_cuda({c.B, c.T, c.N}, at::kHalf, c.x->device(), std::nullopt));
}
// Blocks of the caching allocator belong to the current stream, which is the one the kernels run on.
void make_ws(Call &c, size_t bytes)
{
    if (!c.has_ws && bytes)
        c.ws = at::Tensor(at::detail::empty_cuda({static_cast<int64_t>(bytes < 16 ? 16 : bytes)}, at::kByte, c.x->device(), std::nullopt));
}

// C++ exceptions become the classes that torch's own calls raise: torch.OutOfMemoryError where an allocation fails.
template <class Fn>
PyObject *guarded(Fn fn)
{
    HANDLE_TH_ERRORS
    return fn();
    END_HANDLE_TH_ERRORS
}

// y on success (the caller's object where one was passed), the status as an int otherwise.
PyObject *answer(const Call &c, ptq_status_t st, PyObject *y_arg)
{
    if (st != PTQ_OK) return PyLong_FromLong(st);
    if (!c.has_y) return THPVariable_Wrap(c.y);
    Py_INCREF(y_arg);
    return y_arg;
}

PyObject *py_forward(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        Call c;
        if (!read_call(args, n, c)) return nullptr;
        make_y(c);
        if (!c.has_ws) make_ws(c, f_ws(c.h, static_cast<int>(c.B), 0));
        const size_t bytes = c.ws.defined() ? c.ws.nbytes() : 0;
        void *ws = c.ws.defined() ? c.ws.data_ptr() : nullptr;
        void *stream = c10::cuda::getCurrentCUDAStream().stream();
        const void *x = c.x->const_data_ptr();
        void *y = c.y.data_ptr();
        ptq_status_t st;
        Py_BEGIN_ALLOW_THREADS
        st = f_forward(c.h, x, static_cast<int>(c.B), y, ws, bytes, PTQ_FLAG_NONE, stream);
        Py_END_ALLOW_THREADS
        return answer(c, st, args[5]);
    });
}

PyObject *py_forward_dynamic(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        Call c;
        if (!read_call(args, n, c)) return nullptr;
        make_y(c);
        if (!c.has_ws) make_ws(c, f_ws_dynamic(c.h, static_cast<int>(c.B)));
        const size_t bytes = c.ws.defined() ? c.ws.nbytes() : 0;
        void *ws = c.ws.defined() ? c.ws.data_ptr() : nullptr;
        void *stream = c10::cuda::getCurrentCUDAStream().stream();
        const void *x = c.x->const_data_ptr();
        void *y = c.y.data_ptr();
        ptq_status_t st;
        Py_BEGIN_ALLOW_THREADS
        st = f_dynamic(c.h, x, static_cast<int>(c.B), y, ws, bytes, stream);
        Py_END_ALLOW_THREADS
        return answer(c, st, args[5]);
    });
}

PyObject *py_forward_static(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        Call c;
        if (!read_call(args, n, c)) return nullptr;
        if (!c.has_y || c.y.dim() != 3 || c.y.size(0) != c.B || c.y.size(1) != c.T || c.y.size(2) != c.N ||
            c.y.scalar_type() != at::kHalf || !c.y.is_contiguous() || !c.y.is_cuda()) {
            PyErr_SetString(PyExc_ValueError, "y must be a contiguous CUDA float16 tensor [B,T,N]");
            return nullptr;
        }
        void *stream = c10::cuda::getCurrentCUDAStream().stream();
        const void *x = c.x->const_data_ptr();
        void *y = c.y.data_ptr();
        ptq_status_t st;
        Py_BEGIN_ALLOW_THREADS
        st = f_static(c.h, x, static_cast<int>(c.B), y, stream);
        Py_END_ALLOW_THREADS
        return answer(c, st, args[5]);
    });
}

// Memory of a contiguous host array (buffer protocol), or null for None.
struct Host {
    Py_buffer view;
    bool held = false;
    void *ptr = nullptr;
    bool read(PyObject *o, bool writable)
    {
        if (o == Py_None) return true;
        if (PyObject_GetBuffer(o, &view, writable ? PyBUF_WRITABLE | PyBUF_C_CONTIGUOUS : PyBUF_C_CONTIGUOUS) != 0) return false;
        held = true;
        ptr = view.buf;
        return true;
    }
    Host() = default;
    Host(const Host &) = delete;
    Host &operator=(const Host &) = delete;
    ~Host()
    {
        if (held) PyBuffer_Release(&view);
    }
};

// The integers, the two tensors (activations, workspace) and the host arrays of an offline step: two that the library reads, three
// that it writes.  Shapes and types are the binding's to check.
struct Offline {
    int v[5];
    const void *x;
    void *ws, *stream;
    size_t ws_bytes;
    Host h[5];
};
bool read_offline(PyObject *const *args, Py_ssize_t n, Offline &o)
{
    if (n != 12 || !THPVariable_Check(args[5]) || !THPVariable_Check(args[6])) {
        PyErr_SetString(PyExc_TypeError, "five integers, two tensors and five arrays are wanted");
        return false;
    }
    for (int i = 0; i < 5; ++i) o.v[i] = static_cast<int>(PyLong_AsLong(args[i]));
    if (PyErr_Occurred()) return false;
    for (int i = 0; i < 5; ++i)
        if (!o.h[i].read(args[7 + i], i >= 2)) return false;
    const at::Tensor &ws = THPVariable_Unpack(args[6]);
    o.x = THPVariable_Unpack(args[5]).const_data_ptr();
    o.ws = ws.data_ptr();
    o.ws_bytes = ws.nbytes();
    o.stream = c10::cuda::getCurrentCUDAStream().stream();
    return true;
}

// calibrate(scheme, K, N, T, Bc, xcal, workspace, w, w_step, s, dx, z) -> status
PyObject *py_calibrate(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        Offline o;
        if (!read_offline(args, n, o)) return nullptr;
        ptq_status_t st;
        Py_BEGIN_ALLOW_THREADS
        st = f_calibrate(o.v[0], o.v[1], o.v[2], o.v[3], o.x, o.v[4], o.h[0].ptr, static_cast<const float *>(o.h[1].ptr),
                         static_cast<float *>(o.h[2].ptr), static_cast<float *>(o.h[3].ptr), static_cast<int32_t *>(o.h[4].ptr), o.ws,
                         o.ws_bytes, o.stream);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(st);
    });
}

// search(K, T, Bc, n_grid, j_lo, xcal, workspace, s, base, dx, best, loss) -> status
PyObject *py_search(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        Offline o;
        if (!read_offline(args, n, o)) return nullptr;
        ptq_status_t st;
        Py_BEGIN_ALLOW_THREADS
        st = f_search(o.v[0], o.v[1], o.x, o.v[2], static_cast<const float *>(o.h[0].ptr), static_cast<const float *>(o.h[1].ptr), o.v[3],
                      o.v[4], static_cast<float *>(o.h[2].ptr), static_cast<int32_t *>(o.h[3].ptr), static_cast<double *>(o.h[4].ptr), o.ws,
                      o.ws_bytes, o.stream);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(st);
    });
}

PyObject *py_bind(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (n != 7) {
        PyErr_SetString(PyExc_TypeError, "seven addresses are wanted");
        return nullptr;
    }
    void *p[7];
    for (int i = 0; i < 7; ++i) p[i] = PyLong_AsVoidPtr(args[i]);
    if (PyErr_Occurred()) return nullptr;
    f_forward = reinterpret_cast<decltype(f_forward)>(p[0]);
    f_static = reinterpret_cast<decltype(f_static)>(p[1]);
    f_dynamic = reinterpret_cast<decltype(f_dynamic)>(p[2]);
    f_ws = reinterpret_cast<decltype(f_ws)>(p[3]);
    f_ws_dynamic = reinterpret_cast<decltype(f_ws_dynamic)>(p[4]);
    f_calibrate = reinterpret_cast<decltype(f_calibrate)>(p[5]);
    f_search = reinterpret_cast<decltype(f_search)>(p[6]);
    Py_RETURN_NONE;
}

#define PTQ_METHOD(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fn)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PTQ_METHOD("bind", py_bind), PTQ_METHOD("forward", py_forward),
                         PTQ_METHOD("forward_static", py_forward_static), PTQ_METHOD("forward_dynamic", py_forward_dynamic),
                         PTQ_METHOD("calibrate", py_calibrate), PTQ_METHOD("search", py_search),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_ptq_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__ptq_torch(void) { return PyModule_Create(&module); }
