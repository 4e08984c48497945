// CPython entry points of the calls a program makes per layer or per step.
//
// A small layer runs in a few microseconds, less than ctypes needs to marshal its arguments (measured
// on the benchmark's host: 9.5 us per call through ctypes, of which 2.2 us are the launch).  These
// functions read the tensors' pointers, types and sizes straight from the tensor objects, ask for the
// current stream once, release the interpreter lock around the library call and return its status.
// They take positional arguments only; binding.py holds the documented signatures, the optional
// allocations and the exceptions for statuses.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "prom.h"

namespace {

// What a bad argument raises; caught at the boundary of every entry point.
struct ArgError {};

[[noreturn]] void fail(PyObject *type, const char *fmt, const char *name, const char *detail = "")
{
    PyErr_Format(type, fmt, name, detail);
    throw ArgError();
}

const at::Tensor &tensor(PyObject *o, const char *name)
{
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "%s must be a tensor", name);
    return THPVariable_Unpack(o);
}

const char *dtype_name(at::ScalarType t)
{
    switch (t) {
    case at::kChar: return "torch.int8";
    case at::kByte: return "torch.uint8";
    case at::kInt: return "torch.int32";
    default: return "torch.float32";
    }
}

// A contiguous CUDA tensor of the given type.
const at::Tensor &dev(PyObject *o, at::ScalarType t, const char *name)
{
    const at::Tensor &x = tensor(o, name);
    if (!x.is_cuda()) fail(PyExc_ValueError, "%s must be a CUDA tensor", name);
    if (x.scalar_type() != t || !x.is_contiguous())
        fail(PyExc_ValueError, "%s must be contiguous %s", name, dtype_name(t));
    return x;
}

template <class T> T *ptr(const at::Tensor &t) { return static_cast<T *>(t.data_ptr()); }

void dims(const at::Tensor &t, int64_t n, const char *name)
{
    if (t.dim() != n) {
        PyErr_Format(PyExc_ValueError, "%s must have %d dimensions, not %d", name, (int)n, (int)t.dim());
        throw ArgError();
    }
}

long long integer(PyObject *o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw ArgError();
    return v;
}

int small_int(PyObject *o)
{
    const long long v = integer(o);
    if (v != (int)v) {
        PyErr_SetString(PyExc_OverflowError, "integer argument out of range");
        throw ArgError();
    }
    return (int)v;
}

// A stream handle, or None for the current stream of the current device.
void *stream(PyObject *o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    void *p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) throw ArgError();
    return p;
}

// The binding's ctypes structures, told by it once (register_types).
PyObject *requant_type, *layer_type, *job_type;

// A structure of the given type, or an array of them.
void structure(PyObject *o, PyObject *type, const char *name)
{
    if ((PyObject *)Py_TYPE(o) == type) return;
    static PyObject *const attr = PyUnicode_InternFromString("_type_");
    PyObject *element = PyObject_GetAttr((PyObject *)Py_TYPE(o), attr);       // of an array type
    if (!element) PyErr_Clear();
    const bool ok = element == type || (type && PyObject_IsInstance(o, type) == 1);
    Py_XDECREF(element);
    if (!ok) {
        PyErr_Clear();
        fail(PyExc_TypeError, "%s must be %s", name, type ? ((PyTypeObject *)type)->tp_name : "a registered structure");
    }
}

// The bytes behind a ctypes structure or array (a prom_requant, a layer table, a job table).
class Buffer {
public:
    Buffer(PyObject *o, size_t at_least, PyObject *type, const char *name)
    {
        structure(o, type, name);
        if (PyObject_GetBuffer(o, &view_, PyBUF_SIMPLE) != 0) throw ArgError();
        if ((size_t)view_.len < at_least) {
            PyBuffer_Release(&view_);
            PyErr_SetString(PyExc_ValueError, "structure argument too small");
            throw ArgError();
        }
    }
    ~Buffer() { PyBuffer_Release(&view_); }
    Buffer(const Buffer &) = delete;
    Buffer &operator=(const Buffer &) = delete;
    template <class T> const T *as() const { return static_cast<const T *>(view_.buf); }

private:
    Py_buffer view_;
};

// Runs a library call with the interpreter lock released.
template <class F> PyObject *call(F f)
{
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = (int)f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

template <class F> PyObject *guarded(Py_ssize_t n, Py_ssize_t want, F f)
{
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
        return nullptr;
    }
    try {
        return f();
    } catch (const ArgError &) {
        return nullptr;
    } catch (const std::exception &e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// (x, w_packed, cout, rq, y, variant, stream)
PyObject *pw_conv_i8(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 7, [&] {
        const at::Tensor &x = dev(a[0], at::kChar, "x");
        dims(x, 2, "x");
        const int64_t m = x.size(0);
        const int cin = (int)x.size(1), cout = small_int(a[2]), variant = small_int(a[5]);
        const auto *xp = ptr<const int8_t>(x);
        const auto *wp = ptr<const uint8_t>(dev(a[1], at::kByte, "w_packed"));
        auto *yp = ptr<int8_t>(dev(a[4], at::kChar, "y"));
        const Buffer rq(a[3], sizeof(prom_requant), requant_type, "rq");
        void *st = stream(a[6]);
        return call([&] { return prom_pw_conv_i8(xp, m, cin, wp, cout, rq.as<prom_requant>(), yp, (prom_variant)variant, st); });
    });
}

// (x, w_packed, cout, rq, res, y, variant, stream)
PyObject *pw_conv_i8_res(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 8, [&] {
        const at::Tensor &x = dev(a[0], at::kChar, "x");
        dims(x, 2, "x");
        const int64_t m = x.size(0);
        const int cin = (int)x.size(1), cout = small_int(a[2]), variant = small_int(a[6]);
        const at::Tensor &res = dev(a[4], at::kChar, "res");
        if (res.dim() != 2 || res.size(0) != m || res.size(1) != cout) fail(PyExc_ValueError, "%s must be [m, cout]", "res");
        const auto *xp = ptr<const int8_t>(x);
        const auto *wp = ptr<const uint8_t>(dev(a[1], at::kByte, "w_packed"));
        const auto *rp = ptr<const int8_t>(res);
        auto *yp = ptr<int8_t>(dev(a[5], at::kChar, "y"));
        const Buffer rq(a[3], sizeof(prom_requant), requant_type, "rq");
        void *st = stream(a[7]);
        return call([&] { return prom_pw_conv_i8_res(xp, m, cin, wp, cout, rq.as<prom_requant>(), rp, yp, (prom_variant)variant, st); });
    });
}

// (x, cout, prepared, act_min, act_max, y, stream)
PyObject *pw_conv_i8_prepared(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 7, [&] {
        const at::Tensor &x = dev(a[0], at::kChar, "x");
        dims(x, 2, "x");
        const int64_t m = x.size(0);
        const int cin = (int)x.size(1), cout = small_int(a[1]), lo = small_int(a[3]), hi = small_int(a[4]);
        const auto *xp = ptr<const int8_t>(x);
        const void *pp = ptr<const uint8_t>(dev(a[2], at::kByte, "prepared"));
        auto *yp = ptr<int8_t>(dev(a[5], at::kChar, "y"));
        void *st = stream(a[6]);
        return call([&] { return prom_pw_conv_i8_prepared(xp, m, cin, cout, pp, lo, hi, yp, st); });
    });
}

// (x, batch, w_packed, cout, alpha, gamma_x, q, gamma_y, scale_y, stream)
PyObject *pw_conv_i8_dyn(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 10, [&] {
        const at::Tensor &x = dev(a[0], at::kChar, "x");
        dims(x, 2, "x");
        const int64_t m = x.size(0);
        const int cin = (int)x.size(1), batch = small_int(a[1]), cout = small_int(a[3]);
        if (batch && m % batch) fail(PyExc_ValueError, "%s", "rows must divide evenly into samples");
        const int64_t rows = batch ? m / batch : 1;
        const auto *xp = ptr<const int8_t>(x);
        const auto *wp = ptr<const uint8_t>(dev(a[2], at::kByte, "w_packed"));
        const auto *al = ptr<const float>(dev(a[4], at::kFloat, "alpha"));
        const auto *gx = ptr<const float>(dev(a[5], at::kFloat, "gamma_x"));
        auto *q = ptr<int8_t>(tensor(a[6], "q"));
        auto *gy = ptr<float>(tensor(a[7], "gamma_y"));
        auto *sy = ptr<float>(tensor(a[8], "scale_y"));
        void *st = stream(a[9]);
        return call([&] { return prom_pw_conv_i8_dyn(xp, batch, rows, cin, wp, cout, al, gx, q, gy, sy, st); });
    });
}

// (x, w, rq, stride, y, stream); x is [batch, h, w, c]
PyObject *dw_conv3x3_i8(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 6, [&] {
        const at::Tensor &x = dev(a[0], at::kChar, "x");
        dims(x, 4, "x");
        const int b = (int)x.size(0), h = (int)x.size(1), w = (int)x.size(2), c = (int)x.size(3);
        const int stride = small_int(a[3]);
        const auto *xp = ptr<const int8_t>(x);
        const auto *wp = ptr<const int8_t>(dev(a[1], at::kChar, "w"));
        auto *yp = ptr<int8_t>(dev(a[4], at::kChar, "y"));
        const Buffer rq(a[2], sizeof(prom_requant), requant_type, "rq");
        void *st = stream(a[5]);
        return call([&] { return prom_dw_conv3x3_i8(xp, b, h, w, c, stride, wp, rq.as<prom_requant>(), yp, st); });
    });
}

// (x, q, gamma, scale, stream); x is [batch, ...]
PyObject *quantize_act_absmax(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 5, [&] {
        const at::Tensor &x = tensor(a[0], "x"), &q = tensor(a[1], "q"), &g = tensor(a[2], "gamma"), &s = tensor(a[3], "scale");
        if (!x.is_cuda() || x.scalar_type() != at::kFloat || !x.is_contiguous() || x.dim() < 1)
            fail(PyExc_ValueError, "%s must be a contiguous float32 CUDA tensor", "x");
        const int64_t batch = x.size(0);
        if (q.sizes() != x.sizes() || q.scalar_type() != at::kChar || !q.is_cuda() || g.numel() != batch ||
            s.numel() != batch || g.scalar_type() != at::kFloat || s.scalar_type() != at::kFloat)
            fail(PyExc_ValueError, "%s must be (int8 like x, float32 [batch], float32 [batch]) on the device", "out");
        const int64_t per = batch ? x.numel() / batch : 1;
        const auto *xp = ptr<const float>(x);
        auto *qp = ptr<int8_t>(q);
        auto *gp = ptr<float>(g), *sp = ptr<float>(s);
        void *st = stream(a[4]);
        return call([&] { return prom_quantize_act_absmax(xp, (int)batch, per, qp, gp, sp, st); });
    });
}

// (job table, n, stream)
PyObject *quantize_ternary_batch(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 3, [&] {
        const int jobs = small_int(a[1]);
        const Buffer t(a[0], (size_t)(jobs > 0 ? jobs : 0) * sizeof(prom_quantize_job), job_type, "jobs");
        void *st = stream(a[2]);
        return call([&] { return prom_quantize_ternary_batch(t.as<prom_quantize_job>(), jobs, st); });
    });
}

// (layer table, n, x0, workspace, y, variant, stream); x0 is [batch, h, w, cin]
PyObject *pw_layer_seq(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 7, [&] {
        const int layers = small_int(a[1]), variant = small_int(a[5]);
        const at::Tensor &x = dev(a[2], at::kChar, "x0");
        dims(x, 4, "x0");
        const int b = (int)x.size(0), h = (int)x.size(1), w = (int)x.size(2);
        const at::Tensor &ws = tensor(a[3], "workspace");
        const Buffer t(a[0], (size_t)(layers > 0 ? layers : 0) * sizeof(prom_layer), layer_type, "layers");
        const auto *xp = ptr<const int8_t>(x);
        void *wsp = ws.data_ptr();
        const size_t ws_bytes = (size_t)ws.numel();
        auto *yp = ptr<int8_t>(dev(a[4], at::kChar, "y_out"));
        void *st = stream(a[6]);
        return call([&] { return prom_pw_layer_seq(t.as<prom_layer>(), layers, xp, b, h, w, wsp, ws_bytes, yp, (prom_variant)variant, st); });
    });
}

// (prom_requant, prom_layer, prom_quantize_job as the binding has them); kept for as long as the module
PyObject *register_types(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded(n, 3, [&] {
        for (int i = 0; i < 3; ++i) {
            if (!PyType_Check(a[i])) fail(PyExc_TypeError, "%s", "types are expected");
            Py_INCREF(a[i]);
        }
        requant_type = a[0]; layer_type = a[1]; job_type = a[2];
        Py_RETURN_NONE;
    });
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY(pw_conv_i8), ENTRY(pw_conv_i8_res), ENTRY(pw_conv_i8_prepared), ENTRY(pw_conv_i8_dyn),
                         ENTRY(dw_conv3x3_i8), ENTRY(quantize_act_absmax), ENTRY(quantize_ternary_batch),
                         ENTRY(pw_layer_seq), ENTRY(register_types), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
