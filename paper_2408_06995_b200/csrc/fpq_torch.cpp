// CPython binding of the calls that a running model makes per layer (and that an offline step makes per iteration):
// takes torch tensors, passes their device pointers and the current CUDA stream to the C entry points of fpq.h.
// It marshals arguments and nothing else.
//
// Through ctypes a layer call spent about 9 us in Python (a pointer object per tensor, two structs by value through
// libffi, the stream looked up through three Python frames), more than the kernels of a small layer take; here it is
// well under 1 us.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "fpq.h"

namespace {

PyObject *g_exp_bits, *g_man_bits, *g_exp_bias, *g_sat_mode, *g_data_ptr, *g_numel;

// (torch's accessors report errors as C++ exceptions: they become Python's here; none may leave a call, or run where the
// interpreter lock has been given up)
template <typename F>
bool guarded(F f)
{
    try {
        f();
        return true;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return false;
    }
}

bool stream(void** st)
{
    return guarded([&] { *st = (void*)c10::cuda::getCurrentCUDAStream().stream(); });
}

// device pointer of a tensor, NULL for None
bool pointer(PyObject* o, void** p)
{
    if (o == Py_None) {
        *p = nullptr;
        return true;
    }
    if (THPVariable_Check(o))
        return guarded([&] { *p = THPVariable_Unpack(o).data_ptr(); });
    PyObject* v = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!v)
        return false;
    *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}

bool int_attr(PyObject* o, PyObject* name, int32_t* out)
{
    PyObject* v = PyObject_GetAttr(o, name);
    if (!v)
        return false;
    const long long x = PyLong_AsLongLong(v);
    Py_DECREF(v);
    *out = (int32_t)x;
    return !(x == -1 && PyErr_Occurred());
}

bool format(PyObject* o, fpq_format* f)
{
    return int_attr(o, g_exp_bits, &f->exp_bits) && int_attr(o, g_man_bits, &f->man_bits) &&
           int_attr(o, g_exp_bias, &f->exp_bias) && int_attr(o, g_sat_mode, &f->sat_mode);
}

bool real(PyObject* o, float* out)
{
    const double v = PyFloat_AsDouble(o);
    *out = (float)v;
    return !(v == -1.0 && PyErr_Occurred());
}

bool integer(PyObject* o, int64_t* out)
{
    *out = PyLong_AsLongLong(o);
    return !(*out == -1 && PyErr_Occurred());
}

bool integer(PyObject* o, int* out)
{
    int64_t v;
    if (!integer(o, &v))
        return false;
    *out = (int)v;
    return true;
}

// sizes and elements of a tensor (sparse, nested and traced tensors may throw instead of giving them)
struct Shape {
    int64_t dim, size[4], numel;

    void take(const at::Tensor& t)
    {
        dim = t.dim();
        for (int64_t i = 0; i < 4; ++i)
            size[i] = i < dim ? t.size(i) : 1;
        numel = t.numel();
    }
};

// a contiguous FP32 CUDA tensor of `dim` dimensions (0: any)
bool fp32_cuda(PyObject* o, int64_t dim, Shape* out)
{
    bool fits = false;
    if (THPVariable_Check(o) && !guarded([&] {
            const at::Tensor& t = THPVariable_Unpack(o);
            fits = t.is_cuda() && t.scalar_type() == at::kFloat && t.is_contiguous() && (dim == 0 || t.dim() == dim);
            if (fits)
                out->take(t);
        }))
        return false;
    if (!fits)
        PyErr_SetString(PyExc_AssertionError, "expected a contiguous float32 CUDA tensor of the documented shape");
    return fits;
}

// any tensor: the caller's sizes are taken as they are
bool tensor(PyObject* o, Shape* out)
{
    if (THPVariable_Check(o))
        return guarded([&] { out->take(THPVariable_Unpack(o)); });
    PyErr_SetString(PyExc_TypeError, "expected a tensor");
    return false;
}

// size of a workspace (bytes: its elements are): of any object whose pointer is taken, and never more than it says
bool workspace(PyObject* o, void** p, size_t* bytes)
{
    *bytes = 0;
    if (!pointer(o, p))
        return false;
    if (o == Py_None)
        return true;
    if (THPVariable_Check(o))
        return guarded([&] { *bytes = (size_t)THPVariable_Unpack(o).numel(); });
    PyObject* v = PyObject_CallMethodNoArgs(o, g_numel);
    if (!v)
        return false;
    const long long n = PyLong_AsLongLong(v);
    Py_DECREF(v);
    if (n < 0 && !PyErr_Occurred())
        PyErr_SetString(PyExc_ValueError, "a workspace of negative size");
    *bytes = (size_t)n;
    return n >= 0;
}

bool arguments(Py_ssize_t given, Py_ssize_t wanted)
{
    if (given == wanted)
        return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", wanted, given);
    return false;
}

// linear(x, w_prepared, w_scale, x_scale, fx, fw, bias, N, y, workspace) -> status
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    Shape x;
    void *xp, *w, *ws, *bias, *y, *work, *st;
    size_t work_bytes;
    float xs;
    fpq_format fx, fw;
    int64_t N;
    if (!arguments(n, 10) || !fp32_cuda(a[0], 2, &x) || !pointer(a[1], &w) || !pointer(a[2], &ws) || !real(a[3], &xs) ||
        !format(a[4], &fx) || !format(a[5], &fw) || !pointer(a[6], &bias) || !integer(a[7], &N) || !pointer(a[8], &y) ||
        !workspace(a[9], &work, &work_bytes) || !pointer(a[0], &xp) || !stream(&st))
        return nullptr;
    fpq_status status;
    Py_BEGIN_ALLOW_THREADS
    status = fpq_linear((const float*)xp, w, (const float*)ws, xs, fx, fw, (const float*)bias, (float*)y, x.size[0], N,
                        x.size[1], work, work_bytes, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

// conv2d(x, w_prepared, w_scale, x_scale, fx, fw, bias, C_out, R, S, pad, stride, y, workspace) -> status
PyObject* conv2d(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    Shape x;
    void *xp, *w, *ws, *bias, *y, *work, *st;
    size_t work_bytes;
    float xs;
    fpq_format fx, fw;
    int g[5];
    if (!arguments(n, 14) || !fp32_cuda(a[0], 4, &x) || !pointer(a[1], &w) || !pointer(a[2], &ws) || !real(a[3], &xs) ||
        !format(a[4], &fx) || !format(a[5], &fw) || !pointer(a[6], &bias))
        return nullptr;
    for (int i = 0; i < 5; ++i)
        if (!integer(a[7 + i], &g[i]))
            return nullptr;
    if (!pointer(a[12], &y) || !workspace(a[13], &work, &work_bytes) || !pointer(a[0], &xp) || !stream(&st))
        return nullptr;
    fpq_status status;
    Py_BEGIN_ALLOW_THREADS
    status = fpq_conv2d((const float*)xp, w, (const float*)ws, xs, fx, fw, (const float*)bias, (float*)y, (int)x.size[0],
                        (int)x.size[1], (int)x.size[2], (int)x.size[3], g[0], g[1], g[2], g[3], g[4], work, work_bytes,
                        st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

// conv2d_split(x1, x1_scale, x2, x2_scale, w_prepared, w_scale, fx, fw, bias, y, R, S, pad, stride, workspace) -> status
PyObject* conv2d_split(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    Shape x1, x2, y;
    void *x1p, *x2p, *yp, *w, *ws, *bias, *work, *st;
    size_t work_bytes;
    float s1, s2;
    fpq_format fx, fw;
    int g[4];
    if (!arguments(n, 15) || !tensor(a[0], &x1) || !real(a[1], &s1) || !tensor(a[2], &x2) || !real(a[3], &s2) ||
        !pointer(a[4], &w) || !pointer(a[5], &ws) || !format(a[6], &fx) || !format(a[7], &fw) || !pointer(a[8], &bias) ||
        !tensor(a[9], &y))
        return nullptr;
    if (x1.dim != 4 || x2.dim < 2 || y.dim < 2) {
        PyErr_SetString(PyExc_ValueError, "expected NCHW tensors");
        return nullptr;
    }
    for (int i = 0; i < 4; ++i)
        if (!integer(a[10 + i], &g[i]))
            return nullptr;
    if (!workspace(a[14], &work, &work_bytes) || !pointer(a[0], &x1p) || !pointer(a[2], &x2p) || !pointer(a[9], &yp) || !stream(&st))
        return nullptr;
    fpq_status status;
    Py_BEGIN_ALLOW_THREADS
    status = fpq_conv2d_split((const float*)x1p, (int)x1.size[1], s1, (const float*)x2p, (int)x2.size[1], s2, w,
                              (const float*)ws, fx, fw, (const float*)bias, (float*)yp, (int)x1.size[0],
                              (int)x1.size[2], (int)x1.size[3], (int)y.size[1], g[0], g[1], g[2], g[3], work,
                              work_bytes, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

// search(x, encodings, clip, mse, best, workspace) -> status
PyObject* search(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    Shape x, clip;
    void *xp, *clipp, *mse, *best, *work, *st;
    size_t work_bytes;
    fpq_format enc[16];
    if (!arguments(n, 6) || !fp32_cuda(a[0], 0, &x) || !fp32_cuda(a[2], 0, &clip) || !pointer(a[0], &xp) || !pointer(a[2], &clipp) ||
        !pointer(a[3], &mse) || !pointer(a[4], &best) || !workspace(a[5], &work, &work_bytes) || !stream(&st))
        return nullptr;
    PyObject* seq = PySequence_Fast(a[1], "encodings must be a sequence");
    if (!seq)
        return nullptr;
    // (more encodings than the library takes: the count is passed on and rejected there, before any is read)
    const Py_ssize_t count_enc = PySequence_Fast_GET_SIZE(seq);
    for (Py_ssize_t i = 0; i < count_enc && i < 16; ++i)
        if (!format(PySequence_Fast_GET_ITEM(seq, i), &enc[i])) {
            Py_DECREF(seq);
            return nullptr;
        }
    Py_DECREF(seq);
    const int64_t elements = x.numel;
    const int32_t n_enc = count_enc > 1000000 ? 1000000 : (int32_t)count_enc;
    const int32_t n_clip = clip.numel > 1000000 ? 1000000 : (int32_t)clip.numel;
    fpq_status status;
    Py_BEGIN_ALLOW_THREADS
    status = fpq_search_format((const float*)xp, elements, enc, n_enc, (const float*)clipp, n_clip, (double*)mse, (int32_t*)best,
                               work, work_bytes, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

// learn_step(w, scale, fmt, alpha, a, reg, lr, grad, loss, workspace) -> status
PyObject* learn_step(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    Shape w, scale, alpha, rows;
    void *wp, *scalep, *alphap, *rowsp, *grad, *loss, *work, *st;
    size_t work_bytes;
    fpq_format fmt;
    float reg, lr;
    if (!arguments(n, 10) || !fp32_cuda(a[0], 2, &w) || !fp32_cuda(a[1], 1, &scale) || !format(a[2], &fmt) ||
        !fp32_cuda(a[3], 2, &alpha) || !fp32_cuda(a[4], 2, &rows) || !real(a[5], &reg) || !real(a[6], &lr) || !pointer(a[0], &wp) ||
        !pointer(a[1], &scalep) || !pointer(a[3], &alphap) || !pointer(a[4], &rowsp) || !pointer(a[7], &grad) ||
        !pointer(a[8], &loss) || !workspace(a[9], &work, &work_bytes) || !stream(&st))
        return nullptr;
    const int64_t M = rows.size[0], N = w.size[0], K = w.size[1];
    if (rows.size[1] != K || alpha.size[0] != N || alpha.size[1] != K || scale.size[0] != N) {
        PyErr_SetString(PyExc_AssertionError, "expected w and alpha [N][K], a [M][K], scale [N]");
        return nullptr;
    }
    fpq_status status;
    Py_BEGIN_ALLOW_THREADS
    status = fpq_round_learn_step((const float*)wp, (const float*)scalep, fmt, (float*)alphap, (const float*)rowsp, M, N, K, reg, lr,
                                  (float*)grad, (double*)loss, work, work_bytes, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

PyMethodDef methods[] = {
    {"linear", (PyCFunction)(void (*)(void))linear, METH_FASTCALL, nullptr},
    {"conv2d", (PyCFunction)(void (*)(void))conv2d, METH_FASTCALL, nullptr},
    {"conv2d_split", (PyCFunction)(void (*)(void))conv2d_split, METH_FASTCALL, nullptr},
    {"search", (PyCFunction)(void (*)(void))search, METH_FASTCALL, nullptr},
    {"learn_step", (PyCFunction)(void (*)(void))learn_step, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fpq_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fpq_torch(void)
{
    g_exp_bits = PyUnicode_InternFromString("exp_bits");
    g_man_bits = PyUnicode_InternFromString("man_bits");
    g_exp_bias = PyUnicode_InternFromString("exp_bias");
    g_sat_mode = PyUnicode_InternFromString("sat_mode");
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_numel = PyUnicode_InternFromString("numel");
    return PyModule_Create(&module);
}
