// The host path of the binding's frequent calls, native: the quantized-matrix object and the marshalling of the linear layer's
// entry points.  A small layer's step is bound by the host (1024 x 192 -> 768: 23 us of device work).  Building the ctypes
// structures and converting their arguments cost more of it than the launches do; here a quantized matrix keeps its C
// description inside the object, and a call reads its arguments straight into the C call.  Python time of a call, without
// the launches, in us (ctypes / native): forward with a quantized weight 10.3 / 5.4, forward of a training step 18.5 / 7.4, backward
// 9.1 / 5.0, of which the allocations of the results are 2.7, 4.1 and 2.7.  1024 x 192 -> 768, whole step: 43 -> 33 us.
// The functions take the address of the library's entry point as their first argument: the library itself is loaded, and
// its absence reported, in binding.py.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <structmember.h>

#include "../../include/mxfp4.h"

namespace {

// ---- quantized matrix: the base of binding.QMat ----
struct Mat {
    PyObject_HEAD
    mxfp4_mat_t m;
    PyObject *buf, *data, *scales;   // one buffer for both (data, scales: views of it, made when asked for) or two tensors
    Py_ssize_t at;                   // where the codes start in buf
    PyObject *q4;                    // what binding.linear_fwd made of it besides (see there); gone once the matrix may have changed
};

int mat_traverse(PyObject *o, visitproc visit, void *arg)
{
    Mat *s = reinterpret_cast<Mat *>(o);
    Py_VISIT(s->buf);
    Py_VISIT(s->data);
    Py_VISIT(s->scales);
    Py_VISIT(s->q4);
    return 0;
}
int mat_clear(PyObject *o)
{
    Mat *s = reinterpret_cast<Mat *>(o);
    Py_CLEAR(s->buf);
    Py_CLEAR(s->data);
    Py_CLEAR(s->scales);
    Py_CLEAR(s->q4);
    return 0;
}
void mat_dealloc(PyObject *o)
{
    PyObject_GC_UnTrack(o);
    mat_clear(o);
    Py_TYPE(o)->tp_free(o);
}

PyObject *g_data_ptr;   // the name of the tensors' method

// Once the tensors of a matrix have been handed out (or came from the caller), its addresses are theirs: a program may give a
// tensor another storage.
bool refresh(Mat *s)
{
    if (s->data && s->data != Py_None) {
        PyObject *a = PyObject_CallMethodNoArgs(s->data, g_data_ptr);
        if (!a) return false;
        s->m.data = reinterpret_cast<void *>((uintptr_t)PyLong_AsUnsignedLongLongMask(a));
        Py_DECREF(a);
    }
    if (s->scales && s->scales != Py_None) {
        PyObject *a = PyObject_CallMethodNoArgs(s->scales, g_data_ptr);
        if (!a) return false;
        s->m.scales = reinterpret_cast<uint8_t *>((uintptr_t)PyLong_AsUnsignedLongLongMask(a));
        Py_DECREF(a);
    }
    return !PyErr_Occurred();
}
PyObject *mat_address(PyObject *o, void *scales)
{
    Mat *s = reinterpret_cast<Mat *>(o);
    return refresh(s) ? PyLong_FromVoidPtr(scales ? (void *)s->m.scales : s->m.data) : nullptr;
}
PyGetSetDef mat_getset[] = {{"data_addr", mat_address, nullptr, nullptr, nullptr}, {"scales_addr", mat_address, nullptr, nullptr, (void *)1}, {nullptr, nullptr, nullptr, nullptr, nullptr}};

PyMemberDef mat_members[] = {
    {"rows", T_LONGLONG, offsetof(Mat, m.rows), 0, nullptr},
    {"cols", T_LONGLONG, offsetof(Mat, m.cols), 0, nullptr},
    {"_buf", T_OBJECT, offsetof(Mat, buf), 0, nullptr},
    {"_data", T_OBJECT, offsetof(Mat, data), 0, nullptr},
    {"_scales", T_OBJECT, offsetof(Mat, scales), 0, nullptr},
    {"_at", T_PYSSIZET, offsetof(Mat, at), 0, nullptr},
    {"_q4", T_OBJECT, offsetof(Mat, q4), 0, nullptr},
    {nullptr, 0, 0, 0, nullptr}};

PyTypeObject mat_type = {PyVarObject_HEAD_INIT(nullptr, 0)};

// ---- arguments of a call ----
struct Args {
    PyObject *const *a;
    bool bad = false;

    uint64_t u64(int i)
    {
        const unsigned long long v = PyLong_AsUnsignedLongLongMask(a[i]);
        if (v == (unsigned long long)-1 && PyErr_Occurred()) bad = true;
        return v;
    }
    int64_t i64(int i) { return (int64_t)u64(i); }
    int32_t i32(int i) { return (int32_t)u64(i); }
    template <class T = void> T *ptr(int i) { return given(i) ? reinterpret_cast<T *>((uintptr_t)u64(i)) : nullptr; }
    bool given(int i) const { return a[i] != Py_None; }
    mxfp4_mat_t mat(int i)
    {
        if (PyObject_TypeCheck(a[i], &mat_type)) {
            Mat *s = reinterpret_cast<Mat *>(a[i]);
            if (!bad && !refresh(s)) bad = true;
            return s->m;
        }
        if (given(i) && !bad) {
            PyErr_SetString(PyExc_TypeError, "a quantized matrix (QMat) is expected");
            bad = true;
        }
        return mxfp4_mat_t{nullptr, nullptr, 0, 0};
    }
    // a matrix that the call writes
    mxfp4_mat_t dst(int i)
    {
        const mxfp4_mat_t m = mat(i);
        if (!bad && given(i)) Py_CLEAR(reinterpret_cast<Mat *>(a[i])->q4);
        return m;
    }
    // Runs the call without the interpreter lock and returns its status.
    template <class F> PyObject *run(F &&f)
    {
        if (bad) return nullptr;
        int32_t s;
        Py_BEGIN_ALLOW_THREADS
        s = f();
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(s);
    }
};

bool counted(const char *name, Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "%s: %zd arguments expected, %zd given", name, want, n);
    return false;
}

Py_ssize_t mat_bytes(int64_t rows, int64_t cols)   // codes and scales in one buffer, both on 256-byte boundaries
{
    const int64_t s = ((rows + 127) >> 7) * ((cols + 127) >> 7) * 512;
    return ((rows * (cols / 2) + 255) & ~int64_t(255)) + (s > 256 ? s : 256);
}

// nbytes(rows, cols, ...) -> bytes of one buffer for all of these matrices
PyObject *h_nbytes(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Args r{a};
    Py_ssize_t sum = 0;
    for (int i = 0; i + 1 < n; i += 2) sum += mat_bytes(r.i64(i), r.i64(i + 1));
    return r.bad ? nullptr : PyLong_FromSsize_t(sum);
}

// place(matrix, buf, address of buf, rows, cols): puts the matrix into buf.
// place(class, buf, address of buf, rows, cols, rows, cols, ...) -> tuple of new matrices, one behind the other in buf.
PyObject *h_place(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    const bool one = n == 5 && PyObject_TypeCheck(a[0], &mat_type);
    if (!one && (n < 5 || (n & 1) == 0 || !PyType_Check(a[0]) || !PyType_IsSubtype(reinterpret_cast<PyTypeObject *>(a[0]), &mat_type))) {
        PyErr_SetString(PyExc_TypeError, "place(matrix or class, buf, address, rows, cols, ...)");
        return nullptr;
    }
    Args r{a};
    uint8_t *p = r.ptr<uint8_t>(2);
    const Py_ssize_t count = (n - 3) / 2;
    PyObject *all = one ? Py_NewRef(Py_None) : PyTuple_New(count);
    if (!all) return nullptr;
    Py_ssize_t at = 0;
    for (int i = 0; i < count; i++) {
        const int64_t rows = r.i64(3 + 2 * i), cols = r.i64(4 + 2 * i);
        PyTypeObject *cls = reinterpret_cast<PyTypeObject *>(a[0]);
        PyObject *o = r.bad ? nullptr : one ? a[0] : cls->tp_alloc(cls, 0);
        if (!o) {
            Py_DECREF(all);
            return nullptr;
        }
        Mat *s = reinterpret_cast<Mat *>(o);
        s->m = mxfp4_mat_t{p + at, p + at + ((rows * (cols / 2) + 255) & ~int64_t(255)), rows, cols};
        Py_XSETREF(s->buf, Py_NewRef(a[1]));
        Py_CLEAR(s->data);
        Py_CLEAR(s->scales);
        s->at = at;
        at += mat_bytes(rows, cols);
        if (!one) PyTuple_SET_ITEM(all, i, o);
    }
    return all;
}

PyObject *h_linear_fwd(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    // entry, x, ldx, m, k, w, n, bias, y, ldy, xq, wq, xq_t, wq_t, seed, scale_mode, epilogue, status, stream
    if (!counted("linear_fwd", n, 19)) return nullptr;
    Args r{a};
    const auto f = reinterpret_cast<decltype(&mxfp4_linear_fwd_ex)>(r.ptr(0));
    mxfp4_linear_ctx_t c{r.mat(10), r.given(5) ? r.dst(11) : r.mat(11), r.mat(12), r.u64(14), r.mat(13), r.u64(14)};
    const void *x = r.ptr(1), *w = r.ptr(5), *bias = r.ptr(7);
    void *y = r.ptr(8), *stream = r.ptr(18);
    const int64_t ldx = r.i64(2), m = r.i64(3), k = r.i64(4), nn = r.i64(6), ldy = r.i64(9);
    const int32_t mode = r.i32(15);
    const auto *epi = r.ptr<const mxfp4_epilogue_t>(16);
    auto *status = r.ptr<uint32_t>(17);
    return r.run([&] { return f(x, ldx, m, k, w, nn, bias, y, ldy, &c, mode, epi, status, stream); });
}

PyObject *h_linear_bwd(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    // entry, dy, lddy, dyq, dyq_t, xq, wq, xq_t, wq_t, ctx seed, seed, scale_mode, dx, lddx, dw, lddw, dw dtype, epilogue, workspace,
    // workspace bytes, status, stream
    if (!counted("linear_bwd", n, 22)) return nullptr;
    Args r{a};
    const auto f = reinterpret_cast<decltype(&mxfp4_linear_bwd_ex)>(r.ptr(0));
    const void *dy = r.ptr(1);
    const bool given = r.given(3), given_t = r.given(4);
    const mxfp4_mat_t dyq = r.mat(3), dyq_t = r.mat(4);
    const mxfp4_linear_ctx_t c{r.mat(5), r.mat(6), r.mat(7), r.u64(9), r.mat(8), r.u64(9)};
    const int64_t lddy = r.i64(2), lddx = r.i64(13), lddw = r.i64(15);
    const uint64_t seed = r.u64(10), ws_bytes = r.u64(19);
    const int32_t mode = r.i32(11), dwt = r.i32(16);
    void *dx = r.ptr(12), *dw = r.ptr(14), *ws = r.ptr(18), *stream = r.ptr(21);
    const auto *epi = r.ptr<const mxfp4_epilogue_t>(17);
    auto *status = r.ptr<uint32_t>(20);
    return r.run([&] {
        return f(dy, lddy, given ? &dyq : nullptr, given_t ? &dyq_t : nullptr, &c, seed, mode, dx, lddx, dw, lddw, dwt, epi, ws, ws_bytes, status, stream);
    });
}

PyObject *h_quantize(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    // entry, x, rows, cols, ld, dst, scale_mode, rounding, seed, stream_id, status, stream
    if (!counted("quantize", n, 12)) return nullptr;
    Args r{a};
    const auto f = reinterpret_cast<decltype(&mxfp4_quantize)>(r.ptr(0));
    const mxfp4_qparams_t qp{r.i32(6), r.i32(7), r.u64(8), (uint32_t)r.u64(9), 0u};
    const void *x = r.ptr(1);
    const int64_t rows = r.i64(2), cols = r.i64(3), ld = r.i64(4);
    const mxfp4_mat_t dst = r.dst(5);
    auto *status = r.ptr<uint32_t>(10);
    void *stream = r.ptr(11);
    return r.run([&] { return f(x, rows, cols, ld, dst, &qp, status, stream); });
}

PyObject *h_quantize_t(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    // entry, x, source matrix, rows, cols, ld, dst, scale_mode, rounding, seed, stream_id, status, stream
    if (!counted("quantize_t", n, 13)) return nullptr;
    Args r{a};
    const auto f = reinterpret_cast<decltype(&mxfp4_quantize_t)>(r.ptr(0));
    const mxfp4_qparams_t qp{r.i32(7), r.i32(8), r.u64(9), (uint32_t)r.u64(10), 0u};
    const void *x = r.ptr(1);
    const bool given = r.given(2);
    const mxfp4_mat_t src = r.mat(2), dst = r.dst(6);
    const int64_t rows = r.i64(3), cols = r.i64(4), ld = r.i64(5);
    auto *status = r.ptr<uint32_t>(11);
    void *stream = r.ptr(12);
    return r.run([&] { return f(x, given ? &src : nullptr, rows, cols, ld, dst, &qp, status, stream); });
}

PyObject *h_qema(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    // entry, w, ema, beta, update, n, k, dst, scale_mode, w_prev | None, wq_prev, dist_w, dist_q, status, stream
    if (!counted("qema_quantize", n, 15)) return nullptr;
    Args r{a};
    const auto f = reinterpret_cast<decltype(&mxfp4_qema_quantize)>(r.ptr(0));
    const double beta = PyFloat_AsDouble(a[3]);
    if (beta == -1.0 && PyErr_Occurred()) return nullptr;
    const void *w = r.ptr(1);
    float *ema = r.ptr<float>(2);
    const int32_t update = r.i32(4), mode = r.i32(8);
    const int64_t nn = r.i64(5), k = r.i64(6);
    const mxfp4_mat_t dst = r.dst(7);
    const bool osc = r.given(9);
    const mxfp4_osc_state_t o{r.ptr(9), r.dst(10), r.ptr<float>(11), r.ptr<float>(12)};
    auto *status = r.ptr<uint32_t>(13);
    void *stream = r.ptr(14);
    return r.run([&] { return f(w, ema, (float)beta, update, nn, k, dst, mode, osc ? &o : nullptr, status, stream); });
}

#define FAST(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fn)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST("nbytes", h_nbytes), FAST("place", h_place), FAST("linear_fwd", h_linear_fwd), FAST("linear_bwd", h_linear_bwd),
                         FAST("quantize", h_quantize), FAST("quantize_t", h_quantize_t), FAST("qema_quantize", h_qema), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__host()
{
    mat_type.tp_name = "paper_2502_20853_b200._host.Mat";
    mat_type.tp_basicsize = sizeof(Mat);
    mat_type.tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_BASETYPE | Py_TPFLAGS_HAVE_GC;
    mat_type.tp_new = PyType_GenericNew;
    mat_type.tp_dealloc = mat_dealloc;
    mat_type.tp_traverse = mat_traverse;
    mat_type.tp_clear = mat_clear;
    mat_type.tp_members = mat_members;
    mat_type.tp_getset = mat_getset;
    if (!g_data_ptr && !(g_data_ptr = PyUnicode_InternFromString("data_ptr"))) return nullptr;
    if (PyType_Ready(&mat_type) < 0) return nullptr;
    PyObject *m = PyModule_Create(&module);
    if (m && (PyModule_AddObjectRef(m, "Mat", reinterpret_cast<PyObject *>(&mat_type)) < 0 || PyModule_AddIntConstant(m, "interface", 2) < 0)) Py_CLEAR(m);
    return m;
}
