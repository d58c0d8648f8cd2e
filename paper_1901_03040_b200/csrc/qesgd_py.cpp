// Argument marshalling of the Python binding: one function per entry point that is called per
// round or step.  Each takes the arguments of its C counterpart in order, tensors (anything with
// data_ptr()) or None where that takes a data pointer, and returns its result code.
//
// A codec call on a short vector occupies the GPU for 2 to 4 us; through ctypes its arguments alone
// took 2.1 us (decode) to 4.2 us (encode_batch, sixteen of them), here 0.3 to 0.6 us.
//
// The library is loaded by the Python module (release or debug build), which hands the addresses of
// its functions to bind(); nothing is linked.  A call with an argument that is not taken here goes back
// to that module, which makes it through ctypes: what ctypes converts is accepted, what it refuses is
// refused with its errors.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include "qesgd.h"

namespace {

PyObject *g_data_ptr;   // "data_ptr"
PyObject *g_by_ctypes;  // by_ctypes(name, arguments): the same call through ctypes

// Taken here: integers of any size, of which the low bits count, and what has __index__ (numpy integers,
// tensors of one integer); what has __float__ for a float.
struct Args {
    PyObject *const *a;
    Py_ssize_t n, i;
    bool ok, hand_over;   // hand_over: an argument that is not taken here (no exception is set)
    Args(PyObject *const *args, Py_ssize_t have, Py_ssize_t want) : a(args), n(have), i(0), ok(have == want), hand_over(false)
    {
        if (!ok) PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, have);
    }
    void not_taken()
    {
        PyErr_Clear();
        ok = false;
        hand_over = true;
    }
    uint64_t u64()
    {
        if (!ok) return 0;
        PyObject *const o = a[i++];
        if (PyLong_Check(o)) return PyLong_AsUnsignedLongLongMask(o);
        PyObject *const v = PyNumber_Index(o);
        if (!v) {
            not_taken();
            return 0;
        }
        const uint64_t u = PyLong_AsUnsignedLongLongMask(v);
        Py_DECREF(v);
        return u;
    }
    uint32_t u32() { return (uint32_t)u64(); }
    float f32()
    {
        if (!ok) return 0.0f;
        const double v = PyFloat_AsDouble(a[i++]);
        if (v == -1.0 && PyErr_Occurred()) not_taken();
        return (float)v;
    }
    // address held by an int (the context) ...
    void *address() { return (void *)(uintptr_t)u64(); }
    // ... or by a tensor
    template <typename T>
    T *tensor()
    {
        if (!ok) return nullptr;
        PyObject *const o = a[i++];
        if (o == Py_None) return nullptr;
        PyObject *const p = PyObject_CallMethodNoArgs(o, g_data_ptr);
        if (!p) {
            ok = false;
            return nullptr;
        }
        uint64_t v = 0;
        if (PyLong_Check(p)) v = PyLong_AsUnsignedLongLongMask(p);
        else not_taken();
        Py_DECREF(p);
        return (T *)(uintptr_t)v;
    }
};

#define ENTRIES(X)                                                                                           \
    X(qesgd_encode) X(qesgd_encode_batch) X(qesgd_requantize) X(qesgd_lr_qesgd_step)                         \
    X(qesgd_decode_average_apply) X(qesgd_decode_average_axpy) X(qesgd_decode) X(qesgd_lr_sgd_step)          \
    X(qesgd_lr_gradient) X(qesgd_lr_local_epoch) X(qesgd_lr_local_epoch_batch) X(qesgd_lr_sgd_step_noalloc)
#define DECLARE(name) decltype(&::name) f_##name;
ENTRIES(DECLARE)
#undef DECLARE

// Runs the call without the interpreter lock, as ctypes did.
template <typename F>
PyObject *result(const char *name, Args &args, F call)
{
    if (args.hand_over) {
        PyObject *const all = PyTuple_New(args.n);
        if (!all) return nullptr;
        for (Py_ssize_t i = 0; i < args.n; ++i) PyTuple_SET_ITEM(all, i, Py_NewRef(args.a[i]));
        PyObject *const rc = PyObject_CallFunction(g_by_ctypes, "sO", name, all);
        Py_DECREF(all);
        return rc;
    }
    if (!args.ok) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
#define ENTRY(name, count)                                                                \
    PyObject *py_##name(PyObject *, PyObject *const *args, Py_ssize_t n)                  \
    {                                                                                     \
        Args x(args, n, count);
#define CALL(name, ...)                                                                   \
        return result(#name, x, [&] { return f_##name(__VA_ARGS__); });                          \
    }

ENTRY(qesgd_encode, 14)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *local = x.tensor<const float>(), *anchor = x.tensor<const float>();
    const uint64_t d = x.u64();
    const uint32_t bucket = x.u32(), s = x.u32(), bits = x.u32(), mode = x.u32();
    const float delta = x.f32();
    const uint64_t seed = x.u64();
    const uint32_t worker = x.u32(), epoch = x.u32();
    auto *codes = x.tensor<uint32_t>();
    auto *scales = x.tensor<float>();
CALL(qesgd_encode, ctx, local, anchor, d, bucket, s, bits, mode, delta, seed, worker, epoch, codes, scales)

ENTRY(qesgd_encode_batch, 18)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *local = x.tensor<const float>();
    const uint64_t local_stride = x.u64();
    auto *anchor = x.tensor<const float>();
    const uint64_t d = x.u64();
    const uint32_t K = x.u32(), bucket = x.u32(), s = x.u32(), bits = x.u32(), mode = x.u32();
    const float delta = x.f32();
    const uint64_t seed = x.u64();
    const uint32_t worker0 = x.u32(), epoch = x.u32();
    auto *codes = x.tensor<uint32_t>();
    const uint64_t code_stride = x.u64();
    auto *scales = x.tensor<float>();
    const uint64_t scale_stride = x.u64();
CALL(qesgd_encode_batch, ctx, local, local_stride, anchor, d, K, bucket, s, bits, mode, delta, seed, worker0, epoch,
     codes, code_stride, scales, scale_stride)

ENTRY(qesgd_requantize, 15)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *u = x.tensor<float>();
    auto *anchor = x.tensor<const float>();
    const uint64_t d = x.u64();
    const uint32_t bucket = x.u32(), s = x.u32(), bits = x.u32(), mode = x.u32();
    const float delta = x.f32();
    const uint64_t seed = x.u64();
    const uint32_t worker = x.u32(), step = x.u32();
    auto *zsum = x.tensor<float>();
    auto *codes = x.tensor<uint32_t>();
    auto *scales = x.tensor<float>();
CALL(qesgd_requantize, ctx, u, anchor, d, bucket, s, bits, mode, delta, seed, worker, step, zsum, codes, scales)

ENTRY(qesgd_lr_qesgd_step, 19)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *X = x.tensor<const float>(), *y = x.tensor<const float>();
    const uint32_t m = x.u32();
    const uint64_t d = x.u64();
    const float lr = x.f32();
    auto *u = x.tensor<float>();
    auto *anchor = x.tensor<const float>();
    const uint32_t bucket = x.u32(), s = x.u32(), bits = x.u32(), mode = x.u32();
    const float delta = x.f32();
    const uint64_t seed = x.u64();
    const uint32_t worker = x.u32(), step = x.u32();
    auto *zsum = x.tensor<float>();
    auto *codes = x.tensor<uint32_t>();
    auto *scales = x.tensor<float>();
CALL(qesgd_lr_qesgd_step, ctx, X, y, m, d, lr, u, anchor, bucket, s, bits, mode, delta, seed, worker, step, zsum,
     codes, scales)

ENTRY(qesgd_decode_average_apply, 11)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *param = x.tensor<float>();
    const uint64_t d = x.u64();
    const uint32_t K = x.u32();
    auto *codes = x.tensor<const uint32_t>();
    const uint64_t code_stride = x.u64();
    auto *scales = x.tensor<const float>();
    const uint64_t scale_stride = x.u64();
    const uint32_t bucket = x.u32(), s = x.u32(), bits = x.u32();
CALL(qesgd_decode_average_apply, ctx, param, d, K, codes, code_stride, scales, scale_stride, bucket, s, bits)

ENTRY(qesgd_decode_average_axpy, 12)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *param = x.tensor<float>();
    const uint64_t d = x.u64();
    const uint32_t K = x.u32();
    auto *codes = x.tensor<const uint32_t>();
    const uint64_t code_stride = x.u64();
    auto *scales = x.tensor<const float>();
    const uint64_t scale_stride = x.u64();
    const uint32_t bucket = x.u32(), s = x.u32(), bits = x.u32();
    const float alpha = x.f32();
CALL(qesgd_decode_average_axpy, ctx, param, d, K, codes, code_stride, scales, scale_stride, bucket, s, bits, alpha)

ENTRY(qesgd_decode, 8)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *codes = x.tensor<const uint32_t>();
    auto *scales = x.tensor<const float>();
    const uint64_t d = x.u64();
    const uint32_t bucket = x.u32(), s = x.u32(), bits = x.u32();
    auto *out = x.tensor<float>();
CALL(qesgd_decode, ctx, codes, scales, d, bucket, s, bits, out)

ENTRY(qesgd_lr_sgd_step, 7)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *X = x.tensor<const float>(), *y = x.tensor<const float>();
    const uint32_t m = x.u32();
    const uint64_t d = x.u64();
    const float lr = x.f32();
    auto *u = x.tensor<float>();
CALL(qesgd_lr_sgd_step, ctx, X, y, m, d, lr, u)

ENTRY(qesgd_lr_gradient, 7)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *X = x.tensor<const float>(), *y = x.tensor<const float>();
    const uint32_t m = x.u32();
    const uint64_t d = x.u64();
    auto *w = x.tensor<const float>();
    auto *g = x.tensor<float>();
CALL(qesgd_lr_gradient, ctx, X, y, m, d, w, g)

ENTRY(qesgd_lr_local_epoch, 8)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *X = x.tensor<const float>(), *y = x.tensor<const float>();
    const uint64_t n_local = x.u64(), d = x.u64();
    const uint32_t batch = x.u32();
    const float lr = x.f32();
    auto *u = x.tensor<float>();
CALL(qesgd_lr_local_epoch, ctx, X, y, n_local, d, batch, lr, u)

ENTRY(qesgd_lr_local_epoch_batch, 10)
    auto *ctx = (qesgd_ctx *)x.address();
    auto *X = x.tensor<const float>(), *y = x.tensor<const float>();
    const uint64_t n_local = x.u64(), d = x.u64();
    const uint32_t K = x.u32(), batch = x.u32();
    const float lr = x.f32();
    auto *u = x.tensor<float>();
    const uint64_t u_stride = x.u64();
CALL(qesgd_lr_local_epoch_batch, ctx, X, y, n_local, d, K, batch, lr, u, u_stride)

ENTRY(qesgd_lr_sgd_step_noalloc, 7)
    void *stream = x.address();
    auto *X = x.tensor<const float>(), *y = x.tensor<const float>();
    const uint32_t m = x.u32();
    const uint64_t d = x.u64();
    const float lr = x.f32();
    auto *u = x.tensor<float>();
CALL(qesgd_lr_sgd_step_noalloc, stream, X, y, m, d, lr, u)

// bind({name: address}, by_ctypes): every entry point, before the first call
PyObject *py_bind(PyObject *, PyObject *args)
{
    PyObject *table, *by_ctypes;
    if (!PyArg_ParseTuple(args, "OO", &table, &by_ctypes)) return nullptr;
#define BIND(name)                                                                              \
    {                                                                                           \
        PyObject *v = PyDict_Check(table) ? PyDict_GetItemString(table, #name) : nullptr;       \
        if (!v || !PyLong_Check(v)) return PyErr_Format(PyExc_KeyError, "no address of " #name); \
        f_##name = (decltype(&::name))(uintptr_t)PyLong_AsUnsignedLongLongMask(v);              \
    }
    ENTRIES(BIND)
#undef BIND
    Py_XSETREF(g_by_ctypes, Py_NewRef(by_ctypes));
    Py_RETURN_NONE;
}

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr},
PyMethodDef g_methods[] = {ENTRIES(METHOD){"bind", py_bind, METH_VARARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};
#undef METHOD

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_qesgd_py", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__qesgd_py()
{
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    return g_data_ptr ? PyModule_Create(&g_module) : nullptr;
}
