// Marshalling of the Python calls: tensors, descriptors, integers and the current stream to the C ABI's arguments.
//
// A product of a small layer takes 3.0 us on the GPU and 3.6 us for the C call that enqueues it, so what Python adds to a call
// bounds it.  Through ctypes that was 2.1 us: a handle and an XDesc built field by field, data_ptr() of up to nine tensors, two
// calls for the stream.  No argument is judged here: the library does that, and its status comes back as an integer.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>
#include <tuple>
#include <type_traits>
#include <utility>

#include "bsp.h"

namespace {

struct Failed {};                                              // a Python exception is set

// ---- one Python object to one C argument ----

void *address(PyObject *v)                                     // (takes the reference)
{
    if (v == nullptr) throw Failed();
    void *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) throw Failed();
    return p;
}

void *pointer(PyObject *o)
{
    if (o == Py_None) return nullptr;
    if (THPVariable_CheckExact(o)) return THPVariable_Unpack(o).data_ptr();
    return address(PyObject_CallMethod(o, "data_ptr", nullptr));
}

// An int, as ctypes takes it: nothing that only converts to one.
long long integer(PyObject *o)
{
    if (!PyLong_Check(o)) {
        PyErr_Format(PyExc_TypeError, "int expected instead of %.200s instance", Py_TYPE(o)->tp_name);
        throw Failed();
    }
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
    if (PyErr_Occurred()) throw Failed();
    return (long long)v;
}

// A layer's number of blocks, which may be any object that int() takes (a mask's sum).
long long count(PyObject *o)
{
    if (PyLong_Check(o)) return integer(o);
    PyObject *v = PyNumber_Long(o);
    if (v == nullptr) throw Failed();
    const unsigned long long n = PyLong_AsUnsignedLongLongMask(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) throw Failed();
    return (long long)n;
}

void *stream(PyObject *o)
{
    if (o == Py_None) return (void *)c10::cuda::getCurrentCUDAStream().stream();
    return address(PyObject_GetAttrString(o, "cuda_stream"));
}

// A ctypes structure: its own memory, which the caller's reference keeps for the call.
PyTypeObject *c_data;                                          // the base of all ctypes objects, set by bind()
template <class T>
T *structure(PyObject *o)
{
    if (!PyObject_TypeCheck(o, c_data)) {
        PyErr_Format(PyExc_TypeError, "a ctypes structure expected instead of %.200s instance", Py_TYPE(o)->tp_name);
        throw Failed();
    }
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Failed();
    void *p = view.buf;
    const bool whole = view.len == (Py_ssize_t)sizeof(T);
    PyBuffer_Release(&view);
    if (!whole) {
        PyErr_SetString(PyExc_TypeError, "not the descriptor that this argument takes");
        throw Failed();
    }
    return (T *)p;
}

template <class T>
T convert(PyObject *o)
{
    if constexpr (std::is_same_v<T, const bsp_wdesc *> || std::is_same_v<T, const bsp_xdesc *> || std::is_same_v<T, const bsp_bcsr *>)
        return structure<std::remove_pointer_t<T>>(o);
    else if constexpr (std::is_pointer_v<T>)
        return (T)pointer(o);
    else
        return (T)integer(o);
}

// ---- the library's functions: addresses, set by bind() ----

decltype(&bsp_mask) f_mask;
decltype(&bsp_compact) f_compact;
decltype(&bsp_gemm) f_gemm;
decltype(&bsp_conv2d) f_conv2d;
decltype(&bsp_gemm_q8) f_gemm_q8;
decltype(&bsp_conv2d_q8) f_conv2d_q8;
decltype(&bsp_conv2d_chain) f_chain;
decltype(&bsp_conv2d_chain_q8) f_chain_q8;
decltype(&bsp_spgemm) f_spgemm;

// Runs a body that may raise; the status of the library's call as a Python integer.
template <class F>
PyObject *guarded(F body)
{
    try {
        return PyLong_FromLong((long)body());
    } catch (const Failed &) {
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

bool count_is(Py_ssize_t n, Py_ssize_t want)
{
    if (n != want) PyErr_Format(PyExc_TypeError, "%zd arguments for a call of %zd", n, want);
    return n == want;
}

// The GIL is free during the library's call, as other threads may enqueue on streams of their own.
template <class R, class... A, class... B>
R enqueue(R (*f)(A...), B... b)
{
    PyThreadState *state = PyEval_SaveThread();
    const R r = f(b...);
    PyEval_RestoreThread(state);
    return r;
}

template <class R, class... A, size_t... k>
R spread(R (*f)(A...), PyObject *const *args, std::index_sequence<k...>)
{
    constexpr size_t last = sizeof...(A) - 1;                  // (the last argument of every call is its stream)
    const std::tuple<A...> a{[&] {
        if constexpr (k == last) return (A)stream(args[k]);
        else return convert<A>(args[k]);
    }()...};
    return enqueue(f, std::get<k>(a)...);
}

template <class R, class... A>
PyObject *plain(R (*f)(A...), PyObject *const *args, Py_ssize_t n)
{
    if (!count_is(n, sizeof...(A))) return nullptr;
    return guarded([&] { return spread(f, args, std::make_index_sequence<sizeof...(A)>()); });
}

#define BSP_CALL(name, f) \
    PyObject *name(PyObject *, PyObject *const *args, Py_ssize_t n) { return plain(f, args, n); }
BSP_CALL(mask, f_mask)
BSP_CALL(compact, f_compact)
BSP_CALL(gemm, f_gemm)
BSP_CALL(conv2d, f_conv2d)
BSP_CALL(gemm_q8, f_gemm_q8)
BSP_CALL(conv2d_q8, f_conv2d_q8)
BSP_CALL(conv2d_chain, f_chain)
BSP_CALL(conv2d_chain_q8, f_chain_q8)
BSP_CALL(spgemm, f_spgemm)
#undef BSP_CALL

// ---- the calls of SparseLayer: the handle, the input's shape and the output's type are read here ----
// What is not a plain tensor of the expected rank and type gets None for an answer and is read in Python, as every object with a
// shape, a type and data_ptr() was, with the errors that come from there.

bsp_bcsr handle_of(PyObject *const *a)                         // row_ptr, col_idx, payload, packed, nnz
{
    bsp_bcsr w;
    w.row_ptr = (const int32_t *)pointer(a[0]);
    w.col_idx = (const int32_t *)pointer(a[1]);
    w.payload = pointer(a[2]);
    w.packed = pointer(a[3]);
    w.nnz = count(a[4]);
    return w;
}

bool plain_input(PyObject *x, int64_t dims)
{
    return THPVariable_CheckExact(x) && THPVariable_Unpack(x).dim() == dims;
}

bool type_of(PyObject *y, bsp_dtype &t)
{
    if (!THPVariable_CheckExact(y)) return false;
    switch (THPVariable_Unpack(y).scalar_type()) {
    case at::kFloat: t = BSP_F32; return true;
    case at::kBFloat16: t = BSP_BF16; return true;
    case at::kChar: t = BSP_I8; return true;
    case at::kInt: t = BSP_I32; return true;
    default: return false;
    }
}

// fill_handle(Bcsr, row_ptr, col_idx, payload, packed, nnz): the fields of a handle
PyObject *fill_handle(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!count_is(n, 6)) return nullptr;
    return guarded([&] {
        *structure<bsp_bcsr>(a[0]) = handle_of(a + 1);
        return 0;
    });
}

// layer_gemm(q8, wd, row_ptr, col_idx, payload, packed, nnz, X, bias, shift, Y, ws, stream); shift is read where q8 is true
PyObject *layer_gemm(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!count_is(n, 13)) return nullptr;
    const bool q8 = *a++ == Py_True;
    bsp_dtype yt = BSP_I8;
    if (!plain_input(a[6], 2) || (!q8 && !type_of(a[9], yt))) Py_RETURN_NONE;
    return guarded([&] {
        const bsp_wdesc *wd = structure<bsp_wdesc>(a[0]);
        const bsp_bcsr w = handle_of(a + 1);
        const int64_t P = THPVariable_Unpack(a[6]).size(0);
        const void *X = pointer(a[6]), *bias = pointer(a[7]);
        void *Y = pointer(a[9]), *ws = pointer(a[10]);
        if (q8)
            return enqueue(f_gemm_q8, wd, &w, X, P, (const int32_t *)bias, (const int32_t *)pointer(a[8]), (int8_t *)Y, ws, stream(a[11]));
        return enqueue(f_gemm, wd, &w, X, P, bias, Y, yt, ws, stream(a[11]));
    });
}

// layer_conv2d(q8, wd, row_ptr, col_idx, payload, packed, nnz, X, bias, shift, Y, stride_h, stride_w, pad_h, pad_w, ws, stream)
PyObject *layer_conv2d(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!count_is(n, 17)) return nullptr;
    const bool q8 = *a++ == Py_True;
    bsp_dtype yt = BSP_I8;
    if (!plain_input(a[6], 4) || (!q8 && !type_of(a[9], yt))) Py_RETURN_NONE;
    return guarded([&] {
        const bsp_wdesc *wd = structure<bsp_wdesc>(a[0]);
        const bsp_bcsr w = handle_of(a + 1);
        const at::Tensor &x = THPVariable_Unpack(a[6]);
        bsp_xdesc xd;
        xd.N = (int)x.size(0);
        xd.L = (int)x.size(1);
        xd.J = (int)x.size(2);
        xd.stride_h = (int)integer(a[10]);
        xd.stride_w = (int)integer(a[11]);
        xd.pad_h = (int)integer(a[12]);
        xd.pad_w = (int)integer(a[13]);
        const void *X = pointer(a[6]), *bias = pointer(a[7]);
        void *Y = pointer(a[9]), *ws = pointer(a[14]);
        if (q8)
            return enqueue(f_conv2d_q8, wd, &w, &xd, X, (const int32_t *)bias, (const int32_t *)pointer(a[8]), (int8_t *)Y, ws, stream(a[15]));
        return enqueue(f_conv2d, wd, &w, &xd, X, bias, Y, yt, ws, stream(a[15]));
    });
}

// bind(c_data, mask, compact, gemm, conv2d, gemm_q8, conv2d_q8, chain, chain_q8, spgemm): the base of ctypes objects and the addresses
// of the loaded library's functions
PyObject *bind(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!count_is(n, 10)) return nullptr;
    return guarded([&] {
        if (!PyType_Check(a[0])) {
            PyErr_SetString(PyExc_TypeError, "not a type");
            throw Failed();
        }
        Py_INCREF(a[0]);                                       // (kept as long as the module is)
        c_data = (PyTypeObject *)a[0];
        f_mask = (decltype(f_mask))integer(a[1]);
        f_compact = (decltype(f_compact))integer(a[2]);
        f_gemm = (decltype(f_gemm))integer(a[3]);
        f_conv2d = (decltype(f_conv2d))integer(a[4]);
        f_gemm_q8 = (decltype(f_gemm_q8))integer(a[5]);
        f_conv2d_q8 = (decltype(f_conv2d_q8))integer(a[6]);
        f_chain = (decltype(f_chain))integer(a[7]);
        f_chain_q8 = (decltype(f_chain_q8))integer(a[8]);
        f_spgemm = (decltype(f_spgemm))integer(a[9]);
        return 0;
    });
}

#define BSP_DEF(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {BSP_DEF(bind), BSP_DEF(mask), BSP_DEF(compact), BSP_DEF(gemm), BSP_DEF(conv2d), BSP_DEF(gemm_q8), BSP_DEF(conv2d_q8),
                         BSP_DEF(conv2d_chain), BSP_DEF(conv2d_chain_q8), BSP_DEF(spgemm), BSP_DEF(fill_handle), BSP_DEF(layer_gemm),
                         BSP_DEF(layer_conv2d), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_bspcall", "Argument marshalling of bsp.py.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}   // namespace

PyMODINIT_FUNC PyInit__bspcall(void) { return PyModule_Create(&module_def); }
