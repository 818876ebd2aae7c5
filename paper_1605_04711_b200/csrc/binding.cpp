// CPython binding of the C ABI (include/twn.h): one function per entry point, called by twn.py.
//
// The calls of this library take microseconds on the device, so what a call costs on the host decides
// how fast small layers run.  Marshalling through ctypes cost 7 us per call (a c_int64 object per integer,
// four attribute reads per tensor, 3.2 us for torch.cuda.current_stream()); here the arguments are read
// from the interpreter's own vector, tensors through torch's C++ object and the stream through c10, which
// takes well under a microsecond.  As with ctypes the interpreter lock is released during the call.
//
// A function takes the arguments of its entry point in order, except that a workspace's size is read from
// its tensor.  Pointers are CUDA tensors or None; descriptors and epilogues are objects with the buffer
// protocol (ctypes structures); the stream is None (torch's current stream), a stream object or an integer.
// It returns the status code.
#include <Python.h>

#include <tuple>
#include <type_traits>
#include <utility>
#include <vector>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "twn.h"

namespace {

struct PyError {};      // a Python exception has been set

[[noreturn]] void type_error(const char *what)
{
    PyErr_SetString(PyExc_TypeError, what);
    throw PyError{};
}

struct Args {
    PyObject *const *v;
    Py_ssize_t n, next;
    size_t last_bytes;      // size of the tensor that was read last
    PyObject *take()
    {
        if (next >= n) type_error("too few arguments");
        return v[next++];
    }
};

void *tensor_ptr(PyObject *o, size_t *bytes)
{
    if (o == Py_None) { *bytes = 0; return nullptr; }
    if (!THPVariable_Check(o)) type_error("expected a torch tensor or None");
    const at::Tensor &t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) {
        PyErr_SetString(PyExc_AssertionError, "device tensors must be contiguous CUDA tensors");
        throw PyError{};
    }
    *bytes = t.nbytes();
    return t.data_ptr();
}

// The object outlives the call, so the buffer may be given back before its address is used.
const void *struct_ptr(PyObject *o, size_t size, bool optional)
{
    if (o == Py_None) {
        if (optional) return nullptr;
        type_error("a descriptor is needed");
    }
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw PyError{};
    const void *p = b.buf;
    const bool fits = (size_t)b.len == size;
    PyBuffer_Release(&b);
    if (!fits) type_error("structure of another size");
    return p;
}

twn_stream_t stream_of(PyObject *o)
{
    if (o == Py_None) return reinterpret_cast<twn_stream_t>(c10::cuda::getCurrentCUDAStream().stream());
    PyObject *h = PyLong_Check(o) ? Py_NewRef(o) : PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw PyError{};
    void *p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!p && PyErr_Occurred()) throw PyError{};
    return static_cast<twn_stream_t>(p);
}

long long integer_of(PyObject *o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyError{};
    return v;
}

double real_of(PyObject *o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PyError{};
    return v;
}

template <typename T> T get(Args &a)
{
    if constexpr (std::is_same_v<T, size_t>) return a.last_bytes;       // workspace_bytes follows its workspace
    else if constexpr (std::is_same_v<T, twn_stream_t>) return stream_of(a.next < a.n ? a.take() : Py_None);
    else if constexpr (std::is_same_v<T, const twn_conv_desc_t *>)
        return static_cast<T>(struct_ptr(a.take(), sizeof(twn_conv_desc_t), false));
    else if constexpr (std::is_same_v<T, const twn_epilogue_t *>)
        return static_cast<T>(struct_ptr(a.take(), sizeof(twn_epilogue_t), true));
    else if constexpr (std::is_pointer_v<T>) return static_cast<T>(tensor_ptr(a.take(), &a.last_bytes));
    else if constexpr (std::is_floating_point_v<T>) return static_cast<T>(real_of(a.take()));
    else return static_cast<T>(integer_of(a.take()));
}

template <typename F, typename Tuple> PyObject *finish(F fn, Tuple &&t)
{
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = std::apply(fn, t);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

template <typename... A> PyObject *invoke(int (*fn)(A...), Args &a)
{
    std::tuple<A...> t{get<A>(a)...};       // braces: left to right
    if (a.next != a.n) type_error("too many arguments");
    return finish(fn, t);
}

template <auto Fn> PyObject *entry(PyObject *, PyObject *const *v, Py_ssize_t n)
{
    try {
        Args a{v, n, 0, 0};
        return invoke(Fn, a);
    } catch (const PyError &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// ---- batched calls: a list of tuples, one per tensor ----------------------------------------
template <typename Item> void read_item(Args &a, Item *it);
template <> void read_item(Args &a, twn_ternarize_item_t *it)       // (W, rows, cols, stats, packed, ld_codes, codes_i8)
{
    it->W = get<const float *>(a);
    it->rows = get<int64_t>(a);
    it->cols = get<int64_t>(a);
    it->stats = get<twn_stats_t *>(a);
    it->packed = get<uint32_t *>(a);
    it->ld_codes = get<int64_t>(a);
    it->codes_i8 = get<int8_t *>(a);
}
template <> void read_item(Args &a, twn_sgd_item_t *it)             // (W, dW, V, stats_next)
{
    it->W = get<float *>(a);
    it->n = (int64_t)(a.last_bytes / sizeof(float));
    for (const float **p : {&it->dW, const_cast<const float **>(&it->V)}) {
        *p = get<const float *>(a);
        if ((int64_t)(a.last_bytes / sizeof(float)) != it->n) {
            PyErr_SetString(PyExc_AssertionError, "W, dW and V have the same number of elements");
            throw PyError{};
        }
    }
    it->stats_next = get<twn_stats_t *>(a);
}
template <> void read_item(Args &a, twn_transpose_item_t *it)       // (packed_fwd, ld_fwd, desc, packed_bwd, ld_bwd)
{
    it->packed_fwd = get<const uint32_t *>(a);
    it->ld_fwd = get<int64_t>(a);
    it->desc = *get<const twn_conv_desc_t *>(a);
    it->packed_bwd = get<uint32_t *>(a);
    it->ld_bwd = get<int64_t>(a);
}

template <typename Item, typename... A> PyObject *invoke_batch(int (*fn)(const Item *, int, A...), Args &a)
{
    PyObject *seq = PySequence_Fast(a.take(), "expected a list of tuples");
    if (!seq) throw PyError{};
    std::vector<Item> items((size_t)PySequence_Fast_GET_SIZE(seq));
    try {
        for (size_t i = 0; i < items.size(); ++i) {
            PyObject *row = PySequence_Fast_GET_ITEM(seq, (Py_ssize_t)i);
            if (!PyTuple_Check(row) && !PyList_Check(row)) type_error("expected a list of tuples");
            Args ra{PySequence_Fast_ITEMS(row), PySequence_Fast_GET_SIZE(row), 0, 0};
            read_item(ra, &items[i]);
            if (ra.next != ra.n) type_error("an item has too many fields");
        }
    } catch (...) {
        Py_DECREF(seq);
        throw;
    }
    Py_DECREF(seq);
    std::tuple<const Item *, int, A...> t{items.data(), (int)items.size(), get<A>(a)...};
    if (a.next != a.n) type_error("too many arguments");
    return finish(fn, t);
}

template <auto Fn> PyObject *entry_batch(PyObject *, PyObject *const *v, Py_ssize_t n)
{
    try {
        Args a{v, n, 0, 0};
        return invoke_batch(Fn, a);
    } catch (const PyError &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

#define TWN_ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<twn_##name>)), METH_FASTCALL, nullptr}
#define TWN_BATCH(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry_batch<twn_##name>)), METH_FASTCALL, nullptr}

PyMethodDef methods[] = {
    TWN_ENTRY(ternarize), TWN_ENTRY(ternarize_static), TWN_ENTRY(ternarize_codes), TWN_ENTRY(ternarize_rows), TWN_ENTRY(rows_scale),
    TWN_ENTRY(sgd_update), TWN_ENTRY(pack), TWN_ENTRY(unpack), TWN_ENTRY(transpose_codes),
    TWN_ENTRY(gemm), TWN_ENTRY(conv2d_fwd), TWN_ENTRY(conv2d_fwd_maxpool), TWN_ENTRY(conv2d_fwd_image), TWN_ENTRY(conv2d_fwd_bn), TWN_ENTRY(bn_finalize), TWN_ENTRY(conv2d_bwd_data),
    TWN_ENTRY(conv2d_bwd_weight), TWN_ENTRY(conv2d_fwd_folded), TWN_ENTRY(conv2d_bwd_weight_folded),
    TWN_ENTRY(binarize), TWN_ENTRY(unpack_b1), TWN_ENTRY(transpose_codes_b1), TWN_ENTRY(gemm_b1), TWN_ENTRY(conv2d_fwd_b1),
    TWN_ENTRY(conv2d_bwd_data_b1),
    TWN_ENTRY(im2col), TWN_ENTRY(fold_input), TWN_ENTRY(fold_codes), TWN_ENTRY(maxpool2d_fwd), TWN_ENTRY(maxpool2d_bwd),
    TWN_ENTRY(maxpool2d_bwd_act), TWN_ENTRY(avgpool_fwd), TWN_ENTRY(avgpool_bwd), TWN_ENTRY(act_bwd),
    TWN_BATCH(ternarize_batch), TWN_BATCH(ternarize_codes_batch), TWN_BATCH(sgd_update_batch), TWN_BATCH(transpose_codes_batch),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_twn", "Entry points of libtwn.so.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__twn(void) { return PyModule_Create(&module_def); }
