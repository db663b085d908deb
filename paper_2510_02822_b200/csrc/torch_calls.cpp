// Native marshalling of the calls a program makes per layer (python module _calls): tensors in, C entry points of
// libflexiq, tensors out.  Nothing here computes.
//
// A small layer takes the GPU about 5 us (two launches); marshalled with ctypes and Python attribute look-ups the same two
// calls took 16 us of host time, of which the launches themselves are 5.  Every function
// answers NotImplemented for whatever is not plainly a tensor or a number (duck-typed buffers, odd number types, tensors
// without storage, failed allocations); the caller then takes the general Python path, which accepts or refuses it.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime_api.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <cmath>
#include <memory>
#include <optional>
#include <vector>

#include "flexiq.h"

namespace {

PyObject *g_error_class = nullptr;

PyObject *not_implemented()
{
    PyErr_Clear();
    Py_RETURN_NOTIMPLEMENTED;
}
// the result, or FlexiqError(code, message) in its place
PyObject *finish(int rc, PyObject *result)
{
    if (rc == FLEXIQ_OK) return result;
    Py_XDECREF(result);
    PyObject *e = PyObject_CallFunction(g_error_class, "is", rc, flexiq_last_error());
    if (e) {
        PyErr_SetObject(g_error_class, e);
        Py_DECREF(e);
    }
    return nullptr;
}
void *current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

struct Refused {};   // leave it to the general path

struct Owned {   // a reference given up on every way out but release()
    PyObject *o = nullptr;
    Owned() = default;
    Owned(const Owned &) = delete;
    ~Owned() { Py_XDECREF(o); }
    PyObject *release() { PyObject *r = o; o = nullptr; return r; }
};

const at::Tensor &tensor(PyObject *o)
{
    if (!THPVariable_Check(o)) throw Refused{};
    return THPVariable_Unpack(o);
}
void *pointer(PyObject *o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
float number(PyObject *o)
{
    if (PyFloat_Check(o)) return (float)PyFloat_AS_DOUBLE(o);
    if (PyLong_Check(o)) {
        const double v = PyLong_AsDouble(o);
        if (v == -1.0 && PyErr_Occurred()) throw Refused{};
        return (float)v;
    }
    throw Refused{};
}
long long whole(PyObject *o)
{
    if (!PyLong_Check(o)) throw Refused{};
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    if (over) throw Refused{};
    return v;
}
int whole32(PyObject *o)
{
    const long long v = whole(o);
    if (v < INT32_MIN || v > INT32_MAX) throw Refused{};
    return (int)v;
}
bool truth(PyObject *o)
{
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw Refused{};
    return v != 0;
}
int dtype_code(const at::Tensor &t)
{
    switch (t.scalar_type()) {
        case at::kFloat: return FLEXIQ_DTYPE_F32;
        case at::kHalf: return FLEXIQ_DTYPE_F16;
        case at::kBFloat16: return FLEXIQ_DTYPE_BF16;
        case at::kChar: return FLEXIQ_DTYPE_I8;
        default: throw Refused{};
    }
}
at::ScalarType out_type(int out_mode)
{
    switch (out_mode) {
        case FLEXIQ_OUT_ACC_I32: return at::kInt;
        case FLEXIQ_OUT_REQUANT_I8: return at::kChar;
        case FLEXIQ_OUT_DEQUANT_F32: return at::kFloat;
        case FLEXIQ_OUT_DEQUANT_F16: return at::kHalf;
        case FLEXIQ_OUT_DEQUANT_BF16: return at::kBFloat16;
        default: throw Refused{};
    }
}
template <class F> PyObject *guarded(F f)
{
    try {
        return f();
    } catch (...) {
        return not_implemented();   // what is refused here is refused before a library call, or where the same calls may be made again
    }
}
// the library call with the interpreter released, as ctypes makes it
template <class F> int released(F f)
{
    PyThreadState *s = PyEval_SaveThread();
    const int rc = f();
    PyEval_RestoreThread(s);
    return rc;
}

struct Calls {
    PyObject_HEAD
    flexiq_layer_t h;
    long long K, N, G;
    int conv, stride, pad, R, S;
    int device;
    PyObject *slabs;   // the Layer's dict {rows: (x4, x8)}
};

// at::empty on the layer's device, by the function it dispatches to (1.4 -> 1.05 us of host time)
at::Tensor device_empty(const Calls *c, at::IntArrayRef size, at::ScalarType type)
{
    return at::detail::empty_cuda(size, type, at::Device(at::kCUDA, (c10::DeviceIndex)c->device), std::nullopt);
}
// the (x4, x8) pair for M rows, allocated once per M (borrowed reference)
PyObject *slabs_of(Calls *c, long long M)
{
    PyObject *key = PyLong_FromLongLong(M);
    if (!key) throw Refused{};
    PyObject *pair = PyDict_GetItemWithError(c->slabs, key);
    if (!pair) {
        if (PyErr_Occurred()) { Py_DECREF(key); throw Refused{}; }
        const long long bytes = std::max(M, 1ll) * c->K + 16;
        at::Tensor x4, x8;
        try {
            x4 = device_empty(c, {bytes}, at::kByte);
            x8 = device_empty(c, {bytes}, at::kChar);
        } catch (...) {
            Py_DECREF(key);
            throw;
        }
        PyObject *a = THPVariable_Wrap(x4), *b = THPVariable_Wrap(x8);
        pair = a && b ? PyTuple_Pack(2, a, b) : nullptr;
        Py_XDECREF(a);
        Py_XDECREF(b);
        const bool stored = pair && PyDict_SetItem(c->slabs, key, pair) == 0;
        Py_XDECREF(pair);   // the dict holds it
        if (!stored) { Py_DECREF(key); throw Refused{}; }
    }
    Py_DECREF(key);
    if (!PyTuple_Check(pair) || PyTuple_GET_SIZE(pair) != 2) throw Refused{};
    return pair;
}

// quantize_lower(X, x_scale, dynamic, slabs) -> (x4, x8, positions or None)
PyObject *calls_quantize_lower(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        if (n != 4) throw Refused{};
        Calls *c = reinterpret_cast<Calls *>(self);
        const at::Tensor &X = tensor(args[0]);
        const int dtype = dtype_code(X);
        const float scale = number(args[1]);
        const bool dynamic = truth(args[2]);
        const long long M = X.numel() / c->K;
        void *x = X.data_ptr();
        PyObject *pair = args[3];
        if (pair == Py_None) pair = slabs_of(c, M);
        else if (!PyTuple_Check(pair) || PyTuple_GET_SIZE(pair) != 2) throw Refused{};
        PyObject *x4 = PyTuple_GET_ITEM(pair, 0), *x8 = PyTuple_GET_ITEM(pair, 1);
        void *p4 = pointer(x4), *p8 = pointer(x8);
        at::Tensor shifts, scratch;
        PyObject *positions = Py_None;
        if (dynamic) {
            shifts = device_empty(c, {c->K / c->G}, at::kByte);
            scratch = device_empty(c, {c->K / c->G}, at::kInt);
            positions = THPVariable_Wrap(shifts);
            if (!positions) throw Refused{};
        } else {
            Py_INCREF(positions);
        }
        PyObject *result = PyTuple_Pack(3, x4, x8, positions);
        Py_DECREF(positions);
        if (!result) throw Refused{};
        void *st = current_stream();
        const int rc = released([&] {
            return flexiq_quantize_lower(c->h, x, dtype, M, scale, dynamic, static_cast<uint8_t *>(p4), static_cast<int8_t *>(p8),
                                         dynamic ? static_cast<uint8_t *>(shifts.data_ptr()) : nullptr,
                                         dynamic ? static_cast<uint32_t *>(scratch.data_ptr()) : nullptr, st);
        });
        return finish(rc, result);
    });
}

// mixed_gemm(x4, x8, M, x_scale, y_scale, out_mode, Y, x_shift) -> Y
PyObject *calls_mixed_gemm(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        if (n != 8) throw Refused{};
        Calls *c = reinterpret_cast<Calls *>(self);
        const void *x4 = pointer(args[0]), *x8 = pointer(args[1]), *xs = pointer(args[7]);
        const long long M = whole(args[2]);
        const float x_scale = number(args[3]), y_scale = number(args[4]);
        const int mode = whole32(args[5]);
        PyObject *Y = args[6];
        void *y;
        if (Y == Py_None) {
            const at::Tensor t = device_empty(c, {M, c->N}, out_type(mode));
            y = t.data_ptr();
            if (!(Y = THPVariable_Wrap(t))) throw Refused{};
        } else {
            y = pointer(Y);
            Py_INCREF(Y);
        }
        void *st = current_stream();
        return finish(released([&] {
            return flexiq_mixed_gemm(c->h, static_cast<const uint8_t *>(x4), static_cast<const int8_t *>(x8), static_cast<const uint8_t *>(xs),
                                     M, x_scale, y_scale, mode, y, st);
        }), Y);
    });
}

void out_size(const Calls *c, int H, int W, long long *P, long long *Q)
{
    const long long h = (long long)H + 2 * c->pad - c->R, w = (long long)W + 2 * c->pad - c->S;
    if (!c->conv || h < 0 || w < 0) throw Refused{};
    *P = h / c->stride + 1;
    *Q = w / c->stride + 1;
}

// mixed_conv(x4, x8, Nb, H, W, x_scale, y_scale, out_mode, Y, x_shift) -> Y
PyObject *calls_mixed_conv(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        if (n != 10) throw Refused{};
        Calls *c = reinterpret_cast<Calls *>(self);
        const void *x4 = pointer(args[0]), *x8 = pointer(args[1]), *xs = pointer(args[9]);
        const int Nb = whole32(args[2]), H = whole32(args[3]), W = whole32(args[4]);
        const float x_scale = number(args[5]), y_scale = number(args[6]);
        const int mode = whole32(args[7]);
        long long P, Q;
        out_size(c, H, W, &P, &Q);
        PyObject *Y = args[8];
        void *y;
        if (Y == Py_None) {
            const at::Tensor t = device_empty(c, {Nb, P, Q, c->N}, out_type(mode));
            y = t.data_ptr();
            if (!(Y = THPVariable_Wrap(t))) throw Refused{};
        } else {
            y = pointer(Y);
            Py_INCREF(Y);
        }
        void *st = current_stream();
        return finish(released([&] {
            return flexiq_mixed_conv(c->h, static_cast<const uint8_t *>(x4), static_cast<const int8_t *>(x8), static_cast<const uint8_t *>(xs),
                                     Nb, H, W, x_scale, y_scale, mode, y, st);
        }), Y);
    });
}

extern PyTypeObject CallsType;
Calls *calls_of(PyObject *o)
{
    if (!PyObject_TypeCheck(o, &CallsType)) throw Refused{};
    return reinterpret_cast<Calls *>(o);
}
// a slab of the next layer for M rows: the caller's, or the next layer's own (new reference)
PyObject *next_slab(PyObject *slab, Calls *next, long long M, void **ptr)
{
    if (slab == Py_None) slab = PyTuple_GET_ITEM(slabs_of(next, M), 0);
    *ptr = pointer(slab);
    Py_INCREF(slab);
    return slab;
}

// mixed_gemm_to_slab(x4, x8, M, x_scale, next, next_x_scale, relu, slab, x_shift, out_order) -> slab
PyObject *calls_mixed_gemm_to_slab(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        if (n != 10) throw Refused{};
        Calls *c = reinterpret_cast<Calls *>(self), *next = calls_of(args[4]);
        const void *x4 = pointer(args[0]), *x8 = pointer(args[1]), *xs = pointer(args[8]);
        const long long M = whole(args[2]);
        const float x_scale = number(args[3]), next_scale = number(args[5]);
        const int relu = truth(args[6]), order = whole32(args[9]);
        void *out;
        PyObject *slab = next_slab(args[7], next, M, &out);
        void *st = current_stream();
        return finish(released([&] {
            return flexiq_mixed_gemm_to_slab(c->h, static_cast<const uint8_t *>(x4), static_cast<const int8_t *>(x8), static_cast<const uint8_t *>(xs),
                                             M, x_scale, next->h, next_scale, relu, order, static_cast<uint8_t *>(out), st);
        }), slab);
    });
}

// mixed_conv_to_slab(x4, x8, Nb, H, W, x_scale, next, next_x_scale, relu, slab, x_shift, out_order) -> slab
PyObject *calls_mixed_conv_to_slab(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        if (n != 12) throw Refused{};
        Calls *c = reinterpret_cast<Calls *>(self), *next = calls_of(args[6]);
        const void *x4 = pointer(args[0]), *x8 = pointer(args[1]), *xs = pointer(args[10]);
        const int Nb = whole32(args[2]), H = whole32(args[3]), W = whole32(args[4]);
        const float x_scale = number(args[5]), next_scale = number(args[7]);
        const int relu = truth(args[8]), order = whole32(args[11]);
        long long P, Q;
        out_size(c, H, W, &P, &Q);
        void *out;
        PyObject *slab = next_slab(args[9], next, Nb * P * Q, &out);
        void *st = current_stream();
        return finish(released([&] {
            return flexiq_mixed_conv_to_slab(c->h, static_cast<const uint8_t *>(x4), static_cast<const int8_t *>(x8), static_cast<const uint8_t *>(xs),
                                             Nb, H, W, x_scale, next->h, next_scale, relu, order, static_cast<uint8_t *>(out), st);
        }), slab);
    });
}

PyObject *calls_set_lowbit_ratio(PyObject *self, PyObject *ratio)
{
    return guarded([&]() -> PyObject * {
        const int rc = flexiq_set_lowbit_ratio(reinterpret_cast<Calls *>(self)->h, number(ratio));
        return finish(rc, Py_NewRef(Py_None));
    });
}

struct Bytes {   // a contiguous buffer of single bytes
    Py_buffer view{};
    explicit Bytes(PyObject *o, Py_ssize_t want)
    {
        if (PyObject_GetBuffer(o, &view, PyBUF_C_CONTIGUOUS) != 0) throw Refused{};
        if (view.itemsize != 1 || view.len != want) { PyBuffer_Release(&view); throw Refused{}; }
    }
    ~Bytes() { PyBuffer_Release(&view); }
    Bytes(const Bytes &) = delete;
    const uint8_t *data() const { return static_cast<const uint8_t *>(view.buf); }
};

// The flagged groups first (index order), then the others; *low = their number.
std::vector<int32_t> selection(const Bytes &flags, Py_ssize_t n_g, int32_t *low)
{
    std::vector<int32_t> perm((size_t)n_g);
    *low = 0;
    for (Py_ssize_t g = 0; g < n_g; ++g)
        if (flags.data()[g]) perm[(size_t)(*low)++] = (int32_t)g;
    int32_t at = *low;
    for (Py_ssize_t g = 0; g < n_g; ++g)
        if (!flags.data()[g]) perm[(size_t)at++] = (int32_t)g;
    return perm;
}

// select_groups([(calls, Wq, flags, positions), ...]): every layer laid out with its flagged groups first, at the ratio that
// makes exactly them low -> None
PyObject *select_groups(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        if (n != 1 || !PyList_Check(args[0])) throw Refused{};
        const Py_ssize_t count = PyList_GET_SIZE(args[0]);
        std::vector<Calls *> calls;
        std::vector<flexiq_layer_t> layers;
        std::vector<const int8_t *> weights;
        std::vector<std::vector<int32_t>> perms;
        std::vector<const int32_t *> perm_ptrs;
        std::vector<std::unique_ptr<Bytes>> positions;
        std::vector<const uint8_t *> position_ptrs;
        std::vector<int> low, before((size_t)count);
        for (Py_ssize_t i = 0; i < count; ++i) {
            PyObject *t = PyList_GET_ITEM(args[0], i);
            if (!PyTuple_Check(t) || PyTuple_GET_SIZE(t) != 4) throw Refused{};
            Calls *c = calls_of(PyTuple_GET_ITEM(t, 0));
            const Py_ssize_t n_g = (Py_ssize_t)(c->K / c->G);
            calls.push_back(c);
            layers.push_back(c->h);
            weights.push_back(static_cast<const int8_t *>(pointer(PyTuple_GET_ITEM(t, 1))));
            const Bytes flags(PyTuple_GET_ITEM(t, 2), n_g);
            int32_t l;
            perms.push_back(selection(flags, n_g, &l));
            perm_ptrs.push_back(perms.back().data());
            low.push_back(l);
            positions.push_back(std::make_unique<Bytes>(PyTuple_GET_ITEM(t, 3), n_g));
            position_ptrs.push_back(positions.back()->data());
        }
        auto set_low = [](const Calls *c, int groups) { return flexiq_set_lowbit_ratio(c->h, (float)((double)groups / (double)(c->K / c->G))); };
        // the ratios first, so that the layouts cut the weight blocks that depend on them; a refused layout leaves both as they were
        int rc = FLEXIQ_OK;
        for (size_t i = 0; i < calls.size() && rc == FLEXIQ_OK; ++i) rc = flexiq_get_max_4bit_ch(calls[i]->h, &before[i]);
        for (size_t i = 0; i < calls.size() && rc == FLEXIQ_OK; ++i) rc = set_low(calls[i], low[i]);
        void *st = current_stream();
        if (rc == FLEXIQ_OK) {
            rc = released([&] { return flexiq_layers_set_group_perm((int)count, layers.data(), weights.data(), perm_ptrs.data(), position_ptrs.data(), st); });
            if (rc != FLEXIQ_OK)
                for (size_t i = 0; i < calls.size(); ++i) set_low(calls[i], before[i] / (int)calls[i]->G);
        }
        return finish(rc, Py_NewRef(Py_None));
    });
}

PyMethodDef calls_methods[] = {
    {"quantize_lower", (PyCFunction)(void (*)(void))calls_quantize_lower, METH_FASTCALL, nullptr},
    {"mixed_gemm", (PyCFunction)(void (*)(void))calls_mixed_gemm, METH_FASTCALL, nullptr},
    {"mixed_conv", (PyCFunction)(void (*)(void))calls_mixed_conv, METH_FASTCALL, nullptr},
    {"mixed_gemm_to_slab", (PyCFunction)(void (*)(void))calls_mixed_gemm_to_slab, METH_FASTCALL, nullptr},
    {"mixed_conv_to_slab", (PyCFunction)(void (*)(void))calls_mixed_conv_to_slab, METH_FASTCALL, nullptr},
    {"set_lowbit_ratio", calls_set_lowbit_ratio, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};

int calls_traverse(PyObject *self, visitproc visit, void *arg)
{
    Py_VISIT(reinterpret_cast<Calls *>(self)->slabs);
    return 0;
}
int calls_clear(PyObject *self)
{
    Py_CLEAR(reinterpret_cast<Calls *>(self)->slabs);
    return 0;
}
void calls_dealloc(PyObject *self)
{
    PyObject_GC_UnTrack(self);
    calls_clear(self);
    Py_TYPE(self)->tp_free(self);
}
// Calls(handle, K, N, G, conv, stride, pad, R, S, device, slabs)
PyObject *calls_new(PyTypeObject *type, PyObject *args, PyObject *)
{
    unsigned long long handle;
    long long K, N, G;
    int conv, stride, pad, R, S, device;
    PyObject *slabs;
    if (!PyArg_ParseTuple(args, "KLLLiiiiiiO!", &handle, &K, &N, &G, &conv, &stride, &pad, &R, &S, &device, &PyDict_Type, &slabs)) return nullptr;
    PyObject *self = type->tp_alloc(type, 0);
    if (!self) return nullptr;
    Calls *c = reinterpret_cast<Calls *>(self);
    c->h = reinterpret_cast<flexiq_layer_t>(handle);
    c->K = K; c->N = N; c->G = G; c->conv = conv; c->stride = stride; c->pad = pad; c->R = R; c->S = S; c->device = device;
    c->slabs = Py_NewRef(slabs);
    return self;
}

PyTypeObject CallsType = {PyVarObject_HEAD_INIT(nullptr, 0)};

// static_preparation(X [rows, C], x_scale, Wq, G, conv, batches, coverage or None)
//   -> (perm, x_shift) on the host and (lo, hi, wmax, score, unused_hist) on the device
PyObject *static_preparation(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        if (n != 7) throw Refused{};
        const at::Tensor &X = tensor(args[0]), &Wq = tensor(args[2]);
        const float scale = number(args[1]);
        const long long G = whole(args[3]), batches = whole(args[5]);
        const bool conv = truth(args[4]), cover = args[6] != Py_None;
        if (X.dim() != 2 || !X.is_contiguous() || !X.is_cuda() || !Wq.is_cuda() || Wq.dim() != (conv ? 4 : 2) || G < 1 || batches < 1) throw Refused{};
        if (cover && !(PyFloat_Check(args[6]) && std::isfinite(PyFloat_AS_DOUBLE(args[6])))) throw Refused{};
        const int dtype = dtype_code(X);
        const long long rows = X.size(0), C = X.size(1), n_g = C / G, step = (rows + batches - 1) / batches;
        if (C < 1 || C > INT32_MAX || n_g < 1) throw Refused{};
        const at::TensorOptions opt = at::TensorOptions().device(X.device());
        const at::Tensor work = at::empty({3 * C + 1}, opt.dtype(at::kInt));   // lo, hi, wmax and a scratch word
        // perm int32 [n_g], then x_shift [n_g]: page-locked, written by the device, so that the stream's end is all there is to wait for
        // (one size for most layers: the allocator keeps a block per power of two, and the first of each is a call to the driver)
        const at::Tensor order = at::empty({std::max(5 * n_g, 4096ll)}, at::TensorOptions().dtype(at::kByte).pinned_memory(true));
        void *order_dev = nullptr;
        if (cudaHostGetDevicePointer(&order_dev, order.data_ptr(), 0) != cudaSuccess) { cudaGetLastError(); throw Refused{}; }
        const at::Tensor score = at::empty({n_g}, opt.dtype(at::kLong)), unused = at::empty({5}, opt.dtype(at::kInt));
        at::Tensor hist;
        if (cover) hist = at::empty({C, 256}, opt.dtype(at::kInt));
        const char *x = static_cast<const char *>(X.data_ptr());
        const int8_t *w = static_cast<const int8_t *>(Wq.data_ptr());
        const int N = (int)(conv ? Wq.size(0) : Wq.size(1)), taps = (int)(conv ? Wq.size(1) * Wq.size(2) : 1);
        int32_t *lo_p = work.data_ptr<int32_t>(), *hi_p = lo_p + C, *wmax_p = hi_p + C;
        uint32_t *hist_p = cover ? reinterpret_cast<uint32_t *>(hist.data_ptr<int32_t>()) : nullptr;
        int64_t *score_p = score.data_ptr<int64_t>();
        int32_t *unused_p = unused.data_ptr<int32_t>();
        int32_t *perm_p = static_cast<int32_t *>(order_dev);
        uint8_t *shift_p = static_cast<uint8_t *>(order_dev) + 4 * n_g;
        const long long tail = cover ? (long long)((double)rows * (1.0 - PyFloat_AS_DOUBLE(args[6])) / 2.0) : 0;
        void *st = current_stream();
        const int rc = released([&] {
            int r = FLEXIQ_OK;
            const bool rows_too = batches == 1 && !cover;   // one launch for everything
            for (long long b = 0; b < batches && r == FLEXIQ_OK && !rows_too; ++b) {
                const long long from = std::min(b * step, rows), part = std::min(step, rows - from);
                const void *p = x + (size_t)from * C * X.element_size();
                r = cover ? flexiq_calib_channel_histogram(p, dtype, part, (int)C, scale, b > 0, hist_p, st)
                          : flexiq_calib_channel_ranges(p, dtype, part, (int)C, scale, b > 0, lo_p, hi_p, st);
            }
            if (r == FLEXIQ_OK && (cover || rows_too)) {
                r = flexiq_calib_static(x, dtype, rows, scale, hist_p, tail, (int)C, w, conv, N, taps, (int)G, lo_p, perm_p, shift_p, score_p, unused_p, st);
            } else if (r == FLEXIQ_OK) {
                r = flexiq_calib_weight_absmax(w, conv, (int)C, N, taps, wmax_p, st);
                if (r == FLEXIQ_OK) r = flexiq_calib_prepare(lo_p, hi_p, wmax_p, (int)C, (int)G, perm_p, shift_p, score_p, unused_p, st);
            }
            return r;
        });
        if (rc != FLEXIQ_OK) return finish(rc, nullptr);
        // while the device works: the results' tensors
        Owned result;
        char *perm_host = nullptr, *shift_host = nullptr;
        try {
            const at::Tensor p = at::empty({n_g}, at::kInt), s = at::empty({n_g}, at::kByte);
            perm_host = static_cast<char *>(p.data_ptr());
            shift_host = static_cast<char *>(s.data_ptr());
            const at::Tensor rest[] = {work.narrow(0, 0, C), work.narrow(0, C, C), work.narrow(0, 2 * C, C), score, unused};
            result.o = PyTuple_New(7);
            if (result.o) {
                PyTuple_SET_ITEM(result.o, 0, THPVariable_Wrap(p));
                PyTuple_SET_ITEM(result.o, 1, THPVariable_Wrap(s));
                for (int i = 0; i < 5; ++i) PyTuple_SET_ITEM(result.o, 2 + i, THPVariable_Wrap(rest[i]));
                for (int i = 0; i < 7; ++i)
                    if (!PyTuple_GET_ITEM(result.o, i)) { Py_CLEAR(result.o); break; }
            }
        } catch (...) {
            Py_CLEAR(result.o);
        }
        const int cuda = released([&] { return (int)cudaStreamSynchronize(static_cast<cudaStream_t>(st)); });   // whatever happened: `order` is written until then
        if (cuda) {
            cudaGetLastError();   // reported here, not at whatever torch launches next
            PyErr_SetString(PyExc_RuntimeError, cudaGetErrorString((cudaError_t)cuda));
            return nullptr;
        }
        if (!result.o) {
            if (PyErr_Occurred()) return nullptr;   // the interpreter's own error (no memory) is the caller's to see
            throw Refused{};                        // torch's: the general path makes the calls again, into tensors of its own
        }
        const char *host = static_cast<const char *>(order.data_ptr());
        std::copy(host, host + 4 * n_g, perm_host);
        std::copy(host + 4 * n_g, host + 5 * n_g, shift_host);
        return result.release();
    });
}

// sq_distance_i8(A, B, out, index): out[index] = sum (A - B)^2 -> None
PyObject *sq_distance(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        if (n != 4) throw Refused{};
        const at::Tensor &A = tensor(args[0]), &B = tensor(args[1]), &out = tensor(args[2]);
        const long long i = whole(args[3]);
        if (A.numel() != B.numel() || out.scalar_type() != at::kLong || out.dim() != 1 || i < 0 || i >= out.size(0) || !out.is_contiguous()) throw Refused{};
        const int8_t *a = static_cast<const int8_t *>(A.data_ptr()), *b = static_cast<const int8_t *>(B.data_ptr());
        int64_t *o = out.data_ptr<int64_t>() + i;
        const long long count = A.numel();
        void *st = current_stream();
        return finish(released([&] { return flexiq_sq_distance_i8(a, b, count, o, st); }), Py_NewRef(Py_None));
    });
}

PyObject *set_error_class(PyObject *, PyObject *cls)
{
    Py_XSETREF(g_error_class, Py_NewRef(cls));
    Py_RETURN_NONE;
}

PyMethodDef module_methods[] = {
    {"static_preparation", (PyCFunction)(void (*)(void))static_preparation, METH_FASTCALL, nullptr},
    {"select_groups", (PyCFunction)(void (*)(void))select_groups, METH_FASTCALL, nullptr},
    {"sq_distance_i8", (PyCFunction)(void (*)(void))sq_distance, METH_FASTCALL, nullptr},
    {"set_error_class", set_error_class, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, module_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void)
{
    CallsType.tp_name = "paper_2510_02822_b200._calls.Calls";
    CallsType.tp_basicsize = sizeof(Calls);
    CallsType.tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_GC;
    CallsType.tp_new = calls_new;
    CallsType.tp_dealloc = calls_dealloc;
    CallsType.tp_traverse = calls_traverse;
    CallsType.tp_clear = calls_clear;
    CallsType.tp_free = PyObject_GC_Del;
    CallsType.tp_methods = calls_methods;
    if (PyType_Ready(&CallsType) < 0) return nullptr;
    PyObject *m = PyModule_Create(&module_def);
    if (!m) return nullptr;
    if (PyModule_AddObjectRef(m, "Calls", reinterpret_cast<PyObject *>(&CallsType)) < 0) { Py_DECREF(m); return nullptr; }
    return m;
}
