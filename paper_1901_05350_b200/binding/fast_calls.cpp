// The op calls of the Python binding, marshalled in C++.
//
// A ctypes call with its argument structs, torch.empty and the stream lookup cost 12-16 us of host time, several times
// what the launch itself takes and more than most small ops run on the GPU; the same steps on the C++ side of torch take
// about 2 us.  Every function takes the context's handle as an integer and returns the output tensor, or None whenever an
// argument is not the plain case (contiguous fp32 CUDA tensors of rank 1..4, whole-number options): the caller then takes
// the ctypes path, which raises what there is to raise.  An error that the library reports is raised from here and the
// call is not repeated: a model run, or a call that packs or transposes an operand first, may have enqueued a part of it.
// The library is called through addresses that the caller hands over once, so both paths use one copy of it.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "tfjsb.h"

namespace {

#define FAST_CALLS(X)                                                                                                        \
    X(tfjsb_matmul) X(tfjsb_batch_matmul) X(tfjsb_conv2d) X(tfjsb_depthwise_conv2d) X(tfjsb_avg_pool) X(tfjsb_max_pool)       \
    X(tfjsb_binary) X(tfjsb_softmax) X(tfjsb_bias_act) X(tfjsb_conv2d_backprop_input) X(tfjsb_conv2d_backprop_filter)         \
    X(tfjsb_depthwise_conv2d_backprop_input) X(tfjsb_depthwise_conv2d_backprop_filter) X(tfjsb_act_backprop)                  \
    X(tfjsb_bias_backprop) X(tfjsb_run_model) X(tfjsb_model_layer_output_f32) X(tfjsb_model_layer_shape) X(tfjsb_window_out_shape)       \
    X(tfjsb_last_error)
#define DECLARE(name) decltype(&::name) p_##name = nullptr;
FAST_CALLS(DECLARE)
#undef DECLARE
PyObject* error_type = nullptr;  // called with (status, message)

// An argument list read from left to right; `ok` turns false at the first argument that is not the plain case.
struct Args {
    PyObject* const* at;
    PyObject* const* end;
    bool ok;
    Args(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) : at(args), end(args + n), ok(n == want) {}

    PyObject* next() { return ok ? *at++ : nullptr; }
    long long integer() {
        PyObject* o = next();
        if (!o || !PyLong_Check(o)) { ok = false; return 0; }  // bool is a PyLong
        int overflow = 0;
        const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
        if (overflow) ok = false;
        return v;
    }
    void* handle() {
        PyObject* o = next();
        if (!o || !PyLong_Check(o)) { ok = false; return nullptr; }
        void* p = PyLong_AsVoidPtr(o);
        if (!p) { PyErr_Clear(); ok = false; }
        return p;
    }
    void tensor(tfjsb_tensor* d) {
        PyObject* o = next();
        if (!o || !THPVariable_Check(o)) { ok = false; return; }
        const at::Tensor& t = THPVariable_Unpack(o);
        const int64_t rank = t.dim();
        if (rank < 1 || rank > 4 || !t.is_cuda() || t.scalar_type() != at::kFloat || !t.is_contiguous()) { ok = false; return; }
        d->data = const_cast<void*>(t.const_data_ptr());
        d->rank = (int32_t)rank;
        for (int64_t i = 0; i < rank; ++i) d->dims[i] = t.size(i);
    }
    // a tensor, or None
    const tfjsb_tensor* maybe(tfjsb_tensor* d) {
        if (!ok) return nullptr;
        if (*at == Py_None) { ++at; return nullptr; }
        tensor(d);
        return d;
    }
    // a tuple or list of `count` whole numbers (1..4 of them when count is 0); returns how many
    int integers(int64_t* v, int count) {
        PyObject* o = next();
        const bool tuple = o && PyTuple_Check(o);
        if (!tuple && !(o && PyList_Check(o))) { ok = false; return 0; }
        const Py_ssize_t n = tuple ? PyTuple_GET_SIZE(o) : PyList_GET_SIZE(o);
        if (count ? n != count : (n < 1 || n > 4)) { ok = false; return 0; }
        for (Py_ssize_t i = 0; i < n; ++i) {
            PyObject* e = tuple ? PyTuple_GET_ITEM(o, i) : PyList_GET_ITEM(o, i);
            if (!PyLong_Check(e)) { ok = false; return 0; }
            int overflow = 0;
            v[i] = PyLong_AsLongLongAndOverflow(e, &overflow);
            if (overflow) { ok = false; return 0; }
        }
        return (int)n;
    }
    void pair(int v[2]) {
        int64_t w[2] = {0, 0};
        integers(w, 2);
        for (int i = 0; i < 2; ++i) {
            v[i] = (int)w[i];
            if (v[i] != w[i]) ok = false;
        }
    }
};

// The output: the tensor that the caller passed, or a new one of the given shape.
struct Out {
    PyObject* given = nullptr;
    at::TensorBase made;
    tfjsb_tensor desc;

    bool take(Args& a) {  // the `out` argument; whether one was given
        if (!a.ok) return false;
        if (*a.at == Py_None) { ++a.at; return false; }
        given = *a.at;
        a.tensor(&desc);
        return true;
    }
    void make(Args& a, int device, const int64_t* dims, int rank) {
        for (int i = 0; i < rank; ++i)
            if (dims[i] < 0) a.ok = false;
        if (!a.ok || rank < 1 || rank > 4) { a.ok = false; return; }
        made = at::detail::empty_cuda(at::IntArrayRef(dims, rank), at::kFloat, at::Device(at::kCUDA, (at::DeviceIndex)device), std::nullopt);
        desc.data = const_cast<void*>(made.const_data_ptr());
        desc.rank = rank;
        for (int i = 0; i < rank; ++i) desc.dims[i] = dims[i];
    }
    PyObject* done(tfjsb_ctx* ctx, tfjsb_status st) {
        if (st != TFJSB_OK) {
            PyObject* error = PyObject_CallFunction(error_type, "is", (int)st, p_tfjsb_last_error(ctx));
            if (error) PyErr_SetObject(error_type, error);
            Py_XDECREF(error);
            return nullptr;
        }
        if (given) { Py_INCREF(given); return given; }
        return THPVariable_Wrap(std::move(made));
    }
};

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The library call without the interpreter lock, as ctypes makes it.
template <typename F>
tfjsb_status unlocked(F f) {
    tfjsb_status st;
    Py_BEGIN_ALLOW_THREADS st = f();
    Py_END_ALLOW_THREADS return st;
}

// The Python entry point of an op with N arguments.  What is thrown in it (by an allocation, say), before the library is
// called, goes wrong again on the ctypes path, which reports it.
template <PyObject* (*OP)(Args&), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    try {
        Args a(args, n, N);
        if (!a.ok) Py_RETURN_NONE;
        return OP(a);
    } catch (...) {
        if (PyErr_Occurred()) PyErr_Clear();
        Py_RETURN_NONE;
    }
}

PyObject* bind(PyObject*, PyObject* args) {  // {name: address}, the type of the errors
    PyObject *addresses, *type;
    if (!PyArg_ParseTuple(args, "O!O", &PyDict_Type, &addresses, &type)) return nullptr;
    Py_INCREF(type);
    Py_XSETREF(error_type, type);
#define TAKE(name)                                                                         \
    {                                                                                      \
        PyObject* o = PyDict_GetItemString(addresses, #name);                              \
        void* p = o ? PyLong_AsVoidPtr(o) : nullptr;                                       \
        if (!p) return PyErr_Format(PyExc_KeyError, "no address for " #name);              \
        std::memcpy(&p_##name, &p, sizeof p);                                              \
    }
    FAST_CALLS(TAKE)
#undef TAKE
    Py_RETURN_NONE;
}

// Every op begins with (handle, device, ...) and ends with `out`.
struct Head {
    tfjsb_ctx* ctx;
    int device;
    explicit Head(Args& a) : ctx(static_cast<tfjsb_ctx*>(a.handle())), device((int)a.integer()) {}
};

// matmul(ctx, device, a, b, transpose_a, transpose_b, out) and the rank-3 form
template <bool BATCH>
PyObject* matmul(Args& a) {
    const Head h(a);
    tfjsb_tensor ta, tb;
    Out out;
    a.tensor(&ta);
    a.tensor(&tb);
    const int x = a.integer() != 0, y = a.integer() != 0;
    constexpr int L = BATCH ? 1 : 0;
    const bool given = out.take(a);
    if (!a.ok || ta.rank != 2 + L || tb.rank != 2 + L) Py_RETURN_NONE;
    if (!given) {
        const int64_t d[3] = {BATCH ? ta.dims[0] : ta.dims[x], BATCH ? ta.dims[1 + x] : tb.dims[1 - y], BATCH ? tb.dims[2 - y] : 0};
        out.make(a, h.device, d, 2 + L);
    }
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return (BATCH ? p_tfjsb_batch_matmul : p_tfjsb_matmul)(h.ctx, &ta, &tb, x, y, &out.desc, s); }));
}

bool window_shape(const tfjsb_tensor& x, const int64_t size[2], const int strides[2], int pad, const int dilations[2], int64_t channels,
                  int64_t d[4]) {
    if (x.rank != 4 || size[0] != (int)size[0] || size[1] != (int)size[1]) return false;
    d[0] = x.dims[0];
    d[3] = channels;
    for (int i = 0; i < 2; ++i)
        if (p_tfjsb_window_out_shape(x.dims[1 + i], (int)size[i], strides[i], dilations[i], (tfjsb_pad)pad, &d[1 + i], nullptr, nullptr) != TFJSB_OK)
            return false;
    return true;
}

// conv2d(ctx, device, x, filter, strides, pad, dilations, bias, act, out) and the depthwise form
template <bool DEPTHWISE>
PyObject* conv2d(Args& a) {
    const Head h(a);
    tfjsb_tensor x, f, b;
    Out out;
    int st[2], dl[2];
    a.tensor(&x);
    a.tensor(&f);
    a.pair(st);
    const int pad = (int)a.integer();
    a.pair(dl);
    const tfjsb_tensor* bias = a.maybe(&b);
    const int act = (int)a.integer();
    const bool given = out.take(a);
    if (!a.ok || f.rank != 4) Py_RETURN_NONE;
    if (!given) {
        int64_t d[4];
        if (!window_shape(x, f.dims, st, pad, dl, DEPTHWISE ? f.dims[2] * f.dims[3] : f.dims[3], d)) Py_RETURN_NONE;
        out.make(a, h.device, d, 4);
    }
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] {
        return (DEPTHWISE ? p_tfjsb_depthwise_conv2d : p_tfjsb_conv2d)(h.ctx, &x, &f, st, (tfjsb_pad)pad, dl, bias, (tfjsb_act)act, &out.desc, s);
    }));
}

// avg_pool / max_pool(ctx, device, x, filter_size, strides, pad, out)
template <bool MAX>
PyObject* pool(Args& a) {
    const Head h(a);
    tfjsb_tensor x;
    Out out;
    int size[2], st[2];
    const int one[2] = {1, 1};
    a.tensor(&x);
    a.pair(size);
    a.pair(st);
    const int pad = (int)a.integer();
    const bool given = out.take(a);
    if (!a.ok || x.rank != 4) Py_RETURN_NONE;
    if (!given) {
        const int64_t w[2] = {size[0], size[1]};
        int64_t d[4];
        if (!window_shape(x, w, st, pad, one, x.dims[3], d)) Py_RETURN_NONE;
        out.make(a, h.device, d, 4);
    }
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return (MAX ? p_tfjsb_max_pool : p_tfjsb_avg_pool)(h.ctx, &x, size, st, (tfjsb_pad)pad, &out.desc, s); }));
}

// binary(ctx, device, op, a, b, out)
PyObject* binary(Args& a) {
    const Head h(a);
    tfjsb_tensor u, v;
    Out out;
    const int op = (int)a.integer();
    a.tensor(&u);
    a.tensor(&v);
    if (!out.take(a) && a.ok) out.make(a, h.device, u.dims, u.rank);
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return p_tfjsb_binary(h.ctx, (tfjsb_binary_op)op, &u, &v, &out.desc, s); }));
}

// softmax(ctx, device, logits, out)
PyObject* softmax(Args& a) {
    const Head h(a);
    tfjsb_tensor x;
    Out out;
    a.tensor(&x);
    if (!out.take(a) && a.ok) out.make(a, h.device, x.dims, x.rank);
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return p_tfjsb_softmax(h.ctx, &x, &out.desc, s); }));
}

// bias_act(ctx, device, x, bias, act, out)
PyObject* bias_act(Args& a) {
    const Head h(a);
    tfjsb_tensor x, b;
    Out out;
    a.tensor(&x);
    const tfjsb_tensor* bias = a.maybe(&b);
    const int act = (int)a.integer();
    if (!out.take(a) && a.ok) out.make(a, h.device, x.dims, x.rank);
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return p_tfjsb_bias_act(h.ctx, &x, bias, (tfjsb_act)act, &out.desc, s); }));
}

// conv_grad(ctx, device, which, shape of the result, first, second, strides, pad, dilations, out): which = 0 conv2d input
// (dy, filter), 1 conv2d filter (x, dy), 2 and 3 the depthwise pair
PyObject* conv_grad(Args& a) {
    const Head h(a);
    tfjsb_tensor u, v;
    Out out;
    int st[2], dl[2];
    int64_t d[4];
    const int which = (int)a.integer();
    const int rank = a.integers(d, 0);
    a.tensor(&u);
    a.tensor(&v);
    a.pair(st);
    const int pad = (int)a.integer();
    a.pair(dl);
    if (!out.take(a) && a.ok) out.make(a, h.device, d, rank);
    if (!a.ok) Py_RETURN_NONE;
    const auto call = which == 0   ? p_tfjsb_conv2d_backprop_input
                      : which == 1 ? p_tfjsb_conv2d_backprop_filter
                      : which == 2 ? p_tfjsb_depthwise_conv2d_backprop_input
                                   : p_tfjsb_depthwise_conv2d_backprop_filter;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return call(h.ctx, &u, &v, st, (tfjsb_pad)pad, dl, &out.desc, s); }));
}

// act_backprop(ctx, device, y, dy, act, out)
PyObject* act_backprop(Args& a) {
    const Head h(a);
    tfjsb_tensor y, g;
    Out out;
    a.tensor(&y);
    a.tensor(&g);
    const int act = (int)a.integer();
    if (!out.take(a) && a.ok) out.make(a, h.device, y.dims, y.rank);
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return p_tfjsb_act_backprop(h.ctx, &y, &g, (tfjsb_act)act, &out.desc, s); }));
}

// bias_backprop(ctx, device, dz, out)
PyObject* bias_backprop(Args& a) {
    const Head h(a);
    tfjsb_tensor g;
    Out out;
    a.tensor(&g);
    if (!out.take(a) && a.ok) out.make(a, h.device, &g.dims[g.rank - 1], 1);
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return p_tfjsb_bias_backprop(h.ctx, &g, &out.desc, s); }));
}

// run_model(ctx, device, model, x, output shape, out)
PyObject* run_model(Args& a) {
    const Head h(a);
    auto* m = static_cast<tfjsb_model*>(a.handle());
    tfjsb_tensor x;
    Out out;
    int64_t d[4];
    a.tensor(&x);
    const int rank = a.integers(d, 0);
    if (!out.take(a) && a.ok) out.make(a, h.device, d, rank);
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return p_tfjsb_run_model(m, &x, &out.desc, s); }));
}

// layer_output_f32(ctx, device, model, layer)
PyObject* layer_output_f32(Args& a) {
    const Head h(a);
    auto* m = static_cast<tfjsb_model*>(a.handle());
    const int layer = (int)a.integer();
    Out out;
    int32_t rank = 0;
    int64_t d[4];
    if (!a.ok || p_tfjsb_model_layer_shape(m, layer, &rank, d) != TFJSB_OK) Py_RETURN_NONE;
    out.make(a, h.device, d, rank);
    if (!a.ok) Py_RETURN_NONE;
    void* s = stream();
    return out.done(h.ctx, unlocked([&] { return p_tfjsb_model_layer_output_f32(m, layer, static_cast<float*>(out.desc.data), s); }));
}

#define METHOD(name, op, n) {name, (PyCFunction)(void (*)(void))(&entry<op, n>), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, nullptr},
    METHOD("matmul", matmul<false>, 7),
    METHOD("batch_matmul", matmul<true>, 7),
    METHOD("conv2d", conv2d<false>, 10),
    METHOD("depthwise_conv2d", conv2d<true>, 10),
    METHOD("avg_pool", pool<false>, 7),
    METHOD("max_pool", pool<true>, 7),
    METHOD("binary", binary, 6),
    METHOD("softmax", softmax, 4),
    METHOD("bias_act", bias_act, 6),
    METHOD("conv_grad", conv_grad, 10),
    METHOD("act_backprop", act_backprop, 6),
    METHOD("bias_backprop", bias_backprop, 4),
    METHOD("run_model", run_model, 6),
    METHOD("layer_output_f32", layer_output_f32, 4),
    {nullptr, nullptr, 0, nullptr},
};
#undef METHOD
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fast_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" PyObject* PyInit__fast_calls() {
    PyObject* m = PyModule_Create(&module);
    if (m) {
        PyObject* names = PyList_New(0);
#define NAME(name)                                     \
    {                                                  \
        PyObject* s = PyUnicode_FromString(#name);     \
        PyList_Append(names, s);                       \
        Py_DECREF(s);                                  \
    }
        FAST_CALLS(NAME)
#undef NAME
        PyModule_AddObject(m, "CALLS", names);
    }
    return m;
}
