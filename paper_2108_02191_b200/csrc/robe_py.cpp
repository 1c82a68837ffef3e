// Native marshalling for the Python binding: tensors in, C-ABI call out.
//
// A small lookup runs for about as long on the GPU as ctypes and torch's Python accessors need to hand
// it over (about 8 us of Python per call, measured with a 128-sample batch; 0.3 us through this module),
// so the calls of a training or serving loop read pointers, types and the current stream from the
// tensors here.  Each function returns the C status of the call it made, or kNotTaken without having
// made it when an argument is not plainly what the call wants; the binding then goes through its
// ctypes path, which does the same call or raises the exception that says what is wrong.
//
// Only the addresses of the C-ABI functions are taken (set_calls), so the module works with whichever
// build of the library the binding has loaded.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/robe.h"

namespace {

constexpr long kNotTaken = 1;  // every robe_status is <= 0

struct Calls {
    decltype(&robe_set_option) set_option;
    decltype(&robe_forward) forward;
    decltype(&robe_forward_keep) forward_keep;
    decltype(&robe_backward) backward;
    decltype(&robe_backward_kept) backward_kept;
    decltype(&robe_backward_adam) backward_adam;
    decltype(&robe_backward_adagrad) backward_adagrad;
    decltype(&robe_apply_sgd) apply_sgd;
} calls;

PyObject* handle_type;  // ctypes.c_void_p

// Reads the arguments of one call; ok turns false at the first one that is not plainly usable.
struct Reader {
    PyObject* const* args;
    bool ok = true;

    const at::Tensor* tensor(int k) {
        if (!THPVariable_Check(args[k])) {
            ok = false;
            return nullptr;
        }
        const at::Tensor& t = THPVariable_Unpack(args[k]);
        if (!t.is_cuda() || !t.has_storage() || !t.is_contiguous()) {
            ok = false;
            return nullptr;
        }
        return &t;
    }
    void* data(int k, at::ScalarType type) {
        const at::Tensor* t = tensor(k);
        if (t == nullptr || t->scalar_type() != type) {
            ok = false;
            return nullptr;
        }
        return t->data_ptr();
    }
    void* data_or_null(int k, at::ScalarType type) { return args[k] == Py_None ? nullptr : data(k, type); }
    void* bytes_or_null(int k, size_t& n) {
        n = 0;
        if (args[k] == Py_None) return nullptr;
        const at::Tensor* t = tensor(k);
        if (t == nullptr) return nullptr;
        n = (size_t)t->numel() * t->element_size();
        return t->data_ptr();
    }
    const void* ids(int k, int64_t& nnz, int& type) {
        const at::Tensor* t = tensor(k);
        if (t == nullptr) return nullptr;
        if (t->scalar_type() == at::kLong) type = ROBE_I64;
        else if (t->scalar_type() == at::kInt) type = ROBE_I32;
        else ok = false;
        nnz = t->numel();
        return t->data_ptr();
    }
    int64_t whole(int k) {
        if (!PyLong_CheckExact(args[k])) {
            ok = false;
            return 0;
        }
        int overflow = 0;
        const long long v = PyLong_AsLongLongAndOverflow(args[k], &overflow);
        if (overflow != 0) ok = false;
        return v;
    }
    float number(int k) {
        if (PyFloat_CheckExact(args[k])) return (float)PyFloat_AS_DOUBLE(args[k]);
        if (!PyLong_CheckExact(args[k])) {
            ok = false;
            return 0.0f;
        }
        const double v = PyLong_AsDouble(args[k]);
        if (v == -1.0 && PyErr_Occurred()) {
            PyErr_Clear();
            ok = false;
        }
        return (float)v;
    }
    // a ctypes.c_void_p and nothing else that has a buffer: its buffer is the pointer
    robe_handle_t handle(int k) {
        Py_buffer b;
        robe_handle_t h = nullptr;
        if ((PyObject*)Py_TYPE(args[k]) != handle_type || PyObject_GetBuffer(args[k], &b, PyBUF_SIMPLE) != 0) {
            PyErr_Clear();
            ok = false;
            return nullptr;
        }
        if (b.len == (Py_ssize_t)sizeof h) memcpy(&h, b.buf, sizeof h);
        PyBuffer_Release(&b);
        if (h == nullptr) ok = false;
        return h;
    }
    // None: the current stream; otherwise a stream object or an address
    void* stream(int k) {
        if (args[k] == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        PyObject* v = PyObject_GetAttrString(args[k], "cuda_stream");
        if (v == nullptr) {
            PyErr_Clear();
            ok = false;
            return nullptr;
        }
        void* p = PyLong_AsVoidPtr(v);
        Py_DECREF(v);
        if (PyErr_Occurred()) {
            PyErr_Clear();
            ok = false;
        }
        return p;
    }
};

// What the interpreter calls.  Torch reports a tensor whose memory cannot be had (sparse, fake, transformed
// ones) or a device it cannot reach by a C++ exception, which must not pass into the interpreter: such a call
// is not taken, and the ctypes path raises what there is to raise.  (Arguments are read before the library is
// called, and the library throws nothing.)
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    try {
        return F(self, args, n);
    } catch (const std::exception&) {
        PyErr_Clear();
        return PyLong_FromLong(kNotTaken);
    }
}

// The call itself, without the interpreter lock: a full launch queue makes a launch wait.
template <class F>
PyObject* made(F&& call) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

PyObject* not_taken() { return PyLong_FromLong(kNotTaken); }

// (h, indices, offsets, batch, out, stream)
PyObject* forward(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 6) return not_taken();
    Reader r{args};
    int64_t nnz = 0;
    int type = ROBE_I64;
    robe_handle_t h = r.handle(0);
    const void* ids = r.ids(1, nnz, type);
    const int64_t* offsets = (const int64_t*)r.data_or_null(2, at::kLong);
    const int64_t batch = r.whole(3);
    float* out = (float*)r.data_or_null(4, at::kFloat);
    void* st = r.stream(5);
    if (!r.ok) return not_taken();
    return made([&] {
        calls.set_option(h, ROBE_OPT_INDEX_TYPE, type);
        return calls.forward(h, ids, offsets, batch, nnz, out, st);
    });
}

// (h, indices, offsets, batch, out, workspace, stream)
PyObject* forward_keep(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 7) return not_taken();
    Reader r{args};
    int64_t nnz = 0;
    size_t ws_bytes = 0;
    int type = ROBE_I64;
    robe_handle_t h = r.handle(0);
    const void* ids = r.ids(1, nnz, type);
    const int64_t* offsets = (const int64_t*)r.data_or_null(2, at::kLong);
    const int64_t batch = r.whole(3);
    float* out = (float*)r.data_or_null(4, at::kFloat);
    void* ws = r.bytes_or_null(5, ws_bytes);
    void* st = r.stream(6);
    if (!r.ok) return not_taken();
    return made([&] {
        calls.set_option(h, ROBE_OPT_INDEX_TYPE, type);
        return calls.forward_keep(h, ids, offsets, batch, nnz, out, ws, ws_bytes, st);
    });
}

// The arguments that every backward call starts with: (h, grad_out, indices, offsets, batch, ...)
struct Backward {
    robe_handle_t h;
    const float* grad_out;
    const void* ids;
    const int64_t* offsets;
    int64_t batch, nnz = 0;
    int type = ROBE_I64;
    explicit Backward(Reader& r) {
        h = r.handle(0);
        grad_out = (const float*)r.data_or_null(1, at::kFloat);
        ids = r.ids(2, nnz, type);
        offsets = (const int64_t*)r.data_or_null(3, at::kLong);
        batch = r.whole(4);
    }
};

// (h, grad_out, indices, offsets, batch, grad_array, lr, workspace, stream)
template <decltype(&robe_backward) Calls::* WHICH>
PyObject* backward(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 9) return not_taken();
    Reader r{args};
    const Backward b(r);
    size_t ws_bytes = 0;
    float* grad_array = (float*)r.data_or_null(5, at::kFloat);
    const float lr = r.number(6);
    void* ws = r.bytes_or_null(7, ws_bytes);
    void* st = r.stream(8);
    if (!r.ok) return not_taken();
    return made([&] {
        calls.set_option(b.h, ROBE_OPT_INDEX_TYPE, b.type);
        return (calls.*WHICH)(b.h, b.grad_out, b.ids, b.offsets, b.batch, b.nnz, grad_array, lr, ws, ws_bytes, st);
    });
}

// (h, grad_out, indices, offsets, batch, m1, m2, lr, beta1, beta2, eps, step, workspace, stream)
PyObject* backward_adam(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 14) return not_taken();
    Reader r{args};
    const Backward b(r);
    size_t ws_bytes = 0;
    float* m1 = (float*)r.data_or_null(5, at::kFloat);
    float* m2 = (float*)r.data_or_null(6, at::kFloat);
    const float lr = r.number(7), beta1 = r.number(8), beta2 = r.number(9), eps = r.number(10);
    const int64_t step = r.whole(11);
    void* ws = r.bytes_or_null(12, ws_bytes);
    void* st = r.stream(13);
    if (!r.ok) return not_taken();
    return made([&] {
        calls.set_option(b.h, ROBE_OPT_INDEX_TYPE, b.type);
        return calls.backward_adam(b.h, b.grad_out, b.ids, b.offsets, b.batch, b.nnz, m1, m2, lr, beta1, beta2, eps,
                                   step, ws, ws_bytes, st);
    });
}

// (h, grad_out, indices, offsets, batch, sum_sq, lr, eps, workspace, stream)
PyObject* backward_adagrad(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 10) return not_taken();
    Reader r{args};
    const Backward b(r);
    size_t ws_bytes = 0;
    float* sum_sq = (float*)r.data_or_null(5, at::kFloat);
    const float lr = r.number(6), eps = r.number(7);
    void* ws = r.bytes_or_null(8, ws_bytes);
    void* st = r.stream(9);
    if (!r.ok) return not_taken();
    return made([&] {
        calls.set_option(b.h, ROBE_OPT_INDEX_TYPE, b.type);
        return calls.backward_adagrad(b.h, b.grad_out, b.ids, b.offsets, b.batch, b.nnz, sum_sq, lr, eps, ws,
                                      ws_bytes, st);
    });
}

// (h, grad_array, lr, zero_grad, stream); zero_grad is True or False
PyObject* apply_sgd(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 5) return not_taken();
    Reader r{args};
    robe_handle_t h = r.handle(0);
    float* grad_array = (float*)r.data_or_null(1, at::kFloat);
    const float lr = r.number(2);
    if (args[3] != Py_True && args[3] != Py_False) return not_taken();
    void* st = r.stream(4);
    if (!r.ok) return not_taken();
    const int zero = args[3] == Py_True ? 1 : 0;
    return made([&] { return calls.apply_sgd(h, grad_array, lr, zero, st); });
}

// (the type of a handle, addresses of the C-ABI functions in the order of Calls)
PyObject* set_calls(PyObject*, PyObject* const* args, Py_ssize_t n) {
    void* p[8];
    if (n != 9) {
        PyErr_SetString(PyExc_TypeError, "set_calls takes a type and eight addresses");
        return nullptr;
    }
    for (int k = 0; k < 8; ++k) {
        p[k] = PyLong_AsVoidPtr(args[k + 1]);
        if (PyErr_Occurred()) return nullptr;
    }
    Py_INCREF(args[0]);
    Py_XSETREF(handle_type, args[0]);
    calls = Calls{(decltype(calls.set_option))p[0],       (decltype(calls.forward))p[1],
                  (decltype(calls.forward_keep))p[2],     (decltype(calls.backward))p[3],
                  (decltype(calls.backward_kept))p[4],    (decltype(calls.backward_adam))p[5],
                  (decltype(calls.backward_adagrad))p[6], (decltype(calls.apply_sgd))p[7]};
    Py_RETURN_NONE;
}

#define FAST(...) ((PyCFunction)(void (*)(void))(&guarded<__VA_ARGS__>))
PyMethodDef methods[] = {
    {"set_calls", FAST(set_calls), METH_FASTCALL, "type of a handle, addresses of the C-ABI functions"},
    {"forward", FAST(forward), METH_FASTCALL, "robe_forward"},
    {"forward_keep", FAST(forward_keep), METH_FASTCALL, "robe_forward_keep"},
    {"backward", FAST(backward<&Calls::backward>), METH_FASTCALL, "robe_backward"},
    {"backward_kept", FAST(backward<&Calls::backward_kept>), METH_FASTCALL, "robe_backward_kept"},
    {"backward_adam", FAST(backward_adam), METH_FASTCALL, "robe_backward_adam"},
    {"backward_adagrad", FAST(backward_adagrad), METH_FASTCALL, "robe_backward_adagrad"},
    {"apply_sgd", FAST(apply_sgd), METH_FASTCALL, "robe_apply_sgd"},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_robe_py", "native marshalling of the binding", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__robe_py() { return PyModule_Create(&module); }
