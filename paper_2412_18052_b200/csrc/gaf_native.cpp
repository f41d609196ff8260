// Argument marshalling of the calls that a training loop makes every step, as a CPython extension over the C ABI of
// include/gaf.h.  With ctypes a filter call on 3 or 4 gradients spent 10 to 13 us in the interpreter (tensor
// attributes one by one, pointer arrays, the current stream, 14 converted arguments), which is longer than the
// GPU needs for a million parameters; here the tensors are read directly.
//
// Every function takes its arguments by position (binding.py has the signatures with defaults), checks what the
// binding has always checked, allocates outputs that were not given and raises the error class that
// binding.py registers.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <vector>

#include "../../include/gaf.h"

namespace {

PyObject *g_error = nullptr;            // GafError(code, where)

struct Failed {};                       // a Python exception is set

[[noreturn]] void fail(PyObject *type, const char *text) {
    PyErr_SetString(type, text);
    throw Failed();
}
[[noreturn]] void fail_code(int code, const char *where) {
    PyObject *e = g_error ? PyObject_CallFunction(g_error, "is", code, where) : nullptr;
    if (e) { PyErr_SetObject(g_error, e); Py_DECREF(e); }
    else if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, where);
    throw Failed();
}
void check(int code, const char *where) {
    if (code != GAF_OK) fail_code(code, where);
}

const at::Tensor &tensor(PyObject *o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a torch tensor");
    return THPVariable_Unpack(o);
}
int dtype_code(const at::Tensor &t) {
    if (t.scalar_type() == at::kFloat) return GAF_F32;
    if (t.scalar_type() == at::kBFloat16) return GAF_BF16;
    PyErr_Format(PyExc_TypeError, "gradients must be float32 or bfloat16, got %s", c10::toString(t.scalar_type()));
    throw Failed();
}
void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

double number(PyObject *o) {
    if (PyFloat_Check(o)) return PyFloat_AS_DOUBLE(o);
    PyObject *f = PyNumber_Float(o);    // what float() takes: numpy and torch scalars, texts
    if (!f) throw Failed();
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return v;
}
int64_t integer(PyObject *o) {
    if (PyLong_Check(o)) {
        const int64_t v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) throw Failed();
        return v;
    }
    PyObject *i = PyNumber_Long(o);     // (numpy integers and the like)
    if (!i) throw Failed();
    const int64_t v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return v;
}

// The items of anything that has a length and, where `indexed`, can be indexed (a generator has neither: its items would be
// used up by one call).  They stay alive as long as this object does.
struct Sequence {
    PyObject *fast;
    Py_ssize_t n;
    explicit Sequence(PyObject *o, bool indexed = false) : fast(nullptr), n(0) {
        if (!PyList_Check(o) && !PyTuple_Check(o)) {
            const Py_ssize_t len = PyObject_Size(o);
            if (len < 0) throw Failed();
            if (indexed && len > 0) {
                PyObject *zero = PyLong_FromLong(0), *item = zero ? PyObject_GetItem(o, zero) : nullptr;
                Py_XDECREF(zero);
                if (!item) throw Failed();
                Py_DECREF(item);
            }
        }
        fast = PySequence_Fast(o, "expected a sequence");
        if (!fast) throw Failed();
        n = PySequence_Fast_GET_SIZE(fast);
    }
    ~Sequence() { Py_DECREF(fast); }
    Sequence(const Sequence &) = delete;
    PyObject *operator[](Py_ssize_t i) const { return PySequence_Fast_GET_ITEM(fast, i); }
};

// The gradients of a call: pointers, length, type, device.  It holds the tensors until the call has been made: a sequence may make
// them as they are asked for, and memory that is freed before the outputs are allocated becomes the outputs.
struct Gradients {
    const Sequence seq;
    std::vector<const void *> ptr;
    int64_t D = 0;
    int dtype = 0;
    at::Device device = at::kCPU;
    Gradients(PyObject *o, bool must_match) : seq(o, true) {
        if (seq.n == 0) fail(PyExc_IndexError, "no gradients");
        ptr.reserve(seq.n);
        const at::Tensor &first = tensor(seq[0]);
        D = first.numel();
        dtype = dtype_code(first);
        device = first.device();
        for (Py_ssize_t i = 0; i < seq.n; ++i) {
            const at::Tensor &t = tensor(seq[i]);
            if (must_match && (t.numel() != D || t.scalar_type() != first.scalar_type() || !t.is_contiguous()))
                fail(PyExc_AssertionError, "gradients must be contiguous tensors of one length and type");
            ptr.push_back(t.data_ptr());
        }
    }
    int K() const { return static_cast<int>(ptr.size()); }
};

// A step order for K gradients, or null for the identity.  What is missing from one that is too short, and a number that no int32
// holds, become -1, which the library refuses; what a longer one has beyond K is not looked at.
struct Order {
    std::vector<int32_t> v;
    const int32_t *ptr = nullptr;
    Order(PyObject *o, int K) {
        if (o == Py_None) return;
        const Sequence seq(o);
        v.assign(K, -1);
        for (Py_ssize_t i = 0; i < seq.n && i < K; ++i) {
            const int64_t x = integer(seq[i]);
            if (x >= 0 && x <= INT32_MAX) v[i] = static_cast<int32_t>(x);
        }
        ptr = v.data();
    }
};

// An output: the given tensor, or a new one.
struct Output {
    PyObject *object;
    void *ptr;
    Output(PyObject *given, at::IntArrayRef shape, at::ScalarType type, at::Device device) {
        if (given != Py_None) {
            ptr = tensor(given).data_ptr();
            object = Py_NewRef(given);
        } else {
            const at::Tensor t = at::empty(shape, at::TensorOptions().dtype(type).device(device));
            ptr = t.data_ptr();
            object = THPVariable_Wrap(t);
            if (!object) throw Failed();
        }
    }
    ~Output() { Py_XDECREF(object); }
    Output(const Output &) = delete;
    PyObject *take() { PyObject *o = object; object = nullptr; return o; }
};
template <typename T> T *as(const Output &o) { return static_cast<T *>(o.ptr); }

struct Workspace {
    void *ptr;
    size_t bytes;
    explicit Workspace(PyObject *o) {
        const at::Tensor &t = tensor(o);
        ptr = t.data_ptr();
        bytes = static_cast<size_t>(t.numel());
    }
};

template <typename F>
int without_gil(F &&f) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return rc;
}
// Runs a body that throws Failed (a Python exception is set) or a torch error.
template <typename F>
PyObject *guarded(Py_ssize_t n, Py_ssize_t want, F &&f) {
    if (n != want) { PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n); return nullptr; }
    try {
        return f();
    } catch (const Failed &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <typename... O>
PyObject *tuple_of(O &...o) {
    PyObject *t = PyTuple_New(sizeof...(o));
    if (!t) throw Failed();
    Py_ssize_t i = 0;
    (PyTuple_SET_ITEM(t, i++, o.take()), ...);
    return t;
}

PyObject *py_filter_accumulate(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 9, [&] {
        const Gradients g(a[0], true);
        const double tau = number(a[1]);
        const Workspace ws(a[2]);
        const Order order(a[3], g.K());
        Output macro(a[4], {g.D}, at::kFloat, g.device), mask(a[5], {g.K()}, at::kByte, g.device),
            dist(a[6], {g.K()}, at::kFloat, g.device), count(a[7], {1}, at::kInt, g.device);
        const int schedule = static_cast<int>(integer(a[8]));
        void *const st = stream();
        check(without_gil([&] {
            return gaf_filter_accumulate(g.ptr.data(), g.K(), g.D, g.dtype, tau, order.ptr, as<float>(macro), as<uint8_t>(mask),
                                         as<float>(dist), as<int32_t>(count), ws.ptr, ws.bytes, schedule, st);
        }), "gaf_filter_accumulate");
        return tuple_of(macro, mask, dist, count);
    });
}

PyObject *py_filter_accumulate_any_seed(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 4, [&] {
        const Gradients g(a[0], false);
        const double tau = number(a[1]);
        const Workspace ws(a[2]);
        Output macro(a[3], {g.D}, at::kFloat, g.device), mask(Py_None, {g.K()}, at::kByte, g.device),
            dist(Py_None, {g.K()}, at::kFloat, g.device), count(Py_None, {1}, at::kInt, g.device),
            seed(Py_None, {1}, at::kInt, g.device);
        void *const st = stream();
        check(without_gil([&] {
            return gaf_filter_accumulate_any_seed(g.ptr.data(), g.K(), g.D, g.dtype, tau, as<float>(macro), as<uint8_t>(mask),
                                                  as<float>(dist), as<int32_t>(count), as<int32_t>(seed), ws.ptr, ws.bytes, st);
        }), "gaf_filter_accumulate_any_seed");
        return tuple_of(macro, mask, dist, count, seed);
    });
}

PyObject *py_filter_accumulate_bucketed(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 6, [&] {
        const Gradients g(a[0], false);
        const double tau = number(a[1]);
        std::vector<int64_t> offsets;
        {
            const Sequence seq(a[2]);
            offsets.reserve(seq.n);
            for (Py_ssize_t i = 0; i < seq.n; ++i) offsets.push_back(integer(seq[i]));
        }
        const int64_t S = static_cast<int64_t>(offsets.size()) - 1;
        if (S < 0) fail(PyExc_ValueError, "no bucket offsets");
        const Workspace ws(a[3]);
        const Order order(a[4], g.K());
        Output macro(a[5], {g.D}, at::kFloat, g.device), mask(Py_None, {S, g.K()}, at::kByte, g.device),
            dist(Py_None, {S, g.K()}, at::kFloat, g.device), count(Py_None, {S}, at::kInt, g.device);
        void *const st = stream();
        check(without_gil([&] {
            return gaf_filter_accumulate_bucketed(g.ptr.data(), g.K(), g.D, g.dtype, tau, order.ptr, static_cast<int>(S),
                                                  offsets.data(), as<float>(macro), as<uint8_t>(mask), as<float>(dist),
                                                  as<int32_t>(count), ws.ptr, ws.bytes, st);
        }), "gaf_filter_accumulate_bucketed");
        return tuple_of(macro, mask, dist, count);
    });
}

PyObject *py_pairwise_cosdist(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 4, [&] {
        const Gradients g(a[0], false);
        const Workspace ws(a[1]);
        Output dist(a[2], {g.K(), g.K()}, at::kFloat, g.device), gram(a[3], {g.K(), g.K()}, at::kDouble, g.device);
        void *const st = stream();
        check(without_gil([&] {
            return gaf_pairwise_cosdist(g.ptr.data(), g.K(), g.D, g.dtype, as<float>(dist), as<double>(gram), ws.ptr, ws.bytes, st);
        }), "gaf_pairwise_cosdist");
        return tuple_of(dist, gram);
    });
}

PyObject *py_cosdist(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 5, [&] {
        const at::Tensor &x = tensor(a[0]), &y = tensor(a[1]);
        if (x.numel() != y.numel() || x.scalar_type() != y.scalar_type())
            fail(PyExc_AssertionError, "the two tensors must have one length and type");
        const int dtype = dtype_code(x);
        const Workspace ws(a[2]);
        Output dist(a[3], {1}, at::kFloat, x.device()), stats(a[4], {3}, at::kDouble, x.device());
        void *const st = stream();
        check(without_gil([&] {
            return gaf_cosdist(x.data_ptr(), y.data_ptr(), x.numel(), dtype, as<float>(dist), as<double>(stats), ws.ptr, ws.bytes, st);
        }), "gaf_cosdist");
        return tuple_of(dist, stats);
    });
}

PyObject *py_stream_begin(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 3, [&] {
        const at::Tensor &seed = tensor(a[0]);
        const int dtype = dtype_code(seed);
        float *const acc = static_cast<float *>(tensor(a[1]).data_ptr());
        const Workspace ws(a[2]);
        void *const st = stream();
        check(without_gil([&] { return gaf_stream_begin(seed.data_ptr(), seed.numel(), dtype, acc, ws.ptr, ws.bytes, st); }),
              "gaf_stream_begin");
        return Py_NewRef(Py_None);
    });
}

PyObject *py_stream_push(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 5, [&] {
        const at::Tensor &g = tensor(a[0]);
        const int dtype = dtype_code(g), t = static_cast<int>(integer(a[1]));
        const double tau = number(a[2]);
        float *const acc = static_cast<float *>(tensor(a[3]).data_ptr());
        const Workspace ws(a[4]);
        void *const st = stream();
        check(without_gil([&] { return gaf_stream_push(g.data_ptr(), t, g.numel(), dtype, tau, acc, ws.ptr, ws.bytes, st); }),
              "gaf_stream_push");
        return Py_NewRef(Py_None);
    });
}

PyObject *py_stream_end(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 3, [&] {
        const int64_t K = integer(a[0]);
        const at::Tensor &acc = tensor(a[1]);
        const Workspace ws(a[2]);
        Output mask(Py_None, {K}, at::kByte, acc.device()), dist(Py_None, {K}, at::kFloat, acc.device()),
            count(Py_None, {1}, at::kInt, acc.device());
        void *const st = stream();
        check(without_gil([&] {
            return gaf_stream_end(static_cast<int>(K), acc.numel(), static_cast<float *>(acc.data_ptr()), as<uint8_t>(mask), as<float>(dist),
                                  as<int32_t>(count), ws.ptr, ws.bytes, st);
        }), "gaf_stream_end");
        return tuple_of(mask, dist, count);
    });
}

PyObject *py_register_error(PyObject *, PyObject *cls) {
    Py_XSETREF(g_error, Py_NewRef(cls));
    return Py_NewRef(Py_None);
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST(filter_accumulate), FAST(filter_accumulate_any_seed), FAST(filter_accumulate_bucketed), FAST(pairwise_cosdist),
    FAST(cosdist), FAST(stream_begin), FAST(stream_push), FAST(stream_end),
    {"register_error", py_register_error, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_gaf_native", "Argument marshalling over the C ABI of gaf.h.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__gaf_native(void) { return PyModule_Create(&module); }
