// bind.cpp -- the marshalling of respec.py's entry points, in C++.
//
// Every function takes the arguments of the Python function of its name, in
// order (tensors, None or integer addresses for the pointers; the workspace
// tensor for (pointer, bytes); a stream, None or an integer handle), calls the
// C entry point of librespec.so without the interpreter lock and returns its
// status.  A call of 25 arguments cost ~10 us through ctypes on the host of a
// GB300 (0.23 us a tensor for three attribute calls, 2.9 us to build a stream
// object, 1.8 us of conversions), more than some of the kernels behind it.
//
// Arguments are converted as ctypes converts them: an int wraps to the C type, an
// instance of the C type or an object whose _as_parameter_ is one will do, and
// anything else is refused.  A tensor subclass answers for itself.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <string.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/version.h>

#include <stdexcept>

#include "respec.h"

#define RS_ENTRIES(X)                                                                                            \
    X(entropy_gate) X(entropy_gate_noalloc) X(entropy_gate_rows) X(match_scan) X(tree_verify_attn) X(accept)     \
    X(match_index_build) X(match_index_append) X(match_scan_indexed) X(tree_sample)

namespace {

PyObject *g_params_type = nullptr, *g_argument_error = nullptr;
PyObject *g_c_int = nullptr, *g_c_int64 = nullptr, *g_c_float = nullptr, *g_c_void_p = nullptr;  // ctypes' types

// The library's entry points, as respec.py has loaded them: linked by file name the
// loader might find another librespec.so first.
struct Library {
#define RS_ENTRY(name) decltype(&rs_##name) name = nullptr;
    RS_ENTRIES(RS_ENTRY)
#undef RS_ENTRY
} lib;

struct PyFail {};  // a Python exception is set

// A reference of our own.
struct Ref {
    PyObject *o;
    explicit Ref(PyObject *x) : o(x) {
        if (!o) throw PyFail{};
    }
    ~Ref() { Py_DECREF(o); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
};

// The arguments of one call, taken in order.
struct Args {
    PyObject *const *v;
    Py_ssize_t n, i = 0;
    PyObject *next() {
        if (i >= n) {
            PyErr_SetString(PyExc_TypeError, "too few arguments");
            throw PyFail{};
        }
        return v[i++];
    }
    [[noreturn]] void refuse(const char *what, PyObject *o) {
        PyErr_Format(g_argument_error, "argument %zd: TypeError: %s instead of %s instance", i, what, Py_TYPE(o)->tp_name);
        throw PyFail{};
    }
    // What stands for o where plain(o) does not hold: the first of o,
    // o._as_parameter_ ... that is an instance of the ctypes type or plain.
    // use(x, is_instance) makes the result of it.
    template <class Plain, class Use>
    auto stand_in(PyObject *o, PyObject *type, const char *what, Plain plain, Use use) {
        PyObject *x = Py_NewRef(o);
        for (int depth = 0;; ++depth) {
            const Ref own(x);
            const int is = PyObject_IsInstance(x, type);
            if (is < 0) throw PyFail{};
            if (is || plain(x)) return use(x, is != 0);
            x = depth < 64 ? PyObject_GetAttrString(x, "_as_parameter_") : nullptr;
            if (!x) {
                PyErr_Clear();
                refuse(what, o);
            }
        }
    }
    // The same for numbers: use(x) with x or an instance's value.
    template <class Plain, class Use>
    auto number_for(PyObject *o, PyObject *type, const char *what, Plain plain, Use use) {
        return stand_in(o, type, what, plain, [use](PyObject *x, bool instance) {
            if (!instance) return use(x);
            const Ref v(PyObject_GetAttrString(x, "value"));
            return use(v.o);
        });
    }
    // A handle: None, an int, a c_void_p or what stands for one.
    void *handle(PyObject *h, const char *what) {
        auto plain = [](PyObject *x) { return x == Py_None || PyLong_Check(x); };
        auto use = [this](PyObject *x) { return x == Py_None ? nullptr : reinterpret_cast<void *>(masked(x)); };
        if (plain(h)) return use(h);
        return number_for(h, g_c_void_p, what, plain, use);
    }
    // The address of a tensor, or of an object with a tensor's attributes; its
    // bytes too where asked for.
    void *address(PyObject *o, size_t *bytes) {
        if (THPVariable_CheckExact(o)) {
            const at::Tensor &t = THPVariable_Unpack(o);
            check(t.is_cuda(), t.is_contiguous(), o);
            if (bytes) *bytes = (size_t)t.numel() * (size_t)t.element_size();
            return t.data_ptr();
        }
        const bool cuda = number(PyObject_GetAttrString(o, "is_cuda")) != 0;
        check(cuda, cuda && number(PyObject_CallMethod(o, "is_contiguous", nullptr)) != 0, o);
        if (bytes)
            *bytes = (size_t)(number(PyObject_CallMethod(o, "numel", nullptr)) *
                              number(PyObject_CallMethod(o, "element_size", nullptr)));
        const Ref p(PyObject_CallMethod(o, "data_ptr", nullptr));
        return handle(p.o, "address expected");
    }
    void check(bool cuda, bool contiguous, PyObject *o) {
        if (!cuda) {
            PyObject *d = PyObject_GetAttrString(o, "device");
            if (d) PyErr_Format(PyExc_ValueError, "expected a CUDA tensor, got one on %S", d);
            Py_XDECREF(d);
            throw PyFail{};
        }
        if (!contiguous) {
            PyErr_SetString(PyExc_ValueError, "expected a contiguous tensor");
            throw PyFail{};
        }
    }
    unsigned long long number(PyObject *x) {  // takes the reference
        const Ref own(x);
        if (PyLong_Check(x)) return masked(x);
        const int yes = PyObject_IsTrue(x);
        if (yes < 0) throw PyFail{};
        return (unsigned long long)yes;
    }
    template <class T>
    T *ptr() {
        PyObject *o = next();
        if (o == Py_None) return nullptr;
        if (PyLong_Check(o)) return reinterpret_cast<T *>(masked(o));
        return static_cast<T *>(address(o, nullptr));
    }
    unsigned long long masked(PyObject *o) {
        const unsigned long long x = PyLong_AsUnsignedLongLongMask(o);
        if (x == (unsigned long long)-1 && PyErr_Occurred()) throw PyFail{};
        return x;
    }
    long long i64() { return integer(g_c_int64); }
    int i32() { return (int)integer(g_c_int); }
    long long integer(PyObject *type) {
        PyObject *o = next();
        if (PyLong_Check(o)) return (long long)masked(o);
        return number_for(o, type, "int expected", [](PyObject *x) { return PyLong_Check(x) != 0; },
                          [this](PyObject *x) { return (long long)masked(x); });
    }
    // whether x converts to a double, without an exception
    static bool real(PyObject *x, double *d) {
        *d = PyFloat_AsDouble(x);
        if (*d != -1.0 || !PyErr_Occurred()) return true;
        PyErr_Clear();
        return false;
    }
    float f32() {
        PyObject *o = next();
        double d;
        if (real(o, &d)) return (float)d;
        return number_for(o, g_c_float, "float expected",
                          [](PyObject *x) {
                              double y;
                              return real(x, &y);
                          },
                          [](PyObject *x) {
                              double y;
                              real(x, &y);
                              return (float)y;
                          });
    }
    rs_params params() {
        return stand_in(next(), g_params_type, "expected rs_params", [](PyObject *) { return false; },
                        [](PyObject *x, bool) { return params_of(x); });
    }
    static rs_params params_of(PyObject *x) {
        Py_buffer b;
        if (PyObject_GetBuffer(x, &b, PyBUF_SIMPLE) != 0) throw PyFail{};
        rs_params p;
        const bool fits = b.len == (Py_ssize_t)sizeof p;
        if (fits) memcpy(&p, b.buf, sizeof p);
        PyBuffer_Release(&b);
        if (!fits) {
            PyErr_SetString(PyExc_TypeError, "rs_params has another size");
            throw PyFail{};
        }
        return p;
    }
    // a tensor as (pointer, bytes); None as (null, 0)
    void *sized(size_t *bytes, bool optional) {
        PyObject *o = next();
        *bytes = 0;
        if (o == Py_None && optional) return nullptr;
        return address(o, bytes);
    }
    void *stream() {
        PyObject *o = next();
        if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        if (PyLong_Check(o)) return reinterpret_cast<void *>(masked(o));
        const Ref h(PyObject_GetAttrString(o, "cuda_stream"));
        return handle(h.o, "stream handle expected");
    }
};

// body(args) converts and returns a callable that makes the C call.
template <class F>
PyObject *guarded(PyObject *const *v, Py_ssize_t n, F body) {
    try {
        Args a{v, n};
        auto call = body(a);
        if (a.i != n) {
            PyErr_SetString(PyExc_TypeError, "too many arguments");
            return nullptr;
        }
        rs_status st;
        Py_BEGIN_ALLOW_THREADS
        st = call();
        Py_END_ALLOW_THREADS
        return PyLong_FromLong((long)st);
    } catch (const PyFail &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

#define RS_BIND(name) PyObject *name(PyObject *, PyObject *const *v, Py_ssize_t n)

RS_BIND(entropy_gate) {
    return guarded(v, n, [](Args &a) {
        auto *logits = a.ptr<const float>();
        const int R = a.i32(), V = a.i32();
        auto *row_off = a.ptr<const int32_t>();
        auto *row_commit = a.ptr<const uint8_t>();
        const int B = a.i32();
        const rs_params p = a.params();
        auto *hist = a.ptr<float>();
        auto *hist_n = a.ptr<int32_t>();
        auto *entropy = a.ptr<float>();
        auto *k_star = a.ptr<int32_t>();
        auto *h_best = a.ptr<float>();
        auto *ok = a.ptr<uint8_t>();
        size_t wb;
        void *ws = a.sized(&wb, true), *st = a.stream();
        return [=] {
            return lib.entropy_gate(logits, R, V, row_off, row_commit, B, p, hist, hist_n, entropy, k_star, h_best, ok, ws, wb, st);
        };
    });
}

RS_BIND(entropy_gate_noalloc) {
    return guarded(v, n, [](Args &a) {
        auto *logits = a.ptr<const float>();
        const int R = a.i32(), V = a.i32();
        auto *row_off = a.ptr<const int32_t>();
        auto *row_commit = a.ptr<const uint8_t>();
        const int B = a.i32();
        const rs_params p = a.params();
        auto *hist = a.ptr<float>();
        auto *hist_n = a.ptr<int32_t>();
        auto *entropy = a.ptr<float>();
        auto *k_star = a.ptr<int32_t>();
        auto *h_best = a.ptr<float>();
        auto *ok = a.ptr<uint8_t>();
        void *st = a.stream();
        return [=] {
            return lib.entropy_gate_noalloc(logits, R, V, row_off, row_commit, B, p, hist, hist_n, entropy, k_star, h_best, ok, st);
        };
    });
}

RS_BIND(entropy_gate_rows) {
    return guarded(v, n, [](Args &a) {
        auto *entropy = a.ptr<const float>();
        auto *row_off = a.ptr<const int32_t>();
        auto *row_commit = a.ptr<const uint8_t>();
        const int B = a.i32();
        const rs_params p = a.params();
        auto *hist = a.ptr<float>();
        auto *hist_n = a.ptr<int32_t>();
        auto *k_star = a.ptr<int32_t>();
        auto *h_best = a.ptr<float>();
        auto *ok = a.ptr<uint8_t>();
        void *st = a.stream();
        return [=] { return lib.entropy_gate_rows(entropy, row_off, row_commit, B, p, hist, hist_n, k_star, h_best, ok, st); };
    });
}

RS_BIND(match_scan) {
    return guarded(v, n, [](Args &a) {
        auto *tokens = a.ptr<const int32_t>();
        auto *tok_off = a.ptr<const int64_t>();
        const int B = a.i32();
        auto *k_star = a.ptr<const int32_t>();
        auto *gate_ok = a.ptr<const uint8_t>();
        auto *scores = a.ptr<const float>();
        const rs_params p = a.params();
        const int cap = a.i32();
        auto *count = a.ptr<int32_t>(), *pos = a.ptr<int32_t>(), *sel_pos = a.ptr<int32_t>(), *sel_len = a.ptr<int32_t>();
        auto *spans = a.ptr<int32_t>(), *n_sel = a.ptr<int32_t>(), *status = a.ptr<int32_t>();
        size_t wb;
        void *ws = a.sized(&wb, true), *st = a.stream();
        return [=] {
            return lib.match_scan(tokens, tok_off, B, k_star, gate_ok, scores, p, cap, count, pos, sel_pos, sel_len, spans, n_sel,
                                 status, ws, wb, st);
        };
    });
}

RS_BIND(tree_verify_attn) {
    return guarded(v, n, [](Args &a) {
        auto *q = a.ptr<const uint16_t>(), *k = a.ptr<const uint16_t>(), *vv = a.ptr<const uint16_t>();
        const int64_t kv_rows = a.i64();
        auto *kv_off = a.ptr<const int64_t>();
        auto *ctx_len = a.ptr<const int32_t>(), *node_off = a.ptr<const int32_t>(), *parents = a.ptr<const int32_t>();
        const int B = a.i32(), R = a.i32(), Hq = a.i32(), Hkv = a.i32(), D = a.i32();
        const float scale = a.f32();
        auto *out = a.ptr<float>(), *lse = a.ptr<float>();
        auto *status = a.ptr<int32_t>();
        size_t wb;
        void *ws = a.sized(&wb, true), *st = a.stream();
        return [=] {
            return lib.tree_verify_attn(q, k, vv, kv_rows, kv_off, ctx_len, node_off, parents, B, R, Hq, Hkv, D, scale, out, lse,
                                       status, ws, wb, st);
        };
    });
}

RS_BIND(accept) {
    return guarded(v, n, [](Args &a) {
        auto *logits = a.ptr<const float>();
        const int R = a.i32(), V = a.i32();
        auto *node_off = a.ptr<const int32_t>();
        const int B = a.i32();
        auto *tokens = a.ptr<const int32_t>(), *parents = a.ptr<const int32_t>();
        auto *source = a.ptr<const uint8_t>();
        auto *chain = a.ptr<const int8_t>();
        auto *sel_pos = a.ptr<const int32_t>();
        auto *tok_off = a.ptr<const int64_t>();
        const rs_params p = a.params();
        const int cap = a.i32();
        auto *argmax = a.ptr<int32_t>(), *topk = a.ptr<int32_t>();
        auto *lse = a.ptr<float>(), *p_tok = a.ptr<float>(), *entropy = a.ptr<float>();
        auto *acc_len = a.ptr<int32_t>(), *acc_nodes = a.ptr<int32_t>(), *bonus = a.ptr<int32_t>(), *winner = a.ptr<int32_t>();
        auto *commit = a.ptr<uint8_t>();
        auto *scores = a.ptr<float>();
        auto *status = a.ptr<int32_t>();
        size_t wb;
        void *ws = a.sized(&wb, true), *st = a.stream();
        return [=] {
            return lib.accept(logits, R, V, node_off, B, tokens, parents, source, chain, sel_pos, tok_off, p, cap, argmax, topk, lse,
                             p_tok, entropy, acc_len, acc_nodes, bonus, winner, commit, scores, status, ws, wb, st);
        };
    });
}

RS_BIND(match_index_build) {
    return guarded(v, n, [](Args &a) {
        auto *tokens = a.ptr<const int32_t>();
        auto *tok_off = a.ptr<const int64_t>();
        const int B = a.i32(), V = a.i32();
        const int64_t total = a.i64();
        size_t ib;
        void *index = a.sized(&ib, false), *st = a.stream();
        return [=] { return lib.match_index_build(tokens, tok_off, B, V, total, index, ib, st); };
    });
}

RS_BIND(match_index_append) {
    return guarded(v, n, [](Args &a) {
        auto *tokens = a.ptr<const int32_t>();
        auto *tok_off = a.ptr<const int64_t>();
        const int B = a.i32(), V = a.i32();
        const int64_t total = a.i64();
        size_t ib;
        void *index = a.sized(&ib, false);
        auto *status = a.ptr<int32_t>();
        void *st = a.stream();
        return [=] { return lib.match_index_append(tokens, tok_off, B, V, total, index, ib, status, st); };
    });
}

RS_BIND(match_scan_indexed) {
    return guarded(v, n, [](Args &a) {
        auto *tokens = a.ptr<const int32_t>();
        auto *tok_off = a.ptr<const int64_t>();
        const int B = a.i32();
        auto *k_star = a.ptr<const int32_t>();
        auto *gate_ok = a.ptr<const uint8_t>();
        auto *scores = a.ptr<const float>();
        const rs_params p = a.params();
        const int cap = a.i32();
        auto *count = a.ptr<int32_t>(), *pos = a.ptr<int32_t>(), *sel_pos = a.ptr<int32_t>(), *sel_len = a.ptr<int32_t>();
        auto *spans = a.ptr<int32_t>(), *n_sel = a.ptr<int32_t>(), *status = a.ptr<int32_t>();
        const int V = a.i32();
        const int64_t total = a.i64();
        size_t ib;
        void *index = a.sized(&ib, false), *st = a.stream();
        return [=] {
            return lib.match_scan_indexed(tokens, tok_off, B, k_star, gate_ok, scores, p, cap, count, pos, sel_pos, sel_len, spans,
                                         n_sel, status, V, total, index, ib, st);
        };
    });
}

RS_BIND(tree_sample) {
    return guarded(v, n, [](Args &a) {
        auto *logits = a.ptr<const float>();
        const int R = a.i32(), V = a.i32();
        auto *node_off = a.ptr<const int32_t>();
        const int B = a.i32();
        auto *tokens = a.ptr<const int32_t>(), *parents = a.ptr<const int32_t>();
        auto *source = a.ptr<const uint8_t>();
        const float T = a.f32();
        auto *uniforms = a.ptr<const float>();
        const int cap = a.i32();
        auto *draw = a.ptr<int32_t>(), *acc_len = a.ptr<int32_t>(), *acc_nodes = a.ptr<int32_t>(), *bonus = a.ptr<int32_t>();
        auto *status = a.ptr<int32_t>();
        size_t wb;
        void *ws = a.sized(&wb, true), *st = a.stream();
        return [=] {
            return lib.tree_sample(logits, R, V, node_off, B, tokens, parents, source, T, uniforms, cap, draw, acc_len, acc_nodes,
                                  bonus, status, ws, wb, st);
        };
    });
}

// setup(rs_params type, {name: address of rs_name}): the type the params argument
// must have and the library's entry points.
PyObject *setup(PyObject *, PyObject *args) {
    PyObject *type, *entries;
    if (!PyArg_ParseTuple(args, "OO!", &type, &PyDict_Type, &entries)) return nullptr;
    Library l;
#define RS_ENTRY(name)                                                                              \
    if (PyObject *a = PyDict_GetItemString(entries, "rs_" #name))                                   \
        l.name = reinterpret_cast<decltype(l.name)>(PyLong_AsVoidPtr(a));                           \
    if (!l.name) {                                                                                  \
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_KeyError, "rs_" #name);                        \
        return nullptr;                                                                             \
    }
    RS_ENTRIES(RS_ENTRY)
#undef RS_ENTRY
    lib = l;
    Py_INCREF(type);
    Py_XSETREF(g_params_type, type);
    Py_RETURN_NONE;
}

#define RS_METHOD(name) {"rs_" #name, reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(name)), METH_FASTCALL, nullptr}
#define RS_ENTRY(name) RS_METHOD(name),
PyMethodDef kMethods[] = {RS_ENTRIES(RS_ENTRY)
                          {"setup", setup, METH_VARARGS, nullptr},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_respec_bind", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__respec_bind() {
    PyObject *ctypes = PyImport_ImportModule("ctypes");
    if (!ctypes) return nullptr;
    g_argument_error = PyObject_GetAttrString(ctypes, "ArgumentError");
    g_c_int = PyObject_GetAttrString(ctypes, "c_int");
    g_c_int64 = PyObject_GetAttrString(ctypes, "c_int64");
    g_c_float = PyObject_GetAttrString(ctypes, "c_float");
    g_c_void_p = PyObject_GetAttrString(ctypes, "c_void_p");
    Py_DECREF(ctypes);
    if (!g_argument_error || !g_c_int || !g_c_int64 || !g_c_float || !g_c_void_p) return nullptr;
    PyObject *m = PyModule_Create(&kModule);
    if (m && PyModule_AddStringConstant(m, "torch_version", TORCH_VERSION) != 0) Py_CLEAR(m);
    return m;
}
