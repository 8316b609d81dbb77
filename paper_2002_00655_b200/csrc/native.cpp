// The part of the Python binding that is called per batch, in native code: argument marshalling only, as in binding.py.
//
// A call through ctypes spends 3 to 4 us on the host around the 2 us of a kernel launch (attribute look-ups on tensors,
// argument conversion, the current stream as a Python object, an output tensor through the Python front end), which
// is most of what a call of a few rows costs.  Each function here has the name and arguments of its counterpart in
// include/ps.h, takes the same arguments, makes the same checks and raises the same errors as the ctypes form; what is not a
// tensor, a plain number or a c_void_p is handed to that form's own conversions (pointers, ctypes numbers, tensor-like
// objects).
// The library is not linked: `setup` is given the addresses of its functions, the exception to raise and the conversions.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "ps.h"

namespace {

// ---- the library's functions ----
#define PS_FUNCTIONS(X)                                                                                                \
    X(ps_pull) X(ps_push) X(ps_localize) X(ps_set_rows) X(ps_step_mf) X(ps_step_kge) X(ps_step_rescal) X(ps_step_sgns) \
        X(ps_step_mf_host) X(ps_step_kge_host) X(ps_step_sgns_host) X(ps_keymap_insert) X(ps_keymap_lookup)
#define X(f) decltype(&::f) lib_##f = nullptr;
PS_FUNCTIONS(X)
#undef X
PyObject* ps_error = nullptr;           // PSError(code, where)
PyObject* s_value = nullptr;            // "value"
PyObject* c_void_p = nullptr;           // ctypes.c_void_p
PyObject* convert = nullptr;            // convert(what, object) -> int, float or (pointer, number of elements), as ctypes and binding.py do

enum Kind { kU32, kU64, kF32, kF64, kU8 };
const char* const kKindNames[] = {"(torch.int32, torch.uint32)", "(torch.int64, torch.uint64)", "(torch.float32,)",
                                  "(torch.float64,)", "(torch.uint8,)"};
bool is_kind(at::ScalarType t, Kind k) {
    switch (k) {
        case kU32: return t == at::kInt || t == at::kUInt32;
        case kU64: return t == at::kLong || t == at::kUInt64;
        case kF32: return t == at::kFloat;
        case kF64: return t == at::kDouble;
        default: return t == at::kByte;
    }
}

// One call's arguments; `bad` after the first that does not fit (a Python error is set then).
struct Args {
    PyObject* const* a;
    Py_ssize_t n, at = 0;
    bool bad = false;

    PyObject* next() { return at < n ? a[at++] : nullptr; }
    void fail() { bad = true; }
    PyObject* converted(const char* what, PyObject* o) { return PyObject_CallFunction(convert, "sO", what, o); }
    template <class T> T* handle() {                        // a ctypes c_void_p, an integer or None
        PyObject* o = next();
        if (bad || !o || o == Py_None) return nullptr;
        PyObject* v = PyLong_Check(o) ? Py_NewRef(o) : (PyObject*)Py_TYPE(o) == c_void_p ? PyObject_GetAttr(o, s_value) : converted("handle", o);
        if (!v) return fail(), nullptr;
        void* p = v == Py_None ? nullptr : PyLong_AsVoidPtr(v);
        Py_DECREF(v);
        if (!p && PyErr_Occurred()) fail();
        return (T*)p;
    }
    // pointer of a contiguous tensor on the GPU (cuda) or the host; None: NULL.  *numel: its number of elements
    template <class T> T* tensor(Kind k, bool cuda = true, uint64_t* numel = nullptr) {
        PyObject* o = next();
        if (bad) return nullptr;
        if (!o || o == Py_None) {
            if (numel) {                                    // (this argument's length is the call's)
                PyErr_SetString(PyExc_AttributeError, "expected a tensor, got None");
                fail();
            }
            return nullptr;
        }
        if (!THPVariable_Check(o)) {
            char what[] = {cuda ? 'd' : 'h', (char)('0' + k), 0};
            PyObject* pair = converted(what, o);
            unsigned long long p = 0, n = 0;
            const bool ok = pair && PyArg_ParseTuple(pair, "KK", &p, &n);
            Py_XDECREF(pair);
            if (!ok) return fail(), nullptr;
            if (numel) *numel = n;
            return (T*)(uintptr_t)p;
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (t.is_cuda() != cuda || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, cuda ? "expected a contiguous CUDA tensor" : "expected a contiguous CPU tensor");
            return fail(), nullptr;
        }
        if (!is_kind(t.scalar_type(), k)) {
            if (PyObject* d = PyObject_GetAttrString(o, "dtype")) {
                PyErr_Format(PyExc_AssertionError, "expected dtype in %s, got %S", kKindNames[k], d);
                Py_DECREF(d);
            }
            return fail(), nullptr;
        }
        if (numel) *numel = (uint64_t)t.numel();
        return (T*)t.data_ptr();
    }
    uint64_t u64(const char* what = "u64") {
        PyObject* o = next();
        if (bad) return 0;
        PyObject* i = !o ? nullptr : PyIndex_Check(o) ? PyNumber_Index(o) : converted(what, o);
        if (!i) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "an integer is missing");
            return fail(), 0;
        }
        const unsigned long long v = PyLong_AsUnsignedLongLongMask(i);
        Py_DECREF(i);
        return v;
    }
    uint32_t u32() { return (uint32_t)u64("u32"); }
    float f32() {
        PyObject* o = next();
        if (bad) return 0.f;
        double v = o ? PyFloat_AsDouble(o) : -1.0;
        if (!o) PyErr_SetString(PyExc_TypeError, "a number is missing");
        if (o && v == -1.0 && PyErr_Occurred()) {               // (a c_float; anything else raises again)
            PyErr_Clear();
            PyObject* f = converted("f32", o);
            v = f ? PyFloat_AsDouble(f) : -1.0;
            Py_XDECREF(f);
        }
        if (PyErr_Occurred()) fail();
        return (float)v;
    }
};

void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

PyObject* done(ps_status_t code, const char* where) {
    if (code == PS_OK) Py_RETURN_NONE;
    PyObject* e = PyObject_CallFunction(ps_error, "is", (int)code, where);
    if (e) {
        PyErr_SetObject(ps_error, e);
        Py_DECREF(e);
    }
    return nullptr;
}

// calls into the library without the interpreter's lock, as ctypes does
#define CALL(name, ...)                     \
    do {                                    \
        if (A.bad) return nullptr;          \
        void* st = stream();                \
        ps_status_t code;                   \
        Py_BEGIN_ALLOW_THREADS;             \
        code = lib_##name(__VA_ARGS__, st); \
        Py_END_ALLOW_THREADS;               \
        return done(code, #name);           \
    } while (0)

#define FUNCTION(f) PyObject* py_##f(PyObject*, PyObject* const* args, Py_ssize_t nargs)
#define BEGIN        \
    HANDLE_TH_ERRORS \
    Args A{args, nargs}
#define END return nullptr; END_HANDLE_TH_ERRORS

FUNCTION(ps_pull) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    uint64_t n = 0;
    auto* keys = A.tensor<uint64_t>(kU64, true, &n);
    auto* out = A.tensor<float>(kF32);
    CALL(ps_pull, ps, keys, n, out);
    END
}
FUNCTION(ps_push) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    uint64_t n = 0;
    auto* keys = A.tensor<uint64_t>(kU64, true, &n);
    auto* upd = A.tensor<float>(kF32);
    CALL(ps_push, ps, keys, n, upd);
    END
}
FUNCTION(ps_set_rows) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    uint64_t n = 0;
    auto* keys = A.tensor<uint64_t>(kU64, true, &n);
    auto* vals = A.tensor<float>(kF32);
    CALL(ps_set_rows, ps, keys, n, vals);
    END
}
FUNCTION(ps_localize) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    const uint32_t worker = A.u32();
    uint64_t n = 0;
    auto* keys = A.tensor<uint64_t>(kU64, true, &n);
    CALL(ps_localize, ps, worker, keys, n);
    END
}
FUNCTION(ps_step_mf) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    uint64_t n = 0;
    auto* i = A.tensor<uint32_t>(kU32, true, &n);
    auto* j = A.tensor<uint32_t>(kU32);
    auto* v = A.tensor<float>(kF32);
    const uint64_t base = A.u64();
    const float lr = A.f32(), lam = A.f32();
    auto* loss = A.tensor<double>(kF64);
    CALL(ps_step_mf, ps, i, j, v, n, base, lr, lam, loss);
    END
}
FUNCTION(ps_step_mf_host) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    uint64_t n = 0;
    auto* i = A.tensor<uint32_t>(kU32, false, &n);
    auto* j = A.tensor<uint32_t>(kU32, false);
    auto* v = A.tensor<float>(kF32, false);
    const uint64_t base = A.u64();
    const float lr = A.f32(), lam = A.f32();
    auto* loss = A.tensor<double>(kF64);
    auto* h_loss = A.tensor<double>(kF64, false);
    CALL(ps_step_mf_host, ps, i, j, v, n, base, lr, lam, loss, h_loss);
    END
}
struct Triples {
    uint32_t *s, *r, *o, *neg;
    uint8_t* side;
    uint64_t n = 0, base;
    uint32_t n_neg, dim;
    float lr, eps;
    Triples(Args& A, bool cuda) {
        s = A.tensor<uint32_t>(kU32, cuda, &n);
        r = A.tensor<uint32_t>(kU32, cuda);
        o = A.tensor<uint32_t>(kU32, cuda);
        neg = A.tensor<uint32_t>(kU32, cuda);
        side = A.tensor<uint8_t>(kU8, cuda);
        n_neg = A.u32();
        base = A.u64();
        dim = A.u32();
        lr = A.f32();
        eps = A.f32();
    }
};
FUNCTION(ps_step_kge) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    const Triples t(A, true);
    auto* loss = A.tensor<double>(kF64);
    CALL(ps_step_kge, ps, t.s, t.r, t.o, t.neg, t.side, t.n, t.n_neg, t.base, t.dim, t.lr, t.eps, loss);
    END
}
FUNCTION(ps_step_rescal) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    const Triples t(A, true);
    auto* loss = A.tensor<double>(kF64);
    CALL(ps_step_rescal, ps, t.s, t.r, t.o, t.neg, t.side, t.n, t.n_neg, t.base, t.dim, t.lr, t.eps, loss);
    END
}
FUNCTION(ps_step_kge_host) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    const Triples t(A, false);
    auto* loss = A.tensor<double>(kF64);
    auto* h_loss = A.tensor<double>(kF64, false);
    CALL(ps_step_kge_host, ps, t.s, t.r, t.o, t.neg, t.side, t.n, t.n_neg, t.base, t.dim, t.lr, t.eps, loss, h_loss);
    END
}
FUNCTION(ps_step_sgns) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    uint64_t corpus = 0;
    auto* tokens = A.tensor<uint32_t>(kU32, true, &corpus);
    const uint64_t first = A.u64(), n = A.u64();
    const uint32_t window = A.u32();
    auto* negs = A.tensor<uint32_t>(kU32);
    const uint32_t n_neg = A.u32();
    const uint64_t base = A.u64();
    const float lr = A.f32();
    auto* loss = A.tensor<double>(kF64);
    CALL(ps_step_sgns, ps, tokens, first, n, corpus, window, negs, n_neg, base, lr, loss);
    END
}
FUNCTION(ps_step_sgns_host) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    uint64_t count = 0, n_negs = 0;
    auto* tokens = A.tensor<uint32_t>(kU32, false, &count);
    const uint64_t tok_first = A.u64(), first = A.u64(), n = A.u64(), corpus = A.u64();
    const uint32_t window = A.u32();
    auto* negs = A.tensor<uint32_t>(kU32, false, &n_negs);
    const uint32_t n_neg = A.u32();
    const uint64_t base = A.u64();
    const float lr = A.f32();
    auto* loss = A.tensor<double>(kF64);
    auto* h_loss = A.tensor<double>(kF64, false);
    CALL(ps_step_sgns_host, ps, tokens, tok_first, count, first, n, corpus, window, negs, n_negs, n_neg, base, lr, loss, h_loss);
    END
}
FUNCTION(ps_keymap_insert) {
    BEGIN;
    auto* m = A.handle<ps_keymap_t>();
    uint64_t n = 0;
    auto* in = A.tensor<uint64_t>(kU64, true, &n);
    auto* out = A.tensor<uint64_t>(kU64);
    CALL(ps_keymap_insert, m, in, n, out);
    END
}
FUNCTION(ps_keymap_lookup) {
    BEGIN;
    auto* m = A.handle<ps_keymap_t>();
    uint64_t n = 0;
    auto* in = A.tensor<uint64_t>(kU64, true, &n);
    auto* out = A.tensor<uint64_t>(kU64);
    CALL(ps_keymap_lookup, m, in, n, out);
    END
}

// ---- calls that return a new tensor: (handle, keys, device ordinal[, row length]) ----
template <class F> PyObject* into_new(at::Tensor out, const char* where, F call) {
    ps_status_t code;
    Py_BEGIN_ALLOW_THREADS;
    code = call();
    Py_END_ALLOW_THREADS;
    if (code == PS_OK) return THPVariable_Wrap(std::move(out));
    return done(code, where);
}
at::TensorOptions on_gpu(uint64_t device, at::ScalarType t) {
    return at::TensorOptions().dtype(t).device(at::kCUDA, (c10::DeviceIndex)device);
}
PyObject* py_pull_rows(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    BEGIN;
    auto* ps = A.handle<ps_store_t>();
    uint64_t n = 0;
    auto* keys = A.tensor<uint64_t>(kU64, true, &n);
    const uint64_t device = A.u64(), row = A.u64();
    if (A.bad) return nullptr;
    at::Tensor out = at::empty({(int64_t)n, (int64_t)row}, on_gpu(device, at::kFloat));
    float* to = (float*)out.data_ptr();
    void* st = stream();
    return into_new(std::move(out), "ps_pull", [&] { return lib_ps_pull(ps, keys, n, to, st); });
    END
}
template <bool kInsert> PyObject* map_keys(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    BEGIN;
    auto* m = A.handle<ps_keymap_t>();
    uint64_t n = 0;
    auto* in = A.tensor<uint64_t>(kU64, true, &n);
    const uint64_t device = A.u64();
    if (A.bad) return nullptr;
    at::Tensor out = at::empty({(int64_t)n}, on_gpu(device, at::kLong));
    uint64_t* to = (uint64_t*)out.data_ptr();
    void* st = stream();
    return into_new(std::move(out), kInsert ? "ps_keymap_insert" : "ps_keymap_lookup",
                    [&] { return (kInsert ? lib_ps_keymap_insert : lib_ps_keymap_lookup)(m, in, n, to, st); });
    END
}

// setup({name: address}, exception class, ctypes.c_void_p, convert)
PyObject* py_setup(PyObject*, PyObject* args) {
    PyObject *addresses, *error, *void_p, *conv;
    if (!PyArg_ParseTuple(args, "O!OOO", &PyDict_Type, &addresses, &error, &void_p, &conv)) return nullptr;
#define X(f)                                                                          \
    {                                                                                 \
        PyObject* v = PyDict_GetItemString(addresses, #f);                            \
        void* p = v ? PyLong_AsVoidPtr(v) : nullptr;                                  \
        if (!p) {                                                                     \
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_KeyError, #f);               \
            return nullptr;                                                           \
        }                                                                             \
        lib_##f = (decltype(lib_##f))p;                                               \
    }
    PS_FUNCTIONS(X)
#undef X
    Py_XSETREF(ps_error, Py_NewRef(error));
    Py_XSETREF(c_void_p, Py_NewRef(void_p));
    Py_XSETREF(convert, Py_NewRef(conv));
    Py_RETURN_NONE;
}

#define METHOD(f) {#f, (PyCFunction)(void (*)(void))py_##f, METH_FASTCALL, nullptr},
PyMethodDef methods[] = {
    {"setup", py_setup, METH_VARARGS, nullptr},
    PS_FUNCTIONS(METHOD)
    {"pull_rows", (PyCFunction)(void (*)(void))py_pull_rows, METH_FASTCALL, nullptr},
    {"map_insert", (PyCFunction)(void (*)(void))map_keys<true>, METH_FASTCALL, nullptr},
    {"map_lookup", (PyCFunction)(void (*)(void))map_keys<false>, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
    s_value = PyUnicode_InternFromString("value");
    PyObject* m = s_value ? PyModule_Create(&module) : nullptr;
    if (m && PyModule_AddStringConstant(m, "torch_version", PS_TORCH_VERSION) < 0) Py_CLEAR(m);
    return m;
}
