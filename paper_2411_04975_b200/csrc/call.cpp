// The host path of the calls that a serving loop makes every step (sd_speculate, sd_step,
// sd_append), from torch tensors to the C entry points.
//
// What bounds it: nothing but the host.  A draft for one request takes the GPU 6.9 us; converting
// the arguments in Python and through ctypes took 6 of the call's 8.8 us (each of up to 13 tensors
// costs four attribute lookups, each argument a converter), so a small batch waited for its launches.
// Here a tensor costs one type check and a few loads: 3.1 us for the call (most of it the launch), and
// 17.6 us (22.6 before) from an idle GPU through one such draft to its end.
//
// Only the usual case is taken here: CUDA tensors, contiguous, of the right type.  Anything else (a
// pinned host tensor, or an argument that is not one) goes to the Python function that `setup` was
// given, which returns the address or raises.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "suffixspec.h"

namespace {

decltype(&sd_speculate) f_speculate;
decltype(&sd_step) f_step;
decltype(&sd_append) f_append;
PyObject* slow_ptr;                                              // binding._ptr(tensor, dtype, name)

struct Field {
    const char* name;
    c10::ScalarType type;
    const char* dtype;                                           // the attribute of torch that names it
    PyObject* key;                                               // interned name
    PyObject* py_dtype;
};

enum { N_DRAFT, TOKENS, PARENTS, POSITIONS, MASK, CHOSEN_TREE, CHOSEN_P, SCORE, STATUS, N_OUT };
enum { SLOTS = N_OUT, OFFSETS, NEW_TOKENS, BUDGET_CAP, APPENDED, RESET, N_FIELDS };

Field fields[N_FIELDS] = {
    {"n_draft", c10::kInt, "int32"}, {"tokens", c10::kInt, "int32"}, {"parents", c10::kInt, "int32"},
    {"positions", c10::kInt, "int32"}, {"mask", c10::kInt, "int32"}, {"chosen_tree", c10::kInt, "int32"},
    {"chosen_p", c10::kInt, "int32"}, {"score", c10::kDouble, "float64"}, {"status", c10::kInt, "int32"},
    {"slots", c10::kInt, "int32"}, {"offsets", c10::kLong, "int64"}, {"new_tokens", c10::kInt, "int32"},
    {"budget_cap", c10::kInt, "int32"}, {"tokens", c10::kInt, "int32"}, {"reset", c10::kByte, "uint8"},
};

// A Python exception is already set where this is thrown.
struct Raised {};

void* address(PyObject* t, int field) {
    if (t == Py_None) return nullptr;
    const Field& f = fields[field];
    if (THPVariable_Check(t)) {
        const at::Tensor& v = THPVariable_Unpack(t);
        if (v.scalar_type() == f.type && v.is_cuda() && v.is_contiguous()) return v.data_ptr();
    }
    PyObject* r = PyObject_CallFunctionObjArgs(slow_ptr, t, f.py_dtype, f.key, nullptr);
    if (!r) throw Raised();
    void* p = r == Py_None ? nullptr : PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    if (!p && PyErr_Occurred()) throw Raised();
    return p;
}

int32_t length(PyObject* t) {
    if (THPVariable_Check(t)) return (int32_t)THPVariable_Unpack(t).numel();
    PyObject* r = PyObject_CallMethod(t, "numel", nullptr);
    if (!r) throw Raised();
    const long long n = PyLong_AsLongLong(r);
    Py_DECREF(r);
    if (n == -1 && PyErr_Occurred()) throw Raised();
    return (int32_t)n;
}

long long integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised();
    return v;
}

double real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised();
    return v;
}

void outputs(PyObject* out, void** p) {
    for (int k = 0; k < N_OUT; ++k) {
        PyObject* t = PyObject_GetItem(out, fields[k].key);
        if (!t) throw Raised();
        try {
            p[k] = address(t, k);
        } catch (...) {
            Py_DECREF(t);
            throw;
        }
        Py_DECREF(t);                                            // `out` holds it on
    }
}

bool count_is(Py_ssize_t n, Py_ssize_t want, const char* name) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "%s: %zd arguments expected, got %zd", name, want, n);
    return false;
}

sd_store* store_of(PyObject* o) {
    if (o == Py_None) return nullptr;                            // a store that was freed
    void* s = PyLong_AsVoidPtr(o);
    if (!s && PyErr_Occurred()) throw Raised();
    return (sd_store*)s;
}

sd_spec_params params(PyObject* const* a) {
    sd_spec_params p = {};
    p.P = (int32_t)integer(a[0]); p.alpha = real(a[1]); p.max_spec = (int32_t)integer(a[2]);
    p.flags = (uint32_t)integer(a[3]); p.tau = real(a[4]);
    return p;
}

// speculate(store, slots, P, alpha, max_spec, flags, tau, budget_cap, out) -> status
PyObject* speculate(PyObject*, PyObject* const* a, Py_ssize_t na) {
    HANDLE_TH_ERRORS
    if (!count_is(na, 9, "speculate")) return nullptr;
    try {
        sd_store* s = store_of(a[0]);
        const int32_t n = length(a[1]);
        const auto* slots = (const int32_t*)address(a[1], SLOTS);
        const sd_spec_params prm = params(a + 2);
        const auto* cap = (const int32_t*)address(a[7], BUDGET_CAP);
        void* o[N_OUT];
        outputs(a[8], o);
        void* st = c10::cuda::getCurrentCUDAStream().stream();
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = f_speculate(s, n, slots, &prm, cap, (int32_t*)o[N_DRAFT], (int32_t*)o[TOKENS], (int32_t*)o[PARENTS],
                         (int32_t*)o[POSITIONS], (uint32_t*)o[MASK], (int32_t*)o[CHOSEN_TREE], (int32_t*)o[CHOSEN_P],
                         (double*)o[SCORE], (int32_t*)o[STATUS], st);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    } catch (const Raised&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// step(store, slots, offsets, new_tokens, P, alpha, max_spec, flags, tau, budget_cap, out) -> status
PyObject* step(PyObject*, PyObject* const* a, Py_ssize_t na) {
    HANDLE_TH_ERRORS
    if (!count_is(na, 11, "step")) return nullptr;
    try {
        sd_store* s = store_of(a[0]);
        const int32_t n = length(a[1]);
        const auto* slots = (const int32_t*)address(a[1], SLOTS);
        const auto* off = (const int64_t*)address(a[2], OFFSETS);
        const auto* tok = (const int32_t*)address(a[3], NEW_TOKENS);
        const sd_spec_params prm = params(a + 4);
        const auto* cap = (const int32_t*)address(a[9], BUDGET_CAP);
        void* o[N_OUT];
        outputs(a[10], o);
        void* st = c10::cuda::getCurrentCUDAStream().stream();
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = f_step(s, n, slots, off, tok, &prm, cap, (int32_t*)o[N_DRAFT], (int32_t*)o[TOKENS], (int32_t*)o[PARENTS],
                    (int32_t*)o[POSITIONS], (uint32_t*)o[MASK], (int32_t*)o[CHOSEN_TREE], (int32_t*)o[CHOSEN_P],
                    (double*)o[SCORE], (int32_t*)o[STATUS], st);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    } catch (const Raised&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// append(store, slots, offsets, tokens, reset) -> status
PyObject* append(PyObject*, PyObject* const* a, Py_ssize_t na) {
    HANDLE_TH_ERRORS
    if (!count_is(na, 5, "append")) return nullptr;
    try {
        sd_store* s = store_of(a[0]);
        const int32_t n = length(a[1]);
        const auto* slots = (const int32_t*)address(a[1], SLOTS);
        const auto* off = (const int64_t*)address(a[2], OFFSETS);
        const auto* tok = (const int32_t*)address(a[3], APPENDED);
        const auto* reset = (const uint8_t*)address(a[4], RESET);
        void* st = c10::cuda::getCurrentCUDAStream().stream();
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = f_append(s, n, slots, off, tok, reset, st);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    } catch (const Raised&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// setup(addresses of sd_speculate, sd_step, sd_append, the slow way to an address)
PyObject* setup(PyObject*, PyObject* const* a, Py_ssize_t na) {
    if (!count_is(na, 4, "setup")) return nullptr;
    void* f[3];
    for (int k = 0; k < 3; ++k) {
        f[k] = PyLong_AsVoidPtr(a[k]);
        if (!f[k]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "setup: no address");
            return nullptr;
        }
    }
    PyObject* torch = PyImport_ImportModule("torch");
    if (!torch) return nullptr;
    for (Field& d : fields) {                                    // (kept for the life of the process)
        if (!d.key && !(d.key = PyUnicode_InternFromString(d.name))) return nullptr;
        if (!d.py_dtype && !(d.py_dtype = PyObject_GetAttrString(torch, d.dtype))) return nullptr;
    }
    Py_DECREF(torch);
    f_speculate = (decltype(f_speculate))f[0]; f_step = (decltype(f_step))f[1]; f_append = (decltype(f_append))f[2];
    Py_INCREF(a[3]);
    Py_XSETREF(slow_ptr, a[3]);
    Py_RETURN_NONE;
}

#define METHOD(F) {#F, (PyCFunction)(void (*)(void))F, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(speculate), METHOD(step), METHOD(append), METHOD(setup), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_call", "The per-step calls, arguments converted natively.", -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__call() { return PyModule_Create(&module_def); }
