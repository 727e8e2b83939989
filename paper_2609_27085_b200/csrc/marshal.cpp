// CPython marshalling of the entry points that a serving loop calls for every layer or every step.
//
// Through ctypes an append + attention pair cost 26.5 us of host time per pass in argument conversion alone - more than
// the library spends on planning and launching a small batch - and a batch of a few short sequences is bound by host
// time.  Here an argument costs a type check and a load: 1.6 us per pair (same machine, both calls refused at once).
// The library itself is loaded by the Python module, which hands over the addresses of its functions (bind); nothing
// here computes or keeps anything.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>
#include <cstring>

#include "../../include/crossflow_attn.h"

namespace {

struct Entries {
    decltype(&cf_kv_append) kv_append;
    decltype(&cf_mixed_attention) mixed_attention;
    decltype(&cf_mixed_attention_shared) mixed_attention_shared;
    decltype(&cf_kv_append_planned) kv_append_planned;
    decltype(&cf_mixed_attention_planned) mixed_attention_planned;
    decltype(&cf_mixed_step_host) mixed_step_host;
    decltype(&cf_host_steps_flush) host_steps_flush;
    decltype(&cf_decode_attention_static) decode_attention_static;
} lib;
PyObject* to_int32 = nullptr;      // Python function: anything array-like -> contiguous int32 array
PyObject *s_data_ptr = nullptr, *s_cuda_stream = nullptr;

bool integer(PyObject* o, uint64_t* out)
{
    if (PyLong_Check(o)) {
        *out = (uint64_t)PyLong_AsUnsignedLongLongMask(o);
        return !PyErr_Occurred();
    }
    PyObject* n = PyNumber_Long(o);
    if (!n) return false;
    *out = (uint64_t)PyLong_AsUnsignedLongLongMask(n);
    Py_DECREF(n);
    return !PyErr_Occurred();
}

// device or host address: None, an integer, or an object with data_ptr() (a torch tensor)
template <class T>
bool address(PyObject* o, T* out)
{
    uint64_t v = 0;
    if (o != Py_None) {
        if (PyLong_Check(o)) {
            if (!integer(o, &v)) return false;
        } else {
            PyObject* r = PyObject_CallMethodNoArgs(o, s_data_ptr);
            if (!r) {
                if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
                PyErr_Clear();
                if (!integer(o, &v)) return false;
            } else {
                const bool ok = integer(r, &v);
                Py_DECREF(r);
                if (!ok) return false;
            }
        }
    }
    *out = (T)(uintptr_t)v;
    return true;
}

// opaque handle: None, an integer, or a ctypes.c_void_p
template <class T>
bool handle(PyObject* o, T** out)
{
    uint64_t v = 0;
    if (o != Py_None) {
        if (PyLong_Check(o)) {
            if (!integer(o, &v)) return false;
        } else {
            Py_buffer b;
            if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
            const bool ok = b.len == (Py_ssize_t)sizeof(void*);
            if (ok) std::memcpy(&v, b.buf, sizeof v);
            PyBuffer_Release(&b);
            if (!ok) {
                PyErr_SetString(PyExc_TypeError, "a handle returned by this module is wanted");
                return false;
            }
        }
    }
    *out = (T*)(uintptr_t)v;
    return true;
}

bool int32(PyObject* o, int32_t* out)
{
    uint64_t v;
    if (!integer(o, &v)) return false;
    *out = (int32_t)v;
    return true;
}

bool stream_of(PyObject* o, void** out)
{
    uint64_t v = 0;
    if (o != Py_None) {
        if (PyLong_Check(o)) {
            if (!integer(o, &v)) return false;
        } else {
            PyObject* r = PyObject_GetAttr(o, s_cuda_stream);
            if (!r) {
                if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
                PyErr_Clear();
                if (!integer(o, &v)) return false;
            } else {
                const bool ok = integer(r, &v);
                Py_DECREF(r);
                if (!ok) return false;
            }
        }
    }
    *out = (void*)(uintptr_t)v;
    return true;
}

// A buffer held for the length of a call: the cache descriptor, or an int32 length array (converted if it is not one).
struct Held {
    Py_buffer b;
    bool held = false;
    ~Held()
    {
        if (held) PyBuffer_Release(&b);
    }
    bool desc(PyObject* o, const cf_cache_desc** out)
    {
        if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
        held = true;
        if (b.len != (Py_ssize_t)sizeof(cf_cache_desc)) {
            PyErr_SetString(PyExc_TypeError, "a CacheDesc is wanted");
            return false;
        }
        *out = (const cf_cache_desc*)b.buf;
        return true;
    }
    bool lengths(PyObject* o, const int32_t** out, int32_t* n)
    {
        if (PyObject_GetBuffer(o, &b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) == 0) held = true;
        else PyErr_Clear();
        if (!held || b.itemsize != 4 || b.ndim < 1 || !b.format || b.format[0] != 'i' || b.format[1] != 0) {
            if (held) {
                PyBuffer_Release(&b);
                held = false;
            }
            PyObject* a = PyObject_CallOneArg(to_int32, o);
            if (!a) return false;
            const int rc = PyObject_GetBuffer(a, &b, PyBUF_C_CONTIGUOUS);
            Py_DECREF(a);                          // the buffer keeps the array alive
            if (rc != 0) return false;
            held = true;
            if (b.ndim < 1) {
                PyErr_SetString(PyExc_TypeError, "a sequence of lengths is wanted");
                return false;
            }
        }
        *out = (const int32_t*)b.buf;
        *n = (int32_t)b.shape[0];
        return true;
    }
};

bool arity(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments are wanted, got %zd", want, n);
    return false;
}

// context_len says how many sequences there are; the other arrays have a value for each of them (or more: a caller may hand
// over the front of padded arrays)
bool enough(int32_t seqs, int32_t n)
{
    if (n >= seqs) return true;
    PyErr_SetString(PyExc_ValueError, "a length array is shorter than context_len");
    return false;
}

template <class F>
PyObject* status(F call)
{
    cf_status st;
    Py_BEGIN_ALLOW_THREADS
    st = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

PyObject* py_kv_append(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    cf_ctx* ctx; const cf_cache_desc* d; void *k, *v, *s; const void *kn, *vn; const int32_t *bt, *lc, *lq; int32_t mb, S, S2;
    Held hd, hc, hq;
    if (!arity(n, 11) || !handle(a[0], &ctx) || !hd.desc(a[1], &d) || !address(a[2], &k) || !address(a[3], &v) || !address(a[4], &kn) ||
        !address(a[5], &vn) || !address(a[6], &bt) || !int32(a[7], &mb) || !hc.lengths(a[8], &lc, &S) || !hq.lengths(a[9], &lq, &S2) ||
        !enough(S, S2) || !stream_of(a[10], &s))
        return nullptr;
    return status([&] { return lib.kv_append(ctx, d, k, v, kn, vn, bt, mb, lc, lq, S, s); });
}

PyObject* py_mixed_attention(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    cf_ctx* ctx; const cf_cache_desc* d; void *out, *s; const void *q, *k, *v; float* lse; const int32_t *bt, *lc, *lq; int32_t mb, S, S2;
    Held hd, hc, hq;
    if (!arity(n, 12) || !handle(a[0], &ctx) || !hd.desc(a[1], &d) || !address(a[2], &q) || !address(a[3], &k) || !address(a[4], &v) ||
        !address(a[5], &bt) || !int32(a[6], &mb) || !hc.lengths(a[7], &lc, &S) || !hq.lengths(a[8], &lq, &S2) || !enough(S, S2) ||
        !address(a[9], &out) || !address(a[10], &lse) || !stream_of(a[11], &s))
        return nullptr;
    return status([&] { return lib.mixed_attention(ctx, d, q, k, v, bt, mb, lc, lq, S, out, lse, s); });
}

PyObject* py_mixed_attention_shared(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    cf_ctx* ctx; const cf_cache_desc* d; void *out, *s; const void *q, *k, *v; float* lse; const int32_t *bt, *lc, *lq, *sg, *sl;
    int32_t mb, S, S2, S3, S4;
    Held hd, hc, hq, hg, hl;
    if (!arity(n, 14) || !handle(a[0], &ctx) || !hd.desc(a[1], &d) || !address(a[2], &q) || !address(a[3], &k) || !address(a[4], &v) ||
        !address(a[5], &bt) || !int32(a[6], &mb) || !hc.lengths(a[7], &lc, &S) || !hq.lengths(a[8], &lq, &S2) || !enough(S, S2) ||
        !hg.lengths(a[9], &sg, &S3) || !enough(S, S3) || !hl.lengths(a[10], &sl, &S4) || !enough(S, S4) || !address(a[11], &out) ||
        !address(a[12], &lse) || !stream_of(a[13], &s))
        return nullptr;
    return status([&] { return lib.mixed_attention_shared(ctx, d, q, k, v, bt, mb, lc, lq, sg, sl, S, out, lse, s); });
}

PyObject* py_kv_append_planned(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    cf_plan* plan; void *k, *v, *s; const void *kn, *vn; const int32_t* bt;
    if (!arity(n, 7) || !handle(a[0], &plan) || !address(a[1], &k) || !address(a[2], &v) || !address(a[3], &kn) || !address(a[4], &vn) ||
        !address(a[5], &bt) || !stream_of(a[6], &s))
        return nullptr;
    return status([&] { return lib.kv_append_planned(plan, k, v, kn, vn, bt, s); });
}

PyObject* py_mixed_attention_planned(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    cf_plan* plan; void *out, *s; const void *q, *k, *v; float* lse; const int32_t* bt;
    if (!arity(n, 8) || !handle(a[0], &plan) || !address(a[1], &q) || !address(a[2], &k) || !address(a[3], &v) || !address(a[4], &bt) ||
        !address(a[5], &out) || !address(a[6], &lse) || !stream_of(a[7], &s))
        return nullptr;
    return status([&] { return lib.mixed_attention_planned(plan, q, k, v, bt, out, lse, s); });
}

PyObject* py_mixed_step_host(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    cf_ctx* ctx; const cf_cache_desc* d; void *out, *k, *v, *s; const void *q, *kn, *vn; const int32_t *bt, *lc, *lq; int32_t mb, S, S2;
    Held hd, hc, hq;
    if (!arity(n, 13) || !handle(a[0], &ctx) || !hd.desc(a[1], &d) || !address(a[2], &q) || !address(a[3], &kn) || !address(a[4], &vn) ||
        !address(a[5], &k) || !address(a[6], &v) || !address(a[7], &bt) || !int32(a[8], &mb) || !hc.lengths(a[9], &lc, &S) ||
        !hq.lengths(a[10], &lq, &S2) || !enough(S, S2) || !address(a[11], &out) || !stream_of(a[12], &s))
        return nullptr;
    return status([&] { return lib.mixed_step_host(ctx, d, q, kn, vn, k, v, bt, mb, lc, lq, S, out, s); });
}

PyObject* py_host_steps_flush(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    cf_ctx* ctx; void* s;
    if (!arity(n, 2) || !handle(a[0], &ctx) || !stream_of(a[1], &s)) return nullptr;
    return status([&] { return lib.host_steps_flush(ctx, s); });
}

PyObject* py_decode_attention_static(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    const cf_cache_desc* d; void *out, *s; const void *q, *k, *v; float* lse; const int32_t *bt, *lc; int32_t mb, S;
    Held hd, hc;
    if (!arity(n, 10) || !hd.desc(a[0], &d) || !address(a[1], &q) || !address(a[2], &k) || !address(a[3], &v) || !address(a[4], &bt) ||
        !int32(a[5], &mb) || !hc.lengths(a[6], &lc, &S) || !address(a[7], &out) || !address(a[8], &lse) || !stream_of(a[9], &s))
        return nullptr;
    return status([&] { return lib.decode_attention_static(d, q, k, v, bt, mb, lc, S, out, lse, s); });
}

// bind(to_int32, addresses of the eight entry points in the order of Entries)
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    void* f[8];
    static_assert(sizeof f == sizeof lib, "one address per entry");
    if (!arity(n, 9)) return nullptr;
    for (int i = 0; i < 8; ++i)
        if (!address(a[1 + i], &f[i])) return nullptr;
    std::memcpy(&lib, f, sizeof lib);
    Py_XSETREF(to_int32, Py_NewRef(a[0]));
    Py_RETURN_NONE;
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY(kv_append), ENTRY(mixed_attention), ENTRY(mixed_attention_shared), ENTRY(kv_append_planned),
                         ENTRY(mixed_attention_planned), ENTRY(mixed_step_host), ENTRY(host_steps_flush),
                         ENTRY(decode_attention_static), ENTRY(bind), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!s_data_ptr || !s_cuda_stream) return nullptr;
    return PyModule_Create(&module);
}
