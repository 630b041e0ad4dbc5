// CPython entry points of the calls a model makes once per layer and step: the functions of
// include/evln.h by their C names, taking torch tensors.
//
// A step of a few tokens keeps the GPU busy for less time than ctypes needs to marshal its call
// (a 16-argument evlnStep: 9 us of argument conversion around 7 us of kernel launches), so these
// calls read the tensors' addresses, strides and the current stream straight from the C++ objects.
// Measured per evlnStep call on the host, three launches included: 16.5 us through ctypes, see the
// figure beside kHotCalls in binding.py for this file.  No arithmetic happens here.
#include <torch/csrc/autograd/python_variable.h>

#include <c10/cuda/CUDAStream.h>

#include <string.h>

#include <vector>

#include "../../include/evln.h"

namespace {

// what binding.py hands over once (configure): the parameter structures, the exceptions
PyTypeObject* g_step_type = nullptr;
PyTypeObject* g_paged_type = nullptr;
PyTypeObject* g_packed_type = nullptr;
PyTypeObject* g_gather_type = nullptr;
PyObject* g_error = nullptr;             // EvlnError(status, where)
PyObject* g_argument_error = nullptr;    // a parameter structure of the wrong type

// ---- arguments -------------------------------------------------------------------------------

constexpr int kMaxArgs = 16;

// Positional and keyword arguments of a call into `slots` (in the order of `names`, which ends with
// nullptr); the first `required` must be given.
bool take_args(const char* where, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames, const char* const* names,
               int required, PyObject** slots)
{
    int count = 0;
    while (names[count]) { slots[count] = nullptr; ++count; }
    if (nargs > count) {
        PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", where, count, nargs);
        return false;
    }
    for (Py_ssize_t i = 0; i < nargs; ++i) slots[i] = args[i];
    const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nkw; ++k) {
        PyObject* name = PyTuple_GET_ITEM(kwnames, k);
        int at = -1;
        for (int i = 0; i < count && at < 0; ++i)
            if (PyUnicode_CompareWithASCIIString(name, names[i]) == 0) at = i;
        if (at < 0) {
            PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", where, name);
            return false;
        }
        if (slots[at]) {
            PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%U'", where, name);
            return false;
        }
        slots[at] = args[nargs + k];
    }
    for (int i = 0; i < required; ++i) {
        if (!slots[i]) {
            PyErr_Format(PyExc_TypeError, "%s() missing required argument '%s'", where, names[i]);
            return false;
        }
    }
    for (int i = required; i < count; ++i)
        if (slots[i] == Py_None) slots[i] = nullptr;
    return true;
}

bool is_none(PyObject* o) { return o == nullptr || o == Py_None; }

bool as_long(PyObject* o, long* v)
{
    if (PyLong_Check(o)) {
        *v = PyLong_AsLong(o);
    } else {
        PyObject* n = PyNumber_Long(o);       // whatever int() takes
        if (!n) return false;
        *v = PyLong_AsLong(n);
        Py_DECREF(n);
    }
    return !(*v == -1 && PyErr_Occurred());
}

bool as_int(PyObject* o, int* v)
{
    long l;
    if (!as_long(o, &l)) return false;
    *v = (int)l;
    return true;
}

// Address of a tensor (or of anything with data_ptr()), None -> NULL; plain integers pass through.
bool as_pointer(PyObject* o, void** p)
{
    if (is_none(o)) { *p = nullptr; return true; }
    if (THPVariable_Check(o)) { *p = THPVariable_Unpack(o).data_ptr(); return true; }
    if (PyLong_Check(o)) {
        *p = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
        return !PyErr_Occurred();
    }
    PyObject* r = PyObject_CallMethod(o, "data_ptr", nullptr);
    if (!r) return false;
    *p = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(r);
    Py_DECREF(r);
    return !PyErr_Occurred();
}

// The memory of a ctypes object (a parameter structure, a c_void_p).
bool ctypes_memory(PyObject* o, void* to, size_t bytes)
{
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
    const bool fits = (size_t)b.len == bytes;
    if (fits) memcpy(to, b.buf, bytes);
    PyBuffer_Release(&b);
    if (!fits) PyErr_SetString(g_argument_error, "unexpected size of a ctypes argument");
    return fits;
}

template <typename P>
bool as_params(PyObject* o, PyTypeObject* type, P* p)
{
    if (!type || !PyObject_TypeCheck(o, type)) {
        PyErr_Format(g_argument_error ? g_argument_error : PyExc_TypeError, "expected %s, got %s", type ? type->tp_name : "params",
                     Py_TYPE(o)->tp_name);
        return false;
    }
    return ctypes_memory(o, p, sizeof(P));
}

bool as_handle(PyObject* o, evlnHandle_t* h)
{
    if (is_none(o)) { *h = nullptr; return true; }
    if (PyLong_Check(o)) {
        *h = (evlnHandle_t)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
        return !PyErr_Occurred();
    }
    void* v = nullptr;
    if (!ctypes_memory(o, &v, sizeof(v))) return false;
    *h = (evlnHandle_t)v;
    return true;
}

// None: the current stream of the current device; an integer; or a torch stream.
bool as_stream(PyObject* o, void** st)
{
    if (is_none(o)) { *st = (void*)c10::cuda::getCurrentCUDAStream().stream(); return true; }
    if (PyLong_Check(o)) {
        *st = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
        return !PyErr_Occurred();
    }
    PyObject* r = PyObject_GetAttrString(o, "cuda_stream");
    if (!r) return false;
    *st = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(r);
    Py_DECREF(r);
    return !PyErr_Occurred();
}

bool as_ints(PyObject* o, std::vector<int>* v)
{
    PyObject* seq = PySequence_Fast(o, "expected a sequence of integers");
    if (!seq) return false;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    v->resize((size_t)n);
    bool ok = true;
    for (Py_ssize_t i = 0; i < n && ok; ++i) ok = as_int(PySequence_Fast_GET_ITEM(seq, i), &(*v)[(size_t)i]);
    Py_DECREF(seq);
    return ok;
}

// stride(0) of a tensor argument
bool token_stride(PyObject* o, long* s)
{
    if (THPVariable_Check(o)) { *s = (long)THPVariable_Unpack(o).stride(0); return true; }
    PyObject* r = PyObject_CallMethod(o, "stride", "i", 0);
    if (!r) return false;
    const bool ok = as_long(r, s);
    Py_DECREF(r);
    return ok;
}

// strides of q, k, v: the `strides` argument or the tensors' own
bool token_strides(PyObject* strides, PyObject* q, PyObject* k, PyObject* v, long* s)
{
    if (is_none(strides)) return token_stride(q, &s[0]) && token_stride(k, &s[1]) && token_stride(v, &s[2]);
    PyObject* seq = PySequence_Fast(strides, "strides: three token strides");
    if (!seq) return false;
    bool ok = PySequence_Fast_GET_SIZE(seq) >= 3;
    if (!ok) PyErr_SetString(PyExc_IndexError, "strides: three token strides");
    for (int i = 0; i < 3 && ok; ++i) ok = as_long(PySequence_Fast_GET_ITEM(seq, i), &s[i]);
    Py_DECREF(seq);
    return ok;
}

// bytes of a buffer argument: given, or those of the tensor
bool buffer_bytes(PyObject* given, PyObject* t, size_t* bytes)
{
    if (!is_none(given)) {
        long v;
        if (!as_long(given, &v)) return false;
        *bytes = (size_t)v;
        return true;
    }
    if (t && THPVariable_Check(t)) { *bytes = THPVariable_Unpack(t).nbytes(); return true; }
    long numel = 0, each = 0;
    for (int i = 0; i < 2; ++i) {
        PyObject* r = PyObject_CallMethod(t ? t : Py_None, i == 0 ? "numel" : "element_size", nullptr);
        if (!r) return false;
        const bool ok = as_long(r, i == 0 ? &numel : &each);
        Py_DECREF(r);
        if (!ok) return false;
    }
    *bytes = (size_t)numel * (size_t)each;
    return true;
}

PyObject* finish(int status, const char* where)
{
    if (status == EVLN_OK) Py_RETURN_NONE;
    PyObject* e = g_error ? PyObject_CallFunction(g_error, "is", status, where) : nullptr;
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    } else if (!PyErr_Occurred()) {
        PyErr_Format(PyExc_RuntimeError, "%s: status %d", where, status);
    }
    return nullptr;
}

// A call into the library without the interpreter lock (a launch blocks when the stream's queue is full).
template <typename F>
int unlocked(F&& call)
{
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = (int)call();
    Py_END_ALLOW_THREADS
    return s;
}

// Runs an entry point; a C++ exception (no CUDA device, a tensor without storage) becomes RuntimeError.
template <typename F>
PyObject* guarded(F&& f)
{
    try {
        return f();
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// ---- the entry points ----------------------------------------------------------------------------

#define EVLN_ENTRY(fn) PyObject* fn(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames)

EVLN_ENTRY(py_rope_table)
{
    static const char* const names[] = {"handle", "head_dim", "rope_theta", "first_pos", "count", "table", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnRopeTable", args, nargs, kwnames, names, 6, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        int head_dim, first, count;
        void *table, *st;
        if (!as_handle(a[0], &h) || !as_int(a[1], &head_dim)) return nullptr;
        const double theta = PyFloat_AsDouble(a[2]);
        if (theta == -1.0 && PyErr_Occurred()) return nullptr;
        if (!as_int(a[3], &first) || !as_int(a[4], &count) || !as_pointer(a[5], &table) || !as_stream(a[6], &st)) return nullptr;
        return finish(unlocked([&] { return evlnRopeTable(h, head_dim, theta, first, count, table, st); }), "evlnRopeTable");
    });
}

EVLN_ENTRY(py_rope_append)
{
    static const char* const names[] = {"handle", "params", "q_new", "k_new", "v_new", "q_rot", "k_cache", "v_cache", "stream", "strides", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnRopeAppend", args, nargs, kwnames, names, 8, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnStepParams p;
        void* t[6];
        void* st;
        long s[3];
        if (!token_strides(a[9], a[2], a[3], a[4], s) || !as_handle(a[0], &h) || !as_params(a[1], g_step_type, &p)) return nullptr;
        for (int i = 0; i < 6; ++i)
            if (!as_pointer(a[2 + i], &t[i])) return nullptr;
        if (!as_stream(a[8], &st)) return nullptr;
        return finish(unlocked([&] { return evlnRopeAppend(h, &p, t[0], t[1], t[2], s[0], s[1], s[2], t[3], t[4], t[5], st); }), "evlnRopeAppend");
    });
}

EVLN_ENTRY(py_step_attention)
{
    static const char* const names[] = {"handle", "params", "q_rot", "k_cache", "v_cache", "workspace", "workspace_bytes", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnStepAttention", args, nargs, kwnames, names, 6, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnStepParams p;
        void* t[4];
        void* st;
        size_t bytes;
        if (!buffer_bytes(a[6], a[5], &bytes) || !as_handle(a[0], &h) || !as_params(a[1], g_step_type, &p)) return nullptr;
        for (int i = 0; i < 4; ++i)
            if (!as_pointer(a[2 + i], &t[i])) return nullptr;
        if (!as_stream(a[7], &st)) return nullptr;
        return finish(unlocked([&] { return evlnStepAttention(h, &p, t[0], t[1], t[2], t[3], bytes, st); }), "evlnStepAttention");
    });
}

EVLN_ENTRY(py_step_combine)
{
    static const char* const names[] = {"handle", "params", "workspace", "out", "lse_out", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnStepCombine", args, nargs, kwnames, names, 4, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnStepParams p;
        void *ws, *out, *lse, *st;
        if (!as_handle(a[0], &h) || !as_params(a[1], g_step_type, &p) || !as_pointer(a[2], &ws) || !as_pointer(a[3], &out) ||
            !as_pointer(a[4], &lse) || !as_stream(a[5], &st))
            return nullptr;
        return finish(unlocked([&] { return evlnStepCombine(h, &p, ws, out, (float*)lse, st); }), "evlnStepCombine");
    });
}

EVLN_ENTRY(py_step)
{
    static const char* const names[] = {"handle", "params", "q_new", "k_new", "v_new", "q_rot", "k_cache", "v_cache", "workspace",
                                        "out", "lse_out", "workspace_bytes", "stream", "strides", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnStep", args, nargs, kwnames, names, 10, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnStepParams p;
        void* t[9];
        void* st;
        long s[3];
        size_t bytes;
        if (!token_strides(a[13], a[2], a[3], a[4], s) || !buffer_bytes(a[11], a[8], &bytes) || !as_handle(a[0], &h) ||
            !as_params(a[1], g_step_type, &p))
            return nullptr;
        for (int i = 0; i < 9; ++i)
            if (!as_pointer(a[2 + i], &t[i])) return nullptr;
        if (!as_stream(a[12], &st)) return nullptr;
        return finish(unlocked([&] {
            return evlnStep(h, &p, t[0], t[1], t[2], s[0], s[1], s[2], t[3], t[4], t[5], t[6], bytes, t[7], (float*)t[8], st);
        }), "evlnStep");
    });
}

// the host arrays of a paged call: batch lengths, batch + 1 offsets
bool paged_arrays(const evlnPagedParams& p, PyObject* lens_o, PyObject* offs_o, std::vector<int>* lens, std::vector<int>* offs)
{
    if (!as_ints(lens_o, lens) || !as_ints(offs_o, offs)) return false;
    if ((long)lens->size() < (long)p.batch || (long)offs->size() < (long)p.batch + 1) {
        PyErr_SetString(PyExc_ValueError, "cache_lens needs batch entries and new_offsets batch + 1");
        return false;
    }
    return true;
}

EVLN_ENTRY(py_paged_rope_append)
{
    static const char* const names[] = {"handle", "params", "q_new", "k_new", "v_new", "cache_lens", "new_offsets", "page_table",
                                        "q_rot", "k_pool", "v_pool", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnPagedRopeAppend", args, nargs, kwnames, names, 11, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnPagedParams p;
        std::vector<int> lens, offs;
        void *q, *k, *v, *table, *q_rot, *kp, *vp, *st;
        if (!as_handle(a[0], &h) || !as_params(a[1], g_paged_type, &p) || !paged_arrays(p, a[5], a[6], &lens, &offs) ||
            !as_pointer(a[2], &q) || !as_pointer(a[3], &k) || !as_pointer(a[4], &v) || !as_pointer(a[7], &table) ||
            !as_pointer(a[8], &q_rot) || !as_pointer(a[9], &kp) || !as_pointer(a[10], &vp) || !as_stream(a[11], &st))
            return nullptr;
        return finish(unlocked([&] {
            return evlnPagedRopeAppend(h, &p, q, k, v, lens.data(), offs.data(), (const int*)table, q_rot, kp, vp, st);
        }), "evlnPagedRopeAppend");
    });
}

EVLN_ENTRY(py_paged_step_attention)
{
    static const char* const names[] = {"handle", "params", "q_rot", "k_pool", "v_pool", "cache_lens", "new_offsets", "page_table",
                                        "workspace", "workspace_bytes", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnPagedStepAttention", args, nargs, kwnames, names, 9, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnPagedParams p;
        std::vector<int> lens, offs;
        void *q_rot, *kp, *vp, *table, *ws, *st;
        size_t bytes;
        if (!buffer_bytes(a[9], a[8], &bytes) || !as_handle(a[0], &h) || !as_params(a[1], g_paged_type, &p) ||
            !paged_arrays(p, a[5], a[6], &lens, &offs) || !as_pointer(a[2], &q_rot) || !as_pointer(a[3], &kp) ||
            !as_pointer(a[4], &vp) || !as_pointer(a[7], &table) || !as_pointer(a[8], &ws) || !as_stream(a[10], &st))
            return nullptr;
        return finish(unlocked([&] {
            return evlnPagedStepAttention(h, &p, q_rot, kp, vp, lens.data(), offs.data(), (const int*)table, ws, bytes, st);
        }), "evlnPagedStepAttention");
    });
}

EVLN_ENTRY(py_paged_step_combine)
{
    static const char* const names[] = {"handle", "params", "workspace", "cache_lens", "new_offsets", "out", "lse_out", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnPagedStepCombine", args, nargs, kwnames, names, 6, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnPagedParams p;
        std::vector<int> lens, offs;
        void *ws, *out, *lse, *st;
        if (!as_handle(a[0], &h) || !as_params(a[1], g_paged_type, &p) || !paged_arrays(p, a[3], a[4], &lens, &offs) ||
            !as_pointer(a[2], &ws) || !as_pointer(a[5], &out) || !as_pointer(a[6], &lse) || !as_stream(a[7], &st))
            return nullptr;
        return finish(unlocked([&] { return evlnPagedStepCombine(h, &p, ws, lens.data(), offs.data(), out, (float*)lse, st); }),
                      "evlnPagedStepCombine");
    });
}

EVLN_ENTRY(py_packed_forward)
{
    static const char* const names[] = {"handle", "params", "q", "k", "v", "k_cache", "v_cache", "workspace", "out", "lse_out", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnPackedForward", args, nargs, kwnames, names, 9, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnPackedParams p;
        void* t[8];
        void* st;
        long s[3];
        size_t bytes;
        if (!token_strides(nullptr, a[2], a[3], a[4], s) || !buffer_bytes(nullptr, a[7], &bytes) || !as_handle(a[0], &h) ||
            !as_params(a[1], g_packed_type, &p))
            return nullptr;
        for (int i = 0; i < 8; ++i)
            if (!as_pointer(a[2 + i], &t[i])) return nullptr;
        if (!as_stream(a[10], &st)) return nullptr;
        return finish(unlocked([&] {
            return evlnPackedForward(h, &p, t[0], t[1], t[2], s[0], s[1], s[2], t[3], t[4], t[5], bytes, t[6], (float*)t[7], st);
        }), "evlnPackedForward");
    });
}

EVLN_ENTRY(py_step_attention_no_alloc)
{
    static const char* const names[] = {"params", "q_rot", "k_cache", "v_cache", "out", "lse_out", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnStepAttentionNoAlloc", args, nargs, kwnames, names, 5, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnStepParams p;
        void* t[5];
        void* st;
        if (!as_params(a[0], g_step_type, &p)) return nullptr;
        for (int i = 0; i < 5; ++i)
            if (!as_pointer(a[1 + i], &t[i])) return nullptr;
        if (!as_stream(a[6], &st)) return nullptr;
        return finish(unlocked([&] { return evlnStepAttentionNoAlloc(&p, t[0], t[1], t[2], t[3], (float*)t[4], st); }),
                      "evlnStepAttentionNoAlloc");
    });
}

EVLN_ENTRY(py_store_append)
{
    static const char* const names[] = {"handle", "params", "k_new", "v_new", "store_len", "k_store", "v_store", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnStoreAppend", args, nargs, kwnames, names, 7, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnGatherParams p;
        void *k, *v, *ks, *vs, *st;
        long sk, sv;
        int len, n;
        if (!token_stride(a[2], &sk) || !token_stride(a[3], &sv) || !as_handle(a[0], &h) || !as_params(a[1], g_gather_type, &p)) return nullptr;
        if (THPVariable_Check(a[2])) {
            n = (int)THPVariable_Unpack(a[2]).size(0);
        } else {
            PyObject* r = PyObject_CallMethod(a[2], "size", "i", 0);
            const bool ok = r && as_int(r, &n);
            Py_XDECREF(r);
            if (!ok) return nullptr;
        }
        if (!as_pointer(a[2], &k) || !as_pointer(a[3], &v) || !as_int(a[4], &len) || !as_pointer(a[5], &ks) || !as_pointer(a[6], &vs) ||
            !as_stream(a[7], &st))
            return nullptr;
        return finish(unlocked([&] { return evlnStoreAppend(h, &p, k, v, sk, sv, len, n, ks, vs, st); }), "evlnStoreAppend");
    });
}

EVLN_ENTRY(py_gather_rope)
{
    static const char* const names[] = {"handle", "params", "seg_src", "seg_len", "k_store", "v_store", "k_work", "v_work", "stream", nullptr};
    PyObject* a[kMaxArgs];
    if (!take_args("evlnGatherRope", args, nargs, kwnames, names, 8, a)) return nullptr;
    return guarded([&]() -> PyObject* {
        evlnHandle_t h;
        evlnGatherParams p;
        std::vector<int> src, len;
        void* t[4];
        void* st;
        int total = 0;
        if (!as_handle(a[0], &h) || !as_params(a[1], g_gather_type, &p) || !as_ints(a[2], &src) || !as_ints(a[3], &len)) return nullptr;
        if (len.size() < src.size()) {
            PyErr_SetString(PyExc_ValueError, "seg_len needs an entry for every segment");
            return nullptr;
        }
        for (int i = 0; i < 4; ++i)
            if (!as_pointer(a[4 + i], &t[i])) return nullptr;
        if (!as_stream(a[8], &st)) return nullptr;
        const int s = unlocked([&] {
            return evlnGatherRope(h, &p, (int)src.size(), src.data(), len.data(), t[0], t[1], t[2], t[3], &total, st);
        });
        if (s != EVLN_OK) return finish(s, "evlnGatherRope");
        return PyLong_FromLong(total);
    });
}

// configure(step_type, paged_type, packed_type, gather_type, EvlnError, ArgumentError)
PyObject* py_configure(PyObject*, PyObject* args)
{
    PyObject *s, *g, *k, *q, *e, *ae;
    if (!PyArg_ParseTuple(args, "O!O!O!O!OO", &PyType_Type, &s, &PyType_Type, &g, &PyType_Type, &k, &PyType_Type, &q, &e, &ae)) return nullptr;
    for (PyObject* o : {s, g, k, q, e, ae}) Py_INCREF(o);      // kept for the life of the process
    g_step_type = (PyTypeObject*)s;
    g_paged_type = (PyTypeObject*)g;
    g_packed_type = (PyTypeObject*)k;
    g_gather_type = (PyTypeObject*)q;
    g_error = e;
    g_argument_error = ae;
    Py_RETURN_NONE;
}

#define EVLN_METHOD(name, fn, doc) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL | METH_KEYWORDS, doc}

PyMethodDef kMethods[] = {
    {"configure", py_configure, METH_VARARGS, nullptr},
    EVLN_METHOD("evlnRopeTable", py_rope_table, "(cos, sin) of the positions first_pos .. first_pos+count-1 into `table` (device memory)."),
    EVLN_METHOD("evlnRopeAppend", py_rope_append, "q_new/k_new/v_new: [n,H,D] tensors (last two dims contiguous) or raw addresses + strides."),
    EVLN_METHOD("evlnStepAttention", py_step_attention, "Step attention into the split partials of `workspace`."),
    EVLN_METHOD("evlnStepCombine", py_step_combine, "Merges the split partials into `out`."),
    EVLN_METHOD("evlnStep", py_step, "The three calls of a step in one."),
    EVLN_METHOD("evlnPagedRopeAppend", py_paged_rope_append, "evlnRopeAppend for a batch of episodes on a page pool."),
    EVLN_METHOD("evlnPagedStepAttention", py_paged_step_attention, "evlnStepAttention for a batch of episodes on a page pool."),
    EVLN_METHOD("evlnPagedStepCombine", py_paged_step_combine, "evlnStepCombine for a batch of episodes on a page pool."),
    EVLN_METHOD("evlnPackedForward", py_packed_forward, "A packed sequence I, v_1, a_1, ..., v_N, a_N under the action-isolating mask, in one call."),
    EVLN_METHOD("evlnStepAttentionNoAlloc", py_step_attention_no_alloc,
                "Attention + combine without a handle or a caller workspace: the split partials go to a scratch array built into the "
                "library (at most EVLN_NOALLOC_SCRATCH_BYTES); calls sharing a device must not overlap."),
    EVLN_METHOD("evlnStoreAppend", py_store_append, "The new frame's un-rotated keys and values to the store."),
    EVLN_METHOD("evlnGatherRope", py_gather_rope, "Lays the kept store segments out in the working cache; returns the number of tokens laid out."),
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_evln_native", "The per-layer calls of libevln.so on torch tensors.", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__evln_native() { return PyModule_Create(&kModule); }
