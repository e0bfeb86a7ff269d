// Native half of the Python binding: turns a call's tensors into the C ABI's pointer tables and makes the call.
//
// What bounds an eagerly launched small collective is the host: the kernel runs 1.5-4 us, cudaLaunchKernelEx costs
// 1.7 (dependent launch) to 2.1 us (plain), and marshalling 2 * nranks tensors in Python around a ctypes call cost
// 7-12 us more (a data_ptr() method call and a ctypes item store per tensor, 3.2 us for torch.cuda.current_stream()).
// Here a tensor's address is read from the tensor object itself and the current stream from c10.  Measured back to
// back, before -> now: 2 ranks x 8 KiB one-shot 10.1 -> 2.3 us, 8 ranks x 512 KiB allreduce 11.9 -> 2.5, 16 ranks x
// 64 KiB allgather 15.1 -> 3.35; a call that only validates (count 0) costs 0.25 us at 2 ranks, 0.38 us at 16.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <exception>
#include <memory>
#include <new>

#include "../../../include/nuna.h"

namespace {

typedef int (*CollectiveFn)(const void* const*, void* const*, int, size_t, int, unsigned, void*);
typedef int (*StaticFn)(const void* const*, void* const*, int, size_t, int, void*);
typedef int (*HostFn)(const void* const*, void* const*, int, size_t, int, unsigned, int);

// The six collectives of one signature (the order of _COLLECTIVES in binding.py).
constexpr int kCollectives = 6;
CollectiveFn g_collective[kCollectives] = {};
const char* const kNames[kCollectives] = {"nuna_allreduce", "nuna_allreduce_oneshot", "nuna_allreduce_twoshot",
                                          "nuna_reduce_scatter", "nuna_allgather", "nuna_alltoall"};
// Argument names of the module's functions, interned, and how many of them a call has to give.
struct Signature {
    const char* text[8];
    int n, required;
    PyObject* name[8];
};
Signature g_count = {{"src", "dst", "count", "dtype", "flags", "stream", "check", "nranks"}, 8, 3, {}};
Signature g_shard = {{"src", "dst", "shard_count", "dtype", "flags", "stream", "check", "nranks"}, 8, 3, {}};
Signature g_block = {{"src", "dst", "block_count", "dtype", "flags", "stream", "check", "nranks"}, 8, 3, {}};
Signature g_fixed = {{"src", "dst", "count", "dtype", "stream", "check"}, 6, 3, {}};
Signature g_hosts = {{"src", "dst", "count", "dtype", "flags", "two_shot", "check"}, 7, 3, {}};
const Signature* const kSignature[kCollectives] = {&g_count, &g_count, &g_count, &g_shard, &g_shard, &g_block};
StaticFn g_static = nullptr;
HostFn g_host = nullptr;
PyObject* g_error = nullptr;               // binding.NunaError
PyObject *g_s_data_ptr = nullptr, *g_s_cuda_stream = nullptr, *g_s_ctypes = nullptr, *g_s_data = nullptr;

// int(x) as an address; wraps like a ctypes void pointer does.
bool to_address(PyObject* x, void** out)
{
    PyObject* i = PyNumber_Long(x);
    if (!i) return false;
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) return false;
    *out = reinterpret_cast<void*>((uintptr_t)v);
    return true;
}

// Takes over `x` if it is not null.
bool to_address_owned(PyObject* x, void** out)
{
    if (!x) return false;
    const bool ok = to_address(x, out);
    Py_DECREF(x);
    return ok;
}

// A rank buffer: a torch tensor, an object with data_ptr(), (host = true) an array with .ctypes.data, or an address.
bool address_of(PyObject* x, bool host, void** out)
{
    if (THPVariable_CheckExact(x)) {       // subclasses may override data_ptr: they take the method call below
        try {
            *out = THPVariable_Unpack(x).mutable_data_ptr();
            return true;
        } catch (const std::exception& e) {
            PyErr_SetString(PyExc_RuntimeError, e.what());
            return false;
        }
    }
    if (PyLong_CheckExact(x)) return to_address(x, out);
    if (host) {
        if (PyObject* c = PyObject_GetAttr(x, g_s_ctypes)) {
            PyObject* d = PyObject_GetAttr(c, g_s_data);
            Py_DECREF(c);
            return to_address_owned(d, out);
        }
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
        PyErr_Clear();
    }
    if (PyObject* m = PyObject_GetAttr(x, g_s_data_ptr)) {
        PyObject* d = PyObject_CallNoArgs(m);
        Py_DECREF(m);
        return to_address_owned(d, out);
    }
    if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
    PyErr_Clear();
    return to_address(x, out);
}

// The addresses of a sequence of rank buffers.  The table has at least NUNA_MAX_RANKS entries, null beyond the
// sequence, so that an explicit `nranks` larger than the sequence reads nulls (an argument error), not the stack.
// It keeps the sequence until the call is made: an iterator's buffers may have no other owner.
struct Table {
    void* fixed[NUNA_MAX_RANKS] = {};
    std::unique_ptr<void*[]> heap;
    void** p = fixed;
    Py_ssize_t n = 0;
    PyObject* seq = nullptr;

    ~Table() { Py_XDECREF(seq); }

    bool fill(PyObject* bufs, bool host)
    {
        seq = PySequence_Fast(bufs, "rank buffers must be a sequence");
        if (!seq) return false;
        n = PySequence_Fast_GET_SIZE(seq);
        if (n > NUNA_MAX_RANKS) {
            heap.reset(new (std::nothrow) void*[(size_t)n]());
            if (!heap) {
                PyErr_NoMemory();
                return false;
            }
            p = heap.get();
        }
        bool ok = true;
        // by index with the size read again: an element's own Python code may change a list meanwhile
        for (Py_ssize_t i = 0; ok && i < n && i < PySequence_Fast_GET_SIZE(seq); ++i) {
            PyObject* x = PySequence_Fast_GET_ITEM(seq, i);
            Py_INCREF(x);
            ok = address_of(x, host, &p[i]);
            Py_DECREF(x);
        }
        return ok;
    }
};

bool to_u64(PyObject* x, unsigned long long* out)
{
    if (PyLong_CheckExact(x)) {
        *out = PyLong_AsUnsignedLongLongMask(x);
        return true;
    }
    PyObject* i = PyNumber_Index(x);
    if (!i) return false;
    *out = PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    return true;
}

// None = torch's current stream on the current device; an object with .cuda_stream; or the handle itself.
bool to_stream(PyObject* x, void** out)
{
    if (x == Py_None) {
        try {
            *out = c10::cuda::getCurrentCUDAStream().stream();
            return true;
        } catch (const std::exception& e) {
            PyErr_SetString(PyExc_RuntimeError, e.what());
            return false;
        }
    }
    if (PyLong_CheckExact(x)) return to_address(x, out);
    if (PyObject* h = PyObject_GetAttr(x, g_s_cuda_stream)) return to_address_owned(h, out);
    if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
    PyErr_Clear();
    return to_address(x, out);
}

PyObject* finish(int status, const char* what, PyObject* check)
{
    if (status != NUNA_OK) {
        const int c = PyObject_IsTrue(check);
        if (c < 0) return nullptr;
        if (c) {
            if (PyObject* e = PyObject_CallFunction(g_error, "is", status, what)) {
                PyErr_SetObject(g_error, e);
                Py_DECREF(e);
            }
            return nullptr;
        }
    }
    return PyLong_FromLong(status);
}

// Sorts a call's arguments, positional and by name, into out[0 ... sig.n), null where none was given.
bool arguments(const char* what, const Signature& sig, PyObject* const* args, Py_ssize_t npos, PyObject* kwnames, PyObject** out)
{
    if (npos > sig.n) {
        PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", what, sig.n, npos);
        return false;
    }
    for (int i = 0; i < sig.n; ++i) out[i] = i < npos ? args[i] : nullptr;
    for (Py_ssize_t k = 0, nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0; k < nkw; ++k) {
        PyObject* key = PyTuple_GET_ITEM(kwnames, k);
        int at = 0;
        while (at < sig.n && key != sig.name[at]) ++at;             // names in a call's source are interned
        if (at == sig.n)
            for (at = 0; at < sig.n && PyUnicode_Compare(key, sig.name[at]) != 0;) ++at;
        if (at == sig.n || out[at]) {
            PyErr_Format(PyExc_TypeError, at == sig.n ? "%s() got an unexpected keyword argument '%U'"
                                                      : "%s() got multiple values for argument '%U'", what, key);
            return false;
        }
        out[at] = args[npos + k];
    }
    for (int i = 0; i < sig.required; ++i)
        if (!out[i]) {
            PyErr_Format(PyExc_TypeError, "%s() missing required argument: '%s'", what, sig.text[i]);
            return false;
        }
    return true;
}

bool to_u64_or(PyObject* x, unsigned long long fallback, unsigned long long* out)
{
    if (x) return to_u64(x, out);
    *out = fallback;
    return true;
}

template <int kOp>
PyObject* collective(PyObject*, PyObject* const* args, Py_ssize_t npos, PyObject* kwnames)
{
    PyObject* a[8];
    if (!arguments(kNames[kOp], *kSignature[kOp], args, npos, kwnames, a)) return nullptr;
    Table src, dst;
    unsigned long long count, dtype, flags, nranks;
    void* stream;
    if (!src.fill(a[0], false) || !dst.fill(a[1], false) || !to_u64(a[2], &count) || !to_u64_or(a[3], NUNA_BF16, &dtype) ||
        !to_u64_or(a[4], 0, &flags) || !to_stream(a[5] ? a[5] : Py_None, &stream))
        return nullptr;
    nranks = (unsigned long long)src.n;
    if (a[7] && a[7] != Py_None && !to_u64(a[7], &nranks)) return nullptr;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = g_collective[kOp](src.p, dst.p, (int)nranks, (size_t)count, (int)dtype, (unsigned)flags, stream);
    Py_END_ALLOW_THREADS
    return finish(st, kNames[kOp], a[6] ? a[6] : Py_True);
}

PyObject* twoshot_static(PyObject*, PyObject* const* args, Py_ssize_t npos, PyObject* kwnames)
{
    PyObject* a[8];
    if (!arguments("nuna_allreduce_twoshot_static", g_fixed, args, npos, kwnames, a)) return nullptr;
    Table src, dst;
    unsigned long long count, dtype;
    void* stream;
    if (!src.fill(a[0], false) || !dst.fill(a[1], false) || !to_u64(a[2], &count) || !to_u64_or(a[3], NUNA_BF16, &dtype) ||
        !to_stream(a[4] ? a[4] : Py_None, &stream))
        return nullptr;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = g_static(src.p, dst.p, (int)src.n, (size_t)count, (int)dtype, stream);
    Py_END_ALLOW_THREADS
    return finish(st, "nuna_allreduce_twoshot_static", a[5] ? a[5] : Py_True);
}

PyObject* host(PyObject*, PyObject* const* args, Py_ssize_t npos, PyObject* kwnames)
{
    PyObject* a[8];
    if (!arguments("nuna_allreduce_host", g_hosts, args, npos, kwnames, a)) return nullptr;
    Table src, dst;
    unsigned long long count, dtype, flags;
    if (!src.fill(a[0], true) || !dst.fill(a[1], true) || !to_u64(a[2], &count) || !to_u64_or(a[3], NUNA_BF16, &dtype) ||
        !to_u64_or(a[4], 0, &flags))
        return nullptr;
    const int two = a[5] ? PyObject_IsTrue(a[5]) : 0;
    if (two < 0) return nullptr;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = g_host(src.p, dst.p, (int)src.n, (size_t)count, (int)dtype, (unsigned)flags, two);
    Py_END_ALLOW_THREADS
    return finish(st, "nuna_allreduce_host", a[6] ? a[6] : Py_True);
}

// stream_handle(stream) -> handle as an integer, the way `stream` arguments are read
PyObject* stream_handle(PyObject*, PyObject* x)
{
    void* s;
    if (!to_stream(x, &s)) return nullptr;
    return PyLong_FromVoidPtr(s);
}

// bind(addresses of the six collectives, static, host, NunaError)
PyObject* bind(PyObject*, PyObject* args)
{
    PyObject *fns, *err;
    unsigned long long st, ho;
    if (!PyArg_ParseTuple(args, "O!KKO", &PyTuple_Type, &fns, &st, &ho, &err)) return nullptr;
    if (PyTuple_GET_SIZE(fns) != kCollectives) {
        PyErr_SetString(PyExc_ValueError, "bind: wrong number of entry points");
        return nullptr;
    }
    for (int i = 0; i < kCollectives; ++i) {
        void* p;
        if (!to_address(PyTuple_GET_ITEM(fns, i), &p)) return nullptr;
        g_collective[i] = reinterpret_cast<CollectiveFn>(p);
    }
    g_static = reinterpret_cast<StaticFn>((uintptr_t)st);
    g_host = reinterpret_cast<HostFn>((uintptr_t)ho);
    Py_INCREF(err);
    Py_XSETREF(g_error, err);
    Py_RETURN_NONE;
}

#define NUNA_KW(fn) (PyCFunction)(void (*)(void))(fn), METH_FASTCALL | METH_KEYWORDS
#define NUNA_REST ", dtype=0, flags=0, stream=None, check=True, nranks=None)\n--\n\n"

PyMethodDef methods[] = {
    {"nuna_allreduce", NUNA_KW(collective<0>), "nuna_allreduce(src, dst, count" NUNA_REST},
    {"nuna_allreduce_oneshot", NUNA_KW(collective<1>), "nuna_allreduce_oneshot(src, dst, count" NUNA_REST},
    {"nuna_allreduce_twoshot", NUNA_KW(collective<2>), "nuna_allreduce_twoshot(src, dst, count" NUNA_REST},
    {"nuna_reduce_scatter", NUNA_KW(collective<3>), "nuna_reduce_scatter(src, dst, shard_count" NUNA_REST},
    {"nuna_allgather", NUNA_KW(collective<4>), "nuna_allgather(src, dst, shard_count" NUNA_REST},
    {"nuna_alltoall", NUNA_KW(collective<5>), "nuna_alltoall(src, dst, block_count" NUNA_REST},
    {"nuna_allreduce_twoshot_static", NUNA_KW(twoshot_static),
     "nuna_allreduce_twoshot_static(src, dst, count, dtype=0, stream=None, check=True)\n--\n\n"},
    {"nuna_allreduce_host", NUNA_KW(host),
     "nuna_allreduce_host(src, dst, count, dtype=0, flags=0, two_shot=False, check=True)\n--\n\n"},
    {"stream_handle", (PyCFunction)stream_handle, METH_O, nullptr},
    {"bind", (PyCFunction)bind, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_nuna_py", "Marshalling of the nuna C ABI's calls.", -1, methods,
                          nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__nuna_py()
{
    g_s_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    g_s_ctypes = PyUnicode_InternFromString("ctypes");
    g_s_data = PyUnicode_InternFromString("data");
    for (Signature* sig : {&g_count, &g_shard, &g_block, &g_fixed, &g_hosts})
        for (int i = 0; i < sig->n; ++i) sig->name[i] = PyUnicode_InternFromString(sig->text[i]);
    return PyModule_Create(&module_def);
}
