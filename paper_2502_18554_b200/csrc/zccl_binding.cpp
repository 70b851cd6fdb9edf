// CPython module over the C boundary for the calls a program makes per message: argument checks and marshalling in
// native code.  A codec call on a small message is a few microseconds of GPU work, so the host's share decides how many
// such calls fit a second: through ctypes and torch's Python-level stream objects a call's marshalling took 5.5 us
// (3.3 us of it the look-up of the current stream), here it takes 0.4 us.  The calls themselves are the C boundary's.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/DynamicTypes.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/zccl.h"

namespace {

// The data pointer of a contiguous CUDA tensor of type `dt`; false with a Python error set otherwise.
bool dev_ptr(PyObject* o, c10::ScalarType dt, void** p, size_t* numel = nullptr)
{
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_ValueError, "expected a contiguous CUDA tensor");
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "expected a contiguous CUDA tensor");
        return false;
    }
    if (t.scalar_type() != dt) {
        PyErr_Format(PyExc_ValueError, "expected dtype %S, got %S", (PyObject*)torch::getTHPDtype(dt), (PyObject*)torch::getTHPDtype(t.scalar_type()));
        return false;
    }
    *p = t.data_ptr();
    if (numel) *numel = (size_t)t.numel();
    return true;
}
bool opt_dev_ptr(PyObject* o, c10::ScalarType dt, void** p, size_t* numel = nullptr)
{
    *p = nullptr;
    if (numel) *numel = 0;
    return o == Py_None || dev_ptr(o, dt, p, numel);
}
size_t numel_of(PyObject* o)
{
    return THPVariable_Check(o) ? (size_t)THPVariable_Unpack(o).numel() : 1;
}
// An empty input or output tensor need not be anything in particular: it counts as a null pointer.
bool ptr_unless_empty(PyObject* o, c10::ScalarType dt, void** p, size_t* numel)
{
    *p = nullptr;
    *numel = numel_of(o);
    return *numel == 0 || dev_ptr(o, dt, p, numel);
}

bool stream_of(PyObject* o, void** st)
{
    if (o == Py_None) {
        *st = (void*)c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) return false;
    *st = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

zccl_ctx* ctx_of(PyObject* o) { return (zccl_ctx*)PyLong_AsVoidPtr(o); }

bool nargs_are(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}

// Runs a boundary call without the interpreter lock and hands its status back.
template <class F>
PyObject* status(F&& f)
{
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

using Args = PyObject* const*;

PyObject* current_stream(PyObject*, PyObject*)
{
    return PyLong_FromVoidPtr((void*)c10::cuda::getCurrentCUDAStream().stream());
}

// (ctx, x, eb_mode, eb, out, out_bytes, stream, n)
PyObject* compress(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 8)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    size_t n = a[7] == Py_None ? numel_of(a[1]) : PyLong_AsSize_t(a[7]), cap;
    const int mode = (int)PyLong_AsLong(a[2]);
    const float eb = (float)PyFloat_AsDouble(a[3]);
    if (PyErr_Occurred()) return nullptr;
    void *x = nullptr, *out, *nb, *st;
    if (n && !dev_ptr(a[1], c10::kFloat, &x)) return nullptr;
    if (!dev_ptr(a[4], c10::kByte, &out, &cap) || !dev_ptr(a[5], c10::kLong, &nb) || !stream_of(a[6], &st)) return nullptr;
    return status([&] { return zccl_compress(c, (const float*)x, n, mode, eb, out, cap, (size_t*)nb, st); });
}

// (ctx, stream_bytes, in_bytes_max, y, stream)
PyObject* decompress(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 5)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    void *in, *y, *st;
    size_t cap, n;
    if (!dev_ptr(a[1], c10::kByte, &in, &cap)) return nullptr;
    if (a[2] != Py_None) cap = PyLong_AsSize_t(a[2]);
    if (PyErr_Occurred() || !ptr_unless_empty(a[3], c10::kFloat, &y, &n) || !stream_of(a[4], &st)) return nullptr;
    return status([&] { return zccl_decompress(c, in, cap, (float*)y, n, st); });
}

// (ctx, in_c, n, out_c, out_bytes, local, local_c, raw_out, flags, stream)
PyObject* hop(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 10)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    const size_t n = PyLong_AsSize_t(a[2]);
    const unsigned flags = (unsigned)PyLong_AsUnsignedLong(a[8]);
    if (PyErr_Occurred()) return nullptr;
    void *in, *out, *nb, *local, *local_c, *raw, *st;
    size_t in_cap, out_cap, local_cap;
    if (!dev_ptr(a[1], c10::kByte, &in, &in_cap) || !dev_ptr(a[3], c10::kByte, &out, &out_cap) || !dev_ptr(a[4], c10::kLong, &nb) ||
        !opt_dev_ptr(a[5], c10::kFloat, &local) || !opt_dev_ptr(a[6], c10::kByte, &local_c, &local_cap) ||
        !opt_dev_ptr(a[7], c10::kFloat, &raw) || !stream_of(a[9], &st))
        return nullptr;
    return status([&] {
        return zccl_decompress_reduce_compress(c, in, in_cap, (const float*)local, local_c, local_cap, n, out, out_cap, (size_t*)nb, (float*)raw, flags, st);
    });
}

// (ctx, x, eb_mode, eb, out, out_bytes, stream)
PyObject* compress_f64(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 7)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    const int mode = (int)PyLong_AsLong(a[2]);
    const double eb = PyFloat_AsDouble(a[3]);
    if (PyErr_Occurred()) return nullptr;
    void *x, *out, *nb, *st;
    size_t n, cap;
    if (!ptr_unless_empty(a[1], c10::kDouble, &x, &n) || !dev_ptr(a[4], c10::kByte, &out, &cap) || !dev_ptr(a[5], c10::kLong, &nb) || !stream_of(a[6], &st))
        return nullptr;
    return status([&] { return zccl_compress_f64(c, (const double*)x, n, mode, eb, out, cap, (size_t*)nb, st); });
}

// (ctx, in_c, y, stream)
PyObject* decompress_f64(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 4)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    void *in, *y, *st;
    size_t cap, n;
    if (!dev_ptr(a[1], c10::kByte, &in, &cap) || !ptr_unless_empty(a[2], c10::kDouble, &y, &n) || !stream_of(a[3], &st)) return nullptr;
    return status([&] { return zccl_decompress_f64(c, in, cap, (double*)y, n, st); });
}

// (ctx, x, eb_mode, eb, tile, out, out_bytes, stream)
PyObject* compress_tiled(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 8)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    const int mode = (int)PyLong_AsLong(a[2]);
    const float eb = (float)PyFloat_AsDouble(a[3]);
    const unsigned tile = (unsigned)PyLong_AsUnsignedLong(a[4]);
    if (PyErr_Occurred()) return nullptr;
    void *x, *out, *nb, *st;
    size_t n, cap;
    if (!ptr_unless_empty(a[1], c10::kFloat, &x, &n) || !dev_ptr(a[5], c10::kByte, &out, &cap) || !dev_ptr(a[6], c10::kLong, &nb) || !stream_of(a[7], &st))
        return nullptr;
    return status([&] { return zccl_compress_tiled(c, (const float*)x, n, mode, eb, tile, out, cap, (size_t*)nb, st); });
}

// (ctx, stream_bytes, tile, y, stream)
PyObject* decompress_tiled(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 5)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    const unsigned tile = (unsigned)PyLong_AsUnsignedLong(a[2]);
    if (PyErr_Occurred()) return nullptr;
    void *in, *y, *st;
    size_t cap, n;
    if (!dev_ptr(a[1], c10::kByte, &in, &cap) || !ptr_unless_empty(a[3], c10::kFloat, &y, &n) || !stream_of(a[4], &st)) return nullptr;
    return status([&] { return zccl_decompress_tiled(c, in, cap, tile, (float*)y, n, st); });
}

// The float pointers of a sequence of tensors.
struct Pointers {
    void* p[ZCCL_MAX_RANKS];
    int count = 0;
    size_t first = 0;   // elements of the first
};
bool pointers(PyObject* seq, Pointers& out)
{
    PyObject* f = PySequence_Fast(seq, "expected a sequence of tensors");
    if (!f) return false;
    const Py_ssize_t k = PySequence_Fast_GET_SIZE(f);
    bool ok = true;
    // more buffers than the library knows ranks: the boundary call refuses the count
    for (Py_ssize_t i = 0; ok && i < k && i < ZCCL_MAX_RANKS; ++i)
        ok = dev_ptr(PySequence_Fast_GET_ITEM(f, i), c10::kFloat, &out.p[i], i == 0 ? &out.first : nullptr);
    out.count = (int)k;
    Py_DECREF(f);
    return ok;
}

bool same_count(const Pointers& s, const Pointers& r)
{
    if (r.count >= s.count) return true;
    PyErr_SetString(PyExc_ValueError, "fewer receive buffers than send buffers");
    return false;
}

using SimFn = int (*)(zccl_ctx*, const float* const*, float* const*, int, size_t, int, float, void*);
// (ctx, send, recv, eb_mode, eb, stream)
template <SimFn FN>
PyObject* sim(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 6)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    const int mode = (int)PyLong_AsLong(a[3]);
    const float eb = (float)PyFloat_AsDouble(a[4]);
    if (PyErr_Occurred()) return nullptr;
    Pointers s, r;
    void* st;
    if (!pointers(a[1], s) || !pointers(a[2], r) || !same_count(s, r) || !stream_of(a[5], &st)) return nullptr;
    return status([&] { return FN(c, (const float* const*)s.p, (float* const*)r.p, s.count, s.first, mode, eb, st); });
}
// (ctx, send, recv, eb_mode, eb, flags, stream)
PyObject* sim_allreduce(PyObject*, Args a, Py_ssize_t na)
{
    if (!nargs_are(na, 7)) return nullptr;
    zccl_ctx* c = ctx_of(a[0]);
    const int mode = (int)PyLong_AsLong(a[3]);
    const float eb = (float)PyFloat_AsDouble(a[4]);
    const unsigned flags = (unsigned)PyLong_AsUnsignedLong(a[5]);
    if (PyErr_Occurred()) return nullptr;
    Pointers s, r;
    void* st;
    if (!pointers(a[1], s) || !pointers(a[2], r) || !same_count(s, r) || !stream_of(a[6], &st)) return nullptr;
    return status([&] { return zccl_sim_allreduce(c, (const float* const*)s.p, (float* const*)r.p, s.count, s.first, mode, eb, flags, st); });
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"current_stream", current_stream, METH_NOARGS, nullptr},
    FAST(compress), FAST(decompress), FAST(hop), FAST(compress_f64), FAST(decompress_f64), FAST(compress_tiled), FAST(decompress_tiled), FAST(sim_allreduce),
    {"sim_allgather", (PyCFunction)(void (*)(void))sim<zccl_sim_allgather>, METH_FASTCALL, nullptr},
    {"sim_reduce_scatter", (PyCFunction)(void (*)(void))sim<zccl_sim_reduce_scatter>, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_zccl", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__zccl(void) { return PyModule_Create(&module); }
