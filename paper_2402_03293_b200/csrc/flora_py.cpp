// Native side of binding.py: unpacks tensors and seed arrays and calls the C ABI (include/flora.h).
//
// What bounds the calls on small matrices is the host: a kernel launch takes about 3 us, and marshalling one call through
// ctypes took 10 to 15 us more (a flora_mat per tensor from seven attribute reads: 1.7 us each; the current stream: 3.5 us).
// Reading the tensor's C++ object instead takes tens of nanoseconds (one 256 x 384 compression at r = 32: 18.6 us per call
// before, launch included).  Nothing here computes: every operation runs in libflora.so.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <vector>

#include "../../include/flora.h"

namespace {

// The view of a 2-D float32 or bfloat16 tensor with unit column stride (binding.mat, with the same checks).
bool mat(PyObject* o, flora_mat* out)
{
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a tensor");
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.dim() != 2) {
        PyErr_SetString(PyExc_ValueError, "expected a 2-D tensor");
        return false;
    }
    const int64_t rows = t.size(0), cols = t.size(1), ld = t.stride(0);
    const bool some = rows * cols != 0;
    if (some && t.stride(1) != 1) {
        PyErr_SetString(PyExc_ValueError, "expected unit stride along columns");
        return false;
    }
    const at::ScalarType dt = t.scalar_type();
    if (dt != at::kFloat && dt != at::kBFloat16) {
        PyErr_SetString(PyExc_ValueError, "expected float32 or bfloat16");
        return false;
    }
    if (some && !t.is_cuda()) {
        PyErr_SetString(PyExc_ValueError, "expected a CUDA tensor");
        return false;
    }
    out->data = some ? t.data_ptr() : nullptr;
    out->rows = rows;
    out->cols = cols;
    out->ld = ((rows > 1 || some) && ld > cols) ? ld : cols;
    out->dtype = dt == at::kBFloat16 ? FLORA_BF16 : FLORA_F32;
    return true;
}

// None: the current stream; an object with .cuda_stream; or the address as a number.
bool stream(PyObject* o, void** out)
{
    if (o == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) {
        PyErr_Clear();
        v = Py_NewRef(o);
    }
    PyObject* n = PyNumber_Long(v);
    Py_DECREF(v);
    if (!n) return false;
    *out = PyLong_AsVoidPtr(n);
    Py_DECREF(n);
    return !PyErr_Occurred();
}

bool seed(PyObject* o, uint64_t* out)
{
    *out = PyLong_AsUnsignedLongLongMask(o);
    return !PyErr_Occurred();
}
bool number(PyObject* o, float* out)
{
    *out = (float)PyFloat_AsDouble(o);
    return !PyErr_Occurred();
}
bool integer(PyObject* o, int64_t* out)
{
    *out = PyLong_AsLongLong(o);
    return !PyErr_Occurred();
}
bool handle(PyObject* o, flora_set** out)
{
    *out = static_cast<flora_set*>(PyLong_AsVoidPtr(o));
    return !PyErr_Occurred();
}
// A host array of 64-bit seeds, one per matrix of the set (anything with the buffer protocol: the arrays of binding.seed_array).
struct Seeds {
    Py_buffer b{};
    bool held = false;
    bool get(PyObject* o, Py_ssize_t count)
    {
        if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE)) return false;
        held = true;
        if (b.len < count * (Py_ssize_t)sizeof(uint64_t)) {
            PyErr_SetString(PyExc_ValueError, "expected one seed per matrix");
            return false;
        }
        return true;
    }
    const uint64_t* data() const { return static_cast<const uint64_t*>(b.buf); }
    ~Seeds()
    {
        if (held) PyBuffer_Release(&b);
    }
};

bool args(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}
// Runs a call of the C ABI without the interpreter lock (a first call that plans, or a launch into a full queue, may block)
// and returns its status.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};
template <typename F>
PyObject* run(F&& call)
{
    flora_status s;
    {
        Unlocked unlocked;
        s = call();
    }
    return PyLong_FromLong((long)s);
}

#define FN(name) PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n)

FN(compress_accumulate)              // G, C, seed, r, stream
{
    flora_mat g, c;
    uint64_t s;
    int64_t r;
    void* st;
    if (!args(n, 5) || !mat(a[0], &g) || !mat(a[1], &c) || !seed(a[2], &s) || !integer(a[3], &r) || !stream(a[4], &st)) return nullptr;
    return run([&] { return flora_compress_accumulate(&g, &c, s, (int)r, st); });
}
FN(decompress_apply)                 // W, C, seed, lr, scale, stream
{
    flora_mat w, c;
    uint64_t s;
    float lr, scale;
    void* st;
    if (!args(n, 6) || !mat(a[0], &w) || !mat(a[1], &c) || !seed(a[2], &s) || !number(a[3], &lr) || !number(a[4], &scale) || !stream(a[5], &st))
        return nullptr;
    return run([&] { return flora_decompress_apply(&w, &c, s, lr, scale, st); });
}
FN(momentum_step)                    // G, M, beta, seed, stream
{
    flora_mat g, m;
    uint64_t s;
    float beta;
    void* st;
    if (!args(n, 5) || !mat(a[0], &g) || !mat(a[1], &m) || !number(a[2], &beta) || !seed(a[3], &s) || !stream(a[4], &st)) return nullptr;
    return run([&] { return flora_momentum_step(&g, &m, beta, s, st); });
}
FN(momentum_step_resampled)          // G, M, beta, seed_old, seed_new, stream
{
    flora_mat g, m;
    uint64_t so, sn;
    float beta;
    void* st;
    if (!args(n, 6) || !mat(a[0], &g) || !mat(a[1], &m) || !number(a[2], &beta) || !seed(a[3], &so) || !seed(a[4], &sn) || !stream(a[5], &st))
        return nullptr;
    return run([&] { return flora_momentum_step_resampled(&g, &m, beta, so, sn, st); });
}
FN(resample_transfer)                // M, m, operand, seed_old, seed_new, stream
{
    flora_mat m;
    int64_t cols, op;
    uint64_t so, sn;
    void* st;
    if (!args(n, 6) || !mat(a[0], &m) || !integer(a[1], &cols) || !integer(a[2], &op) || !seed(a[3], &so) || !seed(a[4], &sn) || !stream(a[5], &st))
        return nullptr;
    return run([&] { return flora_resample_transfer(&m, cols, (int32_t)op, so, sn, st); });
}
FN(transfer_axpby)                   // dst, src, m, operand, seed_old, seed_new, a, b, stream
{
    flora_mat d, s;
    int64_t cols, op;
    uint64_t so, sn;
    float ca, cb;
    void* st;
    if (!args(n, 9) || !mat(a[0], &d) || !mat(a[1], &s) || !integer(a[2], &cols) || !integer(a[3], &op) || !seed(a[4], &so) || !seed(a[5], &sn) ||
        !number(a[6], &ca) || !number(a[7], &cb) || !stream(a[8], &st))
        return nullptr;
    return run([&] { return flora_transfer_axpby(&d, &s, cols, (int32_t)op, so, sn, ca, cb, st); });
}
FN(derive_seed)                      // base, matrix, epoch
{
    uint64_t b, m, e;
    if (!args(n, 3) || !seed(a[0], &b) || !seed(a[1], &m) || !seed(a[2], &e)) return nullptr;
    return PyLong_FromUnsignedLongLong(flora_derive_seed(b, m, e));
}
FN(derive_seeds)                     // base, count, epoch: (list of the seeds of matrices 0 .. count-1, the same as bytes)
{
    uint64_t b, e;
    int64_t count;
    if (!args(n, 3) || !seed(a[0], &b) || !integer(a[1], &count) || !seed(a[2], &e)) return nullptr;
    PyObject* list = PyList_New(count);
    PyObject* bytes = list ? PyBytes_FromStringAndSize(nullptr, count * (Py_ssize_t)sizeof(uint64_t)) : nullptr;
    if (!bytes) {
        Py_XDECREF(list);
        return nullptr;
    }
    uint64_t* raw = reinterpret_cast<uint64_t*>(PyBytes_AS_STRING(bytes));
    for (int64_t i = 0; i < count; ++i) {
        raw[i] = flora_derive_seed(b, (uint64_t)i, e);
        PyObject* v = PyLong_FromUnsignedLongLong(raw[i]);
        if (!v) {
            Py_DECREF(list);
            Py_DECREF(bytes);
            return nullptr;
        }
        PyList_SET_ITEM(list, i, v);
    }
    return Py_BuildValue("(NN)", list, bytes);
}
FN(set_rebind)                       // handle, tensors, stream
{
    flora_set* h;
    void* st;
    if (!args(n, 3) || !handle(a[0], &h) || !stream(a[2], &st)) return nullptr;
    THPObjectPtr seq(PySequence_Fast(a[1], "expected a sequence of tensors"));
    if (!seq) return nullptr;
    std::vector<flora_mat> g((size_t)PySequence_Fast_GET_SIZE(seq.get()));
    for (size_t i = 0; i < g.size(); ++i)
        if (!mat(PySequence_Fast_GET_ITEM(seq.get(), (Py_ssize_t)i), &g[i])) return nullptr;
    return run([&] { return flora_set_rebind_gradients(h, g.data(), st); });
}
FN(set_compress_accumulate)          // handle, count, seeds, stream
{
    flora_set* h;
    int64_t count;
    Seeds s;
    void* st;
    if (!args(n, 4) || !handle(a[0], &h) || !integer(a[1], &count) || !s.get(a[2], count) || !stream(a[3], &st)) return nullptr;
    return run([&] { return flora_set_compress_accumulate(h, s.data(), st); });
}
FN(set_momentum_step)                // handle, count, beta, seeds, stream
{
    flora_set* h;
    int64_t count;
    float beta;
    Seeds s;
    void* st;
    if (!args(n, 5) || !handle(a[0], &h) || !integer(a[1], &count) || !number(a[2], &beta) || !s.get(a[3], count) || !stream(a[4], &st)) return nullptr;
    return run([&] { return flora_set_momentum_step(h, beta, s.data(), st); });
}
FN(set_decompress_apply)             // handle, count, seeds, lr, scale, stream
{
    flora_set* h;
    int64_t count;
    float lr, scale;
    Seeds s;
    void* st;
    if (!args(n, 6) || !handle(a[0], &h) || !integer(a[1], &count) || !s.get(a[2], count) || !number(a[3], &lr) || !number(a[4], &scale) ||
        !stream(a[5], &st))
        return nullptr;
    return run([&] { return flora_set_decompress_apply(h, s.data(), lr, scale, st); });
}
FN(set_resample_transfer)            // handle, count, seeds_old, seeds_new, stream
{
    flora_set* h;
    int64_t count;
    Seeds so, sn;
    void* st;
    if (!args(n, 5) || !handle(a[0], &h) || !integer(a[1], &count) || !so.get(a[2], count) || !sn.get(a[3], count) || !stream(a[4], &st)) return nullptr;
    return run([&] { return flora_set_resample_transfer(h, so.data(), sn.data(), st); });
}
FN(set_transfer_axpby)               // dst, src, count, seeds_old, seeds_new, a, b, stream
{
    flora_set *d, *s;
    int64_t count;
    Seeds so, sn;
    float ca, cb;
    void* st;
    if (!args(n, 8) || !handle(a[0], &d) || !handle(a[1], &s) || !integer(a[2], &count) || !so.get(a[3], count) || !sn.get(a[4], count) ||
        !number(a[5], &ca) || !number(a[6], &cb) || !stream(a[7], &st))
        return nullptr;
    return run([&] { return flora_set_transfer_axpby(d, s, so.data(), sn.data(), ca, cb, st); });
}
FN(set_momentum_step_resampled)      // handle, count, beta, seeds_old, seeds_new, stream
{
    flora_set* h;
    int64_t count;
    float beta;
    Seeds so, sn;
    void* st;
    if (!args(n, 6) || !handle(a[0], &h) || !integer(a[1], &count) || !number(a[2], &beta) || !so.get(a[3], count) || !sn.get(a[4], count) ||
        !stream(a[5], &st))
        return nullptr;
    return run([&] { return flora_set_momentum_step_resampled(h, beta, so.data(), sn.data(), st); });
}

// Reading a tensor or asking for the current stream may throw (a tensor without strides, a machine without a GPU): the C++ exception
// becomes a Python one here, instead of passing through the interpreter's C frames, which ends the process.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    return F(self, a, n);
    END_HANDLE_TH_ERRORS
}

#define ROW(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<name>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    ROW(compress_accumulate), ROW(decompress_apply), ROW(momentum_step), ROW(momentum_step_resampled), ROW(resample_transfer),
    ROW(transfer_axpby), ROW(derive_seed), ROW(derive_seeds), ROW(set_rebind), ROW(set_compress_accumulate), ROW(set_momentum_step),
    ROW(set_decompress_apply), ROW(set_resample_transfer), ROW(set_transfer_axpby), ROW(set_momentum_step_resampled),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling of binding.py (see flora_py.cpp).", -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
