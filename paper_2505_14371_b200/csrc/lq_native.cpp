// Python entry of the calls that a program makes every iteration: torch tensors -> raw device pointers -> the C
// functions of lq.h on torch's current stream.  The checks are those of binding.py's ctypes route, which still serves the
// calls made once.  What bounds a small iteration is the host: per call the ctypes route took about
// 8 us (eight attribute look-ups and conversions per tensor), this one takes well under 1 us beside the launches.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "lq.h"

namespace {

PyObject* g_error = nullptr;              // binding.LqError

bool fail(const char* msg)
{
    PyErr_SetString(g_error ? g_error : PyExc_RuntimeError, msg);
    return false;
}

// The tensor's device pointer, or NULL for None; false with an exception set when it is not a contiguous CUDA tensor
// of `type`.
template <typename T>
bool pointer(PyObject* o, at::ScalarType type, T** out)
{
    *out = nullptr;
    if (o == Py_None) return true;
    if (!THPVariable_Check(o)) return fail("expected a contiguous CUDA tensor");
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) return fail("expected a contiguous CUDA tensor");
    if (t.scalar_type() != type) {
        PyErr_Format(g_error ? g_error : PyExc_RuntimeError, "expected dtype %s, got %s", c10::toString(type),
                     c10::toString(t.scalar_type()));
        return false;
    }
    *out = reinterpret_cast<T*>(t.data_ptr());
    return true;
}

bool arity(Py_ssize_t got, Py_ssize_t want)
{
    if (got == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
    return false;
}

bool plan_of(PyObject* o, lq_plan** out)
{
    if (o == Py_None) { *out = nullptr; return true; }       // a closed plan: the C function reports it
    *out = static_cast<lq_plan*>(PyLong_AsVoidPtr(o));
    return !(*out == nullptr && PyErr_Occurred());
}

bool int_of(PyObject* o, int32_t* out)
{
    *out = static_cast<int32_t>(PyLong_AsUnsignedLongMask(o));       // (ctypes takes the low 32 bits as well)
    return !PyErr_Occurred();
}

PyObject* done(int code)
{
    if (code == LQ_OK) Py_RETURN_NONE;
    PyErr_Format(g_error ? g_error : PyExc_RuntimeError, "%s (%d): %s", lq_error_string(code), code, lq_last_error());
    return nullptr;
}

// Runs a C function on torch's current stream, without the interpreter lock (a full launch queue blocks the caller).
template <typename F>
PyObject* call(F&& f)
{
    void* s = static_cast<void*>(c10::cuda::getCurrentCUDAStream().stream());
    int code;
    Py_BEGIN_ALLOW_THREADS
    try { code = f(s); } catch (...) { code = LQ_ENOMEM; }    // (nothing but an allocation can throw there)
    Py_END_ALLOW_THREADS
    return done(code);
}

constexpr at::ScalarType kF32 = at::kFloat, kI32 = at::kInt, kI16 = at::kShort, kF64 = at::kDouble;

PyObject* quantize_pack(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; float *grads, *norms, *prev_norms; uint32_t *packed, *hist, *prev;
    if (!arity(n, 8) || !plan_of(a[0], &p) || !pointer(a[1], kF32, &grads)) return nullptr;
    const uint32_t step = static_cast<uint32_t>(PyLong_AsUnsignedLongMask(a[2]));
    if (PyErr_Occurred()) return nullptr;
    if (!pointer(a[3], kI32, &packed) || !pointer(a[4], kF32, &norms) || !pointer(a[5], kI32, &hist) ||
        !pointer(a[6], kI32, &prev) || !pointer(a[7], kF32, &prev_norms)) return nullptr;
    return call([&](void* s) { return lq_quantize_pack(p, grads, step, packed, norms, hist, prev, prev_norms, s); });
}

PyObject* step_qoda(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; uint32_t* packed; float *norms, *X1, *Y, *Xhalf, *X, *gbar;
    if (!arity(n, 8) || !plan_of(a[0], &p) || !pointer(a[1], kI32, &packed) || !pointer(a[2], kF32, &norms) ||
        !pointer(a[3], kF32, &X1) || !pointer(a[4], kF32, &Y) || !pointer(a[5], kF32, &Xhalf) || !pointer(a[6], kF32, &X) ||
        !pointer(a[7], kF32, &gbar)) return nullptr;
    return call([&](void* s) { return qoda_step(p, packed, norms, X1, Y, Xhalf, X, gbar, s); });
}

PyObject* layer_norms(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; float *grads, *norms;
    if (!arity(n, 3) || !plan_of(a[0], &p) || !pointer(a[1], kF32, &grads) || !pointer(a[2], kF32, &norms)) return nullptr;
    return call([&](void* s) { return lq_layer_norms(p, grads, norms, s); });
}

PyObject* decode_aggregate(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; uint32_t* packed; float *norms, *gbar;
    if (!arity(n, 4) || !plan_of(a[0], &p) || !pointer(a[1], kI32, &packed) || !pointer(a[2], kF32, &norms) ||
        !pointer(a[3], kF32, &gbar)) return nullptr;
    return call([&](void* s) { return lq_decode_aggregate(p, packed, norms, gbar, s); });
}

PyObject* fit_levels(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; uint32_t* hist; float* norms; int32_t z;
    if (!arity(n, 4) || !plan_of(a[0], &p) || !pointer(a[1], kI32, &hist) || !pointer(a[2], kF32, &norms) || !int_of(a[3], &z))
        return nullptr;
    return call([&](void* s) { return lq_fit_levels(p, hist, norms, z, s); });
}

PyObject* level_probabilities(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; uint32_t* hist; float* norms; double* probs; int32_t z;
    if (!arity(n, 6) || !plan_of(a[0], &p) || !pointer(a[1], kI32, &hist) || !pointer(a[2], kF32, &norms) || !int_of(a[3], &z) ||
        !pointer(a[5], kF64, &probs)) return nullptr;
    const int staged = PyObject_IsTrue(a[4]);
    if (staged < 0) return nullptr;
    return call([&](void* s) { return lq_level_probabilities(p, hist, norms, z, staged, probs, s); });
}

PyObject* symbol_counts(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; uint32_t *packed, *counts;
    if (!arity(n, 3) || !plan_of(a[0], &p) || !pointer(a[1], kI32, &packed) || !pointer(a[2], kI32, &counts)) return nullptr;
    return call([&](void* s) { return lq_symbol_counts(p, packed, counts, s); });
}

// words per row of the [K][capacity] stream buffer
bool capacity_of(PyObject* o, int64_t* out)
{
    if (!THPVariable_Check(o) || THPVariable_Unpack(o).dim() < 2) return fail("stream_words must be a [K][capacity] tensor");
    *out = THPVariable_Unpack(o).size(1);
    return true;
}

PyObject* entropy_encode(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; uint32_t *packed, *words, *off; uint16_t* runs; int64_t cap;
    if (!arity(n, 5) || !plan_of(a[0], &p) || !pointer(a[1], kI32, &packed) || !pointer(a[2], kI32, &words) ||
        !capacity_of(a[2], &cap) || !pointer(a[3], kI32, &off) || !pointer(a[4], kI16, &runs)) return nullptr;
    return call([&](void* s) { return lq_entropy_encode(p, packed, words, cap, off, runs, s); });
}

PyObject* entropy_decode(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    lq_plan* p; uint32_t *packed, *words, *off; uint16_t* runs; int64_t cap;
    if (!arity(n, 5) || !plan_of(a[0], &p) || !pointer(a[1], kI32, &words) || !capacity_of(a[1], &cap) ||
        !pointer(a[2], kI32, &off) || !pointer(a[3], kI16, &runs) || !pointer(a[4], kI32, &packed)) return nullptr;
    return call([&](void* s) { return lq_entropy_decode(p, words, cap, off, runs, packed, s); });
}

PyObject* vector_norm_static(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    float *v, *out; uint32_t* st; int32_t q;
    if (!arity(n, 4) || (a[0] == Py_None && !fail("expected a contiguous CUDA tensor")) || !pointer(a[0], kF32, &v) || !int_of(a[1], &q) || !pointer(a[2], kF32, &out) || !pointer(a[3], kI32, &st))
        return nullptr;
    const int64_t len = THPVariable_Unpack(a[0]).numel();
    return call([&](void* s) { return lq_vector_norm_static(v, len, q, out, st, s); });
}

PyObject* register_error(PyObject*, PyObject* cls)
{
    Py_INCREF(cls);
    Py_XDECREF(g_error);
    g_error = cls;
    Py_RETURN_NONE;
}

// Every entry runs inside this: torch's accessors throw for tensors without plain memory (sparse ones, subclasses that answer
// for their layout themselves), and no C++ exception may leave through the interpreter's C frames.
template <PyObject* (*kEntry)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    return kEntry(self, a, n);
    END_HANDLE_TH_ERRORS
}

#define LQ_FAST(name, fn) {name, (PyCFunction)(void (*)(void))guarded<fn>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {LQ_FAST("lq_quantize_pack", quantize_pack), LQ_FAST("qoda_step", step_qoda),
                         LQ_FAST("lq_layer_norms", layer_norms), LQ_FAST("lq_decode_aggregate", decode_aggregate),
                         LQ_FAST("lq_fit_levels", fit_levels), LQ_FAST("lq_level_probabilities", level_probabilities),
                         LQ_FAST("lq_symbol_counts", symbol_counts), LQ_FAST("lq_entropy_encode", entropy_encode),
                         LQ_FAST("lq_entropy_decode", entropy_decode),
                         LQ_FAST("lq_vector_norm_static", vector_norm_static),
                         {"register_error", register_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
#undef LQ_FAST

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
