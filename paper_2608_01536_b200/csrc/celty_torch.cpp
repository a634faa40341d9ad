// The calls of the Python binding that a decoder makes once per token and layer, as functions of a CPython module: they
// take torch tensors, check them, make the result where the caller gave none, and call the C ABI on the current stream.
// Nothing is computed here.  A call on a small layer is bound by the host: 6.1 to 6.4 us through ctypes and Python attribute
// look-ups, 3.6 this way, of which the launch itself is 2.4 (1024 x 1024, y made by the call).
//
// Every function gives the result tensor, or the library's status as an int where it is not CELTY_OK.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "celty.h"

namespace {

const at::Tensor &tensor(PyObject *o)
{
    TORCH_CHECK_TYPE(THPVariable_Check(o), "a torch tensor is wanted, not ", Py_TYPE(o)->tp_name);
    return THPVariable_Unpack(o);
}

struct Failed {};                                                 // a Python exception is set

void demand(bool ok, const char *wanted)
{
    if (ok) return;
    PyErr_SetString(PyExc_AssertionError, wanted);
    throw Failed();
}

int64_t integer(PyObject *o)
{
    const int64_t v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return v;
}

float real(PyObject *o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Failed();
    return (float)v;
}

celty_matrix *handle(PyObject *o)
{
    if (o == Py_None) return nullptr;
    void *p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) throw Failed();
    return static_cast<celty_matrix *>(p);
}

struct Ref {
    PyObject *o;
    ~Ref() { Py_XDECREF(o); }
};

Ref attribute(PyObject *o, const char *name)
{
    PyObject *a = PyObject_GetAttrString(o, name);
    if (!a) throw Failed();
    return Ref{a};
}

celty_stream_t stream_of(PyObject *o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    const Ref s = attribute(o, "cuda_stream");
    void *p = PyLong_AsVoidPtr(s.o);
    if (!p && PyErr_Occurred()) throw Failed();
    return p;
}

// The library gets bare pointers and cannot tell how long a vector is or where it lies, so all of that is checked here.
// A kernel reaches GPU memory, and host memory that is page-locked.
bool reachable(const at::Tensor &t) { return t.is_cuda() || (t.is_cpu() && t.is_pinned()); }

void *vector(const at::Tensor &t, at::ScalarType type, int64_t n, const char *wanted)
{
    demand(t.scalar_type() == type && t.numel() == n && t.is_contiguous() && reachable(t), wanted);
    return t.data_ptr();
}

// The same for one that may be longer than what is read or written.
void *long_vector(const at::Tensor &t, at::ScalarType type, int64_t n, const char *wanted)
{
    demand(t.scalar_type() == type && t.numel() >= n && t.is_contiguous() && reachable(t), wanted);
    return t.data_ptr();
}

constexpr char kWantX[] = "x: K float16, contiguous, on the GPU", kWantY[] = "y: M float32, contiguous, on the GPU",
               kWantFp16[] = "fp16_out: M float16, contiguous, on the GPU";

// The result: the caller's y, checked, or a new vector of M on `like`'s device.
struct Result {
    at::Tensor made;
    PyObject *given = nullptr;
    void *data = nullptr;
    Result(PyObject *y, int64_t M, const at::Tensor &like, bool may_be_longer = false)
    {
        if (y == Py_None) {
            made = at::empty({M}, at::TensorOptions().dtype(at::kFloat).device(like.device()));
            data = vector(made, at::kFloat, M, kWantY);
        } else {
            given = y;
            data = (may_be_longer ? long_vector : vector)(tensor(y), at::kFloat, M, kWantY);
        }
    }
    PyObject *give(int status)
    {
        if (status != CELTY_OK) return PyLong_FromLong(status);
        if (given) {
            Py_INCREF(given);
            return given;
        }
        return THPVariable_Wrap(std::move(made));
    }
};

// (The interpreter's lock is given back while the library launches, as ctypes does.)
template <typename Call>
int without_lock(Call call)
{
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return rc;
}

// FP16 copy of y (a tensor or None) as an epilogue
bool fp16_epilogue(PyObject *out, int64_t M, celty_epilogue *ep, bool may_be_longer = false)
{
    *ep = celty_epilogue{};
    if (out == Py_None) return false;
    ep->kind = CELTY_EPILOGUE_FP16;
    ep->out_fp16 = (may_be_longer ? long_vector : vector)(tensor(out), at::kHalf, M, kWantFp16);
    return true;
}

// FP16 values of a survivor list, as such or as their bit patterns
uint16_t *list_values(const at::Tensor &t, int64_t n, const char *wanted)
{
    return static_cast<uint16_t *>(long_vector(t, t.scalar_type() == at::kHalf ? at::kHalf : at::kShort, n, wanted));
}

template <PyObject *(*body)(PyObject *const *)>
PyObject *guarded(PyObject *, PyObject *const *a, Py_ssize_t n, Py_ssize_t wanted)
{
    HANDLE_TH_ERRORS
    if (n != wanted) {
        PyErr_Format(PyExc_TypeError, "%zd arguments wanted, %zd given", wanted, n);
        return nullptr;
    }
    try {
        return body(a);
    } catch (const Failed &) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

#define CELTY_METHOD(name, wanted) \
    PyObject *name##_call(PyObject *self, PyObject *const *a, Py_ssize_t n) { return guarded<name>(self, a, n, wanted); }

// handle, M, K, x, tau, y, stream
PyObject *spmspv(PyObject *const *a)
{
    celty_matrix *m = handle(a[0]);
    const int64_t M = integer(a[1]), K = integer(a[2]);
    const at::Tensor &x = tensor(a[3]);
    const float tau = real(a[4]);
    const void *xp = vector(x, at::kHalf, K, kWantX);
    Result y(a[5], M, x);
    const celty_stream_t st = stream_of(a[6]);
    return y.give(without_lock([&] { return celty_spmspv(m, xp, tau, y.data, st); }));
}
CELTY_METHOD(spmspv, 7)

// handle, M, K, x, tau, y, stream, image
PyObject *spmspv_static(PyObject *const *a)
{
    celty_matrix *m = handle(a[0]);
    const int64_t M = integer(a[1]), K = integer(a[2]);
    const at::Tensor &x = tensor(a[3]);
    const float tau = real(a[4]);
    const void *xp = vector(x, at::kHalf, K, kWantX);
    Result y(a[5], M, x);
    const at::Tensor &packed = tensor(a[7]);
    demand(reachable(packed), "the packed image on the GPU");
    const void *image = packed.data_ptr();
    const celty_stream_t st = stream_of(a[6]);
    return y.give(without_lock([&] { return celty_spmspv_static(m, image, xp, tau, y.data, st); }));
}
CELTY_METHOD(spmspv_static, 8)

// handle, M, K, x, tau, y, stream, fp16_out, swiglu
PyObject *spmspv_ex(PyObject *const *a)
{
    celty_matrix *m = handle(a[0]);
    const int64_t M = integer(a[1]), K = integer(a[2]);
    const at::Tensor &x = tensor(a[3]);
    const float tau = real(a[4]);
    const void *xp = vector(x, at::kHalf, K, kWantX);
    Result y(a[5], M, x);
    celty_epilogue ep{};
    bool with = false;
    if (a[8] != Py_None) {
        const Ref t = attribute(a[8], "tau"), h = attribute(a[8], "h"), idx = attribute(a[8], "idx"), val = attribute(a[8], "val"),
                  count = attribute(a[8], "count");
        ep.kind = CELTY_EPILOGUE_SWIGLU;
        ep.tau = real(t.o);
        ep.out_fp16 = long_vector(tensor(h.o), at::kHalf, M / 2, "swiglu.h: M / 2 float16, contiguous, on the GPU");
        ep.list_idx = static_cast<int32_t *>(long_vector(tensor(idx.o), at::kInt, M / 2, "swiglu.idx: M / 2 int32, contiguous, on the GPU"));
        ep.list_val = list_values(tensor(val.o), M / 2, "swiglu.val: M / 2 FP16 values or bit patterns, contiguous, on the GPU");
        ep.list_count = static_cast<int32_t *>(long_vector(tensor(count.o), at::kInt, 1, "swiglu.count: an int32 on the GPU"));
        with = true;
    } else {
        with = fp16_epilogue(a[7], M, &ep);
    }
    const celty_stream_t st = stream_of(a[6]);
    return y.give(without_lock([&] { return celty_spmspv_ex(m, xp, tau, y.data, with ? &ep : nullptr, st); }));
}
CELTY_METHOD(spmspv_ex, 9)

// handle, M, K, gate_up, tau, y, stream, h_out, fp16_out
PyObject *spmspv_swiglu(PyObject *const *a)
{
    celty_matrix *m = handle(a[0]);
    const int64_t M = integer(a[1]), K = integer(a[2]);
    const at::Tensor &gate_up = tensor(a[3]);
    const float tau = real(a[4]);
    const float *in = static_cast<const float *>(vector(gate_up, at::kFloat, 2 * K, "gate_up: 2 K float32, contiguous, on the GPU"));
    Result y(a[5], M, gate_up, true);
    celty_epilogue ep;
    const bool with = fp16_epilogue(a[8], M, &ep, true);
    void *h = a[7] == Py_None ? nullptr : long_vector(tensor(a[7]), at::kHalf, K, "h_out: K float16, contiguous, on the GPU");
    const celty_stream_t st = stream_of(a[6]);
    return y.give(without_lock([&] { return celty_spmspv_swiglu(m, in, tau, y.data, h, with ? &ep : nullptr, st); }));
}
CELTY_METHOD(spmspv_swiglu, 9)

// handle, M, idx, val, count, y, stream, fp16_out
PyObject *spmspv_list(PyObject *const *a)
{
    celty_matrix *m = handle(a[0]);
    const int64_t M = integer(a[1]);
    // (how many columns are listed is known on the GPU only: the two vectors have to be as long as the list)
    const at::Tensor &idx = tensor(a[2]);
    const int32_t *ip = static_cast<const int32_t *>(long_vector(idx, at::kInt, 0, "idx: int32, contiguous, on the GPU"));
    const uint16_t *vp = list_values(tensor(a[3]), 0, "val: FP16 values or bit patterns, contiguous, on the GPU");
    const int32_t *np = static_cast<const int32_t *>(long_vector(tensor(a[4]), at::kInt, 1, "count: an int32 on the GPU"));
    Result y(a[5], M, idx, true);
    celty_epilogue ep;
    const bool with = fp16_epilogue(a[7], M, &ep);
    const celty_stream_t st = stream_of(a[6]);
    return y.give(without_lock([&] { return celty_spmspv_list(m, ip, vp, np, y.data, with ? &ep : nullptr, st); }));
}
CELTY_METHOD(spmspv_list, 8)

// handle, M, K, x, tau, y, stream, scratch
PyObject *spmspv_batch(PyObject *const *a)
{
    celty_matrix *m = handle(a[0]);
    const int64_t M = integer(a[1]), K = integer(a[2]);
    const at::Tensor &x = tensor(a[3]);
    const float tau = real(a[4]);
    demand(x.scalar_type() == at::kHalf && x.dim() == 2 && x.size(1) == K && x.stride(1) == 1 && reachable(x),
           "x: N rows of K float16 on the GPU, the values of a row side by side");
    const int64_t N = x.size(0);
    at::Tensor made;
    PyObject *given = a[5];
    if (given == Py_None) made = at::empty({N, M}, at::TensorOptions().dtype(at::kFloat).device(x.device()));
    const at::Tensor &y = given == Py_None ? made : tensor(given);
    demand(y.scalar_type() == at::kFloat && y.dim() == 2 && y.size(0) == N && y.size(1) == M && y.stride(1) == 1 && reachable(y),
           "y: N rows of M float32 on the GPU, the values of a row side by side");
    const at::Tensor &scratch = tensor(a[7]);
    demand(reachable(scratch), "the scratch on the GPU");
    const void *xp = x.data_ptr();
    void *yp = y.data_ptr(), *sp = scratch.data_ptr();
    const int64_t ldx = x.stride(0), ldy = y.stride(0);
    const size_t bytes = (size_t)scratch.numel();
    const celty_stream_t st = stream_of(a[6]);
    const int rc = without_lock([&] { return celty_spmspv_batch(m, xp, ldx, (int32_t)N, tau, yp, ldy, sp, bytes, st); });
    if (rc != CELTY_OK) return PyLong_FromLong(rc);
    if (given == Py_None) return THPVariable_Wrap(std::move(made));
    Py_INCREF(given);
    return given;
}
CELTY_METHOD(spmspv_batch, 8)

#define CELTY_ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name##_call)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {CELTY_ENTRY(spmspv),        CELTY_ENTRY(spmspv_static), CELTY_ENTRY(spmspv_ex), CELTY_ENTRY(spmspv_swiglu),
                         CELTY_ENTRY(spmspv_list),   CELTY_ENTRY(spmspv_batch),  {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_celty_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// What the build looks for in the file; the binding compares the version with torch's before the first call.
const char built_with[] = "built with torch " TORCH_VERSION;

PyMODINIT_FUNC PyInit__celty_torch(void)
{
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_with", built_with) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
