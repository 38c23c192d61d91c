// Native half of the Python binding: the calls of a training or serving loop take tensors straight to the C ABI.
// Marshalling them through ctypes (a Python call per pointer, some twelve of them, and two Python objects for the
// stream) cost 8 to 11 us a call, as much as the kernels of a small batch.  Nothing is kept between calls; the checks
// are those of binding.py.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <algorithm>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include "dqrm.h"

namespace {

// addresses of the C ABI, handed over once by binding.py (which has loaded the library)
struct Abi {
    decltype(&dqrm_scale_refresh) scale_refresh;
    decltype(&dqrm_emb_fwd) emb_fwd;
    decltype(&dqrm_emb_bwd) emb_bwd;
    decltype(&dqrm_grad_quant_int8_bounded) grad_quant_int8;
    decltype(&dqrm_row_update) row_update;
    decltype(&dqrm_train_step) train_step;
    decltype(&dqrm_sort_batch) sort_batch;
    decltype(&dqrm_train_step_sorted) train_step_sorted;
    decltype(&dqrm_train_step_host) train_step_host;
    decltype(&dqrm_pack_tables) pack_tables;
    decltype(&dqrm_packed_fwd) packed_fwd;
} abi;

const char *name_of(at::ScalarType t)
{
    switch (t) {
    case at::kFloat: return "torch.float32";
    case at::kInt: return "torch.int32";
    case at::kChar: return "torch.int8";
    case at::kByte: return "torch.uint8";
    default: return c10::toString(t);
    }
}

// Arguments of one call, taken in order; the first that does not fit leaves a Python error
struct Reader {
    PyObject *const *args;
    Py_ssize_t n, at = 0;
    bool ok;
    int64_t numel = 0;                                  // of the tensor read last

    Reader(PyObject *const *a, Py_ssize_t count, Py_ssize_t want) : args(a), n(count), ok(count == want)
    {
        if (!ok) PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, count);
    }
    void fail(const char *text)
    {
        if (ok) PyErr_SetString(PyExc_AssertionError, text);
        ok = false;
    }
    void *pointer(at::ScalarType dtype, bool device = true)
    {
        if (!ok) return nullptr;
        PyObject *o = args[at++];
        if (o == Py_None) return nullptr;
        if (!THPVariable_Check(o)) { fail("expected a torch tensor"); return nullptr; }
        const at::Tensor &t = THPVariable_Unpack(o);
        if (!t.is_contiguous()) { fail("tensor must be contiguous"); return nullptr; }
        if (t.scalar_type() != dtype) {
            PyErr_Format(PyExc_AssertionError, "expected %s, got %s", name_of(dtype), name_of(t.scalar_type()));
            ok = false;
            return nullptr;
        }
        if (t.is_cuda() != device) { fail(device ? "expected a CUDA tensor" : "expected a host tensor"); return nullptr; }
        numel = t.numel();
        return t.data_ptr();
    }
    float *f32() { return static_cast<float *>(pointer(at::kFloat)); }
    int32_t *i32() { return static_cast<int32_t *>(pointer(at::kInt)); }
    int8_t *i8() { return static_cast<int8_t *>(pointer(at::kChar)); }
    uint8_t *u8() { return static_cast<uint8_t *>(pointer(at::kByte)); }
    float *h_f32() { return static_cast<float *>(pointer(at::kFloat, false)); }
    int32_t *h_i32() { return static_cast<int32_t *>(pointer(at::kInt, false)); }
    int64_t integer()
    {
        if (!ok) return 0;
        PyObject *o = PyNumber_Long(args[at++]);       // (int(...) of whatever the caller passed)
        const int64_t v = o ? PyLong_AsLongLong(o) : -1;
        Py_XDECREF(o);
        if (v == -1 && PyErr_Occurred()) ok = false;
        return v;
    }
    int int32()
    {
        const int64_t v = integer();
        if (ok && (v < INT32_MIN || v > INT32_MAX)) { PyErr_SetString(PyExc_OverflowError, "integer out of range"); ok = false; }
        return (int)v;
    }
    float number()
    {
        if (!ok) return 0.f;
        PyObject *o = PyNumber_Float(args[at++]);      // (float(...) of whatever the caller passed)
        const double v = o ? PyFloat_AsDouble(o) : -1.0;
        Py_XDECREF(o);
        if (v == -1.0 && PyErr_Occurred()) ok = false;
        return (float)v;
    }
    void *address()                                     // an address held as a Python integer
    {
        if (!ok) return nullptr;
        void *p = PyLong_AsVoidPtr(args[at++]);
        if (!p && PyErr_Occurred()) ok = false;
        return p;
    }
    void *stream()                                      // a torch stream, or None for the current one
    {
        if (!ok) return nullptr;
        PyObject *o = args[at++];
        if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        PyObject *raw = PyObject_GetAttrString(o, "cuda_stream");
        void *p = raw ? PyLong_AsVoidPtr(raw) : nullptr;
        Py_XDECREF(raw);
        if (PyErr_Occurred()) ok = false;
        return p;
    }
};

// The interpreter's lock is given back for the call, and taken again whichever way the call is left
struct WithoutGil {
    PyThreadState *state = PyEval_SaveThread();
    ~WithoutGil() { PyEval_RestoreThread(state); }
};

// (arguments are read in the order of the braces, which is the order of the C ABI)
// torch's own calls may throw (a tensor without storage under tracing or vmap, no CUDA device for the current stream):
// nothing may leave through the interpreter's C frames, so exceptions become Python errors here
#define DQ_CALL(NAME, COUNT, ...)                                                   \
    PyObject *py_##NAME(PyObject *, PyObject *const *args, Py_ssize_t n)            \
    {                                                                               \
        HANDLE_TH_ERRORS                                                            \
        Reader r(args, n, COUNT);                                                   \
        dqrm_ctx *ctx = static_cast<dqrm_ctx *>(r.address());                       \
        __VA_ARGS__                                                                 \
        END_HANDLE_TH_ERRORS                                                        \
    }
#define DQ_RETURN(CALL)                                                             \
    if (!r.ok) return nullptr;                                                      \
    int status;                                                                     \
    {                                                                               \
        WithoutGil released;                                                        \
        status = CALL;                                                              \
    }                                                                               \
    return PyLong_FromLong(status)

DQ_CALL(scale_refresh, 8,
    float *tables = r.f32(); int32_t *bits = r.i32(); float *scales = r.f32(); float *minmax = r.f32();
    void *ws = r.address(); size_t bytes = (size_t)r.integer(); void *st = r.stream();
    DQ_RETURN(abi.scale_refresh(ctx, tables, bits, scales, minmax, ws, bytes, st));)

DQ_CALL(emb_fwd, 11,
    float *tables = r.f32(); int32_t *idx = r.i32(); int32_t *off = r.i32(); float *scales = r.f32(); int32_t *bits = r.i32();
    float *out = r.f32(); int8_t *codes = r.i8(); int B = r.int32(); int64_t L = r.integer(); void *st = r.stream();
    DQ_RETURN(abi.emb_fwd(ctx, tables, idx, off, scales, bits, out, codes, B, L, st));)

DQ_CALL(emb_bwd, 12,
    float *go = r.f32(); int32_t *idx = r.i32(); int32_t *off = r.i32(); int32_t *ur = r.i32(); int32_t *uo = r.i32();
    float *gr = r.f32(); int B = r.int32(); int64_t L = r.integer(); void *ws = r.address(); size_t bytes = (size_t)r.integer();
    void *st = r.stream();
    DQ_RETURN(abi.emb_bwd(ctx, go, idx, off, ur, uo, gr, B, L, ws, bytes, st));)

DQ_CALL(grad_quant_int8, 8,
    float *gr = r.f32(); int64_t room = r.numel; int32_t *uo = r.i32(); int8_t *codes = r.i8(); room = std::min(room, r.numel);
    float *gs = r.f32(); void *ws = r.address(); size_t bytes = (size_t)r.integer(); void *st = r.stream();
    DQ_RETURN(abi.grad_quant_int8(ctx, gr, uo, codes, gs, room, ws, bytes, st));)

DQ_CALL(row_update, 8,
    float *tables = r.f32(); int32_t *ur = r.i32(); int32_t *uo = r.i32(); int8_t *codes = r.i8(); float *gs = r.f32();
    float lr = r.number(); void *st = r.stream();
    DQ_RETURN(abi.row_update(ctx, tables, ur, uo, codes, gs, lr, st));)

#define DQ_STEP(NAME)                                                                                                      \
    DQ_CALL(NAME, 19,                                                                                                      \
        float *tables = r.f32(); int32_t *idx = r.i32(); int32_t *off = r.i32(); float *go = r.f32();                      \
        float *scales = r.f32(); int32_t *bits = r.i32(); float *out = r.f32(); int32_t *ur = r.i32();                     \
        int32_t *uo = r.i32(); float *gr = r.f32(); int8_t *codes = r.i8(); float *gs = r.f32(); float lr = r.number();    \
        int B = r.int32(); int64_t L = r.integer(); void *ws = r.address(); size_t bytes = (size_t)r.integer();            \
        void *st = r.stream();                                                                                             \
        DQ_RETURN(abi.NAME(ctx, tables, idx, off, go, scales, bits, out, ur, uo, gr, codes, gs, lr, B, L, ws, bytes, st));)
DQ_STEP(train_step)
DQ_STEP(train_step_sorted)

DQ_CALL(sort_batch, 10,
    int32_t *idx = r.i32(); int32_t *off = r.i32(); int32_t *ur = r.i32(); int32_t *uo = r.i32(); int B = r.int32();
    int64_t L = r.integer(); void *ws = r.address(); size_t bytes = (size_t)r.integer(); void *st = r.stream();
    DQ_RETURN(abi.sort_batch(ctx, idx, off, ur, uo, B, L, ws, bytes, st));)

DQ_CALL(train_step_host, 14,
    float *tables = r.f32(); int32_t *idx = r.h_i32(); int32_t *off = r.h_i32(); float *go = r.h_f32(); float *scales = r.f32();
    int32_t *bits = r.i32(); float *out = r.h_f32(); float lr = r.number(); int B = r.int32(); int64_t L = r.integer();
    void *ws = r.address(); size_t bytes = (size_t)r.integer(); void *st = r.stream();
    DQ_RETURN(abi.train_step_host(ctx, tables, idx, off, go, scales, bits, out, lr, B, L, ws, bytes, st));)

DQ_CALL(pack_tables, 6,
    float *tables = r.f32(); float *scales = r.f32(); int bits = r.int32(); uint8_t *packed = r.u8(); void *st = r.stream();
    DQ_RETURN(abi.pack_tables(ctx, tables, scales, bits, packed, st));)

DQ_CALL(packed_fwd, 10,
    uint8_t *packed = r.u8(); int32_t *idx = r.i32(); int32_t *off = r.i32(); float *scales = r.f32(); int bits = r.int32();
    float *out = r.f32(); int B = r.int32(); int64_t L = r.integer(); void *st = r.stream();
    DQ_RETURN(abi.packed_fwd(ctx, packed, idx, off, scales, bits, out, B, L, st));)

// bind(addresses): the functions' addresses in the order of Abi's members
PyObject *py_bind(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    static_assert(sizeof(Abi) % sizeof(void *) == 0, "");
    constexpr Py_ssize_t want = sizeof(Abi) / sizeof(void *);
    if (n != want) return PyErr_Format(PyExc_TypeError, "expected %zd addresses, got %zd", want, n);
    void *p[want];
    for (Py_ssize_t i = 0; i < want; ++i) {
        p[i] = PyLong_AsVoidPtr(args[i]);
        if (!p[i]) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_ValueError, "null address");
    }
    memcpy(&abi, p, sizeof(abi));
    Py_RETURN_NONE;
}

#define DQ_METHOD(NAME) {#NAME, (PyCFunction)(void (*)(void))py_##NAME, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    DQ_METHOD(bind), DQ_METHOD(scale_refresh), DQ_METHOD(emb_fwd), DQ_METHOD(emb_bwd), DQ_METHOD(grad_quant_int8),
    DQ_METHOD(row_update), DQ_METHOD(train_step), DQ_METHOD(sort_batch), DQ_METHOD(train_step_sorted),
    DQ_METHOD(train_step_host), DQ_METHOD(pack_tables), DQ_METHOD(packed_fwd), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_dqrm_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__dqrm_native(void) { return PyModule_Create(&module); }
