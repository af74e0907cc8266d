// Python calls of the device entry points: unpacks tensors, messages and integers and calls the C ABI.
//
// A ctypes call of an encoder costs 9 us of Python (attribute look-ups on three tensors, a Stream object, nine
// argument conversions), five times what the library call itself takes; a kernel for a small gradient is done in
// less.  Here the same work takes 0.3 us for an encode, and 0.4 us plus 0.1 us per message for a decode.  The GIL is
// released around the library call, which may block while the stream's launch queue is full.
//
// Every function returns the dq_status; errors of the arguments' types raise TypeError, as the ctypes calls do.  What torch
// throws while a tensor is looked at (one under vmap has no storage, for instance) is raised as the Python exception
// that the tensor's own methods raise.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <vector>

#include "dq.h"

namespace {

PyObject *s_packed, *s_scale, *s_seed, *s_worker, *s_kind, *s_params, *s_cuda_stream;

// An owned reference.
struct Ref {
    PyObject* v;
    explicit Ref(PyObject* owned) : v(owned) {}
    ~Ref() { Py_XDECREF(v); }
    Ref(const Ref&) = delete;
    Ref& operator=(const Ref&) = delete;
};

// The GIL is released while one of these lives.
struct WithoutGil {
    PyThreadState* state = PyEval_SaveThread();
    ~WithoutGil() { PyEval_RestoreThread(state); }
};

const char* type_name(at::ScalarType t)
{
    return t == at::kFloat ? "torch.float32" : t == at::kInt ? "torch.int32" : t == at::kLong ? "torch.int64"
                                                                                             : "torch.uint8";
}

// Address of a contiguous CUDA tensor of the given type; None is a null pointer, which the library judges -- but not where
// the call's length is the tensor's (`numel` given).  False: an exception is set.
bool device_pointer(PyObject* o, at::ScalarType type, const char* what, void** out, int64_t* numel = nullptr)
{
    *out = nullptr;
    if (o == Py_None && !numel) return true;
    if (THPVariable_Check(o)) {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (t.is_cuda() && t.is_contiguous() && t.scalar_type() == type) {
            *out = t.data_ptr();
            if (numel) *numel = t.numel();
            return true;
        }
    }
    PyErr_Format(PyExc_TypeError, "%s: expected a contiguous CUDA tensor of %s", what, type_name(type));
    return false;
}

// Integers wrap to their width, as ctypes converts them.
bool as_u64(PyObject* o, uint64_t* out)
{
    *out = PyLong_AsUnsignedLongLongMask(o);
    return !(*out == (uint64_t)-1 && PyErr_Occurred());
}

bool as_u32(PyObject* o, uint32_t* out)
{
    uint64_t v;
    if (!as_u64(o, &v)) return false;
    *out = (uint32_t)v;
    return true;
}

bool as_params(PyObject* o, dq_params* out)
{
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
    const bool fits = b.len == (Py_ssize_t)sizeof(dq_params);
    if (fits) memcpy(out, b.buf, sizeof(dq_params));
    PyBuffer_Release(&b);
    if (!fits) PyErr_SetString(PyExc_TypeError, "params: expected a DqParams");
    return fits;
}

// None: the current device's current stream; else an object with a cuda_stream address.
bool as_stream(PyObject* o, void** out)
{
    if (o == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    Ref a(PyObject_GetAttr(o, s_cuda_stream));
    uint64_t v;
    if (!a.v || !as_u64(a.v, &v)) return false;
    *out = reinterpret_cast<void*>(v);
    return true;
}

bool as_message(PyObject* o, dq_msg* m)
{
    void* p;
    uint32_t kind;
    {
        Ref a(PyObject_GetAttr(o, s_packed));
        if (!a.v || !device_pointer(a.v, at::kInt, "packed", &p)) return false;
        m->packed = static_cast<const uint32_t*>(p);
    }
    {
        Ref a(PyObject_GetAttr(o, s_scale));
        if (!a.v || !device_pointer(a.v, at::kFloat, "scale", &p)) return false;
        m->scale = static_cast<const float*>(p);
    }
    Ref seed(PyObject_GetAttr(o, s_seed));
    if (!seed.v) return false;
    Ref worker(PyObject_GetAttr(o, s_worker));
    if (!worker.v) return false;
    Ref k(PyObject_GetAttr(o, s_kind));
    if (!k.v) return false;
    Ref params(PyObject_GetAttr(o, s_params));
    if (!params.v) return false;
    if (!as_u64(seed.v, &m->seed) || !as_u32(worker.v, &m->worker) || !as_u32(k.v, &kind)) return false;
    m->kind = static_cast<dq_kind>(kind);
    return as_params(params.v, &m->p);
}

PyObject* wrong_count(const char* name)
{
    PyErr_Format(PyExc_TypeError, "%s: wrong number of arguments", name);
    return nullptr;
}

// encode(kind, grad, first_element, seed, worker, step, params, out_packed, out_scale, stream); -1: an output buffer is
// too small.
PyObject* encode(PyObject*, PyObject* const* a, Py_ssize_t n_args)
{
    if (n_args != 10) return wrong_count("encode");
    uint32_t kind, worker;
    uint64_t first, seed, step;
    int64_t n = 0, have_words = 0, have_scales = 0;
    void *grad, *packed, *scale, *stream;
    dq_params p;
    if (!as_u32(a[0], &kind) || !device_pointer(a[1], at::kFloat, "grad", &grad, &n) || !as_u64(a[2], &first) ||
        !as_u64(a[3], &seed) || !as_u32(a[4], &worker) || !as_u64(a[5], &step) || !as_params(a[6], &p) ||
        !device_pointer(a[7], at::kInt, "out_packed", &packed, &have_words) ||
        !device_pointer(a[8], at::kFloat, "out_scale", &scale, &have_scales) || !as_stream(a[9], &stream))
        return nullptr;
    if ((uint64_t)have_words < dq_packed_words((uint64_t)n, p.bits) ||
        (uint64_t)have_scales < dq_num_buckets((uint64_t)n, p.bucket))
        return PyLong_FromLong(-1);
    dq_status s;
    {
        WithoutGil released;
        s = (kind == DQ_KIND_DQSG ? dqsg_encode_range : ndqsg_encode_range)(
            static_cast<const float*>(grad), (uint64_t)n, first, seed, worker, step, &p, static_cast<uint32_t*>(packed),
            static_cast<float*>(scale), stream);
    }
    return PyLong_FromLong(s);
}

enum Decode : uint32_t { kDqsg = 0, kNdqsg = 1, kRange = 2, kHalfDithered = 3, kRunning = 4, kSideFirst = 5 };

// decode(how, msgs, n, first_element, step, side_info, out_avg, status_word, stream)
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n_args)
{
    if (n_args != 9) return wrong_count("decode");
    uint32_t how;
    uint64_t n, first, step;
    void *side, *out, *status, *stream;
    if (!as_u32(a[0], &how) || !as_u64(a[2], &n) || !as_u64(a[3], &first) || !as_u64(a[4], &step) ||
        !device_pointer(a[5], at::kFloat, "side_info", &side) || !device_pointer(a[6], at::kFloat, "out_avg", &out) ||
        !device_pointer(a[7], at::kInt, "status_word", &status) || !as_stream(a[8], &stream))
        return nullptr;
    Ref seq(PySequence_Tuple(a[1]));         // (a list could change while its messages' attributes are read)
    if (!seq.v) return nullptr;
    const Py_ssize_t W = PyTuple_GET_SIZE(seq.v);
    dq_msg few[DQ_MAX_WORKERS];
    std::vector<dq_msg> many;
    dq_msg* m = few;
    if (W > (Py_ssize_t)DQ_MAX_WORKERS) {
        many.resize((size_t)W);
        m = many.data();
    }
    for (Py_ssize_t w = 0; w < W; ++w) {
        if (!as_message(PyTuple_GET_ITEM(seq.v, w), m + w)) return nullptr;
    }
    float* o = static_cast<float*>(out);
    uint32_t* st = static_cast<uint32_t*>(status);
    dq_status s = DQ_ERR_INVALID_ARG;
    {
        WithoutGil released;
        switch (how) {
            case kDqsg: s = dqsg_decode_aggregate(m, (uint32_t)W, n, step, o, stream); break;
            case kNdqsg:
                s = ndqsg_decode_aggregate(m, (uint32_t)W, n, step, static_cast<const float*>(side), o, st, stream);
                break;
            case kRange:
                s = ndqsg_decode_aggregate_range(m, (uint32_t)W, n, first, step, static_cast<const float*>(side), o, st,
                                                 stream);
                break;
            case kHalfDithered: s = dqsg_decode_aggregate_half_dithered(m, (uint32_t)W, n, o, stream); break;
            case kRunning: s = ndqsg_decode_aggregate_running(m, (uint32_t)W, n, step, o, st, stream); break;
            case kSideFirst: s = ndqsg_decode_aggregate_side_first(m, (uint32_t)W, n, step, o, st, stream); break;
            default: break;
        }
    }
    return PyLong_FromLong(s);
}

// code_histogram(packed, n, bits, hist, stream)
PyObject* code_histogram(PyObject*, PyObject* const* a, Py_ssize_t n_args)
{
    if (n_args != 5) return wrong_count("code_histogram");
    uint64_t n;
    uint32_t bits;
    void *packed, *hist, *stream;
    if (!device_pointer(a[0], at::kInt, "packed", &packed) || !as_u64(a[1], &n) || !as_u32(a[2], &bits) ||
        !device_pointer(a[3], at::kLong, "hist", &hist) || !as_stream(a[4], &stream))
        return nullptr;
    dq_status s;
    {
        WithoutGil released;
        s = dq_code_histogram(static_cast<const uint32_t*>(packed), n, bits, static_cast<uint64_t*>(hist), stream);
    }
    return PyLong_FromLong(s);
}

// ternary_pack(packed, n, out, status_word, stream)
PyObject* ternary_pack(PyObject*, PyObject* const* a, Py_ssize_t n_args)
{
    if (n_args != 5) return wrong_count("ternary_pack");
    uint64_t n;
    void *packed, *out, *status, *stream;
    if (!device_pointer(a[0], at::kInt, "packed", &packed) || !as_u64(a[1], &n) ||
        !device_pointer(a[2], at::kByte, "out", &out) || !device_pointer(a[3], at::kInt, "status_word", &status) ||
        !as_stream(a[4], &stream))
        return nullptr;
    dq_status s;
    {
        WithoutGil released;
        s = dq_ternary_pack(static_cast<const uint32_t*>(packed), n, static_cast<uint8_t*>(out),
                            static_cast<uint32_t*>(status), stream);
    }
    return PyLong_FromLong(s);
}

// ternary_unpack(data, n, out, stream)
PyObject* ternary_unpack(PyObject*, PyObject* const* a, Py_ssize_t n_args)
{
    if (n_args != 4) return wrong_count("ternary_unpack");
    uint64_t n;
    void *data, *out, *stream;
    if (!device_pointer(a[0], at::kByte, "data", &data) || !as_u64(a[1], &n) ||
        !device_pointer(a[2], at::kInt, "out", &out) || !as_stream(a[3], &stream))
        return nullptr;
    dq_status s;
    {
        WithoutGil released;
        s = dq_ternary_unpack(static_cast<const uint8_t*>(data), n, static_cast<uint32_t*>(out), stream);
    }
    return PyLong_FromLong(s);
}

// No C++ exception may leave through the interpreter's C frames.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n_args)
{
    HANDLE_TH_ERRORS
    return F(self, a, n_args);
    END_HANDLE_TH_ERRORS
}

#define DQ_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<f>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {DQ_METHOD(encode),       DQ_METHOD(decode),         DQ_METHOD(code_histogram),
                         DQ_METHOD(ternary_pack), DQ_METHOD(ternary_unpack), {nullptr, nullptr, 0, nullptr}};
#undef DQ_METHOD

PyModuleDef module = {PyModuleDef_HEAD_INIT, "dq_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_dq_calls()
{
    s_packed = PyUnicode_InternFromString("packed");
    s_scale = PyUnicode_InternFromString("scale");
    s_seed = PyUnicode_InternFromString("seed");
    s_worker = PyUnicode_InternFromString("worker");
    s_kind = PyUnicode_InternFromString("kind");
    s_params = PyUnicode_InternFromString("params");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module);
}
