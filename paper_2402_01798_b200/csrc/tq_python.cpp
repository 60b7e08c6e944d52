// Argument marshalling of the Python binding (binding.py): tensors, optional streams and sequences become the plain
// pointers and numbers of include/tq.h.  Nothing else happens here; the functions called are libtq.so's, whose addresses
// binding.py hands over once.  Through ctypes and tensor attributes a call spent 2 to 3.7 us of host time beyond the 2.2 to
// 2.6 us of the launch, which bounds rounds of short gradients.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <exception>
#include <vector>

#include "tq.h"

namespace {

struct Functions {
    decltype(&tq_stats) stats;
    decltype(&tq_stats_hinted) stats_hinted;
    decltype(&tq_stats_static) stats_static;
    decltype(&tq_params_batch) params_batch;
    decltype(&tq_params_device) params_device;
    decltype(&tq_compress) compress;
    decltype(&tq_compress_device_params) compress_device_params;
    decltype(&tq_decompress_aggregate) decompress_aggregate;
    decltype(&tq_decompress_aggregate_rows) decompress_aggregate_rows;
    decltype(&tq_decompress_aggregate_apply) decompress_aggregate_apply;
    decltype(&tq_decompress_aggregate_device_params) decompress_aggregate_device_params;
    decltype(&tq_stats_segments) stats_segments;
    decltype(&tq_stats_hinted_segments) stats_hinted_segments;
    decltype(&tq_compress_segments) compress_segments;
    decltype(&tq_decompress_aggregate_segments) decompress_aggregate_segments;
} F;

struct Failed {};                              // a Python exception is set

[[noreturn]] void fail(PyObject* type, const char* what) {
    PyErr_SetString(type, what);
    throw Failed();
}

// Calls the library with the interpreter lock released, as ctypes does: a launch may wait for room in a full queue, behind a host
// callback that needs the lock.  Arguments are ready before; what they point to is held by the caller's arguments or by Args.
template <class... P, class... A>
tq_status call(tq_status (*f)(P...), const A&... args) {
    struct Unlocked {
        PyThreadState* state = PyEval_SaveThread();
        ~Unlocked() { PyEval_RestoreThread(state); }
    } unlocked;
    return f(args...);
}

// Device address of a tensor, or of anything else with a data_ptr() (a storage, say).
void* address_of(PyObject* o) {
    if (THPVariable_Check(o)) return THPVariable_Unpack(o).data_ptr();
    PyObject* v = PyObject_CallMethod(o, "data_ptr", nullptr);
    if (!v) {
        if (PyErr_ExceptionMatches(PyExc_AttributeError)) fail(PyExc_TypeError, "a tensor is needed");
        throw Failed();
    }
    void* p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) throw Failed();
    return p;
}

// One call's positional arguments, taken in order.
class Args {
public:
    Args(PyObject* const* args, Py_ssize_t n) : args_(args), n_(n) {}
    ~Args() { for (Py_buffer& b : held_) PyBuffer_Release(&b); }
    Args(const Args&) = delete;
    Args& operator=(const Args&) = delete;

    PyObject* next() {
        if (at_ >= n_) fail(PyExc_TypeError, "too few arguments");
        return args_[at_++];
    }
    const at::Tensor& tensor() {
        PyObject* o = next();
        if (!THPVariable_Check(o)) fail(PyExc_TypeError, "a tensor is needed");
        return THPVariable_Unpack(o);
    }
    void* address() {                          // nullptr for None
        PyObject* o = next();
        return o == Py_None ? nullptr : address_of(o);
    }
    // a ctypes array (or anything else with a buffer): its address and size
    void* buffer(Py_ssize_t* bytes = nullptr) {
        held_.emplace_back();
        if (PyObject_GetBuffer(next(), &held_.back(), PyBUF_SIMPLE) != 0) { held_.pop_back(); throw Failed(); }
        if (bytes) *bytes = held_.back().len;
        return held_.back().buf;
    }
    uint64_t u64() {                           // wraps, as a C conversion does; the library checks ranges
        const uint64_t v = PyLong_AsUnsignedLongLongMask(next());
        if (v == ~0ull && PyErr_Occurred()) throw Failed();
        return v;
    }
    uint32_t u32() { return static_cast<uint32_t>(u64()); }
    double f64() {
        const double v = PyFloat_AsDouble(next());
        if (v == -1.0 && PyErr_Occurred()) throw Failed();
        return v;
    }
    float f32() { return static_cast<float>(f64()); }
    // None: torch's current stream; else a stream object, or a raw handle: anything that int() takes (other libraries' handles do)
    void* stream() {
        PyObject* o = next();
        if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        PyObject* handle = PyObject_HasAttrString(o, "cuda_stream") ? PyObject_GetAttrString(o, "cuda_stream") : PyNumber_Long(o);
        if (!handle) throw Failed();
        void* s = PyLong_AsVoidPtr(handle);
        Py_DECREF(handle);
        if (PyErr_Occurred()) throw Failed();
        return s;
    }
    // None, or up to n values that float() takes, the rest zeros.  Only the first TQ_MAX_WORKERS are kept: the library refuses more rows before
    // it reads a weight.
    const float* weights(uint32_t n) {
        PyObject* o = next();
        if (o == Py_None) return nullptr;
        PyObject* seq = PySequence_Fast(o, "weights must be a sequence of numbers");
        if (!seq) throw Failed();
        const Py_ssize_t have = PySequence_Fast_GET_SIZE(seq);
        for (Py_ssize_t i = 0; i < have; ++i) {
            PyObject* w = PyNumber_Float(PySequence_Fast_GET_ITEM(seq, i));
            if (!w) break;
            if (i < TQ_MAX_WORKERS) weights_[i] = static_cast<float>(PyFloat_AS_DOUBLE(w));
            Py_DECREF(w);
        }
        Py_DECREF(seq);
        if (PyErr_Occurred()) throw Failed();
        if (have > n) fail(PyExc_IndexError, "invalid index");
        for (Py_ssize_t i = have; i < TQ_MAX_WORKERS; ++i) weights_[i] = 0.0f;
        return weights_;
    }

private:
    PyObject* const* args_;
    Py_ssize_t n_, at_ = 0;
    std::vector<Py_buffer> held_;
    float weights_[TQ_MAX_WORKERS];
};

// A [N, stride] or [d] gradient block.
struct Grad {
    void* data;
    tq_dtype dtype;
    uint64_t width, stride;
    uint32_t n;
};
Grad gradient(Args& a) {
    const at::Tensor& t = a.tensor();
    if (!t.is_cuda()) fail(PyExc_ValueError, "gradient must be a CUDA tensor");
    const int64_t dims = t.dim();
    if ((dims != 1 && dims != 2) || t.stride(dims - 1) != 1) fail(PyExc_ValueError, "gradient must be [N, stride] with unit inner stride");
    Grad g;
    if (t.scalar_type() == at::kFloat) g.dtype = TQ_F32;
    else if (t.scalar_type() == at::kBFloat16) g.dtype = TQ_BF16;
    else fail(PyExc_TypeError, "gradient must be float32 or bfloat16");
    g.data = t.data_ptr();
    g.n = dims == 2 ? static_cast<uint32_t>(t.size(0)) : 1u;
    g.width = static_cast<uint64_t>(t.size(dims - 1));
    g.stride = g.n > 1 ? static_cast<uint64_t>(t.stride(0)) : g.width;
    return g;
}
uint64_t elements(Args& a, const Grad& g) {     // None: the whole width
    PyObject* o = a.next();
    if (o == Py_None) return g.width;
    const uint64_t v = PyLong_AsUnsignedLongLongMask(o);
    if (v == ~0ull && PyErr_Occurred()) throw Failed();
    return v;
}
// A [N, words] block of packed rows.
struct Packed {
    uint32_t* data;
    size_t stride;
    uint32_t n;
};
Packed packed_rows(const at::Tensor& t) {       // in any memory the GPU reads (pinned host memory too); a row may have several dimensions
    if (t.dim() < 1) fail(PyExc_ValueError, "packed must have a row per worker");
    return Packed{static_cast<uint32_t*>(t.data_ptr()), static_cast<size_t>(t.size(0) > 1 ? t.stride(0) : t.size(1)), static_cast<uint32_t>(t.size(0))};
}
Packed packed_out(Args& a, uint32_t n) {        // as many rows as the gradient has; one row may be given as a vector
    const at::Tensor& t = a.tensor();
    const bool rows = t.dim() == 2 && n > 1;
    return Packed{static_cast<uint32_t*>(t.data_ptr()), static_cast<size_t>(rows ? t.stride(0) : t.size(t.dim() - 1)), n};
}
const tq_params_t* host_params(Args& a, uint32_t n, bool or_more = false) {
    Py_ssize_t bytes = 0;
    void* p = a.buffer(&bytes);
    const Py_ssize_t need = static_cast<Py_ssize_t>(n * sizeof(tq_params_t));
    if (or_more ? bytes < need : bytes != need) fail(PyExc_ValueError, "one Params per worker");
    return static_cast<const tq_params_t*>(p);
}
const tq_segment_t* segments(Args& a, uint32_t* n) {
    Py_ssize_t bytes = 0;
    void* p = a.buffer(&bytes);
    *n = static_cast<uint32_t>(bytes / sizeof(tq_segment_t));
    return static_cast<const tq_segment_t*>(p);
}
struct Scratch { void* data; size_t bytes; };
Scratch scratch(Args& a) {
    const at::Tensor& t = a.tensor();
    return Scratch{t.data_ptr(), static_cast<size_t>(t.numel())};
}

tq_status stats(Args& a) {                      // grad, d, g_min, kappa, stats, workspace, stream
    const Grad g = gradient(a);
    const uint64_t d = elements(a, g);
    const float g_min = a.f32(), kappa = a.f32();
    void* st = a.address();
    const Scratch ws = scratch(a);
    return call(F.stats, g.data, g.dtype, d, g.stride, g.n, g_min, kappa, static_cast<tq_stats_t*>(st), ws.data, ws.bytes, a.stream());
}
tq_status stats_hinted(Args& a) {               // grad, d, kappa, hint, stats, workspace, stream
    const Grad g = gradient(a);
    const uint64_t d = elements(a, g);
    const float kappa = a.f32();
    void* hint = a.address();
    void* st = a.address();
    const Scratch ws = scratch(a);
    return call(F.stats_hinted, g.data, g.dtype, d, g.stride, g.n, kappa, static_cast<tq_gmin_hint_t*>(hint), static_cast<tq_stats_t*>(st), ws.data,
                          ws.bytes, a.stream());
}
tq_status stats_static(Args& a) {               // grad, d, g_min, kappa, stats, stream
    const Grad g = gradient(a);
    const uint64_t d = elements(a, g);
    const float g_min = a.f32(), kappa = a.f32();
    void* st = a.address();
    return call(F.stats_static, g.data, g.dtype, d, g.stride, g.n, g_min, kappa, static_cast<tq_stats_t*>(st), a.stream());
}
tq_status params_batch(Args& a) {               // address of the records, n, num_levels, mode, gamma, rule, alpha_user, out
    PyObject* src = a.next();
    const void* records = THPVariable_Check(src) ? THPVariable_Unpack(src).data_ptr() : PyLong_AsVoidPtr(src);
    if (PyErr_Occurred()) throw Failed();
    const uint32_t n = a.u32(), levels = a.u32(), mode = a.u32();
    const double gamma = a.f64();
    const uint32_t rule = a.u32();
    const double alpha = a.f64();
    return call(F.params_batch, static_cast<const tq_stats_t*>(records), n, levels, static_cast<tq_mode>(mode), gamma, static_cast<tq_alpha_rule>(rule),
                          alpha, static_cast<tq_params_t*>(a.buffer()));
}
tq_status params_device(Args& a) {              // stats, n, num_levels, mode, gamma, rule, alpha_user, params, stream
    void* st = a.address();
    const uint32_t n = a.u32(), levels = a.u32(), mode = a.u32();
    const double gamma = a.f64();
    const uint32_t rule = a.u32();
    const double alpha = a.f64();
    void* out = a.address();
    return call(F.params_device, static_cast<tq_stats_t*>(st), n, levels, static_cast<tq_mode>(mode), gamma, static_cast<tq_alpha_rule>(rule), alpha,
                           static_cast<tq_params_t*>(out), a.stream());
}
tq_status compress(Args& a) {                   // grad, d, params, seed, first_worker, packed, stream
    const Grad g = gradient(a);
    const uint64_t d = elements(a, g);
    const tq_params_t* params = host_params(a, g.n);
    const uint64_t seed = a.u64();
    const uint32_t first = a.u32();
    const Packed p = packed_out(a, g.n);
    return call(F.compress, g.data, g.dtype, d, g.stride, g.n, params, seed, first, p.data, p.stride, a.stream());
}
tq_status compress_device_params(Args& a) {     // grad, d, params, num_levels, mode, seed, first_worker, packed, stream
    const Grad g = gradient(a);
    const uint64_t d = elements(a, g);
    void* params = a.address();
    const uint32_t levels = a.u32(), mode = a.u32();
    const uint64_t seed = a.u64();
    const uint32_t first = a.u32();
    const Packed p = packed_out(a, g.n);
    return call(F.compress_device_params, g.data, g.dtype, d, g.stride, g.n, static_cast<tq_params_t*>(params), levels, static_cast<tq_mode>(mode), seed,
                                    first, p.data, p.stride, a.stream());
}
tq_status decompress_aggregate(Args& a) {       // packed, d, params, weights, out, stream
    const at::Tensor& t = a.tensor();
    if (!t.is_cuda() || t.dim() != 2) fail(PyExc_ValueError, "packed must be a [N, words] CUDA tensor");
    const Packed p = packed_rows(t);
    const uint64_t d = a.u64();
    const tq_params_t* params = host_params(a, p.n);
    const float* w = a.weights(p.n);
    void* out = a.address();
    return call(F.decompress_aggregate, p.data, p.stride, p.n, d, params, w, static_cast<float*>(out), a.stream());
}
tq_status decompress_aggregate_rows(Args& a) {  // rows (tensors or addresses), d, params, weights, out, stream
    PyObject* seq = PySequence_Fast(a.next(), "rows must be a sequence");
    if (!seq) throw Failed();
    const uint32_t* rows[TQ_MAX_WORKERS];
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    try {
        for (Py_ssize_t i = 0; i < n && i < TQ_MAX_WORKERS; ++i) {
            PyObject* r = PySequence_Fast_GET_ITEM(seq, i);
            rows[i] = static_cast<const uint32_t*>(PyLong_Check(r) ? PyLong_AsVoidPtr(r) : address_of(r));
            if (PyErr_Occurred()) throw Failed();
        }
    } catch (...) {
        Py_DECREF(seq);
        throw;
    }
    Py_DECREF(seq);
    const uint64_t d = a.u64();
    const tq_params_t* params = host_params(a, static_cast<uint32_t>(n));
    if (n > TQ_MAX_WORKERS) return TQ_ERR_INVALID_ARG;
    const float* w = a.weights(static_cast<uint32_t>(n));
    void* out = a.address();
    return call(F.decompress_aggregate_rows, rows, static_cast<uint32_t>(n), d, params, w, static_cast<float*>(out), a.stream());
}
tq_status decompress_aggregate_apply(Args& a) { // packed, d, params, weights, theta, momentum, lr, mu, weight_decay, stream
    const Packed p = packed_rows(a.tensor());
    const uint64_t d = a.u64();
    const tq_params_t* params = host_params(a, p.n, true);
    const float* w = a.weights(p.n);
    void* theta = a.address();
    void* momentum = a.address();
    const float lr = a.f32(), mu = a.f32(), wd = a.f32();
    return call(F.decompress_aggregate_apply, p.data, p.stride, p.n, d, params, w, static_cast<float*>(theta), static_cast<float*>(momentum), lr, mu, wd,
                                        a.stream());
}
tq_status decompress_aggregate_device_params(Args& a) {      // packed, d, params, num_levels, weights, out, stream
    const Packed p = packed_rows(a.tensor());
    const uint64_t d = a.u64();
    void* params = a.address();
    const uint32_t levels = a.u32();
    const float* w = a.weights(p.n);
    void* out = a.address();
    return call(F.decompress_aggregate_device_params, p.data, p.stride, p.n, d, static_cast<tq_params_t*>(params), levels, w, static_cast<float*>(out),
                                                a.stream());
}
tq_status stats_segments(Args& a) {             // grad, segments, g_min, kappa, stats, workspace, stream
    const Grad g = gradient(a);
    uint32_t n_seg;
    const tq_segment_t* seg = segments(a, &n_seg);
    const float g_min = a.f32(), kappa = a.f32();
    void* st = a.address();
    const Scratch ws = scratch(a);
    return call(F.stats_segments, g.data, g.dtype, g.stride, g.n, seg, n_seg, g_min, kappa, static_cast<tq_stats_t*>(st), ws.data, ws.bytes, a.stream());
}
tq_status stats_hinted_segments(Args& a) {      // grad, segments, kappa, hint, stats, workspace, stream
    const Grad g = gradient(a);
    uint32_t n_seg;
    const tq_segment_t* seg = segments(a, &n_seg);
    const float kappa = a.f32();
    void* hint = a.address();
    void* st = a.address();
    const Scratch ws = scratch(a);
    return call(F.stats_hinted_segments, g.data, g.dtype, g.stride, g.n, seg, n_seg, kappa, static_cast<tq_gmin_hint_t*>(hint), static_cast<tq_stats_t*>(st),
                                   ws.data, ws.bytes, a.stream());
}
tq_status compress_segments(Args& a) {          // grad, segments, params, num_levels, mode, seed, first_worker, packed, stream
    const Grad g = gradient(a);
    uint32_t n_seg;
    const tq_segment_t* seg = segments(a, &n_seg);
    void* params = a.address();
    const uint32_t levels = a.u32(), mode = a.u32();
    const uint64_t seed = a.u64();
    const uint32_t first = a.u32();
    const Packed p = packed_out(a, g.n);
    return call(F.compress_segments, g.data, g.dtype, g.stride, g.n, seg, n_seg, static_cast<tq_params_t*>(params), levels, static_cast<tq_mode>(mode), seed,
                               first, p.data, p.stride, a.stream());
}
tq_status decompress_aggregate_segments(Args& a) {           // packed, segments, params, num_levels, weights, out, stream
    const Packed p = packed_rows(a.tensor());
    uint32_t n_seg;
    const tq_segment_t* seg = segments(a, &n_seg);
    void* params = a.address();
    const uint32_t levels = a.u32();
    const float* w = a.weights(p.n);
    void* out = a.address();
    return call(F.decompress_aggregate_segments, p.data, p.stride, p.n, seg, n_seg, static_cast<tq_params_t*>(params), levels, w, static_cast<float*>(out),
                                           a.stream());
}

template <tq_status (*CALL)(Args&)>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    try {
        Args a(args, n);
        return PyLong_FromLong(CALL(a));
    } catch (const Failed&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// bind([addresses in the order of Functions])
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    constexpr Py_ssize_t count = sizeof(Functions) / sizeof(void*);
    if (n != 1 || !PyList_Check(args[0]) || PyList_GET_SIZE(args[0]) != count) {
        PyErr_SetString(PyExc_TypeError, "a list of function addresses is needed");
        return nullptr;
    }
    void* p[count];
    for (Py_ssize_t i = 0; i < count; ++i) p[i] = PyLong_AsVoidPtr(PyList_GET_ITEM(args[0], i));
    if (PyErr_Occurred()) return nullptr;
    memcpy(&F, p, sizeof(F));
    Py_RETURN_NONE;
}

#define TQ_ENTRY(name) {#name, reinterpret_cast<PyCFunction>(entry<name>), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(bind), METH_FASTCALL, nullptr},
    TQ_ENTRY(stats), TQ_ENTRY(stats_hinted), TQ_ENTRY(stats_static), TQ_ENTRY(params_batch), TQ_ENTRY(params_device), TQ_ENTRY(compress),
    TQ_ENTRY(compress_device_params), TQ_ENTRY(decompress_aggregate), TQ_ENTRY(decompress_aggregate_rows), TQ_ENTRY(decompress_aggregate_apply),
    TQ_ENTRY(decompress_aggregate_device_params), TQ_ENTRY(stats_segments), TQ_ENTRY(stats_hinted_segments), TQ_ENTRY(compress_segments),
    TQ_ENTRY(decompress_aggregate_segments), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module{PyModuleDef_HEAD_INIT, "_tq_python", "Argument marshalling for libtq.so.", -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__tq_python() { return PyModule_Create(&module); }
