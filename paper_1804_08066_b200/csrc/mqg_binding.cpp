// The Python entry points that enqueue work, as native functions over the C ABI of include/mqgrad.h: they
// take torch tensors, read the device pointers and torch's current stream, and make the call.
//
// Why native: a call's work on the device takes 2 to 4 us for gradients up to a million elements, and a
// launch about as long on the host.  Marshalling through ctypes (a Python frame, a type check and a
// data_ptr() call per tensor, a pointer table per list, a stream object, argument conversion) took 7 us for
// the call with the fewest arguments and 22 us for one that takes three lists of eight tensors, so the
// device waited for the host.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <vector>

#include "../../include/mqgrad.h"

namespace {

constexpr int kMaxArgs = 16;

// One entry point's parameters, in order; the last `ndefaults` may be left out (a null slot).
struct Signature {
    const char* function;
    int nargs, ndefaults;
    const char* names[kMaxArgs];
    PyObject* interned[kMaxArgs];
};

// Positional and keyword arguments of a call into slots (borrowed references).
bool bind_arguments(Signature& sig, PyObject* const* args, Py_ssize_t npos, PyObject* kwnames, PyObject** slot)
{
    if (npos > sig.nargs) {
        PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", sig.function, sig.nargs, npos);
        return false;
    }
    for (int i = 0; i < sig.nargs; ++i) slot[i] = i < npos ? args[i] : nullptr;
    const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nkw; ++k) {
        PyObject* key = PyTuple_GET_ITEM(kwnames, k);
        int at = -1;
        for (int i = 0; i < sig.nargs && at < 0; ++i)
            if (key == sig.interned[i]) at = i;
        for (int i = 0; i < sig.nargs && at < 0; ++i)
            if (PyUnicode_CompareWithASCIIString(key, sig.names[i]) == 0) at = i;
        if (at < 0) {
            PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", sig.function, key);
            return false;
        }
        if (slot[at]) {
            PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%s'", sig.function, sig.names[at]);
            return false;
        }
        slot[at] = args[npos + k];
    }
    for (int i = 0; i < sig.nargs - sig.ndefaults; ++i)
        if (!slot[i]) {
            PyErr_Format(PyExc_TypeError, "%s() missing required argument: '%s'", sig.function, sig.names[i]);
            return false;
        }
    return true;
}

// Thrown with a Python error set.
struct PythonError {};

uint64_t to_u64(PyObject* o, uint64_t absent = 0)
{
    if (!o) return absent;
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);      // wraps like a C conversion
    if (v == (unsigned long long)-1 && PyErr_Occurred()) throw PythonError();
    return v;
}
uint32_t to_u32(PyObject* o) { return (uint32_t)to_u64(o); }
int to_int(PyObject* o) { return (int)(uint32_t)to_u64(o); }
float to_float(PyObject* o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PythonError();
    return (float)v;
}
bool to_bool(PyObject* o)
{
    if (!o) return false;
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw PythonError();
    return v != 0;
}

// THPVariable_Check asks isinstance(), which an object can answer without being a tensor.
bool is_tensor(PyObject* o) { return PyObject_TypeCheck(o, reinterpret_cast<PyTypeObject*>(THPVariableClass)); }

// Device pointer of a contiguous CUDA tensor.  `index` >= 0: the tensor is that item of a list.
void* device_ptr(PyObject* o, const char* what, Py_ssize_t index = -1)
{
    char name[64];
    auto called = [&]() -> const char* {
        if (index < 0) return what;
        snprintf(name, sizeof(name), "%s[%zd]", what, index);
        return name;
    };
    if (!is_tensor(o) || !THPVariable_Unpack(o).is_cuda()) {
        PyErr_Format(PyExc_TypeError, "%s must be a CUDA tensor (libmqgrad has no CPU path)", called());
        throw PythonError();
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_contiguous()) {
        PyErr_Format(PyExc_ValueError, "%s must be contiguous", called());
        throw PythonError();
    }
    return t.data_ptr();
}

mqg_dtype grad_dtype(PyObject* o)
{
    if (is_tensor(o)) {
        const at::ScalarType s = THPVariable_Unpack(o).scalar_type();
        if (s == at::kFloat) return MQG_F32;
        if (s == at::kBFloat16) return MQG_BF16;
        PyErr_Format(PyExc_TypeError, "grad must be float32 or bfloat16, got %s", c10::toString(s));
    } else {
        PyErr_SetString(PyExc_TypeError, "grad must be a tensor");
    }
    throw PythonError();
}

// A list (or tuple, or any iterable) of W tensors as a table of device pointers.  Everything that is wanted of the
// items is read at once: later arguments may run Python code that changes the list.
struct PointerTable {
    void* ptr[MQG_MAX_WORKERS];
    PyObject* items = nullptr;
    Py_ssize_t count = 0;
    ~PointerTable() { Py_XDECREF(items); }

    // `exact`: the list has to hold exactly W tensors; otherwise at least W.
    void read(PyObject* o, const char* what, int W, bool exact)
    {
        items = PySequence_Fast(o, "a list of tensors is expected");
        if (!items) throw PythonError();
        count = PySequence_Fast_GET_SIZE(items);
        // a worker count outside the library's range is the C ABI's to reject: it reads no table then
        if (exact ? count != W : count < W && W <= MQG_MAX_WORKERS) {
            PyErr_Format(PyExc_ValueError, "%s must hold %s%d tensors, got %zd", what, exact ? "" : "at least ", W, count);
            throw PythonError();
        }
        const Py_ssize_t n = count < MQG_MAX_WORKERS ? count : MQG_MAX_WORKERS;
        for (Py_ssize_t i = 0; i < n; ++i) ptr[i] = device_ptr(PySequence_Fast_GET_ITEM(items, i), what, i);
    }
    template <typename T> T* const* as() const { return reinterpret_cast<T* const*>(ptr); }
};

struct GradientTable : PointerTable {
    mqg_dtype dtype;

    // `all_alike`: every gradient must have the first one's type.
    void read(PyObject* o, int W, bool exact, bool all_alike)
    {
        PointerTable::read(o, "grads", W, exact);
        if (count == 0) {
            if (all_alike) PyErr_SetString(PyExc_TypeError, "all gradients must have the same dtype: there are none");
            else PyErr_SetString(PyExc_IndexError, "grads is empty");
            throw PythonError();
        }
        dtype = grad_dtype(PySequence_Fast_GET_ITEM(items, 0));
        for (Py_ssize_t i = 1; all_alike && i < count; ++i)
            if (grad_dtype(PySequence_Fast_GET_ITEM(items, i)) != dtype) {
                PyErr_SetString(PyExc_TypeError, "all gradients must have the same dtype");
                throw PythonError();
            }
    }
};

struct Reference {
    PyObject* object;
    ~Reference() { Py_XDECREF(object); }
};

// A segment table: 64-bit integers from an array that exposes them, or from any sequence of numbers.  Copied: the
// library checks the table and then uses it, without the interpreter lock.
struct OffsetTable {
    uint64_t inline_store[65];
    std::vector<uint64_t> store;
    const uint64_t* data = nullptr;
    Py_ssize_t count = 0;

    void read(PyObject* o)
    {
        if (!PyList_Check(o) && !PyTuple_Check(o) && PyObject_CheckBuffer(o) && read_buffer(o)) return;
        const Reference items = {PySequence_Tuple(o)};  // a list could change while its items are converted
        if (!items.object) throw PythonError();
        uint64_t* to = room(PyTuple_GET_SIZE(items.object));
        for (Py_ssize_t i = 0; i < count; ++i) {
            PyObject* v = PyTuple_GET_ITEM(items.object, i);
            const Reference whole = {PyLong_CheckExact(v) ? Py_NewRef(v) : PyNumber_Long(v)};
            if (!whole.object) throw PythonError();
            to[i] = to_u64(whole.object);
        }
    }

private:
    uint64_t* room(Py_ssize_t n)
    {
        uint64_t* to = inline_store;
        if (n > 65) { store.resize((size_t)n); to = store.data(); }
        data = to;
        count = n;
        return to;
    }
    bool read_buffer(PyObject* o)
    {
        struct View : Py_buffer { ~View() { PyBuffer_Release(this); } } view;       // (releasing an empty one does nothing)
        if (PyObject_GetBuffer(o, &view, PyBUF_FORMAT | PyBUF_C_CONTIGUOUS) != 0) {
            PyErr_Clear();
            return false;
        }
        const bool offsets = view.ndim == 1 && view.itemsize == 8 && view.format && view.format[0] != '\0' &&
                             view.format[1] == '\0' && std::strchr("lLqQ", view.format[0]);
        if (offsets) std::memcpy(room(view.len / 8), view.buf, (size_t)view.len);
        return offsets;
    }
};

// seg_off and code_off of a call; returns the number of segments.
int read_segments(PyObject* seg_off, PyObject* code_off, OffsetTable& seg, OffsetTable& code)
{
    seg.read(seg_off);
    code.read(code_off);
    if (code.count < seg.count) {
        PyErr_Format(PyExc_ValueError, "code_off holds %zd offsets, seg_off %zd", code.count, seg.count);
        throw PythonError();
    }
    return (int)seg.count - 1;
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

PyObject* g_error_class = nullptr;      // MqgError of the package

// None, or the package's MqgError with the library's message.
PyObject* finish(mqg_status st)
{
    if (st == MQG_OK) Py_RETURN_NONE;
    PyObject* e = PyObject_CallFunction(g_error_class, "is", (int)st, mqg_last_error());
    if (e) { PyErr_SetObject(g_error_class, e); Py_DECREF(e); }
    return nullptr;
}

// The call itself runs without the interpreter lock: a full launch queue blocks it.  The lock is back whichever way
// the call ends.
struct WithoutLock {
    PyThreadState* state = PyEval_SaveThread();
    ~WithoutLock() { PyEval_RestoreThread(state); }
};
template <typename Fn> PyObject* enqueue(Fn&& fn)
{
    mqg_status st;
    {
        const WithoutLock unlocked;
        st = fn();
    }
    return finish(st);
}

// Defines the native function `name`: binds the arguments to `v[]` and runs the body that follows.
#define MQG_ENTRY(name, ndefaults, nargs, ...)                                                                      \
    Signature sig_##name = {#name, nargs, ndefaults, {__VA_ARGS__}, {}};                                            \
    PyObject* body_##name(PyObject** v);                                                                            \
    PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t npos, PyObject* kwnames)                       \
    {                                                                                                               \
        PyObject* v[kMaxArgs];                                                                                      \
        if (!bind_arguments(sig_##name, args, npos, kwnames, v)) return nullptr;                                    \
        try {                                                                                                       \
            return body_##name(v);                                                                                  \
        } catch (const PythonError&) {                                                                              \
        } catch (const std::exception& e) {                                                                         \
            PyErr_SetString(PyExc_RuntimeError, e.what());                                                          \
        }                                                                                                           \
        return nullptr;                                                                                             \
    }                                                                                                               \
    PyObject* body_##name(PyObject** v)

MQG_ENTRY(mqg_quantize, 3, 10, "grad", "n", "bits", "bucket", "seed", "codes", "scales", "worker", "step", "elem_offset")
{
    const uint64_t n = to_u64(v[1]), bucket = to_u64(v[3]), seed = to_u64(v[4]), off = to_u64(v[9]);
    const int bits = to_int(v[2]);
    const uint32_t worker = to_u32(v[7]), step = to_u32(v[8]);
    const mqg_dtype dt = grad_dtype(v[0]);
    const void* grad = n ? device_ptr(v[0], "grad") : nullptr;
    uint32_t* codes = n ? static_cast<uint32_t*>(device_ptr(v[5], "codes")) : nullptr;
    float* scales = n ? static_cast<float*>(device_ptr(v[6], "scales")) : nullptr;
    void* s = stream();
    return enqueue([=] { return mqg_quantize(grad, n, bits, bucket, seed, codes, scales, dt, worker, step, off, s); });
}

MQG_ENTRY(mqg_quantize_l2, 3, 10, "grad", "n", "bits", "bucket", "seed", "codes", "scales", "worker", "step", "elem_offset")
{
    const uint64_t n = to_u64(v[1]), bucket = to_u64(v[3]), seed = to_u64(v[4]), off = to_u64(v[9]);
    const int bits = to_int(v[2]);
    const uint32_t worker = to_u32(v[7]), step = to_u32(v[8]);
    const void* grad = device_ptr(v[0], "grad");
    const mqg_dtype dt = grad_dtype(v[0]);
    uint32_t* codes = static_cast<uint32_t*>(device_ptr(v[5], "codes"));
    float* scales = static_cast<float*>(device_ptr(v[6], "scales"));
    void* s = stream();
    return enqueue([=] { return mqg_quantize_l2(grad, n, bits, bucket, seed, codes, scales, dt, worker, step, off, s); });
}

template <typename Fn> PyObject* quantize_workers(PyObject** v, Fn fn)
{
    const int W = to_int(v[1]), bits = to_int(v[3]);
    const uint64_t n = to_u64(v[2]), bucket = to_u64(v[4]), seed = to_u64(v[5]), off = to_u64(v[10]);
    const uint32_t first = to_u32(v[8]), step = to_u32(v[9]);
    GradientTable g;
    PointerTable c, sc;
    g.read(v[0], W, true, true);
    c.read(v[6], "codes", W, true);
    sc.read(v[7], "scales", W, true);
    void* s = stream();
    return enqueue([&] { return fn(g.as<const void>(), W, n, bits, bucket, seed, c.as<uint32_t>(), sc.as<float>(), g.dtype,
                                   first, step, off, s); });
}

MQG_ENTRY(mqg_quantize_workers, 3, 11, "grads", "W", "n", "bits", "bucket", "seed", "codes", "scales", "first_worker",
          "step", "elem_offset")
{
    return quantize_workers(v, ::mqg_quantize_workers);
}

MQG_ENTRY(mqg_quantize_workers_l2, 3, 11, "grads", "W", "n", "bits", "bucket", "seed", "codes", "scales", "first_worker",
          "step", "elem_offset")
{
    return quantize_workers(v, ::mqg_quantize_workers_l2);
}

MQG_ENTRY(mqg_quantize_workers_minmax, 0, 7, "grads", "W", "n", "bits", "bucket", "codes", "ranges")
{
    const int W = to_int(v[1]), bits = to_int(v[3]);
    const uint64_t n = to_u64(v[2]), bucket = to_u64(v[4]);
    GradientTable g;
    PointerTable c, r;
    g.read(v[0], W, true, true);
    c.read(v[5], "codes", W, true);
    r.read(v[6], "ranges", W, true);
    void* s = stream();
    return enqueue([&] { return ::mqg_quantize_workers_minmax(g.as<const void>(), W, n, bits, bucket, c.as<uint32_t>(),
                                                              r.as<float>(), g.dtype, s); });
}

MQG_ENTRY(mqg_quantize_minmax, 0, 6, "grad", "n", "bits", "bucket", "codes", "ranges")
{
    const uint64_t n = to_u64(v[1]), bucket = to_u64(v[3]);
    const int bits = to_int(v[2]);
    const mqg_dtype dt = grad_dtype(v[0]);
    const void* grad = n ? device_ptr(v[0], "grad") : nullptr;
    uint32_t* codes = n ? static_cast<uint32_t*>(device_ptr(v[4], "codes")) : nullptr;
    float* ranges = n ? static_cast<float*>(device_ptr(v[5], "ranges")) : nullptr;
    void* s = stream();
    return enqueue([=] { return mqg_quantize_minmax(grad, n, bits, bucket, codes, ranges, dt, s); });
}

MQG_ENTRY(mqg_quantize_1bit_ef, 0, 6, "grad", "residual", "n", "bucket", "codes", "ranges")
{
    const uint64_t n = to_u64(v[2]), bucket = to_u64(v[3]);
    const void* grad = device_ptr(v[0], "grad");
    float* residual = static_cast<float*>(device_ptr(v[1], "residual"));
    uint32_t* codes = static_cast<uint32_t*>(device_ptr(v[4], "codes"));
    float* ranges = static_cast<float*>(device_ptr(v[5], "ranges"));
    const mqg_dtype dt = grad_dtype(v[0]);
    void* s = stream();
    return enqueue([=] { return mqg_quantize_1bit_ef(grad, residual, n, bucket, codes, ranges, dt, s); });
}

template <typename Fn> PyObject* dequant_accumulate(PyObject** v, const char* second, Fn fn)
{
    const int W = to_int(v[2]), bits = to_int(v[3]);
    const uint64_t n = to_u64(v[4]), bucket = to_u64(v[6]);
    const int add = to_bool(v[7]) ? 1 : 0;
    PointerTable c, sc;
    c.read(v[0], "codes", W, false);
    sc.read(v[1], second, W, false);
    float* acc = n ? static_cast<float*>(device_ptr(v[5], "acc")) : nullptr;
    void* s = stream();
    return enqueue([&] { return fn(c.as<const uint32_t>(), sc.as<const float>(), W, bits, n, acc, bucket, add, s); });
}

MQG_ENTRY(mqg_dequant_accumulate, 1, 8, "codes", "scales", "W", "bits", "n", "acc", "bucket", "add_into_acc")
{
    return dequant_accumulate(v, "scales", ::mqg_dequant_accumulate);
}

MQG_ENTRY(mqg_dequant_accumulate_minmax, 1, 8, "codes", "ranges", "W", "bits", "n", "acc", "bucket", "add_into_acc")
{
    return dequant_accumulate(v, "ranges", ::mqg_dequant_accumulate_minmax);
}

float* optional_ptr(PyObject* o, const char* what)
{
    return o && o != Py_None ? static_cast<float*>(device_ptr(o, what)) : nullptr;
}

template <typename Fn> PyObject* server_step(PyObject** v, const char* second, Fn fn)
{
    const int W = to_int(v[2]), bits = to_int(v[3]);
    const uint64_t n = to_u64(v[4]), bucket = to_u64(v[5]);
    const float lr = to_float(v[7]);
    PointerTable c, sc;
    c.read(v[0], "codes", W, false);
    sc.read(v[1], second, W, false);
    float* params = n ? static_cast<float*>(device_ptr(v[6], "params")) : nullptr;
    float* acc = optional_ptr(v[8], "acc_out");
    void* s = stream();
    return enqueue([&] { return fn(c.as<const uint32_t>(), sc.as<const float>(), W, bits, n, bucket, params, lr, acc, s); });
}

MQG_ENTRY(mqg_server_step, 1, 9, "codes", "scales", "W", "bits", "n", "bucket", "params", "lr", "acc_out")
{
    return server_step(v, "scales", ::mqg_server_step);
}

MQG_ENTRY(mqg_server_step_minmax, 1, 9, "codes", "ranges", "W", "bits", "n", "bucket", "params", "lr", "acc_out")
{
    return server_step(v, "ranges", ::mqg_server_step_minmax);
}

MQG_ENTRY(mqg_apply, 0, 4, "params", "acc", "lr", "n")
{
    const uint64_t n = to_u64(v[3]);
    const float lr = to_float(v[2]);
    float* params = n ? static_cast<float*>(device_ptr(v[0], "params")) : nullptr;
    const float* acc = n ? static_cast<const float*>(device_ptr(v[1], "acc")) : nullptr;
    void* s = stream();
    return enqueue([=] { return mqg_apply(params, acc, lr, n, s); });
}

MQG_ENTRY(mqg_server_requantize, 2, 12, "codes", "scales", "W", "bits", "n", "bucket", "mean_scale", "seed", "codes_out",
          "scales_out", "worker", "step")
{
    const int W = to_int(v[2]), bits = to_int(v[3]);
    const uint64_t n = to_u64(v[4]), bucket = to_u64(v[5]), seed = to_u64(v[7]);
    const float mean_scale = to_float(v[6]);
    const uint32_t worker = to_u32(v[10]), step = to_u32(v[11]);
    PointerTable c, sc;
    c.read(v[0], "codes", W, false);
    sc.read(v[1], "scales", W, false);
    uint32_t* codes_out = n ? static_cast<uint32_t*>(device_ptr(v[8], "codes_out")) : nullptr;
    float* scales_out = n ? static_cast<float*>(device_ptr(v[9], "scales_out")) : nullptr;
    void* s = stream();
    return enqueue([&] { return ::mqg_server_requantize(c.as<const uint32_t>(), sc.as<const float>(), W, bits, n, bucket,
                                                        mean_scale, seed, codes_out, scales_out, worker, step, s); });
}

MQG_ENTRY(mqg_quantize_segments, 3, 10, "grad", "seg_off", "code_off", "bits", "seed", "codes", "scales", "worker", "step",
          "elem_offset")
{
    OffsetTable seg, code;
    const int nseg = read_segments(v[1], v[2], seg, code), bits = to_int(v[3]);
    const uint64_t seed = to_u64(v[4]), off = to_u64(v[9]);
    const uint32_t worker = to_u32(v[7]), step = to_u32(v[8]);
    const void* grad = device_ptr(v[0], "grad");
    const mqg_dtype dt = grad_dtype(v[0]);
    uint32_t* codes = static_cast<uint32_t*>(device_ptr(v[5], "codes"));
    float* scales = static_cast<float*>(device_ptr(v[6], "scales"));
    void* s = stream();
    return enqueue([&] { return ::mqg_quantize_segments(grad, nseg, seg.data, code.data, bits, seed, codes, scales, dt,
                                                        worker, step, off, s); });
}

MQG_ENTRY(mqg_quantize_segments_l2, 3, 11, "grad", "seg_off", "code_off", "bits", "seed", "codes", "scales", "workspace",
          "worker", "step", "elem_offset")
{
    OffsetTable seg, code;
    const int nseg = read_segments(v[1], v[2], seg, code), bits = to_int(v[3]);
    const uint64_t seed = to_u64(v[4]), off = to_u64(v[10]);
    const uint32_t worker = to_u32(v[8]), step = to_u32(v[9]);
    const void* grad = device_ptr(v[0], "grad");
    const mqg_dtype dt = grad_dtype(v[0]);
    uint32_t* codes = static_cast<uint32_t*>(device_ptr(v[5], "codes"));
    float* scales = static_cast<float*>(device_ptr(v[6], "scales"));
    float* workspace = static_cast<float*>(device_ptr(v[7], "workspace"));
    const size_t floats = (size_t)THPVariable_Unpack(v[7]).numel();
    void* s = stream();
    return enqueue([&] { return ::mqg_quantize_segments_l2(grad, nseg, seg.data, code.data, bits, seed, codes, scales, dt,
                                                           worker, step, off, workspace, floats, s); });
}

MQG_ENTRY(mqg_quantize_segments_l2_static, 3, 10, "grad", "seg_off", "code_off", "bits", "seed", "codes", "scales",
          "worker", "step", "elem_offset")
{
    OffsetTable seg, code;
    const int nseg = read_segments(v[1], v[2], seg, code), bits = to_int(v[3]);
    const uint64_t seed = to_u64(v[4]), off = to_u64(v[9]);
    const uint32_t worker = to_u32(v[7]), step = to_u32(v[8]);
    const void* grad = device_ptr(v[0], "grad");
    const mqg_dtype dt = grad_dtype(v[0]);
    uint32_t* codes = static_cast<uint32_t*>(device_ptr(v[5], "codes"));
    float* scales = static_cast<float*>(device_ptr(v[6], "scales"));
    void* s = stream();
    return enqueue([&] { return ::mqg_quantize_segments_l2_static(grad, nseg, seg.data, code.data, bits, seed, codes,
                                                                  scales, dt, worker, step, off, s); });
}

MQG_ENTRY(mqg_quantize_segments_workers, 3, 11, "grads", "W", "seg_off", "code_off", "bits", "seed", "codes", "scales",
          "first_worker", "step", "elem_offset")
{
    OffsetTable seg, code;
    const int W = to_int(v[1]), nseg = read_segments(v[2], v[3], seg, code), bits = to_int(v[4]);
    const uint64_t seed = to_u64(v[5]), off = to_u64(v[10]);
    const uint32_t first = to_u32(v[8]), step = to_u32(v[9]);
    GradientTable g;
    PointerTable c, sc;
    g.read(v[0], W, false, false);
    c.read(v[6], "codes", W, false);
    sc.read(v[7], "scales", W, false);
    void* s = stream();
    return enqueue([&] { return ::mqg_quantize_segments_workers(g.as<const void>(), W, nseg, seg.data, code.data, bits,
                                                                seed, c.as<uint32_t>(), sc.as<float>(), g.dtype, first, step,
                                                                off, s); });
}

MQG_ENTRY(mqg_server_step_segments, 1, 9, "codes", "scales", "W", "bits", "seg_off", "code_off", "params", "lr", "acc_out")
{
    OffsetTable seg, code;
    const int W = to_int(v[2]), bits = to_int(v[3]), nseg = read_segments(v[4], v[5], seg, code);
    const float lr = to_float(v[7]);
    PointerTable c, sc;
    c.read(v[0], "codes", W, false);
    sc.read(v[1], "scales", W, false);
    float* params = static_cast<float*>(device_ptr(v[6], "params"));
    float* acc = optional_ptr(v[8], "acc_out");
    void* s = stream();
    return enqueue([&] { return ::mqg_server_step_segments(c.as<const uint32_t>(), sc.as<const float>(), W, bits, nseg,
                                                           seg.data, code.data, params, lr, acc, s); });
}

PyObject* set_error_class(PyObject*, PyObject* cls)
{
    Py_XSETREF(g_error_class, Py_NewRef(cls));
    Py_RETURN_NONE;
}

#define MQG_METHOD(name, signature, doc)                                                                            \
    {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL | METH_KEYWORDS, #name signature "\n--\n\n" doc}

PyMethodDef kMethods[] = {
    MQG_METHOD(mqg_quantize, "(grad, n, bits, bucket, seed, codes, scales, worker=0, step=0, elem_offset=0)",
               "Quantize(g, K): writes `codes` (uint32/int32 words) and `scales` (float32)."),
    MQG_METHOD(mqg_quantize_workers,
               "(grads, W, n, bits, bucket, seed, codes, scales, first_worker=0, step=0, elem_offset=0)",
               "Quantize(g_p, K) for W workers' gradients (lists of W tensors) in one launch."),
    MQG_METHOD(mqg_quantize_workers_l2,
               "(grads, W, n, bits, bucket, seed, codes, scales, first_worker=0, step=0, elem_offset=0)",
               "The L2-norm scale variant for W workers' gradients (lists of W tensors) in one launch."),
    MQG_METHOD(mqg_dequant_accumulate, "(codes, scales, W, bits, n, acc, bucket, add_into_acc=False)",
               "De-quantize and sum W workers' buffers into `acc`."),
    MQG_METHOD(mqg_apply, "(params, acc, lr, n)", "params <- params - lr * acc."),
    MQG_METHOD(mqg_server_step, "(codes, scales, W, bits, n, bucket, params, lr, acc_out=None)",
               "De-quantize, sum and apply W workers' buffers in one pass."),
    MQG_METHOD(mqg_quantize_workers_minmax, "(grads, W, n, bits, bucket, codes, ranges)",
               "The (min, max) variant for W workers' gradients (lists of W tensors) in one launch."),
    MQG_METHOD(mqg_quantize_minmax, "(grad, n, bits, bucket, codes, ranges)",
               "(min, max) nearest-rounding variant: writes `codes` and `ranges` (lo, hi per bucket)."),
    MQG_METHOD(mqg_dequant_accumulate_minmax, "(codes, ranges, W, bits, n, acc, bucket, add_into_acc=False)",
               "mqg_dequant_accumulate for the (min, max) variant."),
    MQG_METHOD(mqg_server_step_minmax, "(codes, ranges, W, bits, n, bucket, params, lr, acc_out=None)",
               "mqg_server_step for the (min, max) variant."),
    MQG_METHOD(mqg_server_requantize,
               "(codes, scales, W, bits, n, bucket, mean_scale, seed, codes_out, scales_out, worker=0, step=0)",
               "Downlink: de-quantize + sum + scale to the mean + quantize again, in one pass."),
    MQG_METHOD(mqg_quantize_segments,
               "(grad, seg_off, code_off, bits, seed, codes, scales, worker=0, step=0, elem_offset=0)",
               "Quantize with one scale per segment of the flat gradient."),
    MQG_METHOD(mqg_quantize_segments_workers,
               "(grads, W, seg_off, code_off, bits, seed, codes, scales, first_worker=0, step=0, elem_offset=0)",
               "mqg_quantize_segments for W workers' gradients that share one segment table."),
    MQG_METHOD(mqg_server_step_segments, "(codes, scales, W, bits, seg_off, code_off, params, lr, acc_out=None)",
               "mqg_server_step for buffers written by mqg_quantize_segments."),
    MQG_METHOD(mqg_quantize_1bit_ef, "(grad, residual, n, bucket, codes, ranges)",
               "One bit with error feedback; `residual` (float32, n elements) is read and updated in place."),
    MQG_METHOD(mqg_quantize_l2, "(grad, n, bits, bucket, seed, codes, scales, worker=0, step=0, elem_offset=0)",
               "mqg_quantize with the bucket's L2 norm as its scale."),
    MQG_METHOD(mqg_quantize_segments_l2,
               "(grad, seg_off, code_off, bits, seed, codes, scales, workspace, worker=0, step=0, elem_offset=0)",
               "`workspace`: float32 CUDA tensor of at least mqg_l2_workspace_floats(seg_off) elements."),
    MQG_METHOD(mqg_quantize_segments_l2_static,
               "(grad, seg_off, code_off, bits, seed, codes, scales, worker=0, step=0, elem_offset=0)",
               "mqg_quantize_segments_l2 for callers that cannot supply a workspace: the partial sums use an array\n"
               "inside the library (at most MQG_L2_STATIC_WORKSPACE_FLOATS of them); calls that may overlap on the\n"
               "device must be ordered by the caller."),
    {"_set_error_class", set_error_class, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};

Signature* const kSignatures[] = {
    &sig_mqg_quantize, &sig_mqg_quantize_workers, &sig_mqg_quantize_workers_l2, &sig_mqg_dequant_accumulate,
    &sig_mqg_apply, &sig_mqg_server_step, &sig_mqg_quantize_workers_minmax, &sig_mqg_quantize_minmax,
    &sig_mqg_dequant_accumulate_minmax, &sig_mqg_server_step_minmax, &sig_mqg_server_requantize,
    &sig_mqg_quantize_segments, &sig_mqg_quantize_segments_workers, &sig_mqg_server_step_segments,
    &sig_mqg_quantize_1bit_ef, &sig_mqg_quantize_l2, &sig_mqg_quantize_segments_l2,
    &sig_mqg_quantize_segments_l2_static,
};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_binding", "Native entry points of libmqgrad.", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void)
{
    for (Signature* s : kSignatures)
        for (int i = 0; i < s->nargs; ++i) {
            s->interned[i] = PyUnicode_InternFromString(s->names[i]);
            if (!s->interned[i]) return nullptr;
        }
    return PyModule_Create(&kModule);
}
