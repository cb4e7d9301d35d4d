// Python entry of the calls that a program makes once per matrix, token or step: tensors to device pointers, the
// current stream, then the C function, without the interpreter in between.  Building the argument objects in
// Python and going through ctypes took 7 to 11 us a call, more than the kernels of a small matrix.
// Every function returns the library's status code; tensors may be None where the C argument may be NULL.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "qamw.h"

namespace {

struct Failed {};  // a Python error has been set

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a torch tensor, got %s", Py_TYPE(o)->tp_name);
        throw Failed{};
    }
    return THPVariable_Unpack(o);
}
// Memory that the call reads; memory that it writes.  Asking for the second makes a tensor that shares its memory until it
// is written (a lazy clone) take its own.
const void* tensor_ptr(PyObject* o) { return o == Py_None ? nullptr : tensor(o).const_data_ptr(); }
void* written_ptr(PyObject* o) { return o == Py_None ? nullptr : tensor(o).mutable_data_ptr(); }
size_t tensor_bytes(PyObject* o) { return tensor(o).numel() * tensor(o).element_size(); }

// The memory of an object with the buffer interface (a ctypes structure or pointer, a numpy array).
struct Bytes {
    Py_buffer view{};
    explicit Bytes(PyObject* o) {
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Failed{};
    }
    ~Bytes() { PyBuffer_Release(&view); }
    Bytes(const Bytes&) = delete;
    Bytes& operator=(const Bytes&) = delete;
};
// qamw_params of a ctypes structure; the caller's object outlives the call
struct Params {
    Bytes b;
    explicit Params(PyObject* o) : b(o) {
        if (b.view.len != Py_ssize_t(sizeof(qamw_params))) {
            PyErr_SetString(PyExc_TypeError, "expected binding.Params");
            throw Failed{};
        }
    }
    const qamw_params* get() const { return static_cast<const qamw_params*>(b.view.buf); }
};
// a library object's address from its ctypes.c_void_p (None: NULL)
template <class T>
T* handle(PyObject* o) {
    if (o == Py_None) return nullptr;
    Bytes b(o);
    if (b.view.len != Py_ssize_t(sizeof(void*))) {
        PyErr_SetString(PyExc_TypeError, "expected a library handle");
        throw Failed{};
    }
    return *static_cast<T**>(b.view.buf);
}
void* stream_ptr(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) throw Failed{};
    void* p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) throw Failed{};
    return p;
}

// Runs `body` (arguments to C values, then the library call through `call`, which gives up the interpreter
// lock) and turns its status code into a Python integer.
template <class F>
PyObject* guarded(Py_ssize_t got, Py_ssize_t want, F body) {
    if (got != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
        return nullptr;
    }
    try {
        return PyLong_FromLong(body());
    } catch (const Failed&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <class F>
int call(F f) {
    struct Unlocked {  // also when the call throws (out of host memory): guarded() needs the lock to report it
        PyThreadState* save = PyEval_SaveThread();
        ~Unlocked() { PyEval_RestoreThread(save); }
    } unlocked;
    return f();
}
template <class T>
const T* in(PyObject* o) { return static_cast<const T*>(tensor_ptr(o)); }
template <class T>
T* out(PyObject* o) { return static_cast<T*>(written_ptr(o)); }

PyObject* py_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 9, [&] {
        const auto* packed = in<uint8_t>(a[0]);
        const auto *norm = in<float>(a[1]), *scale = in<float>(a[2]), *sigma = in<float>(a[4]);
        const auto* signs = in<int8_t>(a[3]);
        const auto* cb = handle<qamw_codebook>(a[5]);
        const Params p(a[6]);
        void *w_hat = written_ptr(a[7]), *st = stream_ptr(a[8]);
        return call([&] { return qamw_decode(packed, norm, scale, signs, sigma, cb, p.get(), w_hat, st); });
    });
}

PyObject* py_decode_gemv(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 11, [&] {
        const auto* packed = in<uint8_t>(a[0]);
        const auto *norm = in<float>(a[1]), *scale = in<float>(a[2]), *sigma = in<float>(a[4]), *x = in<float>(a[7]);
        const auto* signs = in<int8_t>(a[3]);
        const auto* cb = handle<qamw_codebook>(a[5]);
        const Params p(a[6]);
        auto* y = out<float>(a[8]);
        const int n_vec = int(tensor(a[7]).size(0));
        const size_t ws_bytes = tensor(a[9]).numel();
        void *ws = written_ptr(a[9]), *st = stream_ptr(a[10]);
        return call([&] { return qamw_decode_gemv(packed, norm, scale, signs, sigma, cb, p.get(), x, n_vec, y, ws, ws_bytes, st); });
    });
}

PyObject* py_encode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&] {
        const void* W = tensor_ptr(a[0]);
        const Params p(a[1]);
        const auto *scale = in<float>(a[2]), *sigma = in<float>(a[4]);
        const auto* signs = in<int8_t>(a[3]);
        const auto* cb = handle<qamw_codebook>(a[5]);
        auto* packed = out<uint8_t>(a[6]);
        auto* norm = out<float>(a[7]);
        auto* status = out<int32_t>(a[8]);
        void* st = stream_ptr(a[9]);
        return call([&] { return qamw_encode(W, p.get(), scale, signs, sigma, cb, packed, norm, status, st); });
    });
}

PyObject* py_calibrate(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 8, [&] {
        const void* W = tensor_ptr(a[0]);
        const Params p(a[1]);
        const auto* scale = in<float>(a[2]);
        const auto* signs = in<int8_t>(a[3]);
        auto* sigma = out<float>(a[4]);
        void* ws = written_ptr(a[5]);
        const size_t ws_bytes = ws ? tensor_bytes(a[5]) : 0;
        auto* status = out<int32_t>(a[6]);
        void* st = stream_ptr(a[7]);
        return call([&] { return qamw_calibrate(W, p.get(), scale, signs, sigma, ws, ws_bytes, status, st); });
    });
}

PyObject* py_quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 14, [&] {
        const void* W = tensor_ptr(a[0]);
        const Params p(a[1]);
        const Bytes act(a[2] == Py_None ? a[1] : a[2]);  // float32, checked by the caller
        const auto* act_rms = a[2] == Py_None ? nullptr : static_cast<const float*>(act.view.buf);
        if (act_rms && act.view.len < Py_ssize_t(sizeof(float)) * p.get()->d_in) {
            PyErr_Format(PyExc_ValueError, "%zd activation statistics for %d columns", act.view.len / Py_ssize_t(sizeof(float)), int(p.get()->d_in));
            throw Failed{};
        }
        const float alpha = float(PyFloat_AsDouble(a[3]));
        const uint64_t seed = PyLong_AsUnsignedLongLongMask(a[4]);
        if (PyErr_Occurred()) throw Failed{};
        const auto* cb = handle<qamw_codebook>(a[5]);
        auto* scale = out<float>(a[6]);
        auto* signs = out<int8_t>(a[7]);
        auto *sigma = out<float>(a[8]), *norm = out<float>(a[10]);
        auto* packed = out<uint8_t>(a[9]);
        void* ws = written_ptr(a[11]);
        const size_t ws_bytes = ws ? tensor_bytes(a[11]) : 0;
        auto* status = out<int32_t>(a[12]);
        void* st = stream_ptr(a[13]);
        return call([&] {
            return qamw_quantize(W, p.get(), act_rms, alpha, seed, cb, scale, signs, sigma, packed, norm, ws, ws_bytes, status, st);
        });
    });
}

PyObject* py_calibrate_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 4, [&] {
        const auto* b = handle<qamw_batch>(a[0]);
        void* ws = written_ptr(a[1]);
        const size_t ws_bytes = ws ? tensor_bytes(a[1]) : 0;
        auto* status = out<int32_t>(a[2]);
        void* st = stream_ptr(a[3]);
        return call([&] { return qamw_calibrate_batch(b, ws, ws_bytes, status, st); });
    });
}
PyObject* py_encode_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 3, [&] {
        const auto* b = handle<qamw_batch>(a[0]);
        auto* status = out<int32_t>(a[1]);
        void* st = stream_ptr(a[2]);
        return call([&] { return qamw_encode_batch(b, status, st); });
    });
}
PyObject* py_decode_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 2, [&] {
        const auto* b = handle<qamw_batch>(a[0]);
        void* st = stream_ptr(a[1]);
        return call([&] { return qamw_decode_batch(b, st); });
    });
}
PyObject* py_distortion_batch(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 2, [&] {
        const auto* b = handle<qamw_batch>(a[0]);
        void* st = stream_ptr(a[1]);
        return call([&] { return qamw_distortion_batch(b, st); });
    });
}

PyCFunction fast(_PyCFunctionFast f) { return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)); }

PyMethodDef methods[] = {
    {"decode", fast(py_decode), METH_FASTCALL, nullptr},
    {"decode_gemv", fast(py_decode_gemv), METH_FASTCALL, nullptr},
    {"encode", fast(py_encode), METH_FASTCALL, nullptr},
    {"calibrate", fast(py_calibrate), METH_FASTCALL, nullptr},
    {"quantize", fast(py_quantize), METH_FASTCALL, nullptr},
    {"calibrate_batch", fast(py_calibrate_batch), METH_FASTCALL, nullptr},
    {"encode_batch", fast(py_encode_batch), METH_FASTCALL, nullptr},
    {"decode_batch", fast(py_decode_batch), METH_FASTCALL, nullptr},
    {"distortion_batch", fast(py_distortion_batch), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_qamw", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__qamw(void) { return PyModule_Create(&module); }
