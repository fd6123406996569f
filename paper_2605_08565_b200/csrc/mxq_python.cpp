// The calls of binding.py that sit in a caller's inner loop, with their arguments unpacked in C++ instead of ctypes: a ctypes call of
// fifteen arguments and the tensors' attributes cost 2.5 to 3.5 us, which is what the kernels of a small tensor take on the GPU.  Every function takes what its Python counterpart takes and
// returns the library's status, or -1 for arguments it does not know (anything but None or a contiguous CUDA tensor of
// type Tensor or Parameter for a pointer, an int, a float): the caller then goes through ctypes, which converts or refuses them.  us a call on
// the host's side of a pass, ctypes -> here: abs-max and quantization of 4 x 4096 activations 10.1 -> 5.2, quantize + MSE of 37 K
// elements 8.6 -> 5.1, the seven calls that score a recipe on 130 K elements 32 -> 24.
// The library is not linked: bind() receives the addresses of its functions.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/mxq.h"

namespace {

// The library's functions, by name as bind() finds them.
struct Library {
    decltype(&mxq_quantize_ex) quantize_ex;
    decltype(&mxq_quantize_mse) quantize_mse;
    decltype(&mxq_quantize_batch) quantize_batch;
    decltype(&mxq_fake_quantize) fake_quantize;
    decltype(&mxq_tensor_amax) tensor_amax;
    decltype(&mxq_tensor_mse) tensor_mse;
    decltype(&mxq_dequantize_ex) dequantize_ex;
    decltype(&mxq_block_clip_sse) block_clip_sse;
    decltype(&mxq_histograms) histograms;
    decltype(&mxq_segment_mse) segment_mse;
    decltype(&mxq_set_option) set_option;
} lib;
bool bound = false;

// Arguments of one call, read in order; `ok` falls with the first one that is not of the expected kind.
struct Args {
    PyObject* const* a;
    bool ok;
    Args(PyObject* const* args, Py_ssize_t n, Py_ssize_t expected) : a(args), ok(n == expected) {}

    const at::Tensor* tensor(int i) {
        if (!ok || !THPVariable_CheckExact(a[i])) {
            ok = false;
            return nullptr;
        }
        const at::Tensor& t = THPVariable_Unpack(a[i]);
        if (!t.is_cuda() || !t.is_contiguous()) ok = false;
        return &t;
    }
    void* ptr(int i) {
        if (!ok || a[i] == Py_None) return nullptr;
        const at::Tensor* t = tensor(i);
        return ok ? t->data_ptr() : nullptr;
    }
    int dtype(int i) {   // after ptr(i)
        if (!ok || a[i] == Py_None) {
            ok = false;
            return 0;
        }
        const auto d = THPVariable_Unpack(a[i]).scalar_type();
        if (d != at::kFloat && d != at::kBFloat16) ok = false;
        return d == at::kFloat ? MXQ_F32 : MXQ_BF16;
    }
    size_t bytes(int i) {
        if (!ok || a[i] == Py_None) return 0;
        return THPVariable_Unpack(a[i]).nbytes();
    }
    size_t size(int i) {
        if (!ok || !PyLong_Check(a[i])) {
            ok = false;
            return 0;
        }
        const size_t v = PyLong_AsSize_t(a[i]);
        if (v == (size_t)-1 && PyErr_Occurred()) {
            PyErr_Clear();
            ok = false;
        }
        return v;
    }
    int integer(int i) {
        if (!ok || !PyLong_Check(a[i])) {
            ok = false;
            return 0;
        }
        const long v = PyLong_AsLong(a[i]);
        if ((v == -1 && PyErr_Occurred()) || v != (int)v) {
            PyErr_Clear();
            ok = false;
        }
        return (int)v;
    }
    float number(int i) {
        if (!ok || !PyFloat_Check(a[i])) {   // an int among others
            ok = false;
            return 0.0f;
        }
        return (float)PyFloat_AS_DOUBLE(a[i]);
    }
    // None: the current stream of the device that the tensor a[like] lies on; else an object with a cuda_stream
    void* stream(int i, int like) {
        if (!ok) return nullptr;
        if (a[i] == Py_None) {
            const at::Tensor* t = tensor(like);
            return ok ? (void*)c10::cuda::getCurrentCUDAStream(t->get_device()).stream() : nullptr;
        }
        PyObject* s = PyObject_GetAttrString(a[i], "cuda_stream");
        void* p = s != nullptr && PyLong_Check(s) ? PyLong_AsVoidPtr(s) : nullptr;
        if (s == nullptr || !PyLong_Check(s) || (p == nullptr && PyErr_Occurred())) {
            PyErr_Clear();
            ok = false;
        }
        Py_XDECREF(s);
        return p;
    }
};

// Calls f() without the interpreter's lock, as ctypes does.
template <typename F>
PyObject* status_of(const Args& a, F f) {
    if (!a.ok) return PyLong_FromLong(-1);
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

// A tensor without storage and the like throws where its address is asked for: left to the caller's other path.
template <PyObject* (*BODY)(PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (!bound) return PyLong_FromLong(-1);
    try {
        return BODY(args, n);
    } catch (...) {
        PyErr_Clear();
        return PyLong_FromLong(-1);
    }
}

// The arguments are read into locals first: the lambda runs without the lock and touches no Python object.
PyObject* quantize_ex(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 11);
    const void* x = a.ptr(0);
    const int dt = a.dtype(0);
    const size_t n = a.size(1);
    const int B = a.integer(2), fmt = a.integer(3), recipe = a.integer(4);
    const float g = a.number(5);
    const float* dg = (const float*)a.ptr(6);
    uint8_t *codes = (uint8_t*)a.ptr(7), *scales = (uint8_t*)a.ptr(8);
    float* sse = (float*)a.ptr(9);
    void* s = a.stream(10, 0);
    return status_of(a, [&] { return lib.quantize_ex(x, dt, n, B, fmt, recipe, g, dg, codes, scales, sse, s); });
}

PyObject* quantize_mse(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 13);
    const void* x = a.ptr(0);
    const int dt = a.dtype(0);
    const size_t n = a.size(1);
    const int B = a.integer(2), fmt = a.integer(3), recipe = a.integer(4);
    const float g = a.number(5);
    const float* dg = (const float*)a.ptr(6);
    uint8_t *codes = (uint8_t*)a.ptr(7), *scales = (uint8_t*)a.ptr(8);
    float* sse = (float*)a.ptr(9);
    double* mse = (double*)a.ptr(10);
    void* ws = a.ptr(11);
    const size_t ws_bytes = a.bytes(11);
    void* s = a.stream(12, 0);
    return status_of(a, [&] { return lib.quantize_mse(x, dt, n, B, fmt, recipe, g, dg, codes, scales, sse, mse, ws, ws_bytes, s); });
}

PyObject* quantize_batch(PyObject* const* p, Py_ssize_t np) {   // h_descs: its address
    Args a(p, np, 10);
    const size_t h = a.size(0);
    const mxq_tensor_desc* d = (const mxq_tensor_desc*)a.ptr(1);
    const size_t nt = a.size(2);
    const int dt = a.integer(3), B = a.integer(4), fmt = a.integer(5), recipe = a.integer(6);
    const float g = a.number(7);
    const float* dg = (const float*)a.ptr(8);
    void* s = a.stream(9, 1);
    return status_of(a, [&] { return lib.quantize_batch((const mxq_tensor_desc*)h, d, nt, dt, B, fmt, recipe, g, dg, s); });
}

PyObject* fake_quantize(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 9);
    const void* x = a.ptr(0);
    const int dt = a.dtype(0);
    const size_t n = a.size(1);
    const int B = a.integer(2), fmt = a.integer(3), recipe = a.integer(4);
    const float g = a.number(5);
    const float* dg = (const float*)a.ptr(6);
    void* out = a.ptr(7);
    const int odt = a.dtype(7);
    void* s = a.stream(8, 0);
    return status_of(a, [&] { return lib.fake_quantize(x, dt, n, B, fmt, recipe, g, dg, out, odt, s); });
}

PyObject* tensor_amax(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 5);
    const void* x = a.ptr(0);
    const int dt = a.dtype(0);
    const size_t n = a.size(1);
    float *amax = (float*)a.ptr(2), *g = (float*)a.ptr(3);
    void* s = a.stream(4, 0);
    return status_of(a, [&] { return lib.tensor_amax(x, dt, n, amax, g, s); });
}

PyObject* tensor_mse(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 6);
    const float* sse = (const float*)a.ptr(0);
    const size_t nb = a.size(1), n = a.size(2);
    double* out = (double*)a.ptr(3);
    void* ws = a.ptr(4);
    const size_t ws_bytes = a.bytes(4);
    void* s = a.stream(5, 0);
    return status_of(a, [&] { return lib.tensor_mse(sse, nb, n, out, ws, ws_bytes, s); });
}

PyObject* dequantize_ex(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 9);
    const uint8_t *codes = (const uint8_t*)a.ptr(0), *scales = (const uint8_t*)a.ptr(1);
    const size_t n = a.size(2);
    const int B = a.integer(3), fmt = a.integer(4);
    const float g = a.number(5);
    const float* dg = (const float*)a.ptr(6);
    void* out = a.ptr(7);
    const int odt = a.dtype(7);
    void* s = a.stream(8, 7);
    return status_of(a, [&] { return lib.dequantize_ex(codes, scales, n, B, fmt, g, dg, out, odt, s); });
}

PyObject* block_clip_sse(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 9);
    const void* x = a.ptr(0);
    const int dt = a.dtype(0);
    const size_t n = a.size(1);
    const int B = a.integer(2), fmt = a.integer(3);
    const float g = a.number(4);
    const float* dg = (const float*)a.ptr(5);
    const uint8_t* scales = (const uint8_t*)a.ptr(6);
    float* out = (float*)a.ptr(7);
    void* s = a.stream(8, 0);
    return status_of(a, [&] { return lib.block_clip_sse(x, dt, n, B, fmt, g, dg, scales, out, s); });
}

PyObject* histograms(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 7);
    const uint8_t *codes = (const uint8_t*)a.ptr(0), *scales = (const uint8_t*)a.ptr(1);
    const size_t n = a.size(2);
    const int B = a.integer(3);
    auto *ch = (unsigned long long*)a.ptr(4), *sh = (unsigned long long*)a.ptr(5);
    void* s = a.stream(6, 0);
    return status_of(a, [&] { return lib.histograms(codes, scales, n, B, ch, sh, s); });
}

PyObject* segment_mse(PyObject* const* p, Py_ssize_t np) {
    Args a(p, np, 6);
    const float* sse = (const float*)a.ptr(0);
    const size_t nb = a.size(1), per = a.size(2), elems = a.size(3);
    double* out = (double*)a.ptr(4);
    void* s = a.stream(5, 0);
    return status_of(a, [&] { return lib.segment_mse(sse, nb, per, elems, out, s); });
}

PyObject* set_option(PyObject* const* p, Py_ssize_t np) {   // two ints, taken modulo 2^32 as ctypes takes them
    if (np != 2 || !PyLong_Check(p[0]) || !PyLong_Check(p[1])) return PyLong_FromLong(MXQ_ERR_BAD_ENUM);
    return PyLong_FromLong(lib.set_option((int)PyLong_AsUnsignedLongMask(p[0]), (int)PyLong_AsUnsignedLongMask(p[1])));
}

// bind({"mxq_quantize_ex": address, ...})
PyObject* bind(PyObject*, PyObject* addresses) {
    if (!PyDict_Check(addresses)) {
        PyErr_SetString(PyExc_TypeError, "a dict of addresses is expected");
        return nullptr;
    }
    Library l;
    bool ok = true;
    auto get = [&](const char* name) -> void* {
        PyObject* v = PyDict_GetItemString(addresses, name);
        void* p = v != nullptr && PyLong_Check(v) ? PyLong_AsVoidPtr(v) : nullptr;
        if (p == nullptr) ok = false;
        return p;
    };
    l.quantize_ex = (decltype(l.quantize_ex))get("mxq_quantize_ex");
    l.quantize_mse = (decltype(l.quantize_mse))get("mxq_quantize_mse");
    l.quantize_batch = (decltype(l.quantize_batch))get("mxq_quantize_batch");
    l.fake_quantize = (decltype(l.fake_quantize))get("mxq_fake_quantize");
    l.tensor_amax = (decltype(l.tensor_amax))get("mxq_tensor_amax");
    l.tensor_mse = (decltype(l.tensor_mse))get("mxq_tensor_mse");
    l.dequantize_ex = (decltype(l.dequantize_ex))get("mxq_dequantize_ex");
    l.block_clip_sse = (decltype(l.block_clip_sse))get("mxq_block_clip_sse");
    l.histograms = (decltype(l.histograms))get("mxq_histograms");
    l.segment_mse = (decltype(l.segment_mse))get("mxq_segment_mse");
    l.set_option = (decltype(l.set_option))get("mxq_set_option");
    if (!ok) {
        PyErr_Clear();
        PyErr_SetString(PyExc_ValueError, "an address is missing");
        return nullptr;
    }
    lib = l;
    bound = true;
    Py_RETURN_NONE;
}

#define MXQ_METHOD(f) {#f, (PyCFunction)(void (*)(void))guarded<f>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    MXQ_METHOD(quantize_ex), MXQ_METHOD(quantize_mse), MXQ_METHOD(quantize_batch), MXQ_METHOD(fake_quantize), MXQ_METHOD(tensor_amax),
    MXQ_METHOD(tensor_mse), MXQ_METHOD(dequantize_ex), MXQ_METHOD(block_clip_sse), MXQ_METHOD(histograms), MXQ_METHOD(segment_mse),
    MXQ_METHOD(set_option),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "libmxq's inner-loop calls without ctypes", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
