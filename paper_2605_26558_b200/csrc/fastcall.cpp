// CPython entry points of the calls a serving loop makes: argument marshalling only, as in the ctypes binding beside it.
// ctypes and the Python expressions around it (one object per pointer, three attribute look-ups per tensor, shapes) took 1.5 to
// 2.5 us of host time a call beside a launch of about 4 us: 6.0 -> 4.5 us for a draft GEMV, 16.3 -> 9.1 for a sampled step.
// Every wrapper is generated from its C prototype: a tensor or None or an int (address) for a pointer, the ctypes structure for a
// description, None for the current stream.  The interpreter lock is released around the call, as ctypes does.  What torch throws
// on the way (a tensor without storage, as under vmap; a CUDA that does not come up) becomes a Python exception.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "../../include/cass.h"

namespace {

PyTypeObject* g_c_void_p = nullptr;        // ctypes.c_void_p, the type of session handles
PyObject* g_torch_cuda = nullptr;

bool buffer_address(PyObject* o, Py_ssize_t need, void** out) {
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
    const bool fits = b.len >= need;
    *out = b.buf;
    PyBuffer_Release(&b);                  // the caller's reference keeps a ctypes object's memory where it is
    if (!fits) PyErr_SetString(PyExc_TypeError, "structure of another type");
    return fits;
}

bool device_address(PyObject* o, void** out) {
    if (o == Py_None) { *out = nullptr; return true; }
    if (THPVariable_Check(o)) {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, "device buffers must be contiguous CUDA tensors");
            return false;
        }
        *out = t.data_ptr();
        return true;
    }
    if (PyLong_Check(o)) {
        *out = reinterpret_cast<void*>(PyLong_AsUnsignedLongLongMask(o));
        return !PyErr_Occurred();
    }
    if (Py_TYPE(o) == g_c_void_p) {
        void* at = nullptr;
        if (!buffer_address(o, sizeof(void*), &at)) return false;
        *out = *static_cast<void**>(at);
        return true;
    }
    PyErr_SetString(PyExc_TypeError, "expected a CUDA tensor, an address or None");
    return false;
}

bool stream_handle(PyObject* o, void** out) {
    static bool initialised = false;       // under the interpreter lock
    if (o == Py_None && initialised) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* s = o == Py_None ? PyObject_CallMethod(g_torch_cuda, "current_stream", nullptr) : Py_NewRef(o);   // the first call brings CUDA up
    if (!s) return false;
    PyObject* h = PyObject_GetAttrString(s, "cuda_stream");
    Py_DECREF(s);
    if (!h) return false;
    *out = reinterpret_cast<void*>(PyLong_AsUnsignedLongLongMask(h));
    Py_DECREF(h);
    if (PyErr_Occurred()) return false;
    if (o == Py_None) initialised = true;
    return true;
}

template <class T>
bool convert(PyObject* o, T* out) {
    if constexpr (std::is_pointer_v<T>) {
        using P = std::remove_cv_t<std::remove_pointer_t<T>>;
        void* p = nullptr;
        bool ok;
        if constexpr (std::is_class_v<P>) ok = buffer_address(o, sizeof(P), &p);
        else ok = device_address(o, &p);
        *out = static_cast<T>(p);
        return ok;
    } else if constexpr (std::is_floating_point_v<T>) {
        *out = static_cast<T>(PyFloat_AsDouble(o));
        return !PyErr_Occurred();
    } else {
        *out = static_cast<T>(PyLong_AsLongLong(o));
        return !PyErr_Occurred();
    }
}

template <bool STREAM, class T>
bool argument(PyObject* o, T* out) {
    if constexpr (STREAM) return stream_handle(o, out);
    else return convert(o, out);
}

template <auto F>
struct Entry;
template <class... A, int (*F)(A...)>
struct Entry<F> {
    static constexpr size_t N = sizeof...(A);      // the last parameter of every entry point here is the stream
    template <size_t... I>
    static PyObject* run(PyObject* const* args, std::index_sequence<I...>) {
        std::tuple<A...> v;
        if (!(argument<I + 1 == N>(args[I], &std::get<I>(v)) && ...)) return nullptr;
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = F(std::get<I>(v)...);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    }
    static PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
        HANDLE_TH_ERRORS
        if (n != (Py_ssize_t)N) return PyErr_Format(PyExc_TypeError, "%zd arguments where %zu are wanted", n, N);
        return run(args, std::make_index_sequence<N>{});
        END_HANDLE_TH_ERRORS
    }
};

// (w, x, rows, scratch, y_bf16, y_f32, status, stream): sizes come from the tensors
PyObject* verify_gemm(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 8) return PyErr_Format(PyExc_TypeError, "%zd arguments where 8 are wanted", n);
    for (int i : {0, 1, 3})
        if (!THPVariable_Check(a[i])) return PyErr_Format(PyExc_TypeError, "expected a CUDA tensor");
    const long rows = PyLong_AsLong(a[2]);
    if (PyErr_Occurred()) return nullptr;
    const at::Tensor &w = THPVariable_Unpack(a[0]), &x = THPVariable_Unpack(a[1]), &sc = THPVariable_Unpack(a[3]);
    if (w.dim() != 2 || x.dim() != 2 || x.size(0) != (rows <= 16 ? 16 : rows <= 32 ? 32 : 64) || x.size(1) != w.size(1)) {
        PyErr_SetString(PyExc_AssertionError, "x must have 16, 32 or 64 rows of as many values as w's");
        return nullptr;
    }
    void *wp, *xp, *sp, *y16, *y32, *st, *stream;
    if (!device_address(a[0], &wp) || !device_address(a[1], &xp) || !device_address(a[3], &sp) || !device_address(a[4], &y16) ||
        !device_address(a[5], &y32) || !device_address(a[6], &st) || !stream_handle(a[7], &stream))
        return nullptr;
    const int nn = (int)w.size(0), kk = (int)w.size(1);
    const size_t bytes = sc.nbytes();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = cass_verify_gemm(wp, xp, (int)rows, nn, kk, sp, bytes, y16, static_cast<float*>(y32), static_cast<int32_t*>(st), stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
    END_HANDLE_TH_ERRORS
}

// (stream) -> its handle as an int; None: the current stream's
PyObject* stream_address(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    void* stream;
    if (n != 1) return PyErr_Format(PyExc_TypeError, "%zd arguments where 1 is wanted", n);
    return stream_handle(a[0], &stream) ? PyLong_FromVoidPtr(stream) : nullptr;
    END_HANDLE_TH_ERRORS
}

#define CASS_ENTRY(NAME) {#NAME, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&Entry<&NAME>::call)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    CASS_ENTRY(cass_draft_gemv), CASS_ENTRY(cass_draft_gemv_batch), CASS_ENTRY(cass_draft_gemv_static), CASS_ENTRY(cass_kv_append),
    CASS_ENTRY(cass_set_len), CASS_ENTRY(cass_draft_step), CASS_ENTRY(cass_verify), CASS_ENTRY(cass_draft_attention), CASS_ENTRY(cass_accept),
    CASS_ENTRY(cass_accept_sampling), CASS_ENTRY(cass_softmax), CASS_ENTRY(cass_sample),
    {"cass_verify_gemm", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&verify_gemm)), METH_FASTCALL, nullptr},
    {"stream_address", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&stream_address)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() {
    PyObject* ct = PyImport_ImportModule("ctypes");
    if (!ct) return nullptr;
    g_c_void_p = reinterpret_cast<PyTypeObject*>(PyObject_GetAttrString(ct, "c_void_p"));
    Py_DECREF(ct);
    g_torch_cuda = PyImport_ImportModule("torch.cuda");
    if (!g_c_void_p || !g_torch_cuda) return nullptr;
    return PyModule_Create(&kModule);
}
