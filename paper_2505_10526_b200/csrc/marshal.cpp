// Argument marshalling of the calls a decoding loop makes every step: tensors are checked and their addresses taken here
// instead of by half a dozen attribute reads per tensor in Python (25 tensors a step: about 8 us of 26 on a step whose kernels
// take 20).  The functions called are those of the C ABI library the binding has loaded; bind() hands their addresses in.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "massv.h"

namespace {

decltype(&massv_verify_attn) g_verify_attn = nullptr;
decltype(&massv_accept) g_accept = nullptr;
decltype(&massv_kv_commit) g_kv_commit = nullptr;
decltype(&massv_sample_top_p) g_sample_top_p = nullptr;
decltype(&massv_tvd) g_tvd = nullptr;
PyObject *g_attn_desc = nullptr, *g_accept_desc = nullptr;       // the ctypes structures of the two descriptors

const char* dtype_name(c10::ScalarType t) {
    switch (t) {
        case c10::ScalarType::BFloat16: return "torch.bfloat16";
        case c10::ScalarType::Float: return "torch.float32";
        case c10::ScalarType::Int: return "torch.int32";
        default: return c10::toString(t);
    }
}

// Sets a Python error and leaves by exception, so that one catch per call cleans up.
struct PythonError {};
[[noreturn]] void fail(PyObject* type, const char* text) { PyErr_SetString(type, text); throw PythonError(); }

// Address of a tensor's data; None is a null pointer.  dtype Undefined: any.
void* pointer(PyObject* obj, c10::ScalarType dtype) {
    if (obj == Py_None) return nullptr;
    if (!THPVariable_Check(obj)) fail(PyExc_AttributeError, "massv: tensors expected");
    const at::Tensor& t = THPVariable_Unpack(obj);
    if (!t.is_cuda()) fail(PyExc_ValueError, "massv: tensors must live on a CUDA device");
    if (!t.is_contiguous()) fail(PyExc_ValueError, "massv: tensors must be contiguous");
    if (dtype != c10::ScalarType::Undefined && t.scalar_type() != dtype) {
        PyErr_Format(PyExc_ValueError, "massv: expected %s, got %s", dtype_name(dtype), dtype_name(t.scalar_type()));
        throw PythonError();
    }
    return t.mutable_data_ptr();
}
void* bf16(PyObject* o) { return pointer(o, c10::ScalarType::BFloat16); }
float* f32(PyObject* o) { return static_cast<float*>(pointer(o, c10::ScalarType::Float)); }
int32_t* i32(PyObject* o) { return static_cast<int32_t*>(pointer(o, c10::ScalarType::Int)); }
void* any(PyObject* o) { return pointer(o, c10::ScalarType::Undefined); }
size_t elements(PyObject* o) { return o == Py_None ? 0 : (size_t)THPVariable_Unpack(o).numel(); }      // (behind any(): a tensor)

// A descriptor: the bytes of its ctypes structure (or of one derived from it, which begins with the same fields).
template <typename Desc>
struct DescOf {
    Py_buffer view;
    DescOf(PyObject* o, PyObject* type) {
        const int is = PyObject_IsInstance(o, type);
        if (is < 0) throw PythonError();
        if (is == 0) fail(PyExc_TypeError, "massv: wrong descriptor");
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw PythonError();
        if (view.len < (Py_ssize_t)sizeof(Desc)) { PyBuffer_Release(&view); fail(PyExc_TypeError, "massv: wrong descriptor"); }
    }
    DescOf(const DescOf&) = delete;
    DescOf& operator=(const DescOf&) = delete;
    ~DescOf() { PyBuffer_Release(&view); }
    const Desc* get() const { return static_cast<const Desc*>(view.buf); }
};

massv_stream_t stream() { return reinterpret_cast<massv_stream_t>(c10::cuda::getCurrentCUDAStream().stream()); }

long integer(PyObject* o) { const long v = PyLong_AsLong(o); if (v == -1 && PyErr_Occurred()) throw PythonError(); return v; }
double number(PyObject* o) {                                     // whatever float() takes
    PyObject* f = PyNumber_Float(o);
    if (!f) throw PythonError();
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return v;
}

// Runs `call` (arguments in, status out) with the argument count checked and C++ exceptions turned into Python's; the
// library call itself runs without the interpreter lock.
template <typename Call>
PyObject* guarded(Py_ssize_t given, Py_ssize_t wanted, Call&& call) {
    try {
        if (given != wanted) fail(PyExc_TypeError, "massv: wrong number of arguments");
        return PyLong_FromLong(call());
    } catch (const PythonError&) {
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}
template <typename F>
int unlocked(F&& f) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return rc;
}

PyObject* py_verify_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 13, [&] {
        const DescOf<massv_attn_desc> d(a[0], g_attn_desc);
        void *q = bf16(a[1]), *kn = bf16(a[2]), *vn = bf16(a[3]), *kp = bf16(a[4]), *vp = bf16(a[5]);
        int32_t *table = i32(a[6]), *lens = i32(a[7]);
        void* out = bf16(a[8]);
        float *out32 = f32(a[9]), *lse = f32(a[10]);
        void* ws = any(a[11]);
        const size_t ws_bytes = elements(a[11]);
        int32_t* status = i32(a[12]);
        const massv_stream_t s = stream();
        return unlocked([&] { return g_verify_attn(d.get(), q, kn, vn, kp, vp, table, lens, out, out32, lse, ws, ws_bytes, status, s); });
    });
}
PyObject* py_accept(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 13, [&] {
        const DescOf<massv_accept_desc> d(a[0], g_accept_desc);
        void *h = bf16(a[1]), *w = bf16(a[2]);
        int32_t* drafts = i32(a[3]);
        float *q = f32(a[4]), *ua = f32(a[5]), *us = f32(a[6]);
        int32_t *tokens = i32(a[7]), *lens = i32(a[8]);
        float *logits = f32(a[9]), *probs = f32(a[10]);
        void* ws = any(a[11]);
        const size_t ws_bytes = elements(a[11]);
        int32_t* status = i32(a[12]);
        const massv_stream_t s = stream();
        return unlocked([&] { return g_accept(d.get(), h, w, drafts, q, ua, us, tokens, lens, logits, probs, ws, ws_bytes, status, s); });
    });
}
PyObject* py_kv_commit(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 5, [&] {
        const int32_t batch = (int32_t)integer(a[0]), gamma = (int32_t)integer(a[1]);
        int32_t *lens = i32(a[2]), *seq = i32(a[3]), *status = i32(a[4]);
        const massv_stream_t s = stream();
        return unlocked([&] { return g_kv_commit(batch, gamma, lens, seq, status, s); });
    });
}
PyObject* py_sample_top_p(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 9, [&] {
        const int32_t rows = (int32_t)integer(a[0]), vocab = (int32_t)integer(a[1]);
        const float T = (float)number(a[2]), top_p = (float)number(a[3]);
        float *z = f32(a[4]), *u = f32(a[5]);
        int32_t* tokens = i32(a[6]);
        float* probs = f32(a[7]);
        int32_t* status = i32(a[8]);
        const massv_stream_t s = stream();
        return unlocked([&] { return g_sample_top_p(rows, vocab, T, top_p, z, u, tokens, probs, status, s); });
    });
}
PyObject* py_tvd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 7, [&] {
        const DescOf<massv_accept_desc> d(a[0], g_accept_desc);
        float *z = f32(a[1]), *q = f32(a[2]), *tvd = f32(a[3]), *acc = f32(a[4]);
        void* ws = any(a[5]);
        const size_t ws_bytes = elements(a[5]);
        int32_t* status = i32(a[6]);
        const massv_stream_t s = stream();
        return unlocked([&] { return g_tvd(d.get(), z, q, tvd, acc, ws, ws_bytes, status, s); });
    });
}

PyObject* py_bind(PyObject*, PyObject* args) {
    unsigned long long attn, accept, commit, top_p, tvd;
    PyObject *attn_desc, *accept_desc;
    if (!PyArg_ParseTuple(args, "KKKKKO!O!", &attn, &accept, &commit, &top_p, &tvd, &PyType_Type, &attn_desc, &PyType_Type, &accept_desc)) return nullptr;
    Py_INCREF(attn_desc);
    Py_INCREF(accept_desc);
    Py_XSETREF(g_attn_desc, attn_desc);
    Py_XSETREF(g_accept_desc, accept_desc);
    g_verify_attn = reinterpret_cast<decltype(g_verify_attn)>(attn);
    g_accept = reinterpret_cast<decltype(g_accept)>(accept);
    g_kv_commit = reinterpret_cast<decltype(g_kv_commit)>(commit);
    g_sample_top_p = reinterpret_cast<decltype(g_sample_top_p)>(top_p);
    g_tvd = reinterpret_cast<decltype(g_tvd)>(tvd);
    Py_RETURN_NONE;
}

#define MASSV_FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(f)), METH_FASTCALL
PyMethodDef g_methods[] = {
    {"bind", py_bind, METH_VARARGS, "addresses of the C ABI functions, types of the descriptors"},
    {"verify_attn", MASSV_FAST(py_verify_attn), nullptr},
    {"accept", MASSV_FAST(py_accept), nullptr},
    {"kv_commit", MASSV_FAST(py_kv_commit), nullptr},
    {"sample_top_p", MASSV_FAST(py_sample_top_p), nullptr},
    {"tvd", MASSV_FAST(py_tvd), nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&g_module); }
