// Fast argument path of the Python binding.  A call's tensors are checked and marshalled here instead of in Python, where the
// checks, the ctypes descriptor and the stream lookup cost some 10 us a call: more than the kernels of a one-request decoding step.
// Whatever this code does not recognise as a correct call (a wrong type or shape, a workspace that has to grow, a tensor whose sizes or
// storage torch does not hand out, which it says with a C++ exception: none may pass a C entry) is answered with None: the caller
// then takes the general path in Python, which raises the errors or makes the allocation.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>
#include "gdn_tail_replay.h"

namespace {

using Forward = int32_t (*)(const gdn_desc*, const void*, const void*, const void*, const float*, const float*, const int32_t*,
                            int32_t, void*, float*);
using Decode = int32_t (*)(const gdn_desc*, const void*, const void*, const void*, const float*, const float*, const float*,
                           void*, float*);
Forward g_forward[3] = {};               // gdn_tail_replay, gdn_full_prefill, gdn_tail_replay_static_scratch
Decode g_decode = nullptr;
size_t (*g_workspace_size)(const gdn_desc*) = nullptr;
PyObject *s_by_stream = nullptr, *s_cuda_stream = nullptr, *g_workspace_type = nullptr;

inline const at::Tensor* tensor(PyObject* o) { return THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr; }
// contiguous, of type dt, on the side given by `cuda`, of shape {s...}
template <typename... S>
inline bool fits(const at::Tensor* t, at::ScalarType dt, bool cuda, S... s)
{
    if (!t || t->scalar_type() != dt || t->is_cuda() != cuda || t->dim() != (int64_t)sizeof...(s) || !t->is_contiguous()) return false;
    const int64_t want[] = {(int64_t)s...};
    for (size_t i = 0; i < sizeof...(s); ++i)
        if (t->size((int64_t)i) != want[i]) return false;
    return true;
}
template <typename... S>
inline bool fits_or_none(PyObject* o, const at::Tensor*& t, at::ScalarType dt, bool cuda, S... s)
{
    t = nullptr;
    if (o == Py_None) return true;
    t = tensor(o);
    return fits(t, dt, cuda, s...);
}
inline void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
// the stream argument's handle, or the current stream's
inline bool stream_of(PyObject* o, void*& st)
{
    if (o == Py_None) {
        st = (void*)c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* h = PyObject_GetAttr(o, s_cuda_stream);
    if (h) st = PyLong_AsVoidPtr(h);
    Py_XDECREF(h);
    if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    return true;
}

using Entry = PyObject* (*)(PyObject*, PyObject* const*, Py_ssize_t);
template <Entry F> PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    try {
        return F(self, a, n);
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}
// The library's call, with the other Python threads running: it may copy pageable memory, or wait for room in a launch queue that
// only empties when a host callback of another thread's has run.  (The caller's frame holds the arguments.)
template <typename F> PyObject* without_gil(F call)
{
    int32_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}
struct Ref {                                 // an owned reference, given back on every way out
    PyObject* o;
    ~Ref() { Py_XDECREF(o); }
};

// forward(which, q, k, v, g, beta, cu_tail_lens, chunk, out_o, out_state, init_state, workspace, status_word, kernel, stream, raw)
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 16) Py_RETURN_NONE;
    const long which = PyLong_AsLong(a[0]), chunk = PyLong_AsLong(a[7]), kernel = PyLong_AsLong(a[13]);
    const int raw = PyObject_IsTrue(a[15]);
    if (PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }
    if (which < 0 || which > 2 || chunk != (int32_t)chunk || kernel != (int32_t)kernel) Py_RETURN_NONE;
    const at::Tensor *q = tensor(a[1]), *k = tensor(a[2]), *v = tensor(a[3]), *g = tensor(a[4]), *beta = tensor(a[5]), *cu = tensor(a[6]);
    if (!q || !v || !cu || q->dim() != 3 || v->dim() != 3 || cu->dim() != 1 || cu->size(0) < 1) Py_RETURN_NONE;
    const at::ScalarType dt = q->scalar_type();
    const bool cuda = q->is_cuda();
    const int64_t T = q->size(0), Hq = q->size(1), dk = q->size(2), Hv = v->size(1), dv = v->size(2), N = cu->size(0) - 1;
    if ((dt != at::kBFloat16 && dt != at::kFloat) || N > 0x7fffffff || Hq > 0x7fffffff || Hv > 0x7fffffff || dk > 0x7fffffff || dv > 0x7fffffff)
        Py_RETURN_NONE;
    const at::Tensor *o, *st, *init, *status;
    if (!fits(q, dt, cuda, T, Hq, dk) || !fits(k, dt, cuda, T, Hq, dk) || !fits(v, dt, cuda, T, Hv, dv) ||
        !fits(g, at::kFloat, cuda, T, Hv) || !fits(beta, at::kFloat, cuda, T, Hv) || !fits(cu, at::kInt, cuda, N + 1) ||
        !fits_or_none(a[8], o, dt, cuda, T, Hv, dv) || !fits_or_none(a[9], st, at::kFloat, cuda, N, Hv, dk, dv))
        Py_RETURN_NONE;
    init = status = nullptr;
    if (a[10] != Py_None && (!(init = tensor(a[10])) || init->is_cuda() != cuda || !init->is_contiguous() || init->scalar_type() != at::kFloat ||
                             init->numel() < N * Hv * dk * dv))
        Py_RETURN_NONE;
    if (a[12] != Py_None && (!(status = tensor(a[12])) || !status->is_cuda() || status->nbytes() < 4)) Py_RETURN_NONE;

    gdn_desc d = {};
    d.num_qk_heads = (int32_t)Hq; d.num_v_heads = (int32_t)Hv; d.head_k_dim = (int32_t)dk; d.head_v_dim = (int32_t)dv;
    d.io_dtype = dt == at::kBFloat16 ? GDN_BF16 : GDN_F32;
    d.num_seqs = (int32_t)N; d.total_tokens = T;
    d.memory = cuda ? GDN_MEM_DEVICE : GDN_MEM_HOST;
    d.kernel = (int32_t)kernel;
    d.input_stage = raw ? GDN_INPUT_RAW : GDN_INPUT_READY;
    d.init_state = (const float*)ptr(init);
    if (!stream_of(a[14], d.stream)) Py_RETURN_NONE;
    Ref b{nullptr};
    if (which != 2) {
        // the Workspace's buffer for this stream as it is; making or growing it is the general path's
        if ((PyObject*)Py_TYPE(a[11]) != g_workspace_type) Py_RETURN_NONE;
        const Ref map{PyObject_GetAttr(a[11], s_by_stream)}, key{PyLong_FromVoidPtr(d.stream)};
        if (map.o && key.o && PyDict_Check(map.o)) b.o = PyDict_GetItemWithError(map.o, key.o);
        Py_XINCREF(b.o);                                  // (held over the call: another thread may let the Workspace grow)
        const at::Tensor* buf = b.o ? tensor(b.o) : nullptr;
        const int64_t need = (int64_t)g_workspace_size(&d);
        const bool ok = buf && buf->is_cuda() && buf->element_size() == 1 && buf->numel() >= need;
        if (ok) {
            const uintptr_t base = (uintptr_t)buf->data_ptr(), off = (256 - base % 256) % 256;
            d.workspace = (void*)(base + off);
            d.workspace_bytes = (size_t)buf->numel() - off;
        }
        PyErr_Clear();
        if (!ok) Py_RETURN_NONE;
    }
    d.status_word = (int32_t*)ptr(status);
    const void *pq = q->data_ptr(), *pk = k->data_ptr(), *pv = v->data_ptr(), *pg = g->data_ptr(), *pb = beta->data_ptr(), *pc = cu->data_ptr();
    void *po = ptr(o), *ps = ptr(st);
    return without_gil([&]() { return g_forward[which](&d, pq, pk, pv, (const float*)pg, (const float*)pb, (const int32_t*)pc, (int32_t)chunk, po, (float*)ps); });
}

// decode(q, k, v, g, beta, state_in, out_o, state_out, stream)
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 9) Py_RETURN_NONE;
    const at::Tensor *q = tensor(a[0]), *v = tensor(a[2]), *o;
    if (!q || !v || q->dim() != 3 || v->dim() != 3) Py_RETURN_NONE;
    const at::ScalarType dt = q->scalar_type();
    const int64_t N = q->size(0), Hq = q->size(1), dk = q->size(2), Hv = v->size(1), dv = v->size(2);
    if ((dt != at::kBFloat16 && dt != at::kFloat) || N > 0x7fffffff || Hq > 0x7fffffff || Hv > 0x7fffffff || dk > 0x7fffffff || dv > 0x7fffffff)
        Py_RETURN_NONE;
    const at::Tensor *k = tensor(a[1]), *g = tensor(a[3]), *beta = tensor(a[4]), *in = tensor(a[5]), *out = tensor(a[7]);
    if (!fits(q, dt, true, N, Hq, dk) || !fits(k, dt, true, N, Hq, dk) || !fits(v, dt, true, N, Hv, dv) || !fits(g, at::kFloat, true, N, Hv) ||
        !fits(beta, at::kFloat, true, N, Hv) || !fits(in, at::kFloat, true, N, Hv, dk, dv) || !fits(out, at::kFloat, true, N, Hv, dk, dv) ||
        !fits_or_none(a[6], o, dt, true, N, Hv, dv))
        Py_RETURN_NONE;
    gdn_desc d = {};
    d.num_qk_heads = (int32_t)Hq; d.num_v_heads = (int32_t)Hv; d.head_k_dim = (int32_t)dk; d.head_v_dim = (int32_t)dv;
    d.io_dtype = dt == at::kBFloat16 ? GDN_BF16 : GDN_F32;
    d.num_seqs = (int32_t)N; d.total_tokens = N;
    d.memory = GDN_MEM_DEVICE; d.kernel = GDN_KERNEL_AUTO;
    if (!stream_of(a[8], d.stream)) Py_RETURN_NONE;
    const void *pq = q->data_ptr(), *pk = k->data_ptr(), *pv = v->data_ptr(), *pg = g->data_ptr(), *pb = beta->data_ptr(), *pi = in->data_ptr();
    void *po = ptr(o), *ps = out->data_ptr();
    return without_gil([&]() { return g_decode(&d, pq, pk, pv, (const float*)pg, (const float*)pb, (const float*)pi, po, (float*)ps); });
}

// bind(gdn_tail_replay, gdn_full_prefill, gdn_tail_replay_static_scratch, gdn_decode_step, gdn_workspace_size, Workspace): the addresses of
// the library's functions, and the class whose buffers are looked up here
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 6) { PyErr_SetString(PyExc_TypeError, "five addresses and a class"); return nullptr; }
    void* p[5];
    for (int i = 0; i < 5; ++i) p[i] = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred()) return nullptr;
    for (int i = 0; i < 3; ++i) g_forward[i] = (Forward)p[i];
    g_decode = (Decode)p[3];
    g_workspace_size = (size_t (*)(const gdn_desc*))p[4];
    Py_INCREF(a[5]);
    Py_XSETREF(g_workspace_type, a[5]);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"forward", (PyCFunction)(void (*)(void))guarded<forward>, METH_FASTCALL, nullptr},
    {"decode", (PyCFunction)(void (*)(void))guarded<decode>, METH_FASTCALL, nullptr},
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native()
{
    s_by_stream = PyUnicode_InternFromString("by_stream");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for_torch", BUILT_FOR_TORCH) < 0) { Py_DECREF(m); return nullptr; }
    return m;
}
