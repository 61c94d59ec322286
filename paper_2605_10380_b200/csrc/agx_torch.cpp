// CPython module behind agx.py: turns torch tensors, numpy arrays and streams into the pointers and sizes of the C calls.
//
// A decode step of a 32-layer model is 32 attention calls of 7 us of GPU work each, and through ctypes every call took
// 15.5 us of host time, of which the C function 5: the rest was the conversion of two dozen arguments in Python and
// torch.cuda.current_stream() (3.1 us).  The same conversions here take well under a microsecond: a 32-layer decode step
// over 4096 tokens 489 -> 285 us, a verify step 488 -> 336 us.
//
// No arithmetic and no state beyond the addresses of the C functions, which agx.py passes in once (bind), so that there
// is one copy of the library in the process.  The GIL is released around every C call, as ctypes does.
#include <torch/csrc/autograd/python_variable.h>
#include <torch/version.h>

#include <c10/cuda/CUDAStream.h>

#include <exception>

#include "agx.h"

namespace {

struct Functions {
    decltype(&agx_kv_append) kv_append;
    decltype(&agx_attn_prefixed) attn;
    decltype(&agx_attn_prefixed_append) attn_append;
    decltype(&agx_accept_greedy) accept;
    decltype(&agx_verify_step_host) step;
    decltype(&agx_verify_step_host_enqueue) step_enqueue;
    decltype(&agx_ngram_build) ngram_build;
    decltype(&agx_ngram_draft) ngram_draft;
    decltype(&agx_kv_copy_pages) copy_pages;
} fn;
PyObject* to_i32 = nullptr;   // agx._h_i32: anything array-like -> contiguous numpy int32
PyObject* ndarray = nullptr;  // numpy.ndarray

struct PyFailed : std::exception {};   // a Python error is set

// Exact tensors and arrays take a short way; whatever else has the attributes of one is asked for them, as Python code would.
PyObject* checked(PyObject* o) {
    if (!o) throw PyFailed();
    return o;
}
int64_t integer(PyObject* o) {
    PyObject* n = PyLong_Check(o) ? Py_NewRef(o) : checked(PyNumber_Long(o));   // (int(o))
    const long long v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    if (v == -1 && PyErr_Occurred()) throw PyFailed();
    return v;
}
int64_t taken(PyObject* o) {   // integer(o), and o is done with
    struct Ref { PyObject* o; ~Ref() { Py_DECREF(o); } } ref{checked(o)};
    return integer(o);
}
bool is_array(PyObject* o) { return PyObject_TypeCheck(o, (PyTypeObject*)ndarray); }
// what stands for a device tensor: not a host array
PyObject* device(PyObject* o) {
    if (o == Py_None || is_array(o)) { PyErr_Format(PyExc_TypeError, "expected a torch tensor, got %s", Py_TYPE(o)->tp_name); throw PyFailed(); }
    return o;
}
const at::Tensor* exact(PyObject* o) { return THPVariable_CheckExact(o) ? &THPVariable_Unpack(o) : nullptr; }
int64_t dim(PyObject* o, int i) {
    if (const at::Tensor* t = exact(o)) return t->size(i);
    PyObject* shape = checked(PyObject_GetAttrString(device(o), "shape"));
    PyObject* n = PySequence_GetItem(shape, i);
    Py_DECREF(shape);
    return taken(n);
}
int64_t numel(PyObject* o) {
    if (const at::Tensor* t = exact(o)) return t->numel();
    return taken(PyObject_CallMethod(device(o), "numel", nullptr));
}
int64_t stride0(PyObject* o) {
    if (const at::Tensor* t = exact(o)) return t->stride(0);
    return taken(PyObject_CallMethod(device(o), "stride", "i", 0));
}
size_t bytes(PyObject* o) {
    if (o == Py_None) return 0;
    if (const at::Tensor* t = exact(o)) return t->nbytes();
    return (size_t)(numel(o) * taken(PyObject_CallMethod(o, "element_size", nullptr)));
}

// Address of a tensor's or a numpy array's first element; NULL for None.
void* address(PyObject* o) {
    if (o == Py_None) return nullptr;
    if (const at::Tensor* t = exact(o)) return t->mutable_data_ptr();   // (as Tensor.data_ptr(): a copy-on-write tensor gets its own memory first)
    if (!is_array(o)) return (void*)(intptr_t)taken(PyObject_CallMethod(o, "data_ptr", nullptr));
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_STRIDED_RO) != 0) throw PyFailed();
    void* p = view.buf;
    PyBuffer_Release(&view);
    return p;
}
agx_handle* handle(PyObject* o) {
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) throw PyFailed();
    return (agx_handle*)p;
}

// None: torch's current stream; an int: a cudaStream_t; anything else: its cuda_stream attribute.
void* stream(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    if (PyLong_Check(o)) return (void*)(intptr_t)integer(o);
    return (void*)(intptr_t)taken(PyObject_GetAttrString(o, "cuda_stream"));
}

// Host int32 lengths: a contiguous numpy int32 array as it is, anything else through agx._h_i32.  Their number is the first dimension.
struct Lengths {
    Py_buffer view{};
    const int32_t* data;
    int32_t count;
    explicit Lengths(PyObject* o) {
        if (!PyObject_CheckBuffer(o) || PyObject_GetBuffer(o, &view, PyBUF_CONTIG_RO | PyBUF_FORMAT) != 0 || !plain()) {
            PyErr_Clear();
            if (view.obj) PyBuffer_Release(&view);
            PyObject* a = PyObject_CallOneArg(to_i32, o);
            if (!a) throw PyFailed();
            const int rc = PyObject_GetBuffer(a, &view, PyBUF_CONTIG_RO | PyBUF_FORMAT);
            Py_DECREF(a);   // (the view keeps it)
            if (rc != 0) throw PyFailed();
        }
        data = (const int32_t*)view.buf;
        count = (int32_t)view.shape[0];
    }
    Lengths(const Lengths&) = delete;
    ~Lengths() { if (view.obj) PyBuffer_Release(&view); }
    bool plain() const { return view.itemsize == 4 && view.ndim == 1 && view.format && view.format[0] == 'i' && !view.format[1]; }
};

struct ReleaseGil {
    PyThreadState* s = PyEval_SaveThread();
    ~ReleaseGil() { PyEval_RestoreThread(s); }
};

template <typename F>
PyObject* guarded(const char* name, Py_ssize_t got, Py_ssize_t want, F body) {
    if (got != want) { PyErr_Format(PyExc_TypeError, "%s: %zd arguments instead of %zd", name, got, want); return nullptr; }
    try {
        return PyLong_FromLong((long)body());
    } catch (const PyFailed&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// (handle, q, k_new, v_new, k_pool, v_pool, page_table, prefix, q_len, out, lse, workspace, stream); without an append k_new and v_new are not looked at
PyObject* call_attn(bool append, PyObject* const* a, Py_ssize_t n) {
    return guarded("attn", n, 13, [&] {
        agx_handle* h = handle(a[0]);
        const Lengths P(a[7]), Q(a[8]);
        void *q = address(a[1]), *kn = address(a[2]), *vn = address(a[3]), *kp = address(a[4]), *vp = address(a[5]);
        const int32_t* pt = (const int32_t*)address(a[6]);
        void *out = address(a[9]), *ws = address(a[11]), *st = stream(a[12]);
        float* lse = (float*)address(a[10]);
        const int64_t pages = dim(a[4], 0);
        const int32_t stride = (int32_t)dim(a[6], 1);
        const size_t wsb = bytes(a[11]);
        ReleaseGil gil;
        return append ? fn.attn_append(h, q, kn, vn, kp, vp, pages, pt, stride, P.data, Q.data, P.count, out, lse, ws, wsb, st)
                      : fn.attn(h, q, kp, vp, pages, pt, stride, P.data, Q.data, P.count, out, lse, ws, wsb, st);
    });
}
PyObject* py_attn(PyObject*, PyObject* const* a, Py_ssize_t n) { return call_attn(false, a, n); }
PyObject* py_attn_append(PyObject*, PyObject* const* a, Py_ssize_t n) { return call_attn(true, a, n); }
// (handle, k_pool, v_pool, k_new, v_new, page_table, prefix_len, cu_q, stream)
PyObject* py_kv_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded("kv_append", n, 9, [&] {
        agx_handle* h = handle(a[0]);
        const int64_t pages = dim(a[1], 0);
        const int32_t rows = (int32_t)dim(a[3], 0), stride = (int32_t)dim(a[5], 1), B = (int32_t)dim(a[6], 0);
        void *kp = address(a[1]), *vp = address(a[2]), *kn = address(a[3]), *vn = address(a[4]), *st = stream(a[8]);
        const int32_t *pt = (const int32_t*)address(a[5]), *pl = (const int32_t*)address(a[6]), *cu = (const int32_t*)address(a[7]);
        ReleaseGil gil;
        return fn.kv_append(h, kp, vp, pages, kn, vn, pt, stride, pl, cu, B, rows, st);
    });
}
// (handle, logits, dtype, vocab, drafts, cu_q, accept_len, next_token, argmax, seq_lens, workspace, stream)
PyObject* py_accept(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded("accept", n, 12, [&] {
        agx_handle* h = handle(a[0]);
        const int32_t dt = (int32_t)integer(a[2]), vocab = (int32_t)integer(a[3]), B = (int32_t)dim(a[5], 0) - 1;
        int32_t* p[6];
        for (int i = 0; i < 6; ++i) p[i] = (int32_t*)address(a[4 + i]);
        void *l = address(a[1]), *ws = address(a[10]), *st = stream(a[11]);
        const int64_t row_stride = stride0(a[1]);
        const int32_t rows = (int32_t)dim(a[1], 0);
        const size_t wsb = bytes(a[10]);
        ReleaseGil gil;
        return fn.accept(h, l, dt, row_stride, vocab, p[0], p[1], B, rows, p[2], p[3], p[4], p[5], ws, wsb, st);
    });
}
// (handle, sync, k_pool, v_pool, page_table, prefix, q_len, q, k_new, v_new, logits, dtype, row_stride, vocab, drafts, out, accept_len,
//  next_token, seq_lens, workspace, stream)
PyObject* py_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded("verify_step_host", n, 21, [&] {
        agx_handle* h = handle(a[0]);
        const auto f = integer(a[1]) ? fn.step : fn.step_enqueue;
        const int64_t pages = dim(a[2], 0), row_stride = integer(a[12]);
        const int32_t stride = (int32_t)dim(a[4], 1), dt = (int32_t)integer(a[11]), vocab = (int32_t)integer(a[13]);
        const Lengths P(a[5]), Q(a[6]);
        void *kp = address(a[2]), *vp = address(a[3]), *q = address(a[7]), *kn = address(a[8]), *vn = address(a[9]), *lg = address(a[10]);
        void *out = address(a[15]), *ws = address(a[19]), *st = stream(a[20]);
        const int32_t *pt = (const int32_t*)address(a[4]), *dr = (const int32_t*)address(a[14]);
        int32_t *acc = (int32_t*)address(a[16]), *nxt = (int32_t*)address(a[17]), *sl = (int32_t*)address(a[18]);
        const size_t wsb = bytes(a[19]);
        ReleaseGil gil;
        return f(h, kp, vp, pages, pt, stride, P.data, Q.data, P.count, q, kn, vn, lg, dt, row_stride, vocab, dr, out, acc, nxt, sl, ws, wsb, st);
    });
}
// (handle, tokens, n, lut, workspace, stream)
PyObject* py_ngram_build(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded("ngram_build", n, 6, [&] {
        agx_handle* h = handle(a[0]);
        const int32_t tokens = (int32_t)numel(a[1]), order = (int32_t)integer(a[2]);
        const int32_t* s = (const int32_t*)address(a[1]);
        void *lut = address(a[3]), *ws = address(a[4]), *st = stream(a[5]);
        const size_t lb = bytes(a[3]), wb = bytes(a[4]);
        ReleaseGil gil;
        return fn.ngram_build(h, s, tokens, order, lut, lb, ws, wb, st);
    });
}
// (handle, lut, context, fill, k, drafts, has_draft, stream)
PyObject* py_ngram_draft(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded("ngram_draft", n, 8, [&] {
        agx_handle* h = handle(a[0]);
        const int32_t B = (int32_t)dim(a[6], 0), k = (int32_t)integer(a[4]);
        void *lut = address(a[1]), *st = stream(a[7]);
        int32_t *c = (int32_t*)address(a[2]), *f = (int32_t*)address(a[3]), *d = (int32_t*)address(a[5]), *has = (int32_t*)address(a[6]);
        ReleaseGil gil;
        return fn.ngram_draft(h, lut, c, f, B, k, d, has, st);
    });
}
// (handle, k_pool, v_pool, src, dst, stream)
PyObject* py_copy_pages(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded("kv_copy_pages", n, 6, [&] {
        agx_handle* h = handle(a[0]);
        const int64_t pages = dim(a[1], 0);
        const int32_t count = (int32_t)numel(a[3]);
        void *kp = address(a[1]), *vp = address(a[2]), *st = stream(a[5]);
        const int32_t *src = (const int32_t*)address(a[3]), *dst = (const int32_t*)address(a[4]);
        ReleaseGil gil;
        return fn.copy_pages(h, kp, vp, pages, src, dst, count, st);
    });
}

// bind(to_i32, numpy.ndarray, address of each function in the order of `Functions`)
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded("bind", n, 11, [&] {
        void* p[9];
        for (int i = 0; i < 9; ++i) p[i] = (void*)handle(a[2 + i]);
        fn = Functions{(decltype(fn.kv_append))p[0], (decltype(fn.attn))p[1], (decltype(fn.attn_append))p[2], (decltype(fn.accept))p[3],
                       (decltype(fn.step))p[4], (decltype(fn.step_enqueue))p[5], (decltype(fn.ngram_build))p[6],
                       (decltype(fn.ngram_draft))p[7], (decltype(fn.copy_pages))p[8]};
        Py_XSETREF(to_i32, Py_NewRef(a[0]));
        Py_XSETREF(ndarray, Py_NewRef(a[1]));
        return 0;
    });
}

#define AGX_METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {AGX_METHOD(bind), AGX_METHOD(attn), AGX_METHOD(attn_append), AGX_METHOD(kv_append), AGX_METHOD(accept), AGX_METHOD(step),
                         AGX_METHOD(ngram_build), AGX_METHOD(ngram_draft), AGX_METHOD(copy_pages), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "agx_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_agx_torch() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "torch_version", TORCH_VERSION) != 0) Py_CLEAR(m);   // (agx.py does not use it with another torch)
    return m;
}
