// Python binding of the calls in lte.h: unpacks torch tensors, allocates the outputs and the scratch the caller did not bring
// (torch's allocator, current stream) and makes the C call.  Nothing is computed here.  lte.py holds the signatures; its
// functions hand their arguments on by position.
//
// Why native: a small call is bound by the host.  Marshalled in Python (torch.empty, data_ptr and checks per tensor, ctypes
// conversions) a call took 14 us on the host, of which the launch itself is 3; through here it takes 4 to 5.  The
// interpreter lock is released around the C call, as ctypes does.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "lte.h"

namespace {

PyObject* g_error = nullptr;                                   // lte.LteError(fn, status)
struct PyFailure {};                                           // a Python exception has been set

[[noreturn]] void fail(PyObject* type, const char* text) { PyErr_SetString(type, text); throw PyFailure(); }

// the C struct inside a ctypes object (which the caller holds during the call); never NULL: the callers read its sizes
template <typename S> const S* c_struct(PyObject* o)
{
    if (o == Py_None) fail(PyExc_TypeError, "expected an LteShape and an LteConv, not None");
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) throw PyFailure();
    const void* p = b.buf;
    const bool fits = b.len == (Py_ssize_t)sizeof(S);
    PyBuffer_Release(&b);
    if (!fits) fail(PyExc_TypeError, "expected an LteShape and an LteConv");
    return (const S*)p;
}

const at::Tensor& tensor(PyObject* o)
{
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a torch tensor");
    return THPVariable_Unpack(o);
}

// device pointer of a contiguous CUDA tensor, NULL for None
void* ptr(PyObject* o)
{
    if (o == Py_None) return nullptr;
    const at::Tensor& t = tensor(o);
    if (!t.is_cuda() || !t.is_contiguous()) fail(PyExc_AssertionError, "tensors must be contiguous CUDA tensors");
    return t.data_ptr();
}
void* ptr(PyObject* o, at::ScalarType type)
{
    void* p = ptr(o);
    if (o != Py_None && THPVariable_Unpack(o).scalar_type() != type) fail(PyExc_AssertionError, "a tensor has another dtype than the call expects");
    return p;
}
float* fptr(PyObject* o) { return (float*)ptr(o, at::kFloat); }
int32_t* iptr(PyObject* o) { return (int32_t*)ptr(o, at::kInt); }

void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

// A new tensor where `like` is: the library's kernels work on it, so it has to be on a GPU.
at::Tensor allocate(at::IntArrayRef size, at::ScalarType type, const at::Tensor& like)
{
    if (!like.is_cuda()) fail(PyExc_AssertionError, "tensors must be contiguous CUDA tensors");
    return at::empty(size, like.options().dtype(type));
}

// An output: the tensor the caller brought, or a new one.
class Out {
public:
    Out(PyObject* given, at::IntArrayRef size, at::ScalarType type, const at::Tensor& like, bool checked = true) : given_(given)
    {
        if (given == Py_None) {
            mine_ = allocate(size, type, like);
            p_ = mine_.data_ptr();
        } else {
            p_ = checked ? ptr(given, type) : ptr(given);
        }
    }
    template <typename T> T* as() const { return (T*)p_; }
    PyObject* result() const { return given_ == Py_None ? THPVariable_Wrap(mine_) : Py_NewRef(given_); }
private:
    PyObject* given_;
    at::Tensor mine_;
    void* p_ = nullptr;
};

// Scratch: the tensor the caller brought (its elements count as bytes; `bytes_only`: it has to consist of them), `need` bytes allocated
// here for None, nothing for False.
class Scratch {
public:
    Scratch(PyObject* given, size_t need, const at::Tensor& like, size_t at_least = 0, bool bytes_only = false)
    {
        if (given == Py_False) return;
        if (given == Py_None) {
            n_ = need > at_least ? need : at_least;
            if (n_ == 0) return;
            mine_ = allocate({(int64_t)n_}, at::kByte, like);
            p_ = mine_.data_ptr();
        } else {
            p_ = bytes_only ? ptr(given, at::kByte) : ptr(given);
            n_ = (size_t)THPVariable_Unpack(given).numel();
        }
    }
    void* p() const { return p_; }
    size_t n() const { return n_; }
private:
    at::Tensor mine_;
    void* p_ = nullptr;
    size_t n_ = 0;
};

struct Unlocked {                                              // the interpreter lock given up for a scope, however that ends
    PyThreadState* ts = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(ts); }
};
// the C call on the current stream, without the interpreter lock (torch is asked for the stream, and may throw, before that); a status
// other than LTE_OK becomes an LteError
template <typename F> void call(const char* fn, F&& f)
{
    void* const st = stream();
    const int status = [&] { Unlocked u; return f(st); }();
    if (status == LTE_OK) return;
    if (PyObject* e = PyObject_CallFunction(g_error, "si", fn, status)) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw PyFailure();
}

PyObject* pack(std::initializer_list<PyObject*> items)         // takes the references
{
    PyObject* t = PyTuple_New((Py_ssize_t)items.size());
    Py_ssize_t i = 0;
    for (PyObject* o : items) PyTuple_SET_ITEM(t, i++, o);
    return t;
}

int64_t heads_q(const lte_shape* s) { return (int64_t)s->H * (s->group > 1 ? s->group : 1); }

#define LTE_FN(name, count)                                                              \
    PyObject* name##_impl(PyObject* const* a);                                           \
    PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n)                          \
    {                                                                                    \
        HANDLE_TH_ERRORS                                                                 \
        if (n != count) { PyErr_SetString(PyExc_TypeError, #name ": wrong number of arguments"); return nullptr; } \
        try { return name##_impl(a); } catch (const PyFailure&) { return nullptr; }      \
        END_HANDLE_TH_ERRORS                                                             \
    }                                                                                    \
    PyObject* name##_impl(PyObject* const* a)

// s, c, k, v, z, r, ws
LTE_FN(scores, 7)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const lte_conv* c = c_struct<lte_conv>(a[1]);
    const at::Tensor& k = tensor(a[2]);
    Out z(a[4], {s->B, s->H, s->T}, at::kFloat, k);
    Scratch ws(a[6], a[6] == Py_None ? lte_workspace_bytes(LTE_OP_SCORES, s, c) : 0, k, 0, true);
    const void *kp = ptr(a[2]), *vp = ptr(a[3]);
    float* r = fptr(a[5]);
    call("lte_scores", [&](void* st) { return lte_scores(s, c, kp, vp, z.as<float>(), r, ws.p(), ws.n(), st); });
    return z.result();
}

// s, rule, score, idx, cnt, ncand, a tensor or device to allocate on
LTE_FN(select_rule, 7)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const long rule = PyLong_AsLong(a[1]);
    if (rule == -1 && PyErr_Occurred()) throw PyFailure();
    const at::Tensor& like = tensor(a[6]);
    Out idx(a[3], {s->B, s->H, s->R}, at::kInt, like), cnt(a[4], {s->B, s->H}, at::kInt, like);
    const float* score = fptr(a[2]);
    int32_t* ncand = iptr(a[5]);
    call(rule == LTE_RULE_LEARNED ? "lte_select" : "lte_select_rule", [&](void* st) {
        return lte_select_rule(s, (int)rule, score, idx.as<int32_t>(), cnt.as<int32_t>(), ncand, nullptr, 0, st); });
    return pack({idx.result(), cnt.result()});
}

// s, q, k, lse, idx, cnt, a
LTE_FN(attn_colsum, 7)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    Out out(a[6], {s->B, s->H, s->T}, at::kFloat, tensor(a[1]));
    const void *q = ptr(a[1]), *k = ptr(a[2]);
    const float* lse = fptr(a[3]);
    const int32_t *idx = iptr(a[4]), *cnt = iptr(a[5]);
    call("lte_attn_colsum", [&](void* st) { return lte_attn_colsum(s, q, k, lse, idx, cnt, out.as<float>(), st); });
    return out.result();
}

// s, q, k, v, idx, cnt, o, lse, ws
LTE_FN(attn_prefill, 9)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const at::Tensor& q = tensor(a[1]);
    const void *qp = ptr(a[1]), *k = ptr(a[2]), *v = ptr(a[3]);
    const int32_t *idx = iptr(a[4]), *cnt = iptr(a[5]);
    Out o(a[6], q.sizes(), q.scalar_type(), q, false), lse(a[7], {s->B, heads_q(s), s->T}, at::kFloat, q);
    Scratch ws(a[8], a[8] == Py_None ? lte_workspace_bytes(LTE_OP_PREFILL, s, nullptr) : 0, q);
    call("lte_attn_prefill", [&](void* st) { return lte_attn_prefill(s, qp, k, v, idx, cnt, o.as<void>(), lse.as<float>(), ws.p(), ws.n(), st); });
    return pack({o.result(), lse.result()});
}

// s, c, k, v, z, idx, cnt, cache
LTE_FN(cache_init, 8)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const lte_conv* c = c_struct<lte_conv>(a[1]);
    const void *k = ptr(a[2]), *v = ptr(a[3]);
    const float* z = (const float*)ptr(a[4]);
    const int32_t *idx = (const int32_t*)ptr(a[5]), *cnt = (const int32_t*)ptr(a[6]);
    void* cache = ptr(a[7]);
    call("lte_cache_init", [&](void* st) { return lte_cache_init(s, c, k, v, z, idx, cnt, cache, st); });
    return Py_NewRef(a[7]);
}

// s, c, cache, q1, k1, v1, o1, lse1
LTE_FN(attn_decode, 8)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const lte_conv* c = c_struct<lte_conv>(a[1]);
    const at::Tensor& q = tensor(a[3]);
    void* cache = ptr(a[2]);
    const void *q1 = ptr(a[3]), *k1 = ptr(a[4]), *v1 = ptr(a[5]);
    Out o(a[6], q.sizes(), q.scalar_type(), q, false), lse(a[7], {s->B, heads_q(s)}, at::kFloat, q);
    call("lte_attn_decode", [&](void* st) { return lte_attn_decode(s, c, cache, q1, k1, v1, o.as<void>(), lse.as<float>(), st); });
    return pack({o.result(), lse.result()});
}

// s, c, cache, n_past, q, k, v, o, lse, ws, flags
LTE_FN(attn_prefill_chunk, 11)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const lte_conv* c = c_struct<lte_conv>(a[1]);
    const long n_past = PyLong_AsLong(a[3]), flags = PyLong_AsLong(a[10]);
    if (PyErr_Occurred()) throw PyFailure();
    const at::Tensor& q = tensor(a[4]);
    void* cache = ptr(a[2]);
    const void *qp = ptr(a[4]), *k = ptr(a[5]), *v = ptr(a[6]);
    Out o(a[7], q.sizes(), q.scalar_type(), q, false), lse(a[8], {s->B, heads_q(s), s->T}, at::kFloat, q);
    Scratch ws(a[9], a[9] == Py_None ? lte_workspace_bytes((flags & LTE_CHUNK_STREAMING) ? LTE_OP_CHUNK_STREAM : LTE_OP_CHUNK, s, c) : 0, q, 256);
    call("lte_attn_prefill_chunk", [&](void* st) {
        return lte_attn_prefill_chunk_ex(s, c, cache, (int32_t)n_past, qp, k, v, o.as<void>(), lse.as<float>(), (uint32_t)flags, ws.p(), ws.n(), st); });
    return pack({o.result(), lse.result()});
}

// s, z, lam, ws
LTE_FN(sparsity_stats, 4)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const at::Tensor& z = tensor(a[1]);
    const float *zp = fptr(a[1]), *lam = fptr(a[2]);
    Out count(Py_None, {s->H}, at::kFloat, z), penalty(Py_None, {1}, at::kFloat, z);
    Scratch ws(a[3], a[3] == Py_None ? lte_workspace_bytes(LTE_OP_STATS, s, nullptr) : 0, z, 256);
    call("lte_sparsity_stats", [&](void* st) { return lte_sparsity_stats(s, zp, lam, count.as<float>(), penalty.as<float>(), ws.p(), ws.n(), st); });
    return pack({count.result(), penalty.result()});
}

// s, c, cache, cos, sin, ws
LTE_FN(cache_score, 6)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const lte_conv* c = c_struct<lte_conv>(a[1]);
    const at::Tensor& like = tensor(a[2]);
    void* cache = ptr(a[2]);
    const float *co = fptr(a[3]), *si = fptr(a[4]);
    const int32_t len = co ? (int32_t)THPVariable_Unpack(a[3]).size(0) : 0;
    Scratch ws(a[5], a[5] == Py_None ? lte_workspace_bytes(LTE_OP_DECODE, s, c) : 0, like, 256);
    call(co ? "lte_cache_score_unrope" : "lte_cache_score", [&](void* st) { return lte_cache_score_unrope(s, c, cache, co, si, len, ws.p(), ws.n(), st); });
    Py_RETURN_NONE;
}

// s, c, q, k, v, o, lse, dO, z, idx, cnt, lam, flags, want_dbias, ws, outs (dq, dk, dv, dw, db or None), built-in scratch
LTE_FN(attn_bwd, 17)
{
    const lte_shape* s = c_struct<lte_shape>(a[0]);
    const lte_conv* c = c_struct<lte_conv>(a[1]);
    const at::Tensor &q = tensor(a[2]), &k = tensor(a[3]);
    const void *qp = ptr(a[2]), *kp = ptr(a[3]), *v = ptr(a[4]), *o = ptr(a[5]), *dO = ptr(a[7]);
    const float *lse = fptr(a[6]), *z = fptr(a[8]), *lam = fptr(a[11]);
    const int32_t *idx = iptr(a[9]), *cnt = iptr(a[10]);
    const unsigned long flags = PyLong_AsUnsignedLong(a[12]);
    if (PyErr_Occurred()) throw PyFailure();
    const bool given = a[15] != Py_None, want_db = a[13] == Py_True;
    if (given && (!PyTuple_Check(a[15]) || PyTuple_GET_SIZE(a[15]) != 5)) fail(PyExc_ValueError, "outs: five tensors (dq, dk, dv, dw, dbias)");
    PyObject* outs[5];
    for (int i = 0; i < 5; ++i) outs[i] = given ? PyTuple_GET_ITEM(a[15], i) : Py_None;
    // the scorer's gradients: [H, K, 2d] and [H], or packed like the three-layer stack's parameters
    const int64_t H = s->H, d = s->d;
    const bool stack = c->n_layers == 3;
    const at::DimVector dw_size = stack ? at::DimVector({H * (d * 3 * 2 * d + (d / 2) * 3 * d + (d / 4) * 3 * (d / 2) + d / 4)}) : at::DimVector({H, c->kernel, 2 * d});
    const int64_t db_size = stack ? H * (d + d / 2 + d / 4 + 1) : H;
    Out dq(outs[0], q.sizes(), q.scalar_type(), q, false), dk(outs[1], k.sizes(), k.scalar_type(), k, false), dv(outs[2], k.sizes(), k.scalar_type(), k, false);
    Out dw(outs[3], dw_size, at::kFloat, q, false);
    std::unique_ptr<Out> db;
    if (given ? outs[4] != Py_None : want_db) db.reset(new Out(outs[4], {db_size}, at::kFloat, q, false));
    float* dbp = db ? db->as<float>() : nullptr;
    if (a[16] == Py_True) {
        call("lte_attn_bwd_static", [&](void* st) {
            return lte_attn_bwd_static(s, c, qp, kp, v, o, lse, dO, z, idx, cnt, lam, dq.as<void>(), dk.as<void>(), dv.as<void>(), dw.as<float>(), dbp,
                                       (uint32_t)flags, st); });
    } else {
        Scratch ws(a[14], a[14] == Py_None ? lte_workspace_bytes(LTE_OP_BWD, s, c) : 0, q, 16);
        call("lte_attn_bwd", [&](void* st) {
            return lte_attn_bwd(s, c, qp, kp, v, o, lse, dO, z, idx, cnt, lam, dq.as<void>(), dk.as<void>(), dv.as<void>(), dw.as<float>(), dbp,
                                (uint32_t)flags, ws.p(), ws.n(), st); });
    }
    return pack({dq.result(), dk.result(), dv.result(), dw.result(), db ? db->result() : Py_NewRef(Py_None)});
}

// the exception class for a call's status
PyObject* set_error(PyObject*, PyObject* cls)
{
    Py_XSETREF(g_error, Py_NewRef(cls));
    Py_RETURN_NONE;
}

#define LTE_DEF(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    LTE_DEF(scores), LTE_DEF(select_rule), LTE_DEF(attn_colsum), LTE_DEF(attn_prefill), LTE_DEF(cache_init), LTE_DEF(attn_decode),
    LTE_DEF(attn_prefill_chunk), LTE_DEF(sparsity_stats), LTE_DEF(cache_score), LTE_DEF(attn_bwd),
    {"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding()
{
    PyObject* m = PyModule_Create(&module);
    if (m) PyModule_AddStringConstant(m, "built_for", LTE_BUILT_FOR);
    return m;
}
