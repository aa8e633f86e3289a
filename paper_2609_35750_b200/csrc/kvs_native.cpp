// The calls of a step and of a generated token as one native function each: tensor checks, output tensors, the C-ABI call.
// By ctypes and torch's Python functions the host took 8 us for an append, 18 for a decode step, 12 for a forward and 26 for a
// backward; a turn of 16 tokens is 33 such calls and was bound by them (4 sequences: 448 -> 262 us), and so is every short step.
// No logic of the path is here: binding.py keeps the names, arguments, defaults and errors, and gives the addresses of the
// C-ABI functions of the library it has loaded.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/DynamicTypes.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "kvs.h"

namespace {

// ---- the loaded library -------------------------------------------------------------------------------------------
#define KVS_FUNCTIONS(X) \
    X(kvs_mask_meta_bytes) X(kvs_mask_meta) X(kvs_mask_meta_keys) X(kvs_mask_meta_evicted) X(kvs_attn_fwd) X(kvs_attn_fwd_packed) \
    X(kvs_attn_fwd_dual) X(kvs_attn_bwd) X(kvs_attn_bwd_packed) X(kvs_attn_bwd_workspace_bytes) X(kvs_permute_rows) X(kvs_rope_qk) \
    X(kvs_cache_append) X(kvs_decode_num_splits) X(kvs_decode_workspace_bytes) X(kvs_decode_attn)
#define KVS_POINTER(name) decltype(&::name) name = nullptr;
struct Library {
    KVS_FUNCTIONS(KVS_POINTER)
};
Library lib;
PyObject* error_class = nullptr;        // binding.KvsError(code, where)

// ---- arguments ----------------------------------------------------------------------------------------------------
struct Raised {};                       // a Python error is set

[[noreturn]] void value_error(const char* format, const char* name) {
    PyErr_Format(PyExc_ValueError, format, name);
    throw Raised();
}
int whole(PyObject* o) {
    PyObject* i = PyNumber_Index(o);
    if (!i) throw Raised();
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    if (PyErr_Occurred()) throw Raised();
    return (int)v;
}
float real(PyObject* o) {
    PyObject* f = PyNumber_Float(o);
    if (!f) throw Raised();
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return (float)v;
}
bool given(PyObject* o) { return o != Py_None; }
const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor", name);
        throw Raised();
    }
    return THPVariable_Unpack(o);
}
void* address(const at::Tensor& t, const char* name, at::ScalarType dtype) {
    if (!t.is_cuda()) value_error("%s must be a CUDA tensor (there is no CPU path)", name);
    if (!t.is_contiguous()) value_error("%s must be contiguous", name);
    if (t.scalar_type() != dtype) {
        PyErr_Format(PyExc_ValueError, "%s must be %S, got %S", name, torch::getTHPDtype(dtype), torch::getTHPDtype(t.scalar_type()));
        throw Raised();
    }
    return t.mutable_data_ptr();
}
void dims(const at::Tensor& t, int64_t n, const char* name) {
    if (t.dim() != n) {
        PyErr_Format(PyExc_ValueError, "%s must have %d dimensions, got %d", name, (int)n, (int)t.dim());
        throw Raised();
    }
}
int64_t size1(const at::Tensor& t, const char* name) {
    if (t.dim() < 2) {
        PyErr_Format(PyExc_IndexError, "%s must have a second dimension", name);
        throw Raised();
    }
    return t.size(1);
}
kvs_stream_t stream_of(PyObject* stream) {
    if (!given(stream)) return (kvs_stream_t)c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(stream, "cuda_stream");
    if (!h) throw Raised();
    void* p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (PyErr_Occurred()) throw Raised();
    return (kvs_stream_t)p;
}
// Allocations, like calls into the library, are made without the interpreter lock: the allocator may wait for the device.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};
at::Tensor empty(at::IntArrayRef sizes, const at::Tensor& like, at::ScalarType dtype) {
    Unlocked u;
    return at::empty(sizes, like.options().dtype(dtype));
}
at::Tensor bytes(size_t n, const at::Tensor& like) { return empty({(int64_t)n}, like, at::kByte); }
// the tensor given, or a new one
at::Tensor out_of(PyObject* o, const char* name, at::IntArrayRef sizes, const at::Tensor& like, at::ScalarType dtype) {
    return given(o) ? tensor(o, name) : empty(sizes, like, dtype);
}
at::Tensor out_of(PyObject* o, const char* name, const at::Tensor& like) {
    if (given(o)) return tensor(o, name);
    Unlocked u;
    return at::empty_like(like);
}

void check(int code, const char* where) {
    if (code == KVS_OK) return;
    PyObject* e = PyObject_CallFunction(error_class, "is", code, where);
    if (e) {
        PyErr_SetObject(error_class, e);
        Py_DECREF(e);
    }
    throw Raised();
}
// a call into the library
template <typename F>
void call(const char* where, F f) {
    int rc;
    {
        Unlocked u;
        rc = f();
    }
    check(rc, where);
}
PyObject* wrap(const at::Tensor& t, PyObject* o) {
    if (given(o)) {
        Py_INCREF(o);
        return o;
    }
    return THPVariable_Wrap(t);
}
PyObject* tuple(std::initializer_list<PyObject*> items) {
    PyObject* t = PyTuple_New((Py_ssize_t)items.size());
    Py_ssize_t i = 0;
    for (PyObject* o : items) {
        if (!o || !t) {
            for (PyObject* x : items) Py_XDECREF(x);
            Py_XDECREF(t);
            throw Raised();
        }
        ++i;
    }
    i = 0;
    for (PyObject* o : items) PyTuple_SET_ITEM(t, i++, o);
    return t;
}

// ---- the calls: positional arguments, None for what is left out -----------------------------------------------------
constexpr auto BF16 = at::kBFloat16;
constexpr auto F32 = at::kFloat;
constexpr auto I32 = at::kInt;
constexpr auto U8 = at::kByte;

// (what, first, evict, cu_seqlens, max_seqlen, meta_buf, stream): what 0 plain, 1 keys, 2 evicted
PyObject* mask_meta(PyObject* const* a) {
    const int what = whole(a[0]), max_seqlen = whole(a[4]);
    const char* name = what == 0 ? "evict_at" : "key_evict";
    const at::Tensor &evict = tensor(a[2], name), &cu = tensor(a[3], "cu_seqlens");
    const int batch = (int)(cu.numel() - 1), total = (int)evict.numel();
    const at::Tensor meta = given(a[5]) ? tensor(a[5], "meta_buf") : bytes(lib.kvs_mask_meta_bytes(batch, total, max_seqlen), evict);
    const int32_t* first = what == 1 ? (const int32_t*)address(tensor(a[1], "key_first"), "key_first", I32) : nullptr;
    const int32_t *e = (const int32_t*)address(evict, name, I32), *c = (const int32_t*)address(cu, "cu_seqlens", I32);
    void* m = address(meta, "meta_buf", U8);
    const size_t n = (size_t)meta.numel();
    const kvs_stream_t st = stream_of(a[6]);
    if (what == 1) call("kvs_mask_meta_keys", [&] { return lib.kvs_mask_meta_keys(first, e, c, batch, total, max_seqlen, m, n, st); });
    else if (what == 2) call("kvs_mask_meta_evicted", [&] { return lib.kvs_mask_meta_evicted(e, c, batch, total, max_seqlen, m, n, st); });
    else call("kvs_mask_meta", [&] { return lib.kvs_mask_meta(e, c, batch, total, max_seqlen, m, n, st); });
    return wrap(meta, a[5]);
}

// (q, k, v, meta, batch, max_seqlen, scale, out, lse, stream)
PyObject* attn_fwd(PyObject* const* a) {
    const at::Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v"), &meta = tensor(a[3], "meta_buf");
    dims(q, 3, "q");
    const int total = (int)q.size(0), Hq = (int)q.size(1), d = (int)q.size(2), Hkv = (int)size1(k, "k");
    const int batch = whole(a[4]), max_seqlen = whole(a[5]);
    const float scale = real(a[6]);
    const at::Tensor out = out_of(a[7], "out", q);
    const at::Tensor lse = out_of(a[8], "lse", {Hq, total}, q, F32);
    void *pq = address(q, "q", BF16), *pk = address(k, "k", BF16), *pv = address(v, "v", BF16), *pm = address(meta, "meta_buf", U8),
         *po = address(out, "out", BF16);
    float* pl = (float*)address(lse, "lse", F32);
    const kvs_stream_t st = stream_of(a[9]);
    call("kvs_attn_fwd", [&] { return lib.kvs_attn_fwd(pq, pk, pv, pm, batch, total, max_seqlen, Hq, Hkv, d, scale, po, pl, st); });
    return tuple({wrap(out, a[7]), wrap(lse, a[8])});
}

// (qkv, meta, batch, max_seqlen, Hq, Hkv, scale, out, lse, stream)
PyObject* attn_fwd_packed(PyObject* const* a) {
    const at::Tensor &qkv = tensor(a[0], "qkv"), &meta = tensor(a[1], "meta_buf");
    dims(qkv, 3, "qkv");
    const int total = (int)qkv.size(0), d = (int)qkv.size(2), batch = whole(a[2]), max_seqlen = whole(a[3]), Hq = whole(a[4]), Hkv = whole(a[5]);
    if (qkv.size(1) != (int64_t)Hq + 2 * (int64_t)Hkv) value_error("%s must have Hq + 2 Hkv heads", "qkv");
    const float scale = real(a[6]);
    const at::Tensor out = out_of(a[7], "out", {total, Hq, d}, qkv, BF16), lse = out_of(a[8], "lse", {Hq, total}, qkv, F32);
    void *pq = address(qkv, "qkv", BF16), *pm = address(meta, "meta_buf", U8), *po = address(out, "out", BF16);
    float* pl = (float*)address(lse, "lse", F32);
    const kvs_stream_t st = stream_of(a[9]);
    call("kvs_attn_fwd_packed", [&] { return lib.kvs_attn_fwd_packed(pq, pm, batch, total, max_seqlen, Hq, Hkv, d, scale, po, pl, st); });
    return tuple({wrap(out, a[7]), wrap(lse, a[8])});
}

// (q, k, v, meta_student, meta_evicted, batch, max_seqlen, scale, out_student, lse_student, out_teacher, lse_teacher, stream)
PyObject* attn_fwd_dual(PyObject* const* a) {
    const at::Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v"), &ms = tensor(a[3], "meta_student"),
                     &me = tensor(a[4], "meta_evicted");
    dims(q, 3, "q");
    const int total = (int)q.size(0), Hq = (int)q.size(1), d = (int)q.size(2), Hkv = (int)size1(k, "k");
    const int batch = whole(a[5]), max_seqlen = whole(a[6]);
    const float scale = real(a[7]);
    const at::Tensor os = out_of(a[8], "out_student", q), ls = out_of(a[9], "lse_student", {Hq, total}, q, F32),
                     ot = out_of(a[10], "out_teacher", q), lt = out_of(a[11], "lse_teacher", {Hq, total}, q, F32);
    void *pq = address(q, "q", BF16), *pk = address(k, "k", BF16), *pv = address(v, "v", BF16), *pms = address(ms, "meta_student", U8),
         *pme = address(me, "meta_evicted", U8), *pos = address(os, "out_student", BF16), *pot = address(ot, "out_teacher", BF16);
    float *pls = (float*)address(ls, "lse_student", F32), *plt = (float*)address(lt, "lse_teacher", F32);
    const kvs_stream_t st = stream_of(a[12]);
    call("kvs_attn_fwd_dual", [&] {
        return lib.kvs_attn_fwd_dual(pq, pk, pv, pms, pme, batch, total, max_seqlen, Hq, Hkv, d, scale, pos, pls, pot, plt, st);
    });
    return tuple({wrap(os, a[8]), wrap(ls, a[9]), wrap(ot, a[10]), wrap(lt, a[11])});
}

// (dout, q, k, v, out, lse, meta, batch, max_seqlen, scale, grad_dtype, dq, dk, dv, workspace, stream)
PyObject* attn_bwd(PyObject* const* a) {
    const at::Tensor &dout = tensor(a[0], "dout"), &q = tensor(a[1], "q"), &k = tensor(a[2], "k"), &v = tensor(a[3], "v"), &out = tensor(a[4], "out"),
                     &lse = tensor(a[5], "lse"), &meta = tensor(a[6], "meta_buf");
    dims(q, 3, "q");
    const int total = (int)q.size(0), Hq = (int)q.size(1), d = (int)q.size(2), Hkv = (int)size1(k, "k");
    const int batch = whole(a[7]), max_seqlen = whole(a[8]), grad = whole(a[10]);
    const float scale = real(a[9]);
    const at::ScalarType gdt = grad == KVS_GRAD_FP32 ? F32 : BF16;
    const at::Tensor dq = out_of(a[11], "dq", q.sizes(), q, gdt), dk = out_of(a[12], "dk", k.sizes(), q, gdt), dv = out_of(a[13], "dv", v.sizes(), q, gdt);
    const at::Tensor ws = given(a[14]) ? tensor(a[14], "workspace") : bytes(lib.kvs_attn_bwd_workspace_bytes(total, Hq, Hkv, d, grad), q);
    void *pdo = address(dout, "dout", BF16), *pq = address(q, "q", BF16), *pk = address(k, "k", BF16), *pv = address(v, "v", BF16),
         *po = address(out, "out", BF16), *pm = address(meta, "meta_buf", U8), *pdq = address(dq, "dq", gdt), *pdk = address(dk, "dk", gdt),
         *pdv = address(dv, "dv", gdt), *pw = address(ws, "workspace", U8);
    const float* pl = (const float*)address(lse, "lse", F32);
    const size_t wn = (size_t)ws.numel();
    const kvs_stream_t st = stream_of(a[15]);
    call("kvs_attn_bwd", [&] {
        return lib.kvs_attn_bwd(pdo, pq, pk, pv, po, pl, pm, batch, total, max_seqlen, Hq, Hkv, d, scale, grad, pdq, pdk, pdv, pw, wn, st);
    });
    return tuple({wrap(dq, a[11]), wrap(dk, a[12]), wrap(dv, a[13])});
}

// (dout, qkv, out, lse, meta, batch, max_seqlen, Hq, Hkv, scale, grad_dtype, dqkv, workspace, stream)
PyObject* attn_bwd_packed(PyObject* const* a) {
    const at::Tensor &dout = tensor(a[0], "dout"), &qkv = tensor(a[1], "qkv"), &out = tensor(a[2], "out"), &lse = tensor(a[3], "lse"),
                     &meta = tensor(a[4], "meta_buf");
    dims(qkv, 3, "qkv");
    const int total = (int)qkv.size(0), d = (int)qkv.size(2), batch = whole(a[5]), max_seqlen = whole(a[6]), Hq = whole(a[7]), Hkv = whole(a[8]),
              grad = whole(a[10]);
    const float scale = real(a[9]);
    const at::ScalarType gdt = grad == KVS_GRAD_FP32 ? F32 : BF16;
    const at::Tensor dqkv = out_of(a[11], "dqkv", qkv.sizes(), qkv, gdt);
    const at::Tensor ws = given(a[12]) ? tensor(a[12], "workspace") : bytes(lib.kvs_attn_bwd_workspace_bytes(total, Hq, Hkv, d, grad), qkv);
    void *pdo = address(dout, "dout", BF16), *pq = address(qkv, "qkv", BF16), *po = address(out, "out", BF16), *pm = address(meta, "meta_buf", U8),
         *pg = address(dqkv, "dqkv", gdt), *pw = address(ws, "workspace", U8);
    const float* pl = (const float*)address(lse, "lse", F32);
    const size_t wn = (size_t)ws.numel();
    const kvs_stream_t st = stream_of(a[13]);
    call("kvs_attn_bwd_packed", [&] {
        return lib.kvs_attn_bwd_packed(pdo, pq, po, pl, pm, batch, total, max_seqlen, Hq, Hkv, d, scale, grad, pg, pw, wn, st);
    });
    return wrap(dqkv, a[11]);
}

// (src, perm, dst, inverse, stream)
PyObject* permute_rows(PyObject* const* a) {
    const at::Tensor &src = tensor(a[0], "src"), &perm = tensor(a[1], "perm");
    const at::Tensor dst = out_of(a[2], "dst", src);
    const int inverse = PyObject_IsTrue(a[3]);
    if (inverse < 0) throw Raised();
    if (src.dim() < 1) {
        PyErr_SetString(PyExc_IndexError, "src must have a leading dimension");
        throw Raised();
    }
    const long long n = src.size(0), row_bytes = (long long)(src.numel() / (n > 0 ? n : 1)) * (long long)src.element_size();
    if (!src.is_cuda() || !src.is_contiguous() || !dst.is_contiguous() || dst.sizes() != src.sizes() || dst.scalar_type() != src.scalar_type())
        value_error("%s must be contiguous CUDA tensors of the same shape and dtype", "src and dst");
    const void* ps = src.const_data_ptr();
    void* pd = dst.mutable_data_ptr();
    const int32_t* pp = (const int32_t*)address(perm, "perm", I32);
    const kvs_stream_t st = stream_of(a[4]);
    call("kvs_permute_rows", [&] { return lib.kvs_permute_rows(ps, pp, pd, n, row_bytes, inverse, st); });
    return wrap(dst, a[2]);
}

// (q, k, cu_seqlens, positions, theta_base, inverse, q_out, k_out, stream)
PyObject* rope_qk(PyObject* const* a) {
    const at::Tensor& ref = tensor(given(a[0]) ? a[0] : a[1], given(a[0]) ? "q" : "k");
    dims(ref, 3, given(a[0]) ? "q" : "k");
    const int total = (int)ref.size(0), d = (int)ref.size(2);
    const at::ScalarType dt = ref.scalar_type();
    if (dt != BF16 && dt != F32) {
        PyErr_Format(PyExc_ValueError, "%s must be torch.bfloat16 or torch.float32, got %S", given(a[0]) ? "q" : "k", torch::getTHPDtype(dt));
        throw Raised();
    }
    const float theta = real(a[4]);
    const int inverse = PyObject_IsTrue(a[5]);
    if (inverse < 0) throw Raised();
    const char* names[4] = {"q", "k", "q_out", "k_out"};
    at::Tensor out[2];
    void* p[4] = {nullptr, nullptr, nullptr, nullptr};
    int heads[2] = {0, 0};
    for (int i = 0; i < 2; ++i) {
        if (given(a[i])) {
            const at::Tensor& t = tensor(a[i], names[i]);
            heads[i] = (int)size1(t, names[i]);
            out[i] = out_of(a[6 + i], names[2 + i], t);
            p[i] = address(t, names[i], dt);
            p[2 + i] = address(out[i], names[2 + i], dt);
        } else if (given(a[6 + i])) {
            p[2 + i] = address(tensor(a[6 + i], names[2 + i]), names[2 + i], dt);
        }
    }
    const int32_t* pos = given(a[3]) ? (const int32_t*)address(tensor(a[3], "positions"), "positions", I32) : nullptr;
    const int32_t* cu = given(a[2]) ? (const int32_t*)address(tensor(a[2], "cu_seqlens"), "cu_seqlens", I32) : nullptr;
    const int batch = cu ? (int)(tensor(a[2], "cu_seqlens").numel() - 1) : 0;
    const kvs_stream_t st = stream_of(a[8]);
    const int grad = dt == F32 ? KVS_GRAD_FP32 : KVS_GRAD_BF16;
    call("kvs_rope_qk", [&] {
        return lib.kvs_rope_qk(p[0], p[1], pos, cu, batch, total, heads[0], heads[1], d, theta, grad, inverse, p[2], p[3], st);
    });
    auto result = [&](int i) {
        if (given(a[i]) || given(a[6 + i])) return wrap(out[i], a[6 + i]);
        Py_INCREF(Py_None);
        return Py_None;
    };
    return tuple({result(0), result(1)});
}

// (k_new, v_new, active, num_seqs, Hkv, d, page_size, max_pages, num_pages, block_table, n_tokens, free_list, k_cache, v_cache, stream)
PyObject* cache_append(PyObject* const* a) {
    const void *k = address(tensor(a[0], "k_new"), "k_new", BF16), *v = address(tensor(a[1], "v_new"), "v_new", BF16);
    const uint8_t* active = given(a[2]) ? (const uint8_t*)address(tensor(a[2], "active"), "active", U8) : nullptr;
    int n[6];
    for (int i = 0; i < 6; ++i) n[i] = whole(a[3 + i]);
    void* p[5];
    for (int i = 0; i < 5; ++i) p[i] = tensor(a[9 + i], "a buffer of the cache").mutable_data_ptr();
    const kvs_stream_t st = stream_of(a[14]);
    call("kvs_cache_append", [&] {
        return lib.kvs_cache_append(k, v, active, n[0], n[1], n[2], n[3], n[4], n[5], (int32_t*)p[0], (int32_t*)p[1], (int32_t*)p[2], p[3], p[4], st);
    });
    Py_RETURN_NONE;
}

// (q, scale, num_splits, out, lse, workspace, most_tokens, Hkv, page_size, max_pages, num_pages, block_table, n_tokens, k_cache, v_cache, stream)
PyObject* decode(PyObject* const* a) {
    const at::Tensor& q = tensor(a[0], "q");
    dims(q, 3, "q");
    const int S = (int)q.size(0), Hq = (int)q.size(1), d = (int)q.size(2), Hkv = whole(a[7]);
    const float scale = real(a[1]);
    int splits = whole(a[2]);
    if (splits <= 0) splits = lib.kvs_decode_num_splits(S, Hkv, whole(a[6]));
    const at::Tensor ws = given(a[5]) ? tensor(a[5], "workspace") : bytes(lib.kvs_decode_workspace_bytes(S, Hq, d, splits), q);
    const at::Tensor out = out_of(a[3], "out", q), lse = out_of(a[4], "lse", {S, Hq}, q, F32);
    const void* pq = address(q, "q", BF16);
    void *po = address(out, "out", BF16), *pw = address(ws, "workspace", U8);
    float* pl = (float*)address(lse, "lse", F32);
    int n[3];
    for (int i = 0; i < 3; ++i) n[i] = whole(a[8 + i]);
    void* p[4];
    for (int i = 0; i < 4; ++i) p[i] = tensor(a[11 + i], "a buffer of the cache").mutable_data_ptr();
    const size_t wn = (size_t)ws.numel();
    const kvs_stream_t st = stream_of(a[15]);
    call("kvs_decode_attn", [&] {
        return lib.kvs_decode_attn(pq, p[2], p[3], (const int32_t*)p[0], (const int32_t*)p[1], S, Hq, Hkv, d, n[0], n[1], n[2], scale, splits, po, pl,
                                   pw, wn, st);
    });
    return tuple({wrap(out, a[3]), wrap(lse, a[4])});
}

// ---- the module ---------------------------------------------------------------------------------------------------
// A call's C++ errors (torch's among them) become Python errors, as torch's own functions have them.
template <PyObject* (*F)(PyObject* const*), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %d", N, (int)n);
        return nullptr;
    }
    if (!error_class) {
        PyErr_SetString(PyExc_RuntimeError, "no library: binding.load() comes first");
        return nullptr;
    }
    try {
        return F(args);
    } catch (const Raised&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// bind({name: address}, error_class)
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 2 || !PyDict_Check(args[0])) {
        PyErr_SetString(PyExc_TypeError, "bind(addresses, error_class)");
        return nullptr;
    }
    Library l;
#define KVS_BIND(name)                                                    \
    {                                                                     \
        PyObject* o = PyDict_GetItemString(args[0], #name);               \
        void* p = o ? PyLong_AsVoidPtr(o) : nullptr;                      \
        if (!p) {                                                         \
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_KeyError, #name); \
            return nullptr;                                               \
        }                                                                 \
        l.name = (decltype(l.name))p;                                     \
    }
    KVS_FUNCTIONS(KVS_BIND)
    lib = l;
    Py_INCREF(args[1]);
    Py_XSETREF(error_class, args[1]);
    Py_RETURN_NONE;
}

#define KVS_ENTRY(name, n) {#name, (PyCFunction)(void (*)(void)) & entry<name, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void)) & bind, METH_FASTCALL, nullptr},
    KVS_ENTRY(mask_meta, 7),
    KVS_ENTRY(attn_fwd, 10),
    KVS_ENTRY(attn_fwd_packed, 10),
    KVS_ENTRY(attn_fwd_dual, 13),
    KVS_ENTRY(attn_bwd, 16),
    KVS_ENTRY(attn_bwd_packed, 14),
    KVS_ENTRY(permute_rows, 5),
    KVS_ENTRY(rope_qk, 9),
    KVS_ENTRY(cache_append, 15),
    KVS_ENTRY(decode, 16),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_kvs_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__kvs_native() { return PyModule_Create(&module); }
