// Argument marshalling of binding.py in native code: tensors, ctypes structures and numbers -> one call of the C ABI.
//
// What bounds it: the layer-step of one short sequence is about 10 us on the GPU, and reading some twenty-five
// pointers, strides and sizes through Python attributes and ctypes kept the host busy for longer than that, so eager
// steps were host-bound.  Here a pointer is one load from the tensor's C++ object.  Measured (eager calls back to back,
// one sequence of 4096 tokens): 13.9 us per ha_sparse_decode before, of which the GPU needed 10.5; 5.0 us of host time
// now, launch included, so the GPU is what is waited for.
//
// Every function takes the Python wrapper's arguments positionally and returns the C status; wrong types raise the
// exceptions the wrappers documented (TypeError, ValueError, AssertionError).  The GIL is released around the C call, as
// ctypes does.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/TensorBase.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <string>

#include "hashattn.h"

namespace {

struct Raised {};   // a Python exception is set

[[noreturn]] void raise(PyObject *type, const std::string &what) {
    PyErr_SetString(type, what.c_str());
    throw Raised{};
}

const at::Tensor &tensor(PyObject *o) {
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string("expected a torch tensor, got ") + Py_TYPE(o)->tp_name);
    return THPVariable_Unpack(o);
}
template <typename T>
T *ptr(PyObject *o) { return reinterpret_cast<T *>(tensor(o).data_ptr()); }
template <typename T>
T *ptr_or_null(PyObject *o) { return o == Py_None ? nullptr : ptr<T>(o); }

int32_t i32(PyObject *o) {
    const unsigned long v = PyLong_Check(o) ? PyLong_AsUnsignedLongMask(o) : (unsigned long)PyNumber_AsSsize_t(o, PyExc_OverflowError);
    if (v == (unsigned long)-1 && PyErr_Occurred()) throw Raised{};
    return (int32_t)v;
}

// A ctypes structure's memory.  The object outlives the call (the caller's frame holds it), so the view is released at once.
template <typename T>
const T *structure(PyObject *o) {
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Raised{};
    const T *p = reinterpret_cast<const T *>(view.buf);
    const bool fits = view.len >= (Py_ssize_t)sizeof(T);
    PyBuffer_Release(&view);
    if (!fits) raise(PyExc_TypeError, "structure too small");
    return p;
}
PyObject *g_struct_name = nullptr;
// The ha_mapping of a Mapping / MappingWide object (its `struct` attribute, which the object keeps alive); None -> NULL.
const ha_mapping *mapping(PyObject *o) {
    if (o == Py_None) return nullptr;
    PyObject *s = PyObject_GetAttr(o, g_struct_name);
    if (!s) throw Raised{};
    const ha_mapping *m = nullptr;
    try {
        m = structure<ha_mapping>(s);
    } catch (...) {
        Py_DECREF(s);
        throw;
    }
    Py_DECREF(s);
    return m;
}

// bf16 [B,H,N,128] or [B,H,128] on the device -> ha_tensor (binding.make_tensor)
ha_tensor view(const at::Tensor &t) {
    if (!t.is_cuda() || t.scalar_type() != at::kBFloat16)
        raise(PyExc_TypeError, "tensor: expected a CUDA tensor of torch.bfloat16");
    const auto n = t.dim();
    if ((n != 3 && n != 4) || t.stride(n - 1) != 1) raise(PyExc_ValueError, "expected [B,H,N,128] with a contiguous last dimension");
    ha_tensor r;
    r.ptr = t.data_ptr();
    r.stride_b = t.stride(0);
    r.stride_h = t.stride(1);
    // one token per head: the token stride is never used, but has to be a valid one
    if (n == 3) r.stride_n = t.size(2) * t.stride(2) > 128 ? t.size(2) * t.stride(2) : 128;
    else r.stride_n = t.size(2) > 1 ? t.stride(2) : (t.stride(2) > 128 ? t.stride(2) : 128);
    return r;
}
ha_tensor view(PyObject *o) { return view(tensor(o)); }

void device_type(const at::Tensor &t, at::ScalarType type, const char *name) {
    if (!t.is_cuda() || t.scalar_type() != type) raise(PyExc_TypeError, std::string(name) + ": expected a CUDA tensor of another type");
}
void require(bool ok, const char *what) {
    if (!ok) raise(PyExc_AssertionError, what);
}

PyObject *g_stream_name = nullptr;
// None: torch's current stream on the current device; a torch stream; or the handle as a number
void *stream(PyObject *o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *h = PyObject_GetAttr(o, g_stream_name);
    if (!h) {
        PyErr_Clear();
        h = PyNumber_Long(o);
        if (!h) throw Raised{};
    }
    void *p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!p && PyErr_Occurred()) throw Raised{};
    return p;
}

struct Workspace {
    void *p;
    size_t n;
};
Workspace workspace(PyObject *o) {
    const at::Tensor &t = tensor(o);
    return {t.data_ptr(), (size_t)t.numel() * t.element_size()};
}
// [rows][row][...] output or signature tensor with its two leading strides
template <typename T>
struct Rows {
    T *p;
    int64_t s0, s1;
};
template <typename T>
Rows<T> rows(PyObject *o) {
    const at::Tensor &t = tensor(o);
    return {reinterpret_cast<T *>(t.data_ptr()), t.stride(0), t.stride(1)};
}
// int32 [n_pages, Hkv, page_size] signature pool (binding._pool)
struct Pool {
    uint32_t *p;
    int64_t page, head;
    int32_t size;
};
Pool pool(PyObject *o) {
    const at::Tensor &t = tensor(o);
    device_type(t, at::kInt, "code_pool");
    require(t.dim() == 3 && t.stride(2) == 1, "code_pool: expected int32 [n_pages, Hkv, page_size]");
    return {reinterpret_cast<uint32_t *>(t.data_ptr()), t.stride(0), t.stride(1), (int32_t)t.size(2)};
}
struct Table {
    const int32_t *p;
    int64_t s0;
};
Table table(PyObject *o) {
    const at::Tensor &t = tensor(o);
    return {reinterpret_cast<const int32_t *>(t.data_ptr()), t.stride(0)};
}
const uint16_t *host(PyObject *o) {
    const at::Tensor &t = tensor(o);
    if (t.is_cuda() || !t.is_contiguous()) raise(PyExc_TypeError, "host buffers must be contiguous CPU tensors");
    return reinterpret_cast<const uint16_t *>(t.data_ptr());
}

template <typename F>
PyObject *guarded(Py_ssize_t got, Py_ssize_t want, F body) {
    if (got != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
        return nullptr;
    }
    try {
        return PyLong_FromLong(body());
    } catch (const Raised &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <typename F>
int unlocked(F call) {
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = call();
    Py_END_ALLOW_THREADS
    return st;
}

#define HA_FN(name) PyObject *name(PyObject *, PyObject *const *a, Py_ssize_t n)

// ---------------------------------------------------------------- ENCODE

// mapping, heads_per_kv, x, codes, slot, stream
HA_FN(encode) {
    return guarded(n, 6, [&] {
        const at::Tensor &x = tensor(a[2]), &c = tensor(a[3]);
        const ha_tensor xt = view(x);
        const int32_t B = x.size(0), H = x.size(1), T = x.dim() == 3 ? 1 : x.size(2);
        device_type(c, at::kInt, "codes");
        require(c.dim() == 3 && c.stride(2) == 1, "codes: expected int32 [B,H,T] with a contiguous last dimension");
        const ha_mapping *m = mapping(a[0]);
        const int32_t hpk = i32(a[1]);
        const int32_t *slot = ptr_or_null<const int32_t>(a[4]);
        void *st = stream(a[5]);
        return unlocked([&] {
            return ha_encode(m, hpk, &xt, B, H, T, reinterpret_cast<uint32_t *>(c.data_ptr()), c.stride(0), c.stride(1), slot, st);
        });
    });
}

// mapping, heads_per_kv, x, codes, path, workspace, stream
HA_FN(encode_prefill) {
    return guarded(n, 7, [&] {
        const at::Tensor &x = tensor(a[2]), &c = tensor(a[3]);
        const ha_tensor xt = view(x);
        const int32_t B = x.size(0), H = x.size(1), T = x.dim() == 3 ? 1 : x.size(2);
        device_type(c, at::kInt, "codes");
        require(c.dim() == 3 && c.stride(2) == 1, "codes: expected int32 [B,H,T] with a contiguous last dimension");
        const ha_mapping *m = mapping(a[0]);
        const int32_t hpk = i32(a[1]), path = i32(a[4]);
        void *ws = ptr_or_null<void>(a[5]), *st = stream(a[6]);
        return unlocked([&] {
            return ha_encode_prefill(m, hpk, &xt, B, H, T, reinterpret_cast<uint32_t *>(c.data_ptr()), c.stride(0), c.stride(1), path,
                                     ws, st);
        });
    });
}

// mapping, heads_per_kv, x, codes, n_bits, slot, stream
HA_FN(encode_wide) {
    return guarded(n, 7, [&] {
        const at::Tensor &x = tensor(a[2]), &c = tensor(a[3]);
        const ha_tensor xt = view(x);
        const int32_t B = x.size(0), H = x.size(1), T = x.dim() == 3 ? 1 : x.size(2);
        device_type(c, at::kLong, "codes");
        require(c.dim() == 4 && c.stride(3) == 1 && c.stride(2) == c.size(3) && c.size(3) == i32(a[4]) / 64,
                "codes: expected int64 [B,H,T,n_bits/64], contiguous per token");
        const ha_mapping *m = mapping(a[0]);
        const int32_t hpk = i32(a[1]);
        const int32_t *slot = ptr_or_null<const int32_t>(a[5]);
        void *st = stream(a[6]);
        return unlocked([&] {
            return ha_encode_wide(m, hpk, &xt, B, H, T, reinterpret_cast<uint64_t *>(c.data_ptr()), c.stride(0), c.stride(1), slot, st);
        });
    });
}

// mapping, k_new, code_pool, block_table, seq_lens, stream
HA_FN(encode_append_paged) {
    return guarded(n, 6, [&] {
        const Pool cp = pool(a[2]);
        const at::Tensor &x = tensor(a[1]);
        device_type(x, at::kBFloat16, "k_new");
        require(x.is_contiguous(), "k_new: expected a contiguous tensor");
        const Table bt = table(a[3]);
        const ha_mapping *m = mapping(a[0]);
        const int32_t *lens = ptr<const int32_t>(a[4]);
        void *st = stream(a[5]);
        return unlocked([&] {
            return ha_encode_append_paged(m, reinterpret_cast<const uint16_t *>(x.data_ptr()), (int32_t)x.size(0), cp.p, cp.page, cp.head,
                                          bt.p, bt.s0, cp.size, lens, st);
        });
    });
}

// ---------------------------------------------------------------- SCORE + TOPK

// shape, q_codes, k_codes, seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, idx, count, workspace, hist_out, stream
HA_FN(score_topk) {
    return guarded(n, 13, [&] {
        const ha_shape *s = structure<ha_shape>(a[0]);
        const uint32_t *q = ptr<const uint32_t>(a[1]);
        const Rows<const uint32_t> kc = rows<const uint32_t>(a[2]);
        const int32_t *lens = ptr<const int32_t>(a[3]), *ks = ptr_or_null<const int32_t>(a[4]);
        const int32_t ku = i32(a[5]), nmax = i32(a[6]), kmax = i32(a[7]);
        const Rows<int32_t> idx = rows<int32_t>(a[8]);
        int32_t *cnt = ptr<int32_t>(a[9]), *hist = ptr_or_null<int32_t>(a[11]);
        const Workspace w = workspace(a[10]);
        void *st = stream(a[12]);
        return unlocked([&] {
            return ha_score_topk(s, q, kc.p, kc.s0, kc.s1, lens, ks, ku, nmax, kmax, idx.p, idx.s0, idx.s1, cnt, hist, w.p, w.n, st);
        });
    });
}

// shape, q_codes, k_codes, seq_lens, k_per_seq, k_uniform, k_max, idx, count, hist_out, stream
template <decltype(&ha_score_topk_sum) kEntry>
HA_FN(score_topk_no_workspace) {
    return guarded(n, 11, [&] {
        const ha_shape *s = structure<ha_shape>(a[0]);
        const uint32_t *q = ptr<const uint32_t>(a[1]);
        const Rows<const uint32_t> kc = rows<const uint32_t>(a[2]);
        const int32_t *lens = ptr<const int32_t>(a[3]), *ks = ptr_or_null<const int32_t>(a[4]);
        const int32_t ku = i32(a[5]), kmax = i32(a[6]);
        const Rows<int32_t> idx = rows<int32_t>(a[7]);
        int32_t *cnt = ptr<int32_t>(a[8]), *hist = ptr_or_null<int32_t>(a[9]);
        void *st = stream(a[10]);
        return unlocked([&] { return kEntry(s, q, kc.p, kc.s0, kc.s1, lens, ks, ku, kmax, idx.p, idx.s0, idx.s1, cnt, hist, st); });
    });
}

// shape, q_codes, code_pool, block_table, seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, idx, count, workspace, hist_out, stream
template <decltype(&ha_score_topk_paged) kEntry>
HA_FN(score_topk_paged) {
    return guarded(n, 14, [&] {
        const ha_shape *s = structure<ha_shape>(a[0]);
        const uint32_t *q = ptr<const uint32_t>(a[1]);
        const Pool cp = pool(a[2]);
        const Table bt = table(a[3]);
        const int32_t *lens = ptr<const int32_t>(a[4]), *ks = ptr_or_null<const int32_t>(a[5]);
        const int32_t ku = i32(a[6]), nmax = i32(a[7]), kmax = i32(a[8]);
        const Rows<int32_t> idx = rows<int32_t>(a[9]);
        int32_t *cnt = ptr<int32_t>(a[10]), *hist = ptr_or_null<int32_t>(a[12]);
        const Workspace w = workspace(a[11]);
        void *st = stream(a[13]);
        return unlocked([&] {
            return kEntry(s, q, cp.p, cp.page, cp.head, bt.p, bt.s0, cp.size, lens, ks, ku, nmax, kmax, idx.p, idx.s0, idx.s1, cnt, hist,
                          w.p, w.n, st);
        });
    });
}

// shape, n_bits, q_codes, k_codes, seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, idx, count, workspace, hist_out, stream
HA_FN(score_topk_wide) {
    return guarded(n, 14, [&] {
        const ha_shape *s = structure<ha_shape>(a[0]);
        const int32_t bits = i32(a[1]);
        const at::Tensor &q = tensor(a[2]), &kc = tensor(a[3]);
        device_type(q, at::kLong, "q_codes");
        device_type(kc, at::kLong, "k_codes");
        require(q.is_contiguous() && kc.dim() == 4 && kc.stride(3) == 1 && kc.stride(2) == kc.size(3),
                "signatures: expected contiguous q_codes and k_codes int64 [B,Hkv,N,n_bits/64], contiguous per token");
        const int32_t *lens = ptr<const int32_t>(a[4]), *ks = ptr_or_null<const int32_t>(a[5]);
        const int32_t ku = i32(a[6]), nmax = i32(a[7]), kmax = i32(a[8]);
        const Rows<int32_t> idx = rows<int32_t>(a[9]);
        int32_t *cnt = ptr<int32_t>(a[10]), *hist = ptr_or_null<int32_t>(a[12]);
        const Workspace w = workspace(a[11]);
        void *st = stream(a[13]);
        return unlocked([&] {
            return ha_score_topk_wide(s, bits, reinterpret_cast<const uint64_t *>(q.data_ptr()),
                                      reinterpret_cast<const uint64_t *>(kc.data_ptr()), kc.stride(0), kc.stride(1), lens, ks, ku, nmax,
                                      kmax, idx.p, idx.s0, idx.s1, cnt, hist, w.p, w.n, st);
        });
    });
}

// ---------------------------------------------------------------- attention

// shape, q, K, V, seq_lens, idx, count, k_max, out, workspace, lse, stream
template <decltype(&ha_gather_attn) kEntry>
HA_FN(gather_attn) {
    return guarded(n, 12, [&] {
        const ha_shape *s = structure<ha_shape>(a[0]);
        const uint16_t *q = ptr<const uint16_t>(a[1]);
        const ha_tensor K = view(a[2]), V = view(a[3]);
        const int32_t *lens = ptr<const int32_t>(a[4]);
        const Rows<const int32_t> idx = rows<const int32_t>(a[5]);
        const int32_t *cnt = ptr<const int32_t>(a[6]);
        const int32_t kmax = i32(a[7]);
        uint16_t *out = ptr<uint16_t>(a[8]);
        const Workspace w = workspace(a[9]);
        float *lse = ptr_or_null<float>(a[10]);
        void *st = stream(a[11]);
        return unlocked([&] { return kEntry(s, q, &K, &V, lens, idx.p, idx.s0, idx.s1, cnt, kmax, out, lse, w.p, w.n, st); });
    });
}

// shape, q, K_pool, V_pool, block_table, page_size, seq_lens, idx, count, k_max, out, workspace, lse, stream
template <decltype(&ha_gather_attn_paged) kEntry>
HA_FN(gather_attn_paged) {
    return guarded(n, 14, [&] {
        const ha_shape *s = structure<ha_shape>(a[0]);
        const uint16_t *q = ptr<const uint16_t>(a[1]);
        const ha_tensor K = view(a[2]), V = view(a[3]);
        const Table bt = table(a[4]);
        const int32_t ps = i32(a[5]);
        const int32_t *lens = ptr<const int32_t>(a[6]);
        const Rows<const int32_t> idx = rows<const int32_t>(a[7]);
        const int32_t *cnt = ptr<const int32_t>(a[8]);
        const int32_t kmax = i32(a[9]);
        uint16_t *out = ptr<uint16_t>(a[10]);
        const Workspace w = workspace(a[11]);
        float *lse = ptr_or_null<float>(a[12]);
        void *st = stream(a[13]);
        return unlocked([&] { return kEntry(s, q, &K, &V, bt.p, bt.s0, ps, lens, idx.p, idx.s0, idx.s1, cnt, kmax, out, lse, w.p, w.n, st); });
    });
}

// shape, q, K, V, seq_lens, idx, count, k_max, out, lse, stream
HA_FN(gather_attn_static) {
    return guarded(n, 11, [&] {
        const ha_shape *s = structure<ha_shape>(a[0]);
        const uint16_t *q = ptr<const uint16_t>(a[1]);
        const ha_tensor K = view(a[2]), V = view(a[3]);
        const int32_t *lens = ptr<const int32_t>(a[4]);
        const Rows<const int32_t> idx = rows<const int32_t>(a[5]);
        const int32_t *cnt = ptr<const int32_t>(a[6]);
        const int32_t kmax = i32(a[7]);
        uint16_t *out = ptr<uint16_t>(a[8]);
        float *lse = ptr_or_null<float>(a[9]);
        void *st = stream(a[10]);
        return unlocked([&] { return ha_gather_attn_static(s, q, &K, &V, lens, idx.p, idx.s0, idx.s1, cnt, kmax, out, lse, st); });
    });
}

// shape, q, K, V, seq_lens, max_seq_len, out, workspace, lse, stream
HA_FN(dense_decode) {
    return guarded(n, 10, [&] {
        const ha_shape *s = structure<ha_shape>(a[0]);
        const uint16_t *q = ptr<const uint16_t>(a[1]);
        const ha_tensor K = view(a[2]), V = view(a[3]);
        const int32_t *lens = ptr<const int32_t>(a[4]);
        const int32_t nmax = i32(a[5]);
        uint16_t *out = ptr<uint16_t>(a[6]);
        const Workspace w = workspace(a[7]);
        float *lse = ptr_or_null<float>(a[8]);
        void *st = stream(a[9]);
        return unlocked([&] { return ha_dense_decode(s, q, &K, &V, lens, nmax, out, lse, w.p, w.n, st); });
    });
}

// ---------------------------------------------------------------- the whole layer-step

// what the step entries share: shape, map_q, map_k, q, k_new, K, V at the front; the tail from seq_lens on
struct StepFront {
    const ha_shape *s;
    const ha_mapping *mq, *mk;
    const uint16_t *q, *k_new;
    ha_tensor K, V;
    explicit StepFront(PyObject *const *a)
        : s(structure<ha_shape>(a[0])), mq(mapping(a[1])), mk(mapping(a[2])), q(ptr<const uint16_t>(a[3])),
          k_new(ptr_or_null<const uint16_t>(a[4])), K(view(a[5])), V(view(a[6])) {}
};
struct StepTail {   // seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, q_codes, idx, count, out, workspace, lse, stream
    const int32_t *lens, *ks;
    int32_t ku, nmax, kmax;
    uint32_t *qc;
    Rows<int32_t> idx;
    int32_t *cnt;
    uint16_t *out;
    Workspace w;
    float *lse;
    void *st;
    explicit StepTail(PyObject *const *a)
        : lens(ptr<const int32_t>(a[0])), ks(ptr_or_null<const int32_t>(a[1])), ku(i32(a[2])), nmax(i32(a[3])), kmax(i32(a[4])),
          qc(ptr<uint32_t>(a[5])), idx(rows<int32_t>(a[6])), cnt(ptr<int32_t>(a[7])), out(ptr<uint16_t>(a[8])), w(workspace(a[9])),
          lse(ptr_or_null<float>(a[10])), st(stream(a[11])) {}
};

// shape, map_q, map_k, q, k_new, K, V, k_codes, <tail>
template <decltype(&ha_sparse_decode) kEntry>
HA_FN(sparse_decode) {
    return guarded(n, 20, [&] {
        const StepFront f(a);
        const Rows<uint32_t> kc = rows<uint32_t>(a[7]);
        const StepTail t(a + 8);
        return unlocked([&] {
            return kEntry(f.s, f.mq, f.mk, f.q, f.k_new, &f.K, &f.V, kc.p, kc.s0, kc.s1, t.lens, t.ks, t.ku, t.nmax, t.kmax, t.qc, t.idx.p,
                          t.idx.s0, t.idx.s1, t.cnt, t.out, t.lse, t.w.p, t.w.n, t.st);
        });
    });
}

// shape, map_q, map_k, q, k_new, K_pool, V_pool, block_table, page_size, k_codes, <tail>
HA_FN(sparse_decode_paged) {
    return guarded(n, 22, [&] {
        const StepFront f(a);
        const Table bt = table(a[7]);
        const int32_t ps = i32(a[8]);
        const Rows<uint32_t> kc = rows<uint32_t>(a[9]);
        const StepTail t(a + 10);
        return unlocked([&] {
            return ha_sparse_decode_paged(f.s, f.mq, f.mk, f.q, f.k_new, &f.K, &f.V, bt.p, bt.s0, ps, kc.p, kc.s0, kc.s1, t.lens, t.ks, t.ku,
                                          t.nmax, t.kmax, t.qc, t.idx.p, t.idx.s0, t.idx.s1, t.cnt, t.out, t.lse, t.w.p, t.w.n, t.st);
        });
    });
}

// shape, map_q, map_k, q, k_new, K_pool, V_pool, code_pool, block_table, <tail>
HA_FN(sparse_decode_paged_codes) {
    return guarded(n, 21, [&] {
        const StepFront f(a);
        const Pool cp = pool(a[7]);
        const Table bt = table(a[8]);
        const StepTail t(a + 9);
        return unlocked([&] {
            return ha_sparse_decode_paged_codes(f.s, f.mq, f.mk, f.q, f.k_new, &f.K, &f.V, cp.p, cp.page, cp.head, bt.p, bt.s0, cp.size, t.lens,
                                                t.ks, t.ku, t.nmax, t.kmax, t.qc, t.idx.p, t.idx.s0, t.idx.s1, t.cnt, t.out, t.lse, t.w.p,
                                                t.w.n, t.st);
        });
    });
}

// ---------------------------------------------------------------- host-buffer steps

// Arguments of a host-buffer step: shape, map_q, map_k, q_host, k_new_host, v_new_host, K, V, [block_table, page_size,] k_codes,
// seq_lens, k_per_seq, k_uniform, max_seq_len, k_max, idx, count, out_host, workspace, stream
struct HostStep {
    const ha_shape *s;
    const ha_mapping *mq, *mk;
    const uint16_t *q, *k_new, *v_new;
    uint16_t *out;
    ha_tensor K, V;
    bool paged;
    Table bt;
    int32_t ps;
    Rows<uint32_t> kc;
    const int32_t *lens, *ks;
    int32_t ku, nmax, kmax;
    Rows<int32_t> idx;
    int32_t *cnt;
    Workspace w;
    void *st;
    HostStep(PyObject *const *a, bool is_paged)
        : s(structure<ha_shape>(a[0])), mq(mapping(a[1])), mk(mapping(a[2])), q(host(a[3])), k_new(host(a[4])), v_new(host(a[5])),
          K(view(a[6])), V(view(a[7])), paged(is_paged), bt{nullptr, 0}, ps(0) {
        if (paged) {
            bt = table(a[8]);
            ps = i32(a[9]);
        }
        PyObject *const *t = a + (paged ? 10 : 8);
        kc = rows<uint32_t>(t[0]);
        lens = ptr<const int32_t>(t[1]);
        ks = ptr_or_null<const int32_t>(t[2]);
        ku = i32(t[3]);
        nmax = i32(t[4]);
        kmax = i32(t[5]);
        idx = rows<int32_t>(t[6]);
        cnt = ptr<int32_t>(t[7]);
        out = const_cast<uint16_t *>(host(t[8]));
        w = workspace(t[9]);
        st = stream(t[10]);
    }
    int call() const {
        if (paged)
            return ha_sparse_decode_paged_host(s, mq, mk, q, k_new, v_new, &K, &V, bt.p, bt.s0, ps, kc.p, kc.s0, kc.s1, lens, ks, ku, nmax,
                                               kmax, idx.p, idx.s0, idx.s1, cnt, out, w.p, w.n, st);
        return ha_sparse_decode_host(s, mq, mk, q, k_new, v_new, &K, &V, kc.p, kc.s0, kc.s1, lens, ks, ku, nmax, kmax, idx.p, idx.s0, idx.s1,
                                     cnt, out, w.p, w.n, st);
    }
};

HA_FN(sparse_decode_host) {
    return guarded(n, 19, [&] {
        const HostStep h(a, false);
        return unlocked([&] { return h.call(); });
    });
}
HA_FN(sparse_decode_paged_host) {
    return guarded(n, 21, [&] {
        const HostStep h(a, true);
        return unlocked([&] { return h.call(); });
    });
}

// The arguments of a contiguous host-buffer step, kept for SparseDecodeHostStep (which keeps the objects behind them alive).
const char *const kStepName = "hashattn.host_step";
HA_FN(host_step_prepare) {
    if (n != 19) {
        PyErr_Format(PyExc_TypeError, "expected 19 arguments, got %zd", n);
        return nullptr;
    }
    try {
        return PyCapsule_New(new HostStep(a, false), kStepName,
                             [](PyObject *c) { delete static_cast<HostStep *>(PyCapsule_GetPointer(c, kStepName)); });
    } catch (const Raised &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
PyObject *host_step_run(PyObject *, PyObject *capsule) {
    const HostStep *h = static_cast<const HostStep *>(PyCapsule_GetPointer(capsule, kStepName));
    if (!h) return nullptr;
    return PyLong_FromLong(unlocked([&] { return h->call(); }));
}

#define HA_METHOD(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(fn)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    HA_METHOD("encode", encode),
    HA_METHOD("encode_prefill", encode_prefill),
    HA_METHOD("encode_wide", encode_wide),
    HA_METHOD("encode_append_paged", encode_append_paged),
    HA_METHOD("score_topk", score_topk),
    HA_METHOD("score_topk_sum", score_topk_no_workspace<&ha_score_topk_sum>),
    HA_METHOD("score_topk_per_head", score_topk_no_workspace<&ha_score_topk_per_head>),
    HA_METHOD("score_topk_paged", score_topk_paged<&ha_score_topk_paged>),
    HA_METHOD("score_topk_per_head_paged", score_topk_paged<&ha_score_topk_per_head_paged>),
    HA_METHOD("score_topk_wide", score_topk_wide),
    HA_METHOD("gather_attn", gather_attn<&ha_gather_attn>),
    HA_METHOD("gather_attn_per_head", gather_attn<&ha_gather_attn_per_head>),
    HA_METHOD("gather_attn_paged", gather_attn_paged<&ha_gather_attn_paged>),
    HA_METHOD("gather_attn_per_head_paged", gather_attn_paged<&ha_gather_attn_per_head_paged>),
    HA_METHOD("gather_attn_static", gather_attn_static),
    HA_METHOD("dense_decode", dense_decode),
    HA_METHOD("sparse_decode", sparse_decode<&ha_sparse_decode>),
    HA_METHOD("sparse_decode_pipelined", sparse_decode<&ha_sparse_decode_pipelined>),
    HA_METHOD("sparse_decode_paged", sparse_decode_paged),
    HA_METHOD("sparse_decode_paged_codes", sparse_decode_paged_codes),
    HA_METHOD("sparse_decode_host", sparse_decode_host),
    HA_METHOD("sparse_decode_paged_host", sparse_decode_paged_host),
    HA_METHOD("host_step_prepare", host_step_prepare),
    {"host_step_run", host_step_run, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_hostcall", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

} // namespace

PyMODINIT_FUNC PyInit__hostcall(void) {
    g_struct_name = PyUnicode_InternFromString("struct");
    g_stream_name = PyUnicode_InternFromString("cuda_stream");
    if (!g_struct_name || !g_stream_name) return nullptr;
    return PyModule_Create(&kModule);
}
