// Native half of binding.py: builds the C ABI's argument structs from torch tensors and calls the library, without the library
// being linked (its entry points' addresses are handed over once).  The ctypes marshalling of one call -- some thirty attribute reads and
// struct fields -- took 10 to 15 us of Python, longer than a small layer runs; here it takes about one.  Arguments arrive positionally from
// the wrappers of the same names; every function returns the lisa_status_t.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "lisa.h"

namespace {

struct Raised {};   // a Python exception is set

decltype(&lisa_attn_anchor) p_anchor;
decltype(&lisa_attn_shared_prefill) p_prefill;
decltype(&lisa_attn_shared_prefill_carry) p_carry;
decltype(&lisa_attn_shared_decode) p_decode;
decltype(&lisa_kvcache_append) p_append;
decltype(&lisa_kvcache_append_layer) p_append_layer;
decltype(&lisa_project) p_project;
decltype(&lisa_workspace_bytes) p_workspace_bytes;

PyObject *s_qp, *s_kp, *s_w1, *s_w2, *s_b1, *s_b2, *s_act, *s_integrate, *s_ffn_layers;

[[noreturn]] void fail(PyObject* type, const char* msg) {
    PyErr_SetString(type, msg);
    throw Raised{};
}
const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a torch.Tensor");
    return THPVariable_Unpack(o);
}
int32_t dtype(const at::Tensor& t) {
    if (t.scalar_type() == at::kBFloat16) return LISA_BF16;
    if (t.scalar_type() == at::kFloat) return LISA_F32;
    fail(PyExc_TypeError, "unsupported dtype");
}
lisa_tensor tensor4(const at::Tensor& t) {
    if (t.dim() != 4 || t.stride(3) != 1) fail(PyExc_AssertionError, "expected [B,N,H,x] with contiguous x");
    const auto s = t.strides();
    return lisa_tensor{t.data_ptr(), dtype(t), 0, s[0], s[1], s[2]};
}
void* ptr(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
int64_t integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return v;
}
template <typename T>
T address(PyObject* o) {
    void* v = PyLong_AsVoidPtr(o);
    if (!v && PyErr_Occurred()) throw Raised{};
    return static_cast<T>(v);
}
lisa_stream_t stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

struct Ref {   // an owned reference
    PyObject* o;
    explicit Ref(PyObject* p) : o(p) { if (!o) throw Raised{}; }
    ~Ref() { Py_DECREF(o); }
    Ref(const Ref&) = delete;
};

lisa_link link(PyObject* o) {
    lisa_link l{};
    Ref qp(PyObject_GetAttr(o, s_qp)), kp(PyObject_GetAttr(o, s_kp)), w1(PyObject_GetAttr(o, s_w1)), w2(PyObject_GetAttr(o, s_w2)),
        b1(PyObject_GetAttr(o, s_b1)), b2(PyObject_GetAttr(o, s_b2)), act(PyObject_GetAttr(o, s_act)), integrate(PyObject_GetAttr(o, s_integrate)),
        layers(PyObject_GetAttr(o, s_ffn_layers));
    const at::Tensor& q = tensor(qp.o);
    l.qp = tensor4(q);
    if (kp.o != Py_None) l.kp = tensor4(tensor(kp.o));
    l.w_dtype = LISA_F32;
    if (w1.o != Py_None) {
        const at::Tensor& w = tensor(w1.o);
        l.w_dtype = dtype(w);
        l.m = (int32_t)w.size(1);
    }
    const void** dst[4] = {&l.w1, &l.b1, &l.w2, &l.b2};
    PyObject* src[4] = {w1.o, b1.o, w2.o, b2.o};
    for (int i = 0; i < 4; ++i) {
        if (src[i] == Py_None) continue;
        const at::Tensor& w = tensor(src[i]);
        if (!w.is_contiguous()) fail(PyExc_AssertionError, "aligner weights must be contiguous");
        if (dtype(w) != l.w_dtype) fail(PyExc_AssertionError, "aligner weights must share one dtype");
        *dst[i] = w.data_ptr();
    }
    l.r = (int32_t)q.size(3);
    l.act = (int32_t)integer(act.o);
    l.integrate = (int32_t)integer(integrate.o);
    l.ffn_layers = (int32_t)integer(layers.o);
    return l;
}

// Scratch of a call: the caller's tensor, or one allocated here, which lives until the call's kernels are enqueued (the allocator
// orders its reuse behind them).
struct Scratch {
    at::Tensor own;
    void* p = nullptr;
    size_t bytes = 0;
    lisa_status_t status = LISA_OK;
    Scratch(PyObject* given, int32_t op, const void* args) {
        if (given != Py_None) {
            const at::Tensor& t = tensor(given);
            p = t.data_ptr();
            bytes = (size_t)t.numel();
            return;
        }
        status = p_workspace_bytes(op, args, &bytes);
        if (status != LISA_OK || bytes == 0) return;
        own = at::empty({(int64_t)bytes}, at::TensorOptions().dtype(at::kByte).device(at::kCUDA));
        p = own.data_ptr();
    }
};

template <typename F>
PyObject* call(F f) {
    try {
        return PyLong_FromLong(f());
    } catch (const Raised&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
void expect(Py_ssize_t n, Py_ssize_t want) { if (n != want) fail(PyExc_TypeError, "wrong number of arguments"); }
// The library's calls run without the interpreter lock, as ctypes runs them.
template <typename F>
lisa_status_t unlocked(F f) {
    lisa_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return st;
}

// (q, k, v, cache descriptor's address or 0, L, seq_lens, out, out_scores, workspace)
PyObject* py_anchor(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call([&]() -> long {
        expect(n, 9);
        const at::Tensor& q = tensor(a[0]);
        lisa_anchor_args p{};
        p.struct_size = sizeof(p);
        p.q = tensor4(q);
        p.o = tensor4(tensor(a[6]));
        p.B = (int32_t)q.size(0); p.Nq = (int32_t)q.size(1); p.Hq = (int32_t)q.size(2); p.d = (int32_t)q.size(3); p.L = (int32_t)integer(a[4]);
        p.cache = address<const lisa_kvcache_layer*>(a[3]);
        if (!p.cache) {
            const at::Tensor& k = tensor(a[1]);
            p.k = tensor4(k);
            p.v = tensor4(tensor(a[2]));
            p.Hkv = (int32_t)k.size(2);
        } else {
            p.Hkv = p.cache->Hkv;
            p.seq_lens = static_cast<const int32_t*>(ptr(a[5]));
            if (a[7] != Py_None) {
                const at::Tensor& r = tensor(a[7]);
                if (r.stride(2) != 1) fail(PyExc_AssertionError, "out_scores rows must be contiguous");
                p.out_scores = r.data_ptr(); p.scores_stride_b = r.stride(0); p.scores_stride_h = r.stride(1); p.scores_dtype = dtype(r);
            }
        }
        Scratch ws(a[8], LISA_OP_ANCHOR, &p);
        if (ws.status != LISA_OK) return ws.status;
        p.workspace = ws.p; p.workspace_bytes = ws.bytes;
        lisa_stream_t s = stream();
        return unlocked([&] { return p_anchor(&p, s); });
    });
}

void prefill_shape(lisa_shared_prefill_args& p, const at::Tensor& q0, int64_t Hkv, int32_t chain) {
    p.struct_size = sizeof(p);
    p.B = (int32_t)q0.size(0); p.N = (int32_t)q0.size(1); p.Hq = (int32_t)q0.size(2); p.d = (int32_t)q0.size(3);
    p.Hkv = (int32_t)Hkv; p.chain_len = chain;
}

// (q0, k0, links, v, out, workspace)
PyObject* py_prefill(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call([&]() -> long {
        expect(n, 6);
        Ref seq(PySequence_Fast(a[2], "links must be a sequence"));
        const Py_ssize_t c = PySequence_Fast_GET_SIZE(seq.o);
        std::vector<lisa_link> links;
        for (Py_ssize_t i = 0; i < c; ++i) links.push_back(link(PySequence_Fast_GET_ITEM(seq.o, i)));
        const at::Tensor &q0 = tensor(a[0]), &k0 = tensor(a[1]);
        lisa_shared_prefill_args p{};
        p.q0 = tensor4(q0); p.k0 = tensor4(k0); p.v = tensor4(tensor(a[3])); p.o = tensor4(tensor(a[4]));
        prefill_shape(p, q0, k0.size(2), (int32_t)c);
        p.links = links.data();
        Scratch ws(a[5], LISA_OP_SHARED_PREFILL, &p);
        if (ws.status != LISA_OK) return ws.status;
        p.workspace = ws.p; p.workspace_bytes = ws.bytes;
        lisa_stream_t s = stream();
        return unlocked([&] { return p_prefill(&p, s); });
    });
}

// (q0 or None, k0 or None, link, v, out, scores, first, keep, workspace)
PyObject* py_carry(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call([&]() -> long {
        expect(n, 9);
        lisa_link l = link(a[2]);
        const at::Tensor &v = tensor(a[3]), &out = tensor(a[4]), &scores = tensor(a[5]);
        lisa_shared_prefill_carry_args c{};
        c.struct_size = sizeof(c);
        lisa_shared_prefill_args& p = c.layer;
        p.v = tensor4(v); p.o = tensor4(out);
        if (a[0] == Py_None) {   // not read unless first: zeroed descriptors
            prefill_shape(p, out, v.size(2), 1);
        } else {
            const at::Tensor &q0 = tensor(a[0]), &k0 = tensor(a[1]);
            p.q0 = tensor4(q0); p.k0 = tensor4(k0);
            prefill_shape(p, q0, k0.size(2), 1);
        }
        p.links = &l;
        c.scores = scores.data_ptr(); c.scores_bytes = (size_t)scores.numel() * scores.element_size();
        c.first = (int32_t)integer(a[6]); c.keep = (int32_t)integer(a[7]);
        Scratch ws(a[8], LISA_OP_SHARED_PREFILL_CARRY, &c);
        if (ws.status != LISA_OK) return ws.status;
        p.workspace = ws.p; p.workspace_bytes = ws.bytes;
        lisa_stream_t s = stream();
        return unlocked([&] { return p_carry(&c, s); });
    });
}

// (prev_scores, link, cache descriptor's address, L, seq_lens, out, out_scores, workspace)
PyObject* py_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call([&]() -> long {
        expect(n, 8);
        const at::Tensor& prev = tensor(a[0]);
        if (prev.dim() != 3 || prev.stride(2) != 1) fail(PyExc_AssertionError, "expected score rows [B,Hq,L] with contiguous L");
        lisa_shared_decode_args p{};
        p.struct_size = sizeof(p);
        p.B = (int32_t)prev.size(0); p.Hq = (int32_t)prev.size(1); p.L = (int32_t)integer(a[3]); p.scores_dtype = dtype(prev);
        p.prev_scores = prev.data_ptr(); p.prev_stride_b = prev.stride(0); p.prev_stride_h = prev.stride(1);
        p.link = link(a[1]);
        p.cache = address<const lisa_kvcache_layer*>(a[2]);
        p.seq_lens = static_cast<const int32_t*>(ptr(a[4]));
        p.o = tensor4(tensor(a[5]));
        if (a[6] != Py_None) {
            const at::Tensor& r = tensor(a[6]);
            if (r.scalar_type() != prev.scalar_type() || r.stride(2) != 1) fail(PyExc_AssertionError, "out_scores: prev_scores' type, contiguous rows");
            p.out_scores = r.data_ptr(); p.scores_stride_b = r.stride(0); p.scores_stride_h = r.stride(1);
        }
        Scratch ws(a[7], LISA_OP_SHARED_DECODE, &p);
        if (ws.status != LISA_OK) return ws.status;
        p.workspace = ws.p; p.workspace_bytes = ws.bytes;
        lisa_stream_t s = stream();
        return unlocked([&] { return p_decode(&p, s); });
    });
}

// (cache descriptor's address, k or k', v, seq_lens_before)
PyObject* py_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call([&]() -> long {
        expect(n, 4);
        const at::Tensor& vt = tensor(a[2]);
        const lisa_tensor k = tensor4(tensor(a[1])), v = tensor4(vt);
        const lisa_kvcache_layer* layer = address<const lisa_kvcache_layer*>(a[0]);
        const int32_t* lens = static_cast<const int32_t*>(ptr(a[3]));
        lisa_stream_t s = stream();
        return unlocked([&] { return p_append(layer, &k, &v, lens, (int32_t)vt.size(1), s); });
    });
}

// (multi-layer cache's address, layer, k or k', v, seq_lens_before)
PyObject* py_append_layer(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call([&]() -> long {
        expect(n, 5);
        const at::Tensor& vt = tensor(a[3]);
        const lisa_tensor k = tensor4(tensor(a[2])), v = tensor4(vt);
        const lisa_kvcache* cache = address<const lisa_kvcache*>(a[0]);
        const int32_t layer = (int32_t)integer(a[1]);
        const int32_t* lens = static_cast<const int32_t*>(ptr(a[4]));
        lisa_stream_t s = stream();
        return unlocked([&] { return p_append_layer(cache, layer, &k, &v, lens, (int32_t)vt.size(1), s); });
    });
}

// (x, w, outs)
PyObject* py_project(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call([&]() -> long {
        expect(n, 3);
        const at::Tensor &x = tensor(a[0]), &w = tensor(a[1]);
        Ref seq(PySequence_Fast(a[2], "outs must be a sequence"));
        const Py_ssize_t c = PySequence_Fast_GET_SIZE(seq.o);
        if (c < 1 || c > 4) fail(PyExc_AssertionError, "one to four outputs");
        if (x.dim() != 3 || x.stride(2) != 1 || w.dim() != 2 || !w.is_contiguous() || w.size(0) != x.size(2))
            fail(PyExc_AssertionError, "expected x [B,N,d_in] with contiguous rows and a contiguous w [d_in, n_out]");
        lisa_project_args p{};
        p.struct_size = sizeof(p);
        p.B = (int32_t)x.size(0); p.N = (int32_t)x.size(1); p.d_in = (int32_t)x.size(2); p.n_outputs = (int32_t)c;
        p.x = lisa_tensor{x.data_ptr(), dtype(x), 0, x.stride(0), x.stride(1), 0};
        p.w = w.data_ptr(); p.w_dtype = dtype(w);
        int64_t cols = 0;
        for (Py_ssize_t i = 0; i < c; ++i) {
            const at::Tensor& o = tensor(PySequence_Fast_GET_ITEM(seq.o, i));
            p.outputs[i] = lisa_project_output{tensor4(o), (int32_t)o.size(2), (int32_t)o.size(3)};
            cols += o.size(2) * o.size(3);
        }
        if (cols != w.size(1)) fail(PyExc_AssertionError, "the outputs' columns must add up to w's");
        lisa_stream_t s = stream();
        return unlocked([&] { return p_project(&p, s); });
    });
}

// The addresses of the library's entry points, in this order.
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return call([&]() -> long {
        expect(n, 8);
        p_anchor = reinterpret_cast<decltype(p_anchor)>(address<void*>(a[0]));
        p_prefill = reinterpret_cast<decltype(p_prefill)>(address<void*>(a[1]));
        p_carry = reinterpret_cast<decltype(p_carry)>(address<void*>(a[2]));
        p_decode = reinterpret_cast<decltype(p_decode)>(address<void*>(a[3]));
        p_append = reinterpret_cast<decltype(p_append)>(address<void*>(a[4]));
        p_append_layer = reinterpret_cast<decltype(p_append_layer)>(address<void*>(a[5]));
        p_project = reinterpret_cast<decltype(p_project)>(address<void*>(a[6]));
        p_workspace_bytes = reinterpret_cast<decltype(p_workspace_bytes)>(address<void*>(a[7]));
        return 0;
    });
}

#define LISA_METHOD(name_) {#name_, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name_)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {LISA_METHOD(anchor), LISA_METHOD(prefill), LISA_METHOD(carry), LISA_METHOD(decode), LISA_METHOD(append),
                         LISA_METHOD(append_layer), LISA_METHOD(project), LISA_METHOD(bind), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_lisa_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__lisa_binding(void) {
    s_qp = PyUnicode_InternFromString("qp"); s_kp = PyUnicode_InternFromString("kp");
    s_w1 = PyUnicode_InternFromString("w1"); s_w2 = PyUnicode_InternFromString("w2");
    s_b1 = PyUnicode_InternFromString("b1"); s_b2 = PyUnicode_InternFromString("b2");
    s_act = PyUnicode_InternFromString("act"); s_integrate = PyUnicode_InternFromString("integrate");
    s_ffn_layers = PyUnicode_InternFromString("ffn_layers");
    return PyModule_Create(&module);
}
