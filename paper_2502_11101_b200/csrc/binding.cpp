// Native argument marshalling of the calls a serving loop issues per layer or per token: reads tensors, strides and the
// current stream without going through Python objects, releases the GIL and calls the C ABI.  A call of the ctypes
// binding costs 6 to 12 us of host time (address and stride look-ups, fifteen argument conversions, the current-stream
// query), as much as the kernels it launches run for; here it is well under one.  Functions take their arguments by
// position, in the order of the C ABI with tensors in place of addresses, and return the library's error code;
// binding.py holds the public signatures.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <vector>

#include "cachefocus.h"

namespace {

struct Raised {};                                  // a Python exception is set

[[noreturn]] void fail(PyObject* type, const char* what) {
    PyErr_SetString(type, what);
    throw Raised{};
}
void require(bool ok, const char* what) {
    if (!ok) fail(PyExc_AssertionError, what);
}

// A view of an object's bytes for the duration of a call (ctypes structures, NumPy arrays).
struct Bytes {
    Py_buffer view{};
    bool held = false;
    Bytes() = default;
    Bytes(const Bytes&) = delete;
    void get(PyObject* o) {
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Raised{};
        held = true;
    }
    ~Bytes() {
        if (held) PyBuffer_Release(&view);
    }
};

// The positional arguments of a call, read one after the other.
class Args {
public:
    Args(PyObject* const* a, Py_ssize_t n) : a_(a), n_(n) {}
    PyObject* next() {
        if (i_ >= n_) fail(PyExc_TypeError, "too few arguments");
        return a_[i_++];
    }
    const at::Tensor& tensor() {
        PyObject* o = next();
        if (!THPVariable_Check(o)) fail(PyExc_TypeError, "a torch tensor is expected");
        return THPVariable_Unpack(o);
    }
    // nullptr for None
    const at::Tensor* maybe_tensor() {
        PyObject* o = next();
        if (o == Py_None) return nullptr;
        if (!THPVariable_Check(o)) fail(PyExc_TypeError, "a torch tensor or None is expected");
        return &THPVariable_Unpack(o);
    }
    void* ptr() { return tensor().data_ptr(); }
    // address of a tensor, of a NumPy array or given as a number; None is a null pointer
    void* maybe_ptr() {
        PyObject* o = next();
        if (o == Py_None) return nullptr;
        if (THPVariable_Check(o)) return THPVariable_Unpack(o).data_ptr();
        if (PyObject_CheckBuffer(o)) {
            Bytes b;
            b.get(o);
            return b.view.buf;
        }
        void* p = PyLong_AsVoidPtr(o);
        if (!p && PyErr_Occurred()) throw Raised{};
        return p;
    }
    long long integer() {
        const long long v = PyLong_AsLongLong(next());
        if (v == -1 && PyErr_Occurred()) throw Raised{};
        return v;
    }
    int32_t i32() {
        const long long v = integer();
        if (v < INT32_MIN || v > INT32_MAX) fail(PyExc_OverflowError, "a 32-bit integer is expected");
        return (int32_t)v;
    }
    float real() {
        const double v = PyFloat_AsDouble(next());
        if (v == -1.0 && PyErr_Occurred()) throw Raised{};
        return (float)v;
    }
    template <typename T>
    const T* structure(Bytes& b) {
        b.get(next());
        if (b.view.len != (Py_ssize_t)sizeof(T)) fail(PyExc_TypeError, "a structure of another size is expected");
        return static_cast<const T*>(b.view.buf);
    }
    // a stream object, a raw handle, or None for the current stream
    void* stream() {
        PyObject* o = next();
        if (o == Py_None) return (void*)c10::cuda::getCurrentCUDAStream().stream();
        PyObject* handle = PyObject_HasAttrString(o, "cuda_stream") ? PyObject_GetAttrString(o, "cuda_stream") : PyNumber_Long(o);
        if (!handle) throw Raised{};
        void* p = PyLong_AsVoidPtr(handle);
        Py_DECREF(handle);
        if (!p && PyErr_Occurred()) throw Raised{};
        return p;
    }

private:
    PyObject* const* a_;
    Py_ssize_t n_, i_ = 0;
};

size_t bytes_of(const at::Tensor& t) { return (size_t)t.numel() * t.element_size(); }

template <typename F>
PyObject* guarded(F&& f) {
    try {
        return f();
    } catch (const Raised&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <typename F>
PyObject* call(F&& f) {                            // f() returns a CF_* code and touches no Python object
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

#define NATIVE(name) PyObject* name(PyObject*, PyObject* const* argv, Py_ssize_t argc)

NATIVE(plan_init) {                                // geom, batch, plan, order, kept_count, query_start, score_accum (S = 0) or None, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg, bb;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const cf_batch* b = in.structure<cf_batch>(bb);
        const at::Tensor& plan = in.tensor();
        const int32_t* order = static_cast<const int32_t*>(in.maybe_ptr());
        const int32_t* kept = static_cast<const int32_t*>(in.maybe_ptr());
        const int32_t start = in.i32();
        float* scores = (float*)in.maybe_ptr();
        void* s = in.stream();
        void* p = plan.data_ptr();
        const size_t n = bytes_of(plan);
        return call([&] { return cf_plan_init_scores(g, b, order, kept, start, scores, p, n, s); });
    });
}

NATIVE(prune_topk) {                               // geom, batch, plan, score_accum, keep, keep_per_request, strategy, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg, bb;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const cf_batch* b = in.structure<cf_batch>(bb);
        void* plan = in.ptr();
        const float* scores = static_cast<const float*>(in.ptr());
        const int32_t keep = in.i32();
        const int32_t* per = static_cast<const int32_t*>(in.maybe_ptr());
        const int32_t strategy = in.i32();
        void* s = in.stream();
        return call([&] { return cf_prune_topk(g, b, plan, scores, keep, per, strategy, s); });
    });
}

NATIVE(reposition_keys) {                          // geom, batch, plan, k_in, k_out, n_layers, layer_stride, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg, bb;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const cf_batch* b = in.structure<cf_batch>(bb);
        void *plan = in.ptr(), *ki = in.ptr(), *ko = in.ptr();
        const int32_t n = in.i32();
        const int64_t stride = in.integer();
        void* s = in.stream();
        return call([&] { return cf_reposition_keys(g, b, plan, n, stride, ki, ko, s); });
    });
}

NATIVE(query_prefill_attn) {                       // geom, batch, plan, q, k, v, out, workspace, lse, doc_scores, score_accum, scale, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg, bb;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const cf_batch* b = in.structure<cf_batch>(bb);
        void *plan = in.ptr(), *q = in.ptr(), *k = in.ptr(), *v = in.ptr(), *out = in.ptr();
        const at::Tensor& ws = in.tensor();
        float *lse = (float*)in.maybe_ptr(), *scores = (float*)in.maybe_ptr(), *accum = (float*)in.maybe_ptr();
        const float scale = in.real();
        void *s = in.stream(), *w = ws.data_ptr();
        const size_t n = bytes_of(ws);
        return call([&] { return cf_query_prefill_attn(g, b, plan, q, k, v, scale, out, lse, scores, accum, w, n, s); });
    });
}

NATIVE(query_prefill_attn_slot) {                  // geom, batch, plan, slot, n_slots, q, k, v, out, workspace, lse, scale, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg, bb;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const cf_batch* b = in.structure<cf_batch>(bb);
        void* plan = in.ptr();
        const int32_t slot = in.i32(), n_slots = in.i32();
        void *q = in.ptr(), *k = in.ptr(), *v = in.ptr(), *out = in.ptr();
        const at::Tensor& ws = in.tensor();
        float* lse = (float*)in.maybe_ptr();
        const float scale = in.real();
        void *s = in.stream(), *w = ws.data_ptr();
        const size_t n = bytes_of(ws);
        return call([&] { return cf_query_prefill_attn_slot(g, b, plan, slot, n_slots, q, k, v, scale, out, lse, w, n, s); });
    });
}

NATIVE(accumulate_scores) {                        // geom, batch, plan, n_filled, n_slots, workspace, doc_scores, score_accum, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg, bb;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const cf_batch* b = in.structure<cf_batch>(bb);
        void* plan = in.ptr();
        const int32_t filled = in.i32(), n_slots = in.i32();
        const at::Tensor& ws = in.tensor();
        float *scores = (float*)in.maybe_ptr(), *accum = (float*)in.maybe_ptr();
        void *s = in.stream(), *w = ws.data_ptr();
        const size_t n = bytes_of(ws);
        return call([&] { return cf_accumulate_scores(g, b, plan, filled, n_slots, scores, accum, w, n, s); });
    });
}

NATIVE(assemble_final_cache) {                     // geom, batch, plan, k, v, k_self, v_self, k_out, v_out, final_rows, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg, bb;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const cf_batch* b = in.structure<cf_batch>(bb);
        void* plan = in.ptr();
        const at::Tensor &k = in.tensor(), &v = in.tensor(), &ks = in.tensor(), &vs = in.tensor(), &ko = in.tensor(), &vo = in.tensor(), &rows = in.tensor();
        void* s = in.stream();
        require(ko.is_contiguous() && vo.is_contiguous() && ko.sizes() == vo.sizes(), "k_out and v_out: contiguous, of one shape");
        require(rows.scalar_type() == at::kInt && k.stride(0) == v.stride(0), "final_rows: int32; k_cache and v_cache: one layer stride");
        const int32_t n_layers = (int32_t)k.size(0), out_rows = (int32_t)ko.size(2);
        const int64_t stride = k.stride(0), self_stride = ks.stride(0);
        void *kp = k.data_ptr(), *vp = v.data_ptr(), *ksp = ks.data_ptr(), *vsp = vs.data_ptr(), *kop = ko.data_ptr(), *vop = vo.data_ptr();
        int32_t* rp = (int32_t*)rows.data_ptr();
        return call([&] { return cf_assemble_final_cache(g, b, plan, n_layers, stride, kp, vp, self_stride, ksp, vsp, out_rows, kop, vop, rp, s); });
    });
}

NATIVE(document_prefill_attn) {                    // geom, doc_offsets, max_doc_len, q, k, v, out, k_prefix, v_prefix, lse, scale, token_stride, status, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const at::Tensor& off = in.tensor();
        const int32_t longest = in.i32();
        const at::Tensor &q = in.tensor(), &k = in.tensor(), &v = in.tensor(), &out = in.tensor();
        const at::Tensor *kp = in.maybe_tensor(), *vp = in.maybe_tensor(), *lse = in.maybe_tensor();
        const float scale = in.real();
        PyObject* ts = in.next();
        int32_t* status = (int32_t*)in.maybe_ptr();
        void* s = in.stream();
        const int64_t n = q.size(0), total = q.size(1);
        require(off.scalar_type() == at::kInt && off.is_contiguous(), "doc_offsets: contiguous int32");
        require(k.size(0) == n && v.size(0) == n && out.size(0) == n, "q, k, v and out: one number of layers");
        require(k.stride(0) == v.stride(0) && (!lse || lse->is_contiguous()), "k and v: one layer stride; lse: contiguous");
        const int64_t prefix = kp ? kp->size(1) : 0;
        require(prefix == 0 || (vp && kp->stride(0) == vp->stride(0)), "k_prefix and v_prefix: one layer stride");
        int64_t stride = k.size(2) * k.size(3);
        if (ts != Py_None) {
            stride = PyLong_AsLongLong(ts);
            if (stride == -1 && PyErr_Occurred()) throw Raised{};
        }
        const cf_doc_batch docs = {(int32_t)(off.numel() - 1), longest, (int32_t)prefix, 0, total, stride, (const int32_t*)off.data_ptr()};
        const int64_t qs = q.stride(0), kvs = k.stride(0), os = out.stride(0), ps = prefix ? kp->stride(0) : 0;
        void *qp = q.data_ptr(), *kd = k.data_ptr(), *vd = v.data_ptr(), *op = out.data_ptr();
        void *kpp = prefix ? kp->data_ptr() : nullptr, *vpp = prefix ? vp->data_ptr() : nullptr;
        float* lp = lse ? (float*)lse->data_ptr() : nullptr;
        return call([&] { return cf_document_prefill_attn(g, &docs, (int32_t)n, qp, qs, kd, vd, kvs, kpp, vpp, ps, scale, op, os, lp, status, s); });
    });
}

NATIVE(decode_plan) {                              // geom, n_requests, cache_rows, rows, extra_rows, decode_plan, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const int32_t nb = in.i32(), room = in.i32();
        const int32_t* rows = (const int32_t*)in.ptr();
        const int32_t extra = in.i32();
        const at::Tensor& plan = in.tensor();
        void *s = in.stream(), *p = plan.data_ptr();
        const size_t n = bytes_of(plan);
        return call([&] { return cf_decode_plan(g, nb, room, rows, extra, p, n, s); });
    });
}

NATIVE(decode_attn) {                              // geom, n_requests, cache_rows, decode_plan, q, k, v, out, workspace, lse, scale, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const int32_t nb = in.i32(), room = in.i32();
        void* plan = in.ptr();
        const at::Tensor &q = in.tensor(), &k = in.tensor(), &v = in.tensor(), &out = in.tensor(), &ws = in.tensor();
        const at::Tensor* lse = in.maybe_tensor();
        const float scale = in.real();
        void* s = in.stream();
        const int64_t n = q.size(0);
        require(k.size(0) == n && v.size(0) == n && out.size(0) == n, "q, k_final, v_final and out: one number of layers");
        require(k.stride(0) == v.stride(0) && (!lse || lse->is_contiguous()), "k_final and v_final: one layer stride; lse: contiguous");
        const int64_t qs = q.stride(0), kvs = k.stride(0), os = out.stride(0);
        void *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr(), *op = out.data_ptr(), *w = ws.data_ptr();
        const size_t wn = bytes_of(ws);
        float* lp = lse ? (float*)lse->data_ptr() : nullptr;
        return call([&] { return cf_decode_attn(g, nb, room, plan, (int32_t)n, qp, qs, kp, vp, kvs, scale, op, os, lp, w, wn, s); });
    });
}

NATIVE(decode_append) {                            // geom, n_requests, cache_rows, k_final, v_final, rows, step, k_new, v_new, status, stream
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const int32_t nb = in.i32(), room = in.i32();
        const at::Tensor &k = in.tensor(), &v = in.tensor();
        const int32_t* rows = (const int32_t*)in.ptr();
        const int32_t step = in.i32();
        const at::Tensor &kn = in.tensor(), &vn = in.tensor();
        int32_t* status = (int32_t*)in.maybe_ptr();
        void* s = in.stream();
        const int64_t n = k.size(0);
        require(v.size(0) == n && kn.size(0) == n && vn.size(0) == n, "k_final, v_final, k_new and v_new: one number of layers");
        require(k.stride(0) == v.stride(0) && kn.stride(0) == vn.stride(0), "keys and values: one layer stride");
        const int64_t kvs = k.stride(0), ns = kn.stride(0);
        void *kp = k.data_ptr(), *vp = v.data_ptr(), *knp = kn.data_ptr(), *vnp = vn.data_ptr();
        return call([&] { return cf_decode_append(g, nb, room, (int32_t)n, kp, vp, kvs, rows, step, knp, vnp, ns, status, s); });
    });
}

// A whole stack: geom, batch, plan, workspace, q, k, v, out, score_accum, schedule [(layer, keep), ...], strategy,
// batch_layers, lse, layer_scores, k_final, k_self, v_self, scale, doc_len, req_doc_begin (int32 arrays or None),
// k_prefix, v_prefix, stream.  Returns (code, 0), or (0, bytes) without doing anything when the workspace is smaller
// than that.
NATIVE(run_stack) {
    return guarded([&] {
        Args in(argv, argc);
        Bytes bg, bb, bl, br;
        const cf_geom* g = in.structure<cf_geom>(bg);
        const cf_batch* b = in.structure<cf_batch>(bb);
        const at::Tensor &plan = in.tensor(), &ws = in.tensor(), &q = in.tensor(), &k = in.tensor(), &v = in.tensor(), &out = in.tensor(), &accum = in.tensor();
        PyObject* sched = PySequence_Fast(in.next(), "the schedule is a sequence of (layer, keep) pairs");
        if (!sched) throw Raised{};
        std::vector<std::pair<int, int>> cuts;
        for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(sched); ++i) {
            int layer, keep;
            PyObject* pair = PySequence_Tuple(PySequence_Fast_GET_ITEM(sched, i));
            const bool ok = pair && PyArg_ParseTuple(pair, "ii", &layer, &keep);
            Py_XDECREF(pair);
            if (!ok) {
                Py_DECREF(sched);
                throw Raised{};
            }
            cuts.emplace_back(layer, keep);
        }
        Py_DECREF(sched);
        std::sort(cuts.begin(), cuts.end());
        std::vector<int32_t> layers, keeps;
        for (auto& c : cuts) {
            layers.push_back(c.first);
            keeps.push_back(c.second);
        }
        const int32_t strategy = in.i32();
        const int batched = PyObject_IsTrue(in.next());
        const at::Tensor *lse = in.maybe_tensor(), *scores = in.maybe_tensor(), *kf = in.maybe_tensor(), *ks = in.maybe_tensor(), *vs = in.maybe_tensor();
        const float scale = in.real();
        PyObject *lens = in.next(), *begins = in.next();
        const at::Tensor *kp = in.maybe_tensor(), *vp = in.maybe_tensor();
        void* s = in.stream();
        const int64_t n = q.size(0);
        require(k.size(0) == n && v.size(0) == n && out.size(0) == n && k.stride(0) == v.stride(0), "q, k, v and out: one number of layers; k and v: one layer stride");
        require((!lse || (lse->size(0) == n && lse->is_contiguous())) && (!scores || (scores->size(0) == n && scores->is_contiguous())), "lse and layer_scores: contiguous, one entry per layer");
        require(!kf || (kf->sizes() == k.sizes() && kf->stride(0) == k.stride(0)), "k_final: the layout of the key store");
        require(!ks || (vs && ks->size(0) == n && ks->stride(0) == vs->stride(0)), "k_self and v_self: one entry per layer, one layer stride");
        cf_stack st = {};
        st.n_layers = (int32_t)n;
        st.n_prune = (int32_t)cuts.size();
        st.prune_layer = cuts.empty() ? nullptr : layers.data();
        st.prune_keep = cuts.empty() ? nullptr : keeps.data();
        st.strategy = strategy;
        st.batch_layers = batched ? 1 : 0;
        st.softmax_scale = scale;
        st.q = q.data_ptr();
        st.q_layer_stride = q.stride(0);
        st.k_cache = k.data_ptr();
        st.v_cache = v.data_ptr();
        st.kv_layer_stride = k.stride(0);
        st.k_self = ks ? ks->data_ptr() : nullptr;
        st.v_self = vs ? vs->data_ptr() : nullptr;
        st.self_layer_stride = ks ? ks->stride(0) : 0;
        st.out = out.data_ptr();
        st.out_layer_stride = out.stride(0);
        st.lse = lse ? (float*)lse->data_ptr() : nullptr;
        st.layer_scores = scores ? (float*)scores->data_ptr() : nullptr;
        st.score_accum = (float*)accum.data_ptr();
        st.k_final = kf ? kf->data_ptr() : nullptr;
        if (lens != Py_None && begins != Py_None) {
            bl.get(lens);
            br.get(begins);
            st.doc_len_host = (const int32_t*)bl.view.buf;
            st.req_doc_begin_host = (const int32_t*)br.view.buf;
        }
        st.k_prefix = kp ? kp->data_ptr() : nullptr;
        st.v_prefix = vp ? vp->data_ptr() : nullptr;
        st.prefix_layer_stride = kp ? kp->stride(0) : 0;
        st.prefix_len = kp ? (int32_t)kp->size(1) : 0;
        void *p = plan.data_ptr(), *w = ws.data_ptr();
        const size_t pn = bytes_of(plan), wn = bytes_of(ws);
        size_t need = 0;
        int rc = CF_OK;
        Py_BEGIN_ALLOW_THREADS
        need = cf_run_stack_workspace_bytes(g, b, &st);
        if (need <= wn) {
            need = 0;
            rc = cf_run_stack(g, b, &st, p, pn, w, wn, s);
        }
        Py_END_ALLOW_THREADS
        return Py_BuildValue("in", rc, (Py_ssize_t)need);
    });
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ENTRY(plan_init), ENTRY(prune_topk), ENTRY(reposition_keys), ENTRY(query_prefill_attn),
                         ENTRY(query_prefill_attn_slot), ENTRY(accumulate_scores), ENTRY(assemble_final_cache),
                         ENTRY(document_prefill_attn), ENTRY(decode_plan), ENTRY(decode_attn), ENTRY(decode_append),
                         ENTRY(run_stack), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "argument marshalling of the hot calls", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
