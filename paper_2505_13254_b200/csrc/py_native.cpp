// CPython side of the step calls: reads the tensor bundles of binding.py and makes the C call, without building ctypes
// structures in Python (a step's three calls took 55 us of host time that way, more than the GPU needs for a small
// tree).  Only the CPython API is used: a tensor is asked for its `data_ptr`, `stride` and `size` like any object, so
// the module does not depend on torch's C++ interface.  Every function returns the hs_status as an int.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/heterospec.h"

namespace {

PyObject *n_data_ptr, *n_stride, *n_size, *n_dtype, *o_zero, *o_one, *o_two, *t_f32, *t_bf16;

struct Name {
    const char* text;
    PyObject* str;
};
Name k_tree[] = {{"batch"}, {"n_nodes_total"}, {"node_off"}, {"parent"}, {"token"}};
Name k_quant[] = {{"row_max"}, {"row_lse"}, {"h_full"}, {"i_topk"}, {"i_trunc"}, {"topk_val"}, {"topk_idx"},
                  {"logc"}, {"score"}, {"phi"}, {"depth"}, {"pstar_node"}, {"phi_star"}, {"status"}};
Name k_pruned[] = {{"bin"}, {"d_prime"}, {"n_prime"}, {"n_keep"}, {"keep_off"}, {"keep_idx"}, {"new_parent"},
                   {"new_depth"}, {"keep_rank"}, {"anc_mask"}, {"status"}};
Name k_accept[] = {{"accept_len"}, {"path_nodes"}, {"path_compact"}, {"path_tokens"}, {"bonus_token"},
                   {"terminal_rank"}, {"status"}, {"path_cap"}, {"max_kept_rows"}};
Name k_expand[] = {{"batch"}, {"cap"}, {"top_k"}, {"n_cand"}, {"parent"}, {"token"}, {"depth"}, {"logc"}, {"score"},
                   {"frontier"}, {"n_frontier"}, {"status"}};
Name k_policy[] = {{"thresholds"}, {"d_base"}, {"alpha"}, {"n_default"}, {"top_k"}, {"gamma_pct"}, {"phi_mode"},
                   {"pstar_mode"}, {"entropy_mode"}};

bool intern_all(Name* k, size_t n) {
    for (size_t i = 0; i < n; ++i)
        if (!(k[i].str = PyUnicode_InternFromString(k[i].text))) return false;
    return true;
}

// Reads arguments and fields; after a failed read `bad` stays set, the Python error with it, and reads return 0.
struct Reader {
    bool bad = false;

    long long integer(PyObject* o) {
        if (bad) return 0;
        const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
        if (v == (unsigned long long)-1 && PyErr_Occurred()) bad = true;
        return (long long)v;
    }
    double real(PyObject* o) {
        if (bad) return 0.0;
        const double v = PyFloat_AsDouble(o);
        if (v == -1.0 && PyErr_Occurred()) bad = true;
        return v;
    }
    // device pointer of a tensor, NULL for None
    void* ptr(PyObject* o) {
        if (bad || o == Py_None) return nullptr;
        PyObject* args[] = {nullptr, o};                             // (the call may use the slot ahead of its arguments)
        PyObject* r = PyObject_VectorcallMethod(n_data_ptr, args + 1, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, nullptr);
        if (!r) { bad = true; return nullptr; }
        void* p = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(r);
        Py_DECREF(r);
        return p;
    }
    long long dim(PyObject* name, PyObject* t, PyObject* index) {
        if (bad) return 0;
        PyObject* args[] = {nullptr, t, index};
        PyObject* r = PyObject_VectorcallMethod(name, args + 1, 2 | PY_VECTORCALL_ARGUMENTS_OFFSET, nullptr);
        if (!r) { bad = true; return 0; }
        const long long v = integer(r);
        Py_DECREF(r);
        return v;
    }
    long long size(PyObject* t, PyObject* index) { return dim(n_size, t, index); }
    long long stride(PyObject* t, PyObject* index) { return dim(n_stride, t, index); }
    hs_dtype dtype(PyObject* t) {
        if (bad) return HS_F32;
        PyObject* d = PyObject_GetAttr(t, n_dtype);
        if (!d) { bad = true; return HS_F32; }
        Py_DECREF(d);
        if (d == t_bf16) return HS_BF16;
        if (d == t_f32) return HS_F32;
        bad = true;
        PyErr_Format(PyExc_TypeError, "logits must be float32 or bfloat16, got %S", d);
        return HS_F32;
    }
    void* field_ptr(PyObject* o, const Name& k) {
        if (bad) return nullptr;
        PyObject* v = PyObject_GetAttr(o, k.str);
        if (!v) { bad = true; return nullptr; }
        void* p = ptr(v);
        Py_DECREF(v);
        return p;
    }
    int field_int(PyObject* o, const Name& k) {
        if (bad) return 0;
        PyObject* v = PyObject_GetAttr(o, k.str);
        if (!v) { bad = true; return 0; }
        const int i = (int)integer(v);
        Py_DECREF(v);
        return i;
    }
    // n pointers in declaration order (the C structs start with, or consist of, an unbroken run of pointers)
    void pointers(PyObject* o, const Name* k, int n, void* dst) {
        void** out = (void**)dst;
        for (int i = 0; i < n; ++i) out[i] = field_ptr(o, k[i]);
    }
    void tree(PyObject* o, hs_tree_batch* t) {
        t->batch = field_int(o, k_tree[0]);
        t->n_nodes_total = field_int(o, k_tree[1]);
        t->node_off = (const int32_t*)field_ptr(o, k_tree[2]);
        t->parent = (const int32_t*)field_ptr(o, k_tree[3]);
        t->token = (const int32_t*)field_ptr(o, k_tree[4]);
    }
    void expand(PyObject* o, hs_expand_state* s) {
        s->batch = field_int(o, k_expand[0]);
        s->cap = field_int(o, k_expand[1]);
        s->top_k = field_int(o, k_expand[2]);
        pointers(o, k_expand + 3, 9, &s->n_cand);
    }
    PyObject* item(PyObject* dict, const Name& k) {                  // borrowed
        if (bad) return nullptr;
        PyObject* v = PyDict_GetItemWithError(dict, k.str);
        if (!v) {
            bad = true;
            if (!PyErr_Occurred()) PyErr_SetObject(PyExc_KeyError, k.str);
        }
        return v;
    }
    void policy(PyObject* d, hs_policy* p) {
        for (int which = 0; which < 2 && !bad; ++which) {
            PyObject* v = item(d, k_policy[which ? 5 : 0]);
            if (bad) return;
            PyObject* s = PySequence_Fast(v, "the policy's thresholds and gamma_pct are sequences");
            if (!s) { bad = true; return; }
            const Py_ssize_t n = PySequence_Fast_GET_SIZE(s), want = which ? 3 : 7;
            for (Py_ssize_t i = 0; i < want; ++i) {                  // (missing entries are zero)
                PyObject* x = i < n ? PySequence_Fast_GET_ITEM(s, i) : nullptr;
                if (which) p->gamma_pct[i] = x ? (int)integer(x) : 0;
                else p->thresholds[i] = x ? (float)real(x) : 0.f;
            }
            Py_DECREF(s);
            if (n > want && !bad) { bad = true; PyErr_SetString(PyExc_IndexError, "invalid index"); }
        }
        int* at[] = {&p->d_base, &p->alpha, &p->n_default, &p->top_k};
        for (int i = 0; i < 4; ++i) if (PyObject* v = item(d, k_policy[1 + i])) *at[i] = (int)integer(v);
        int* modes[] = {&p->phi_mode, &p->pstar_mode, &p->entropy_mode};
        for (int i = 0; i < 3; ++i) if (PyObject* v = item(d, k_policy[6 + i])) *modes[i] = (int)integer(v);
    }
    hs_ctx* ctx(PyObject* o) { return (hs_ctx*)(uintptr_t)integer(o); }
    hs_stream stream(PyObject* o) { return (hs_stream)(uintptr_t)integer(o); }
};

static_assert(sizeof(hs_quant_out) == 14 * sizeof(void*), "hs_quant_out is fourteen pointers");
static_assert(sizeof(hs_pruned_tree) == 11 * sizeof(void*), "hs_pruned_tree is eleven pointers");

bool arity(Py_ssize_t got, Py_ssize_t want) {
    if (got == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
    return false;
}

#define HS_NATIVE(name) PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n)
// the C call, with the interpreter lock released (a launch may wait for room in the driver's queue)
#define HS_DONE(call)                                   \
    do {                                                \
        hs_ctx* ctx = r.ctx(a[0]);                      \
        hs_stream stream = r.stream(a[n - 1]);          \
        if (r.bad) return nullptr;                      \
        hs_status st;                                   \
        Py_BEGIN_ALLOW_THREADS                          \
        st = call;                                      \
        Py_END_ALLOW_THREADS                            \
        return PyLong_FromLong((long)st);               \
    } while (0)

// (ctx, tree, logits, policy, quant, stream)
HS_NATIVE(entropy_quantify) {
    if (!arity(n, 6)) return nullptr;
    Reader r;
    hs_tree_batch t; hs_policy p; hs_quant_out q;
    r.tree(a[1], &t); r.policy(a[3], &p); r.pointers(a[4], k_quant, 14, &q);
    const void* x = r.ptr(a[2]);
    const hs_dtype dt = r.dtype(a[2]);
    const long long rs = r.stride(a[2], o_zero), v = r.size(a[2], o_one);
    HS_DONE(hs_entropy_quantify(ctx, &t, x, dt, rs, (int)v, &p, &q, stream));
}
// (ctx, tree, logits, policy, quant, pruned, stream)
HS_NATIVE(entropy_quantify_prune) {
    if (!arity(n, 7)) return nullptr;
    Reader r;
    hs_tree_batch t; hs_policy p; hs_quant_out q; hs_pruned_tree k;
    r.tree(a[1], &t); r.policy(a[3], &p); r.pointers(a[4], k_quant, 14, &q); r.pointers(a[5], k_pruned, 11, &k);
    const void* x = r.ptr(a[2]);
    const hs_dtype dt = r.dtype(a[2]);
    const long long rs = r.stride(a[2], o_zero), v = r.size(a[2], o_one);
    HS_DONE(hs_entropy_quantify_prune(ctx, &t, x, dt, rs, (int)v, &p, &q, &k, stream));
}
// (ctx, tree, quant, policy, pruned, stream)
HS_NATIVE(stratify_prune) {
    if (!arity(n, 6)) return nullptr;
    Reader r;
    hs_tree_batch t; hs_policy p; hs_quant_out q; hs_pruned_tree k;
    r.tree(a[1], &t); r.pointers(a[2], k_quant, 14, &q); r.policy(a[3], &p); r.pointers(a[4], k_pruned, 11, &k);
    HS_DONE(hs_stratify_prune(ctx, &t, &q, &p, &k, stream));
}
// (ctx, tree, quant, policy, slo_class, budget, pruned, stream)
HS_NATIVE(stratify_prune_budget) {
    if (!arity(n, 8)) return nullptr;
    Reader r;
    hs_tree_batch t; hs_policy p; hs_quant_out q; hs_pruned_tree k;
    r.tree(a[1], &t); r.pointers(a[2], k_quant, 14, &q); r.policy(a[3], &p); r.pointers(a[6], k_pruned, 11, &k);
    const int32_t* slo = (const int32_t*)r.ptr(a[4]);
    const int budget = (int)r.integer(a[5]);
    HS_DONE(hs_stratify_prune_budget(ctx, &t, &q, &p, slo, budget, &k, stream));
}
// (ctx, pruned, q, k_tree, v_tree, k_cache, v_cache, kv_off, batch, max_nodes, max_kv_len, layout, node_off | None,
//  sm_scale | None, out, lse | None, stream)
HS_NATIVE(tree_verify_attention) {
    if (!arity(n, 17)) return nullptr;
    Reader r;
    hs_pruned_tree k; hs_attn_desc d;
    r.pointers(a[1], k_pruned, 11, &k);
    d.batch = (int)r.integer(a[8]);
    d.max_rows = (int)r.size(a[2], o_zero);
    d.max_nodes = (int)r.integer(a[9]);
    d.kv_total = (int)r.size(a[5], o_zero);
    d.max_kv_len = (int)r.integer(a[10]);
    d.hq = (int)r.size(a[2], o_one);
    d.hkv = (int)r.size(a[3], o_one);
    d.head_dim = (int)r.size(a[2], o_two);
    d.layout = (int)r.integer(a[11]);
    d.node_off = (const int32_t*)r.ptr(a[12]);
    d.kv_off = (const int32_t*)r.ptr(a[7]);
    d.kv_token_stride = d.kv_total ? r.stride(a[5], o_zero) : (int64_t)d.hkv * d.head_dim;
    d.kv_head_stride = d.kv_total ? r.stride(a[5], o_one) : d.head_dim;
    if (a[13] == Py_None) {
        // 1 / sqrt(head_dim), the default (for the one supported head size a constant)
        d.sm_scale = d.head_dim == HS_HEAD_DIM ? 0.08838834764831845f : 1.f;
    } else {
        d.sm_scale = (float)r.real(a[13]);
    }
    const void *q = r.ptr(a[2]), *kt = r.ptr(a[3]), *vt = r.ptr(a[4]), *kc = r.ptr(a[5]), *vc = r.ptr(a[6]);
    void* out = r.ptr(a[14]);
    float* lse = (float*)r.ptr(a[15]);
    HS_DONE(hs_tree_verify_attention(ctx, &k, &d, q, kt, vt, kc, vc, out, lse, stream));
}
// (ctx, tree, pruned, target, target_layout, draft | None, mode, temperature, seed, offset, uniforms | None, accept, stream)
HS_NATIVE(accept_path) {
    if (!arity(n, 13)) return nullptr;
    Reader r;
    hs_tree_batch t; hs_pruned_tree k; hs_accept_out o;
    r.tree(a[1], &t); r.pointers(a[2], k_pruned, 11, &k); r.pointers(a[11], k_accept, 7, &o);
    o.path_cap = r.field_int(a[11], k_accept[7]);
    o.max_kept_rows = r.field_int(a[11], k_accept[8]);
    const void *x = r.ptr(a[3]), *q = r.ptr(a[5]);
    const hs_dtype dt = r.dtype(a[3]);
    const long long rs = r.stride(a[3], o_zero), v = r.size(a[3], o_one);
    const int layout = (int)r.integer(a[4]);
    const int32_t* mode = (const int32_t*)r.ptr(a[6]);
    const float *temp = (const float*)r.ptr(a[7]), *u = (const float*)r.ptr(a[10]);
    const uint64_t seed = (uint64_t)r.integer(a[8]), offset = (uint64_t)r.integer(a[9]);
    HS_DONE(hs_accept_path(ctx, &t, &k, x, layout, q, dt, rs, (int)v, mode, temp, seed, offset, u, &o, stream));
}
// (ctx, state, stream)
HS_NATIVE(expand_init) {
    if (!arity(n, 3)) return nullptr;
    Reader r;
    hs_expand_state s;
    r.expand(a[1], &s);
    HS_DONE(hs_expand_init(ctx, &s, stream));
}
// (ctx, state, topk_val, topk_idx, row_lse, stream)
HS_NATIVE(expand_level) {
    if (!arity(n, 6)) return nullptr;
    Reader r;
    hs_expand_state s;
    r.expand(a[1], &s);
    const float* tv = (const float*)r.ptr(a[2]);
    const int32_t* ti = (const int32_t*)r.ptr(a[3]);
    const float* lse = (const float*)r.ptr(a[4]);
    const int stride = (int)r.size(a[2], o_one);
    HS_DONE(hs_expand_level(ctx, &s, tv, ti, lse, stride, stream));
}
// (ctx, state, n_top | None, n_default, node_off, parent, token, cand_id, depth, stream)
HS_NATIVE(rerank) {
    if (!arity(n, 10)) return nullptr;
    Reader r;
    hs_expand_state s;
    r.expand(a[1], &s);
    const int32_t* top = (const int32_t*)r.ptr(a[2]);
    const int def = (int)r.integer(a[3]);
    int32_t* o[5];
    for (int i = 0; i < 5; ++i) o[i] = (int32_t*)r.ptr(a[4 + i]);
    HS_DONE(hs_rerank(ctx, &s, top, def, o[0], o[1], o[2], o[3], o[4], stream));
}

// setup(torch.float32, torch.bfloat16)
HS_NATIVE(setup) {
    if (!arity(n, 2)) return nullptr;
    t_f32 = Py_NewRef(a[0]);
    t_bf16 = Py_NewRef(a[1]);
    Py_RETURN_NONE;
}

#define HS_METHOD(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {HS_METHOD(setup), HS_METHOD(entropy_quantify), HS_METHOD(entropy_quantify_prune),
                         HS_METHOD(stratify_prune), HS_METHOD(stratify_prune_budget), HS_METHOD(tree_verify_attention),
                         HS_METHOD(accept_path), HS_METHOD(expand_init), HS_METHOD(expand_level), HS_METHOD(rerank),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    n_data_ptr = PyUnicode_InternFromString("data_ptr");
    n_stride = PyUnicode_InternFromString("stride");
    n_size = PyUnicode_InternFromString("size");
    n_dtype = PyUnicode_InternFromString("dtype");
    o_zero = PyLong_FromLong(0);
    o_one = PyLong_FromLong(1);
    o_two = PyLong_FromLong(2);
    if (!n_data_ptr || !n_stride || !n_size || !n_dtype || !o_zero || !o_one || !o_two ||
        !intern_all(k_tree, 5) || !intern_all(k_quant, 14) || !intern_all(k_pruned, 11) || !intern_all(k_accept, 9) ||
        !intern_all(k_expand, 12) || !intern_all(k_policy, 9))
        return nullptr;
    return PyModule_Create(&module);
}
