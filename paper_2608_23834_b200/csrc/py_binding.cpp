// Python fast path of the calls a decode step makes: argument checks and marshalling in C++, then the C ABI call.
//
// What bounds a small call from Python is not the GPU but the marshalling: 15 attribute and dtype comparisons, a
// dozen ctypes conversions and a Stream object are about 10 us per call (and 8 us per layer of a several-layer
// call), against 3 us for the launch itself.  Here a call costs about 1 us plus the launch.  Every function
// returns 0 (enqueued), a negative mkv_status, or kCheck when an argument is not what the call takes; nothing has
// been enqueued then and the Python caller goes through its own checks, which say what is wrong.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "mkv.h"

namespace {

constexpr long kCheck = 1;

// what the checks of a call need of its pool (held by the Python Pool as a capsule)
struct PoolRef {
    mkv_pool* pool;
    int hkv, hq, d;
};
const char* kCapsule = "mkv.pool_ref";
PyObject *s_workspace, *s_ref, *s_cuda_stream, *s_ws_bytes;

void free_ref(PyObject* capsule) { delete static_cast<PoolRef*>(PyCapsule_GetPointer(capsule, kCapsule)); }

PyObject* pool_ref(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 4) {
        PyErr_SetString(PyExc_TypeError, "pool_ref(handle, kv_heads, q_heads, head_dim)");
        return nullptr;
    }
    auto* r = new PoolRef;
    r->pool = static_cast<mkv_pool*>(PyLong_AsVoidPtr(a[0]));
    r->hkv = (int)PyLong_AsLong(a[1]);
    r->hq = (int)PyLong_AsLong(a[2]);
    r->d = (int)PyLong_AsLong(a[3]);
    if (PyErr_Occurred()) {
        delete r;
        return nullptr;
    }
    return PyCapsule_New(r, kCapsule, free_ref);
}

const PoolRef* ref_of(PyObject* o)
{
    return PyCapsule_IsValid(o, kCapsule) ? static_cast<const PoolRef*>(PyCapsule_GetPointer(o, kCapsule)) : nullptr;
}

// the tensor behind a Python object, or null
const at::Tensor* tensor(PyObject* o) { return o && THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr; }

bool is(const at::Tensor* t, at::ScalarType dtype) { return t && t->scalar_type() == dtype; }
bool is_dense(const at::Tensor* t, at::ScalarType dtype) { return is(t, dtype) && t->is_contiguous(); }
bool shape3(const at::Tensor* t, int64_t a, int64_t b, int64_t c)
{
    return t->dim() == 3 && t->size(0) == a && t->size(1) == b && t->size(2) == c;
}
// a tensor argument that may be None
bool optional(PyObject* o, void** ptr)
{
    *ptr = nullptr;
    if (o == Py_None) return true;
    const at::Tensor* t = tensor(o);
    if (!t) return false;
    *ptr = t->data_ptr();
    return true;
}

// None: the current stream of the current device; else a torch.cuda.Stream
bool stream_of(PyObject* o, void** s)
{
    if (o == Py_None) {
        *s = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* v = PyObject_GetAttr(o, s_cuda_stream);
    if (!v) {
        PyErr_Clear();
        return false;
    }
    *s = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        return false;
    }
    return true;
}

PyObject* result(long rc) { return PyLong_FromLong(rc); }

// the C call with the interpreter lock released
template <typename Call>
PyObject* enqueue(Call call)
{
    long rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return result(rc);
}

// append(ref, k, v, slot_mapping, stream)
PyObject* append(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    const PoolRef* r = n == 5 ? ref_of(a[0]) : nullptr;
    const at::Tensor *k = r ? tensor(a[1]) : nullptr, *v = r ? tensor(a[2]) : nullptr, *slots = r ? tensor(a[3]) : nullptr;
    void* s;
    if (!is_dense(k, at::kBFloat16) || !is_dense(v, at::kBFloat16) || !is(slots, at::kInt) || k->dim() != 3 ||
        !shape3(k, k->size(0), r->hkv, r->d) || !v->sizes().equals(k->sizes()) || !stream_of(a[4], &s))
        return result(kCheck);
    const int tokens = (int)k->size(0);
    const void *kp = k->data_ptr(), *vp = v->data_ptr();
    const auto* sp = static_cast<const int32_t*>(slots->data_ptr());
    return enqueue([=] { return mkv_append(r->pool, kp, vp, sp, tokens, s); });
}

// demote / promote(ref, src, dst, block_table, tier_tag, entry_index, stream)
template <int32_t (*F)(mkv_pool*, const int32_t*, const int32_t*, int32_t, int32_t*, uint8_t*, const int64_t*, int64_t, void*)>
PyObject* convert(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    const PoolRef* r = n == 7 ? ref_of(a[0]) : nullptr;
    const at::Tensor *src = r ? tensor(a[1]) : nullptr, *dst = r ? tensor(a[2]) : nullptr;
    void *bt, *tags, *entry, *s;
    if (!is(src, at::kInt) || !is(dst, at::kInt) || src->numel() != dst->numel() || !optional(a[3], &bt) ||
        !optional(a[4], &tags) || !optional(a[5], &entry) || !stream_of(a[6], &s))
        return result(kCheck);
    if (a[5] != Py_None && (!is(tensor(a[5]), at::kLong) || !is(tensor(a[3]), at::kInt) || !is(tensor(a[4]), at::kByte)))
        return result(kCheck);
    const int64_t entries = a[4] == Py_None ? 0 : tensor(a[4])->numel();
    const int pages = (int)src->numel();
    const auto *sp = static_cast<const int32_t*>(src->data_ptr()), *dp = static_cast<const int32_t*>(dst->data_ptr());
    return enqueue([=] {
        return F(r->pool, sp, dp, pages, static_cast<int32_t*>(bt), static_cast<uint8_t*>(tags), static_cast<const int64_t*>(entry),
                 entries, s);
    });
}

// The arguments that every decode call shares.
struct DecodeArgs {
    const PoolRef* r;
    const void* q;
    const int32_t *bt, *lens;
    const uint8_t* tags;
    int B, max_pages;
    float scale;
    void *out, *lse, *ws, *stream;
    size_t ws_bytes;
};

bool same_shape2(const at::Tensor* t, int64_t a, int64_t b) { return t->dim() == 2 && t->size(0) == a && t->size(1) == b; }

// (ref, q, block_table, tier_tag, seq_lens, scale, out, lse, workspace, stream, ...)
bool decode_args(PyObject* const* a, DecodeArgs& d)
{
    d.r = ref_of(a[0]);
    if (!d.r) return false;
    const at::Tensor *q = tensor(a[1]), *bt = tensor(a[2]), *tags = tensor(a[3]), *lens = tensor(a[4]), *ws = tensor(a[8]);
    if (!is_dense(q, at::kBFloat16) || q->dim() != 3 || !shape3(q, q->size(0), d.r->hq, d.r->d)) return false;
    d.B = (int)q->size(0);
    if (!is_dense(bt, at::kInt) || bt->dim() != 2 || bt->size(0) != d.B) return false;
    if (!is_dense(tags, at::kByte) || !same_shape2(tags, d.B, bt->size(1))) return false;
    if (!is(lens, at::kInt) || lens->numel() != d.B || !ws) return false;
    d.scale = (float)PyFloat_AsDouble(a[5]);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        return false;
    }
    if (a[6] == Py_None || !optional(a[6], &d.out) || !optional(a[7], &d.lse) || !stream_of(a[9], &d.stream)) return false;
    d.max_pages = (int)bt->size(1);
    d.q = q->data_ptr();
    d.bt = static_cast<const int32_t*>(bt->data_ptr());
    d.tags = static_cast<const uint8_t*>(tags->data_ptr());
    d.lens = static_cast<const int32_t*>(lens->data_ptr());
    d.ws = ws->data_ptr();
    d.ws_bytes = (size_t)ws->numel();
    return true;
}

PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    DecodeArgs d;
    if (n != 10 || !decode_args(a, d)) return result(kCheck);
    return enqueue([&] {
        return mkv_decode_attention(d.r->pool, d.q, d.bt, d.tags, d.lens, d.B, d.max_pages, d.scale, static_cast<float*>(d.out),
                                    static_cast<float*>(d.lse), d.ws, d.ws_bytes, d.stream);
    });
}

// as decode, then page_mass
PyObject* decode_scored(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    DecodeArgs d;
    void* mass;
    if (n != 11 || !decode_args(a, d) || a[10] == Py_None || !optional(a[10], &mass)) return result(kCheck);
    return enqueue([&] {
        return mkv_decode_attention_scored(d.r->pool, d.q, d.bt, d.tags, d.lens, d.B, d.max_pages, d.scale,
                                           static_cast<float*>(d.out), static_cast<float*>(d.lse), static_cast<float*>(mass),
                                           d.ws, d.ws_bytes, d.stream);
    });
}

// A Python sequence of at least n items; PySequence_Fast objects are released on destruction.
struct Items {
    PyObject* fast;
    explicit Items(PyObject* o) : fast(PySequence_Fast(o, "")) { if (!fast) PyErr_Clear(); }
    ~Items() { Py_XDECREF(fast); }
    Py_ssize_t size() const { return fast ? PySequence_Fast_GET_SIZE(fast) : -1; }
    PyObject* operator[](Py_ssize_t i) const { return PySequence_Fast_GET_ITEM(fast, i); }
};

// an attribute of a Pool, held while it is looked at (it may be a property that makes a new object)
struct Attr {
    PyObject* o;
    Attr(PyObject* of, PyObject* name) : o(PyObject_GetAttr(of, name)) { if (!o) PyErr_Clear(); }
    Attr(const Attr&) = delete;
    ~Attr() { Py_XDECREF(o); }
};

// decode_layers(pools, qs, block_tables, tier_tags, seq_lens, scale, outs, lses, stream)
PyObject* decode_layers(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 9) return result(kCheck);
    const Items pools(a[0]), qs(a[1]), bts(a[2]), tags(a[3]), outs(a[6]);
    const bool with_lse = a[7] != Py_None;
    const Items lses(with_lse ? a[7] : a[6]);
    const Py_ssize_t L = pools.size();
    void* s;
    const at::Tensor* lens = tensor(a[4]);
    if (L < 1 || L > MKV_MAX_LAYERS_PER_CALL || qs.size() < L || bts.size() < L || tags.size() < L || outs.size() < L ||
        lses.size() < L || !is(lens, at::kInt) || !stream_of(a[8], &s))
        return result(kCheck);
    const float scale = (float)PyFloat_AsDouble(a[5]);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        return result(kCheck);
    }
    mkv_layer_call calls[MKV_MAX_LAYERS_PER_CALL];
    int64_t B = 0, width = 0;
    size_t ws_bytes = 0;
    for (Py_ssize_t i = 0; i < L; ++i) {
        const Attr ref(pools[i], s_ref), workspace(pools[i], s_workspace);
        const PoolRef* r = ref.o ? ref_of(ref.o) : nullptr;
        const at::Tensor *ws = tensor(workspace.o), *q = tensor(qs[i]), *bt = tensor(bts[i]), *tg = tensor(tags[i]),
                         *out = tensor(outs[i]);
        if (!r || !ws || !is_dense(q, at::kBFloat16) || q->dim() != 3 || !is_dense(bt, at::kInt) || bt->dim() != 2)
            return result(kCheck);
        if (i == 0) {
            B = q->size(0);
            width = bt->size(1);
            const Attr nb(pools[0], s_ws_bytes);
            if (!nb.o) return result(kCheck);
            ws_bytes = PyLong_AsSize_t(nb.o);
            if (PyErr_Occurred()) {
                PyErr_Clear();
                return result(kCheck);
            }
        }
        if (!shape3(q, B, r->hq, r->d) || !same_shape2(bt, B, width) || !is_dense(tg, at::kByte) || !same_shape2(tg, B, width) ||
            !is_dense(out, at::kFloat) || !shape3(out, B, r->hq, r->d))
            return result(kCheck);
        void* lse = nullptr;
        if (with_lse && !optional(lses[i], &lse)) return result(kCheck);
        calls[i] = {r->pool, q->data_ptr(), static_cast<const int32_t*>(bt->data_ptr()), static_cast<const uint8_t*>(tg->data_ptr()),
                    static_cast<float*>(out->data_ptr()), static_cast<float*>(lse), ws->data_ptr()};
    }
    if (lens->numel() != B) return result(kCheck);
    const auto* lp = static_cast<const int32_t*>(lens->data_ptr());
    return enqueue([&] {
        return mkv_decode_attention_layers(calls, (int)L, lp, (int)B, (int)width, scale, ws_bytes, s);
    });
}

// append_layers(pools, ks, vs, slot_mapping, stream)
PyObject* append_layers(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 5) return result(kCheck);
    const Items pools(a[0]), ks(a[1]), vs(a[2]);
    const Py_ssize_t L = pools.size();
    void* s;
    const at::Tensor* slots = tensor(a[3]);
    if (L < 1 || L > MKV_MAX_LAYERS_PER_CALL || ks.size() < L || vs.size() < L || !is(slots, at::kInt) || !stream_of(a[4], &s))
        return result(kCheck);
    mkv_layer_append calls[MKV_MAX_LAYERS_PER_CALL];
    const int64_t tokens = slots->numel();
    for (Py_ssize_t i = 0; i < L; ++i) {
        const Attr ref(pools[i], s_ref);
        const PoolRef* r = ref.o ? ref_of(ref.o) : nullptr;
        const at::Tensor *k = tensor(ks[i]), *v = tensor(vs[i]);
        if (!r || !is_dense(k, at::kBFloat16) || !is_dense(v, at::kBFloat16) || !shape3(k, tokens, r->hkv, r->d) ||
            !v->sizes().equals(k->sizes()))
            return result(kCheck);
        calls[i] = {r->pool, k->data_ptr(), v->data_ptr()};
    }
    const auto* sp = static_cast<const int32_t*>(slots->data_ptr());
    return enqueue([&] { return mkv_append_layers(calls, (int)L, sp, (int)tokens, s); });
}

// score_update(page_mass, seq_lens, head_mask, beta, score, stream, page_tokens)
PyObject* score_update(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 7) return result(kCheck);
    const at::Tensor *mass = tensor(a[0]), *lens = tensor(a[1]), *score = tensor(a[4]);
    void* s;
    if (!is_dense(mass, at::kFloat) || mass->dim() != 3 || !is_dense(score, at::kFloat) || !is(lens, at::kInt) ||
        !same_shape2(score, mass->size(0), mass->size(2)) || lens->numel() != mass->size(0) || !stream_of(a[5], &s))
        return result(kCheck);
    const uint64_t mask = PyLong_AsUnsignedLongLong(a[2]);
    const float beta = (float)PyFloat_AsDouble(a[3]);
    const long page = PyLong_AsLong(a[6]);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        return result(kCheck);
    }
    const auto *mp = static_cast<const float*>(mass->data_ptr());
    const auto* lp = static_cast<const int32_t*>(lens->data_ptr());
    auto* sp = static_cast<float*>(score->data_ptr());
    const int B = (int)mass->size(0), hq = (int)mass->size(1), pages = (int)mass->size(2);
    return enqueue([=] { return mkv_page_score_update_paged(mp, lp, B, hq, pages, (int)page, mask, beta, sp, s); });
}

// A C++ exception of a check (an argument that is not an ordinary tensor) becomes kCheck.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    try {
        return F(self, a, n);
    } catch (...) {
        return result(kCheck);
    }
}

#define FAST(name, ...) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<__VA_ARGS__>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST("pool_ref", pool_ref), FAST("append", append), FAST("demote", convert<mkv_demote>), FAST("promote", convert<mkv_promote>),
    FAST("decode", decode), FAST("decode_scored", decode_scored), FAST("decode_layers", decode_layers),
    FAST("append_layers", append_layers), FAST("score_update", score_update), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mkv_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__mkv_native()
{
    s_workspace = PyUnicode_InternFromString("workspace");
    s_ref = PyUnicode_InternFromString("_ref");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_ws_bytes = PyUnicode_InternFromString("ws_bytes");
    return PyModule_Create(&module);
}
