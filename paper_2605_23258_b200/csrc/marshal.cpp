// Argument marshalling of the calls that a serving loop makes, as a CPython module: what binding.py does with ctypes, without a Python
// object for every pointer.  A call here answers the plain case -- tensors of exactly torch's own classes, structs of the binding's
// own classes or of classes that pack like them, numbers that struct.pack and ctypes would take, the current stream or a stream's handle -- and returns None for everything else
// (other classes, a wrong dtype, device or layout, a tensor missing), before anything has been launched: binding.py then takes its own path,
// which raises what it raised before.  What is refused is refused without an exception, at the first argument that is not plain.
// A step of one layer (append and attention, 10.5 us on the device) took 14.2 us of host time, 6.3 of them in the library.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>

#include "vector.h"

namespace {

#define ENTRY_POINTS(X) \
    X(vector_score) X(vector_route) X(vector_route_layer) X(vector_compact) X(vector_compact_layer) X(vector_append) X(vector_decode_attn) \
        X(vector_decode_attn_layer) X(vector_decode_attn_static)
#define POINTER(name) decltype(&::name) p_##name = nullptr;
ENTRY_POINTS(POINTER)

// A class of the binding, and what makes up the packed form that ctypes is given: a class derived from it is read like it where these
// members are still the base's.
struct Class {
    static constexpr int MEMBERS = 2;
    PyTypeObject* type = nullptr;
    PyObject* name[MEMBERS] = {};
    PyObject* member[MEMBERS] = {};
    bool covers(PyObject* o) const {
        if (Py_TYPE(o) == type) return true;
        if (!PyType_IsSubtype(Py_TYPE(o), type)) return false;
        for (int i = 0; i < MEMBERS; ++i)
            if (name[i]) {
                PyObject* m = PyObject_GetAttr((PyObject*)Py_TYPE(o), name[i]);
                Py_XDECREF(m);
                if (m != member[i]) return false;
            }
        return true;
    }
    bool set(PyObject* t, const char* first, const char* second = nullptr) {
        Py_INCREF(t);
        type = (PyTypeObject*)t;
        const char* const names[MEMBERS] = {first, second};
        for (int i = 0; i < MEMBERS; ++i)
            if (names[i] && (!(name[i] = PyUnicode_InternFromString(names[i])) || !(member[i] = PyObject_GetAttr(t, name[i])))) return false;
        return true;
    }
};
Class shape_class, budget_class, cache_class;
enum Name { BATCH, N_LAYERS, N_Q_HEADS, N_KV_HEADS, HEAD_DIM, DTYPE, WINDOW, POOL_KERNEL, SM_SCALE, ROPE_ENABLED, ROPE_THETA, N_TOKENS,
            N_BUDGET_PAIRS, N_A, N_POOL, N_APX, N_RET, N_EVICT, RET_K, RET_V, APX_K, RET_POS, APX_POS, NAMES };
const char* const spelled[NAMES] = {"batch", "n_layers", "n_q_heads", "n_kv_heads", "head_dim", "dtype", "window", "pool_kernel", "sm_scale",
                                    "rope_enabled", "rope_theta", "n_tokens", "n_budget_pairs", "n_a", "n_pool", "n_apx", "n_ret",
                                    "n_evict", "ret_k", "ret_v", "apx_k", "ret_pos", "apx_pos"};
PyObject* name[NAMES];

struct Ref {                                            // an owned reference, or none
    PyObject* o;
    explicit Ref(PyObject* p) : o(p) {}
    ~Ref() { Py_XDECREF(o); }
    Ref(const Ref&) = delete;
};
struct Workspace { void* p = nullptr; size_t n = 0; };
struct Out { void* p = nullptr; int32_t type = 0; };
at::ScalarType type_of(const vector_shape& s) { return s.dtype == VECTOR_BF16 ? at::kBFloat16 : at::kFloat; }

// Reads a call's arguments.  `plain` turns false at the first one that is not: what is read from then on is nothing and means nothing.
struct Reader {
    bool plain = true;
    bool need(bool holds) { return plain = plain && holds; }
    PyObject* attr(PyObject* o, Name n) {               // new, or null
        PyObject* v = plain ? PyObject_GetAttr(o, name[n]) : nullptr;
        need(v);
        return v;
    }
    int64_t integer(PyObject* o) {                      // an argument: ctypes takes an int
        if (!need(o && PyLong_Check(o))) return 0;
        int over = 0;
        const long long v = PyLong_AsLongLongAndOverflow(o, &over);
        need(!over);
        return v;
    }
    int32_t integer32(PyObject* o) {
        const int64_t v = integer(o);
        need(v == (int32_t)v);
        return (int32_t)v;
    }
    int64_t field(PyObject* o, Name n) {                // a struct's field: struct.pack takes whatever is an index
        const Ref v(attr(o, n));
        if (!plain || PyLong_Check(v.o)) return integer(v.o);
        if (!need(PyIndex_Check(v.o))) return 0;
        const Ref i(PyNumber_Index(v.o));
        return need(i.o) ? integer(i.o) : 0;
    }
    int32_t field32(PyObject* o, Name n) {
        const int64_t v = field(o, n);
        need(v == (int32_t)v);
        return (int32_t)v;
    }
    float number(PyObject* o, Name n) {                 // whatever is a float, an integer too
        const Ref v(attr(o, n));
        if (!plain) return 0.f;
        const double x = PyFloat_AsDouble(v.o);
        need(!PyErr_Occurred() && std::isfinite((float)x));
        return (float)x;
    }
    const at::Tensor* tensor(PyObject* o) { return need(o && THPVariable_CheckExact(o)) ? &THPVariable_Unpack(o) : nullptr; }
    void* device(PyObject* o, at::ScalarType type) {
        const at::Tensor* t = tensor(o);
        return t && need(t->is_cuda() && t->is_contiguous() && t->scalar_type() == type) ? t->data_ptr() : nullptr;
    }
    void* optional(PyObject* o, at::ScalarType type) { return o == Py_None ? nullptr : device(o, type); }
    Workspace workspace(PyObject* o) {
        Workspace w;
        w.p = optional(o, at::kByte);
        if (plain && o != Py_None) w.n = (size_t)tensor(o)->numel();
        return w;
    }
    Out output(PyObject* o) {
        Out out;
        const at::Tensor* t = tensor(o);
        if (!t || !need(t->scalar_type() == at::kFloat || t->scalar_type() == at::kBFloat16)) return out;
        out.type = t->scalar_type() == at::kBFloat16 ? VECTOR_BF16 : VECTOR_F32;
        out.p = device(o, t->scalar_type());
        return out;
    }
    void* stream(PyObject* o) {                         // None, the current one, or a handle
        if (!plain) return nullptr;
        if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        if (!need(PyLong_CheckExact(o))) return nullptr;
        void* p = PyLong_AsVoidPtr(o);
        need(!PyErr_Occurred());
        return p;
    }
    vector_shape shape(PyObject* o) {
        vector_shape s = {};
        if (!need(shape_class.covers(o))) return s;
        s.batch = field32(o, BATCH);
        s.n_layers = field32(o, N_LAYERS);
        s.n_q_heads = field32(o, N_Q_HEADS);
        s.n_kv_heads = field32(o, N_KV_HEADS);
        s.head_dim = field32(o, HEAD_DIM);
        s.dtype = field32(o, DTYPE);
        s.window = field32(o, WINDOW);
        s.pool_kernel = field32(o, POOL_KERNEL);
        s.sm_scale = number(o, SM_SCALE);
        s.rope_enabled = field32(o, ROPE_ENABLED);
        s.rope_theta = number(o, ROPE_THETA);
        return s;
    }
    vector_budget budget(PyObject* o) {
        vector_budget b = {};
        if (!need(budget_class.covers(o))) return b;
        b.n_tokens = field(o, N_TOKENS);
        b.n_budget_pairs = field(o, N_BUDGET_PAIRS);
        b.n_a = field(o, N_A);
        b.n_pool = field(o, N_POOL);
        b.n_apx = field(o, N_APX);
        b.n_ret = field(o, N_RET);
        b.n_evict = field(o, N_EVICT);
        return b;
    }
    vector_cache cache(PyObject* o) {
        vector_cache c = {};
        if (!need(cache_class.covers(o))) return c;
        const Ref rk(attr(o, RET_K)), rv(attr(o, RET_V)), ak(attr(o, APX_K)), rp(attr(o, RET_POS)), ap(attr(o, APX_POS));
        const at::Tensor *trk = tensor(rk.o), *trv = tensor(rv.o), *tak = tensor(ak.o), *trp = tensor(rp.o), *tap = tensor(ap.o);
        if (!plain || !need(trk->dim() >= 2 && tak->dim() >= 2)) return c;
        c.ret_k = trk->data_ptr();
        c.ret_v = trv->data_ptr();
        c.apx_k = tak->data_ptr();
        c.ret_pos = (decltype(c.ret_pos))trp->data_ptr();
        c.apx_pos = (decltype(c.apx_pos))tap->data_ptr();
        c.cap_ret = trk->size(1);
        c.cap_apx = tak->size(1);
        c.n_ret = field(o, N_RET);
        c.n_apx = field(o, N_APX);
        return c;
    }
};

// What `call` returns as a Python integer; None where the plain case does not hold.
template <typename F>
PyObject* plain(Py_ssize_t given, Py_ssize_t wanted, F call) {
    if (given != wanted) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; }
    Reader r;
    long rc = 0;
    try {
        rc = call(r);
    } catch (const std::exception&) {                   // torch's refusals: a tensor without storage, say
        r.plain = false;
    }
    if (r.plain) return PyLong_FromLong(rc);
    PyErr_Clear();
    Py_RETURN_NONE;
}
// The library runs without the interpreter's lock, as it does under ctypes; nothing runs where the plain case does not hold.
template <typename F>
long run(const Reader& r, F f) {
    long rc = 0;
    if (!r.plain) return rc;
    Py_BEGIN_ALLOW_THREADS
    rc = (long)f();
    Py_END_ALLOW_THREADS
    return rc;
}

#define METHOD(name) PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n)
METHOD(score) {                                         // shape, Q_obs, K, N, scores, raw_out, ws, stream
    return plain(n, 8, [&](Reader& r) {
        const vector_shape s = r.shape(a[0]);
        void *q = r.device(a[1], type_of(s)), *k = r.device(a[2], type_of(s));
        const int64_t N = r.integer(a[3]);
        float *out = (float*)r.device(a[4], at::kFloat), *raw = (float*)r.optional(a[5], at::kFloat);
        const Workspace w = r.workspace(a[6]);
        void* st = r.stream(a[7]);
        return run(r, [&] { return p_vector_score(&s, q, k, N, out, raw, w.p, w.n, st); });
    });
}
template <typename Fn>
long route_with(Fn fn, Reader& r, PyObject* const* a) { // shape, budget, scores, K, V, W, tier, ret_idx, apx_idx, eps_out, pool_idx_out, ws, stream
    const vector_shape s = r.shape(a[0]);
    const vector_budget b = r.budget(a[1]);
    const at::ScalarType type = type_of(s);
    const float* scores = (const float*)r.device(a[2], at::kFloat);
    void *k = r.device(a[3], type), *v = r.device(a[4], type), *w = r.device(a[5], type);
    uint8_t* tier = (uint8_t*)r.device(a[6], at::kByte);
    int32_t *ret = (int32_t*)r.device(a[7], at::kInt), *apx = (int32_t*)r.device(a[8], at::kInt);
    float* eps = (float*)r.optional(a[9], at::kFloat);
    int32_t* pool = (int32_t*)r.optional(a[10], at::kInt);
    const Workspace ws = r.workspace(a[11]);
    void* st = r.stream(a[12]);
    return run(r, [&] { return fn(&s, &b, scores, k, v, w, tier, ret, apx, eps, pool, ws.p, ws.n, st); });
}
METHOD(route) { return plain(n, 13, [&](Reader& r) { return route_with(p_vector_route, r, a); }); }
METHOD(route_layer) { return plain(n, 13, [&](Reader& r) { return route_with(p_vector_route_layer, r, a); }); }
template <typename Fn>
long compact_with(Fn fn, Reader& r, PyObject* const* a) {      // shape, budget, K, V, ret_idx, apx_idx, cache, stream
    const vector_shape s = r.shape(a[0]);
    const vector_budget b = r.budget(a[1]);
    void *k = r.device(a[2], type_of(s)), *v = r.device(a[3], type_of(s));
    const int32_t *ret = (const int32_t*)r.device(a[4], at::kInt), *apx = (const int32_t*)r.device(a[5], at::kInt);
    const vector_cache c = r.cache(a[6]);
    void* st = r.stream(a[7]);
    return run(r, [&] { return fn(&s, &b, k, v, ret, apx, &c, st); });
}
METHOD(compact) { return plain(n, 8, [&](Reader& r) { return compact_with(p_vector_compact, r, a); }); }
METHOD(compact_layer) { return plain(n, 8, [&](Reader& r) { return compact_with(p_vector_compact_layer, r, a); }); }
METHOD(decode_attn) {                                   // shape, q, cache, W, out, mode, ws, stream
    return plain(n, 8, [&](Reader& r) {
        const vector_shape s = r.shape(a[0]);
        void* q = r.device(a[1], type_of(s));
        const vector_cache c = r.cache(a[2]);
        void* W = r.device(a[3], type_of(s));
        const Out out = r.output(a[4]);
        const int32_t mode = r.integer32(a[5]);
        const Workspace w = r.workspace(a[6]);
        void* st = r.stream(a[7]);
        return run(r, [&] { return p_vector_decode_attn(&s, q, &c, W, out.p, out.type, mode, w.p, w.n, st); });
    });
}
METHOD(decode_attn_layer) {                             // shape, q, cache, W_layer, out, ws, stream
    return plain(n, 7, [&](Reader& r) {
        const vector_shape s = r.shape(a[0]);
        void* q = r.device(a[1], type_of(s));
        const vector_cache c = r.cache(a[2]);
        void* W = r.device(a[3], type_of(s));
        const Out out = r.output(a[4]);
        const Workspace w = r.workspace(a[5]);
        void* st = r.stream(a[6]);
        return run(r, [&] { return p_vector_decode_attn_layer(&s, q, &c, W, out.p, out.type, w.p, w.n, st); });
    });
}
METHOD(decode_attn_static) {                            // shape, q, cache, W, out, mode, stream
    return plain(n, 7, [&](Reader& r) {
        const vector_shape s = r.shape(a[0]);
        void* q = r.device(a[1], type_of(s));
        const vector_cache c = r.cache(a[2]);
        void* W = r.device(a[3], type_of(s));
        const Out out = r.output(a[4]);
        const int32_t mode = r.integer32(a[5]);
        void* st = r.stream(a[6]);
        return run(r, [&] { return p_vector_decode_attn_static(&s, q, &c, W, out.p, out.type, mode, st); });
    });
}
METHOD(append) {                                        // shape, cache, k_new, v_new, pos, stream
    return plain(n, 6, [&](Reader& r) {
        const vector_shape s = r.shape(a[0]);
        const vector_cache c = r.cache(a[1]);
        void *k = r.device(a[2], type_of(s)), *v = r.device(a[3], type_of(s));
        const int32_t pos = r.integer32(a[4]);
        void* st = r.stream(a[5]);
        return run(r, [&] { return p_vector_append(&s, &c, k, v, pos, st); });
    });
}
// Compressor.append's own conditions on top: plain rows of the shape's size on the current device, room for one more, and not what the
// entry point refuses (rows off a 16-byte boundary): those rows are assigned.
METHOD(append_rows) {                                   // shape, cache, k_new, v_new, pos
    return plain(n, 5, [&](Reader& r) {
        const vector_shape s = r.shape(a[0]);
        const vector_cache c = r.cache(a[1]);
        r.need((PyObject*)Py_TYPE(a[2]) == THPVariableClass && (PyObject*)Py_TYPE(a[3]) == THPVariableClass);
        const Ref rk(r.attr(a[1], RET_K)), rv(r.attr(a[1], RET_V)), rp(r.attr(a[1], RET_POS));
        const at::Tensor *trk = r.tensor(rk.o), *trv = r.tensor(rv.o), *trp = r.tensor(rp.o), *tk = r.tensor(a[2]), *tv = r.tensor(a[3]);
        if (!r.plain || !r.need(trk->dim() == 3 && tk->dim() == 2 && tv->dim() == 2)) return 0L;
        const int64_t U = trk->size(0), cap = trk->size(1), d = trk->size(2);
        const bool rows = tk->size(0) == U && tk->size(1) == d && tv->size(0) == U && tv->size(1) == d && d == s.head_dim &&
                          U == (int64_t)s.batch * s.n_layers * s.n_kv_heads;
        const int dev = c10::cuda::current_device();
        const bool here = tk->get_device() == dev && tv->get_device() == dev && trk->get_device() == dev && trv->get_device() == dev;
        r.need(rows && here && c.n_ret < cap && trv->nbytes() == trk->nbytes() && trk->is_contiguous() && trv->is_contiguous() &&
               trp->numel() == U * cap && !tk->requires_grad() && !tv->requires_grad());
        void *k = r.device(a[2], type_of(s)), *v = r.device(a[3], type_of(s));
        const int32_t pos = r.integer32(a[4]);
        void* st = r.stream(Py_None);
        const long rc = run(r, [&] { return p_vector_append(&s, &c, k, v, pos, st); });
        r.need(rc != VECTOR_ERR_SHAPE);
        return rc;
    });
}
// The library's entry points, by the handle of the library that ctypes has loaded, and the classes of the three structs.
METHOD(bind) {
    if (n != 4 || !PyLong_Check(a[0]) || !PyType_Check(a[1]) || !PyType_Check(a[2]) || !PyType_Check(a[3])) {
        PyErr_SetString(PyExc_TypeError, "bind(handle, Shape, Budget, Cache)");
        return nullptr;
    }
    void* handle = PyLong_AsVoidPtr(a[0]);
#define RESOLVE(name)                                                                                             \
    p_##name = (decltype(p_##name))dlsym(handle, #name);                                                          \
    if (!p_##name) { PyErr_SetString(PyExc_ImportError, "libvector.so does not export " #name); return nullptr; }
    ENTRY_POINTS(RESOLVE)
    if (!shape_class.set(a[1], "_p", "torch_dtype") || !budget_class.set(a[2], "_p") || !cache_class.set(a[3], "_p")) return nullptr;
    Py_RETURN_NONE;
}

#define ROW(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ROW(bind), ROW(score), ROW(route), ROW(route_layer), ROW(compact), ROW(compact_layer), ROW(append), ROW(append_rows),
                         ROW(decode_attn), ROW(decode_attn_layer), ROW(decode_attn_static), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
    for (int i = 0; i < NAMES; ++i)
        if (!(name[i] = PyUnicode_InternFromString(spelled[i]))) return nullptr;
    return PyModule_Create(&module);
}
