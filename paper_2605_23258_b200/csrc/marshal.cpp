// Argument marshalling of the calls that a serving loop makes, as a CPython module: what binding.py does with ctypes, without a Python
// object for every pointer.  A call here answers the plain case -- tensors of exactly torch's own classes, structs and counts of exactly
// their own types, the current stream -- and returns None for everything else (other types, a wrong dtype, device or layout, a given
// stream), before anything has been launched: binding.py then takes its own path, which raises what it
// raised before.
// A step of one layer (append and attention, 10.5 us on the device) took 14.2 us of host time, 6.3 of them in the library.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include "vector.h"

namespace {

#define ENTRY_POINTS(X) \
    X(vector_score) X(vector_route) X(vector_route_layer) X(vector_compact) X(vector_compact_layer) X(vector_append) X(vector_decode_attn) \
        X(vector_decode_attn_layer) X(vector_decode_attn_static)
#define POINTER(name) decltype(&::name) p_##name = nullptr;
ENTRY_POINTS(POINTER)

PyTypeObject *shape_type = nullptr, *budget_type = nullptr, *cache_type = nullptr;
enum Name { BATCH, N_LAYERS, N_Q_HEADS, N_KV_HEADS, HEAD_DIM, DTYPE, WINDOW, POOL_KERNEL, SM_SCALE, ROPE_ENABLED, ROPE_THETA, N_TOKENS,
            N_BUDGET_PAIRS, N_A, N_POOL, N_APX, N_RET, N_EVICT, RET_K, RET_V, APX_K, RET_POS, APX_POS, NAMES };
const char* const spelled[NAMES] = {"batch", "n_layers", "n_q_heads", "n_kv_heads", "head_dim", "dtype", "window", "pool_kernel", "sm_scale",
                                    "rope_enabled", "rope_theta", "n_tokens", "n_budget_pairs", "n_a", "n_pool", "n_apx", "n_ret",
                                    "n_evict", "ret_k", "ret_v", "apx_k", "ret_pos", "apx_pos"};
PyObject* name[NAMES];

// The plain case does not hold: the caller's own path decides.
struct Otherwise {};

struct Ref {                                            // an owned reference
    PyObject* o;
    explicit Ref(PyObject* p) : o(p) { if (!p) { PyErr_Clear(); throw Otherwise(); } }
    ~Ref() { Py_DECREF(o); }
    Ref(const Ref&) = delete;
};
Ref attr(PyObject* o, Name n) { return Ref(PyObject_GetAttr(o, name[n])); }

int64_t integer(PyObject* o) {
    if (!PyLong_CheckExact(o)) throw Otherwise();
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    if (over) throw Otherwise();
    return v;
}
int32_t integer32(PyObject* o) {
    const int64_t v = integer(o);
    if (v != (int32_t)v) throw Otherwise();
    return (int32_t)v;
}
float number(PyObject* o) {
    if (!PyFloat_CheckExact(o)) throw Otherwise();
    const double v = PyFloat_AS_DOUBLE(o);
    if (!(v >= -3.4e38 && v <= 3.4e38)) throw Otherwise();
    return (float)v;
}
const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_CheckExact(o)) throw Otherwise();
    return THPVariable_Unpack(o);
}

vector_shape shape_of(PyObject* o) {
    if (Py_TYPE(o) != shape_type) throw Otherwise();
    vector_shape s;
    s.batch = integer32(attr(o, BATCH).o);
    s.n_layers = integer32(attr(o, N_LAYERS).o);
    s.n_q_heads = integer32(attr(o, N_Q_HEADS).o);
    s.n_kv_heads = integer32(attr(o, N_KV_HEADS).o);
    s.head_dim = integer32(attr(o, HEAD_DIM).o);
    s.dtype = integer32(attr(o, DTYPE).o);
    s.window = integer32(attr(o, WINDOW).o);
    s.pool_kernel = integer32(attr(o, POOL_KERNEL).o);
    s.sm_scale = number(attr(o, SM_SCALE).o);
    s.rope_enabled = integer32(attr(o, ROPE_ENABLED).o);
    s.rope_theta = number(attr(o, ROPE_THETA).o);
    return s;
}
vector_budget budget_of(PyObject* o) {
    if (Py_TYPE(o) != budget_type) throw Otherwise();
    vector_budget b;
    b.n_tokens = integer(attr(o, N_TOKENS).o);
    b.n_budget_pairs = integer(attr(o, N_BUDGET_PAIRS).o);
    b.n_a = integer(attr(o, N_A).o);
    b.n_pool = integer(attr(o, N_POOL).o);
    b.n_apx = integer(attr(o, N_APX).o);
    b.n_ret = integer(attr(o, N_RET).o);
    b.n_evict = integer(attr(o, N_EVICT).o);
    return b;
}
vector_cache cache_of(PyObject* o) {
    if (Py_TYPE(o) != cache_type) throw Otherwise();
    const Ref rk = attr(o, RET_K), rv = attr(o, RET_V), ak = attr(o, APX_K), rp = attr(o, RET_POS), ap = attr(o, APX_POS);
    const at::Tensor &trk = tensor(rk.o), &tak = tensor(ak.o);
    if (trk.dim() < 2 || tak.dim() < 2) throw Otherwise();
    vector_cache c;
    c.ret_k = trk.data_ptr();
    c.ret_v = tensor(rv.o).data_ptr();
    c.apx_k = tak.data_ptr();
    c.ret_pos = (decltype(c.ret_pos))tensor(rp.o).data_ptr();
    c.apx_pos = (decltype(c.apx_pos))tensor(ap.o).data_ptr();
    c.cap_ret = trk.size(1);
    c.cap_apx = tak.size(1);
    c.n_ret = integer(attr(o, N_RET).o);
    c.n_apx = integer(attr(o, N_APX).o);
    return c;
}
at::ScalarType type_of(const vector_shape& s) { return s.dtype == VECTOR_BF16 ? at::kBFloat16 : at::kFloat; }
void* device(PyObject* o, at::ScalarType type) {
    if (o == Py_None) return nullptr;
    const at::Tensor& t = tensor(o);
    if (!t.is_cuda() || !t.is_contiguous() || t.scalar_type() != type) throw Otherwise();
    return t.data_ptr();
}
struct Workspace { void* p; size_t n; };
Workspace workspace(PyObject* o) {
    Workspace w = {device(o, at::kByte), 0};
    if (o != Py_None) w.n = (size_t)tensor(o).numel();
    return w;
}
struct Out { void* p; int32_t type; };
Out output(PyObject* o) {
    const at::ScalarType type = tensor(o).scalar_type();
    if (type != at::kFloat && type != at::kBFloat16) throw Otherwise();
    return {device(o, type), type == at::kBFloat16 ? VECTOR_BF16 : VECTOR_F32};
}
void* stream_of(PyObject* o) {
    if (o != Py_None) throw Otherwise();
    return c10::cuda::getCurrentCUDAStream().stream();
}

// What `call` returns as a Python integer; None where the plain case does not hold.  The library runs without the interpreter's lock,
// as it does under ctypes.
template <typename F>
PyObject* plain(Py_ssize_t given, Py_ssize_t wanted, F call) {
    if (given != wanted) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; }
    try {
        return PyLong_FromLong(call());
    } catch (const Otherwise&) {
    } catch (const std::exception&) {                   // torch's refusals: a tensor without storage, say
    }
    PyErr_Clear();
    Py_RETURN_NONE;
}
template <typename F>
long unlocked(F f) {
    long rc;
    Py_BEGIN_ALLOW_THREADS
    rc = (long)f();
    Py_END_ALLOW_THREADS
    return rc;
}

#define METHOD(name) PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n)
METHOD(score) {                                         // shape, Q_obs, K, N, scores, raw_out, ws, stream
    return plain(n, 8, [&] {
        const vector_shape s = shape_of(a[0]);
        void *q = device(a[1], type_of(s)), *k = device(a[2], type_of(s));
        const int64_t N = integer(a[3]);
        float *out = (float*)device(a[4], at::kFloat), *raw = (float*)device(a[5], at::kFloat);
        const Workspace w = workspace(a[6]);
        void* st = stream_of(a[7]);
        return unlocked([&] { return p_vector_score(&s, q, k, N, out, raw, w.p, w.n, st); });
    });
}
template <typename Fn>
long route_with(Fn fn, PyObject* const* a) {            // shape, budget, scores, K, V, W, tier, ret_idx, apx_idx, eps_out, pool_idx_out, ws, stream
    const vector_shape s = shape_of(a[0]);
    const vector_budget b = budget_of(a[1]);
    const at::ScalarType type = type_of(s);
    const float* scores = (const float*)device(a[2], at::kFloat);
    void *k = device(a[3], type), *v = device(a[4], type), *w = device(a[5], type);
    uint8_t* tier = (uint8_t*)device(a[6], at::kByte);
    int32_t *ret = (int32_t*)device(a[7], at::kInt), *apx = (int32_t*)device(a[8], at::kInt);
    float* eps = (float*)device(a[9], at::kFloat);
    int32_t* pool = (int32_t*)device(a[10], at::kInt);
    const Workspace ws = workspace(a[11]);
    void* st = stream_of(a[12]);
    return unlocked([&] { return fn(&s, &b, scores, k, v, w, tier, ret, apx, eps, pool, ws.p, ws.n, st); });
}
METHOD(route) { return plain(n, 13, [&] { return route_with(p_vector_route, a); }); }
METHOD(route_layer) { return plain(n, 13, [&] { return route_with(p_vector_route_layer, a); }); }
template <typename Fn>
long compact_with(Fn fn, PyObject* const* a) {          // shape, budget, K, V, ret_idx, apx_idx, cache, stream
    const vector_shape s = shape_of(a[0]);
    const vector_budget b = budget_of(a[1]);
    void *k = device(a[2], type_of(s)), *v = device(a[3], type_of(s));
    const int32_t *ret = (const int32_t*)device(a[4], at::kInt), *apx = (const int32_t*)device(a[5], at::kInt);
    const vector_cache c = cache_of(a[6]);
    void* st = stream_of(a[7]);
    return unlocked([&] { return fn(&s, &b, k, v, ret, apx, &c, st); });
}
METHOD(compact) { return plain(n, 8, [&] { return compact_with(p_vector_compact, a); }); }
METHOD(compact_layer) { return plain(n, 8, [&] { return compact_with(p_vector_compact_layer, a); }); }
METHOD(decode_attn) {                                   // shape, q, cache, W, out, mode, ws, stream
    return plain(n, 8, [&] {
        const vector_shape s = shape_of(a[0]);
        void* q = device(a[1], type_of(s));
        const vector_cache c = cache_of(a[2]);
        void* W = device(a[3], type_of(s));
        const Out out = output(a[4]);
        const int32_t mode = integer32(a[5]);
        const Workspace w = workspace(a[6]);
        void* st = stream_of(a[7]);
        return unlocked([&] { return p_vector_decode_attn(&s, q, &c, W, out.p, out.type, mode, w.p, w.n, st); });
    });
}
METHOD(decode_attn_layer) {                             // shape, q, cache, W_layer, out, ws, stream
    return plain(n, 7, [&] {
        const vector_shape s = shape_of(a[0]);
        void* q = device(a[1], type_of(s));
        const vector_cache c = cache_of(a[2]);
        void* W = device(a[3], type_of(s));
        const Out out = output(a[4]);
        const Workspace w = workspace(a[5]);
        void* st = stream_of(a[6]);
        return unlocked([&] { return p_vector_decode_attn_layer(&s, q, &c, W, out.p, out.type, w.p, w.n, st); });
    });
}
METHOD(decode_attn_static) {                            // shape, q, cache, W, out, mode, stream
    return plain(n, 7, [&] {
        const vector_shape s = shape_of(a[0]);
        void* q = device(a[1], type_of(s));
        const vector_cache c = cache_of(a[2]);
        void* W = device(a[3], type_of(s));
        const Out out = output(a[4]);
        const int32_t mode = integer32(a[5]);
        void* st = stream_of(a[6]);
        return unlocked([&] { return p_vector_decode_attn_static(&s, q, &c, W, out.p, out.type, mode, st); });
    });
}
METHOD(append) {                                        // shape, cache, k_new, v_new, pos, stream
    return plain(n, 6, [&] {
        const vector_shape s = shape_of(a[0]);
        const vector_cache c = cache_of(a[1]);
        void *k = device(a[2], type_of(s)), *v = device(a[3], type_of(s));
        const int32_t pos = integer32(a[4]);
        void* st = stream_of(a[5]);
        return unlocked([&] { return p_vector_append(&s, &c, k, v, pos, st); });
    });
}
// Compressor.append's own conditions on top: plain rows of the shape's size on the current device, room for one more, and not what the
// entry point refuses (rows off a 16-byte boundary): those rows are assigned.
METHOD(append_rows) {                                   // shape, cache, k_new, v_new, pos
    return plain(n, 5, [&] {
        const vector_shape s = shape_of(a[0]);
        const vector_cache c = cache_of(a[1]);
        if ((PyObject*)Py_TYPE(a[2]) != THPVariableClass || (PyObject*)Py_TYPE(a[3]) != THPVariableClass) throw Otherwise();
        const Ref rk = attr(a[1], RET_K), rv = attr(a[1], RET_V), rp = attr(a[1], RET_POS);
        const at::Tensor &trk = tensor(rk.o), &trv = tensor(rv.o), &tk = tensor(a[2]), &tv = tensor(a[3]);
        if (trk.dim() != 3 || tk.dim() != 2 || tv.dim() != 2) throw Otherwise();
        const int64_t U = trk.size(0), cap = trk.size(1), d = trk.size(2);
        const bool rows = tk.size(0) == U && tk.size(1) == d && tv.size(0) == U && tv.size(1) == d && d == s.head_dim &&
                          U == (int64_t)s.batch * s.n_layers * s.n_kv_heads;
        const int dev = c10::cuda::current_device();
        const bool here = tk.get_device() == dev && tv.get_device() == dev && trk.get_device() == dev && trv.get_device() == dev;
        if (!rows || !here || c.n_ret >= cap || trv.nbytes() != trk.nbytes() || !trk.is_contiguous() || !trv.is_contiguous() ||
            tensor(rp.o).numel() != U * cap || tk.requires_grad() || tv.requires_grad())
            throw Otherwise();
        void *k = device(a[2], type_of(s)), *v = device(a[3], type_of(s));
        const int32_t pos = integer32(a[4]);
        void* st = stream_of(Py_None);
        const long rc = unlocked([&] { return p_vector_append(&s, &c, k, v, pos, st); });
        if (rc == VECTOR_ERR_SHAPE) throw Otherwise();
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
    for (int i = 0; i < 3; ++i) Py_INCREF(a[1 + i]);
    shape_type = (PyTypeObject*)a[1];
    budget_type = (PyTypeObject*)a[2];
    cache_type = (PyTypeObject*)a[3];
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
