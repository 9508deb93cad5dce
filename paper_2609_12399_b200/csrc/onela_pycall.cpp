// Native argument marshalling for the Python binding (binding.py): the calls a decode loop makes, from torch tensors to
// the C ABI of libonela.so.
//
// What bounds it: host time.  Through ctypes a call cost 9 - 20 us of Python (shape tuples, dtype comparisons, one
// ctypes object per pointer, the current stream looked up through torch.cuda) against 2 - 10 us of kernel, so every
// call of a small batch waited for the host: a generation of the 8-beam fp32 workload took 99 us for 19 us of kernels.
// The same checks on the tensors' C++ objects take a fraction of a microsecond: 99 -> 33 us for that generation, 134 ->
// 72 us for the 128-beam one (four calls, 63 us of kernels).
//
// A call returns the library's status, or NOT_TAKEN when an argument is not what the fast path expects; binding.py
// then repeats the call through its own checks, which name the argument that is wrong.  Nothing is launched before all
// arguments have passed.  The library's functions are called through addresses handed over by binding.py, so this
// module works on whichever build of the library the process has loaded.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <initializer_list>

#include "onela.h"

namespace {

constexpr long NOT_TAKEN = 1;

struct Api {
    decltype(&onela_export_chains) export_chains;
    decltype(&onela_init_shared_state) init_state;
    decltype(&onela_init_shared_states) init_states;
    decltype(&onela_prefill_shared_state) prefill;
    decltype(&onela_reorder_beams) reorder;
    decltype(&onela_select_beams) select;
    decltype(&onela_append_records) append;
    decltype(&onela_decode_step) decode;
    decltype(&onela_append_decode_step) append_decode;
    decltype(&onela_export_shared_state) export_state;
    decltype(&onela_release_request) release;
};
constexpr int API_FUNCTIONS = sizeof(Api) / sizeof(void*);

struct Caller {
    PyObject_HEAD
    Api api;
    onela_ctx* ctx;
    onela_config cfg;
    int64_t Hv;
    at::ScalarType rec, out;
};

// ---- arguments ----
bool int_of(PyObject* o, int32_t& v) {
    if (!PyLong_Check(o)) return false;
    const long x = PyLong_AsLong(o);
    if ((x == -1 && PyErr_Occurred()) || x != (int32_t)x) {
        PyErr_Clear();
        return false;
    }
    v = (int32_t)x;
    return true;
}

bool tensor_of(PyObject* o, at::ScalarType type, std::initializer_list<int64_t> shape, void*& p) {
    if (!THPVariable_Check(o)) return false;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.scalar_type() != type || t.layout() != at::kStrided) return false;
    const auto sizes = t.sizes();
    if (sizes.size() != shape.size()) return false;
    size_t i = 0;
    for (const int64_t n : shape)
        if (sizes[i++] != n) return false;
    if (!t.is_contiguous()) return false;
    p = t.data_ptr();
    return true;
}

bool stream_of(PyObject* o, void*& stream) {
    if (o == Py_None) {
        stream = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* raw = PyObject_GetAttrString(o, "cuda_stream");
    if (!raw) {
        PyErr_Clear();
        return false;
    }
    stream = PyLong_AsVoidPtr(raw);
    Py_DECREF(raw);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        return false;
    }
    return true;
}

// beam width (and depth) of a request; 0 when it has none
int32_t width_of(const Caller* c, int32_t request, int32_t* depth = nullptr) {
    int32_t d = 0, w = 0;
    c->api.export_chains(c->ctx, request, nullptr, &d, &w, nullptr);
    if (depth) *depth = d;
    return w;
}

template <class F>
PyObject* call(F f) {
    onela_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}
PyObject* not_taken() { return PyLong_FromLong(NOT_TAKEN); }

// ---- the calls (positional arguments as in binding.py, the stream last) ----
PyObject* init_state(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r, l;
    void *S0, *s;
    if (n != 4 || !int_of(a[0], r) || !int_of(a[1], l) || !tensor_of(a[2], at::kFloat, {c->Hv, c->cfg.dv, c->cfg.dk}, S0) || !stream_of(a[3], s))
        return not_taken();
    return call([&] { return c->api.init_state(c->ctx, r, l, static_cast<const float*>(S0), s); });
}

PyObject* init_states(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r0, nr;
    void *S0, *s;
    if (n != 4 || !int_of(a[0], r0) || !int_of(a[1], nr) ||
        !tensor_of(a[2], at::kFloat, {nr, c->cfg.num_layers, c->Hv, c->cfg.dv, c->cfg.dk}, S0) || !stream_of(a[3], s))
        return not_taken();
    return call([&] { return c->api.init_states(c->ctx, r0, nr, static_cast<const float*>(S0), s); });
}

PyObject* prefill(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r, l;
    void *k, *v, *al, *be, *s;
    if (n != 7 || !int_of(a[0], r) || !int_of(a[1], l) || !THPVariable_Check(a[2])) return not_taken();
    const at::Tensor& kt = THPVariable_Unpack(a[2]);
    if (!kt.defined() || kt.dim() != 3 || kt.size(0) > INT32_MAX) return not_taken();
    const int64_t T = kt.size(0), H = c->cfg.num_heads;
    if (!tensor_of(a[2], c->rec, {T, H, c->cfg.dk}, k) || !tensor_of(a[3], c->rec, {T, H, c->cfg.dv}, v) ||
        !tensor_of(a[4], at::kFloat, {T, H}, al) || !tensor_of(a[5], at::kFloat, {T, H}, be) || !stream_of(a[6], s))
        return not_taken();
    return call([&] {
        return c->api.prefill(c->ctx, r, l, k, v, static_cast<const float*>(al), static_cast<const float*>(be), (int32_t)T, s);
    });
}

PyObject* reorder(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r0, nr, W;
    void *par = nullptr, *s;
    if (n != 5 || !int_of(a[0], r0) || !int_of(a[1], nr) || !int_of(a[3], W) ||
        (a[2] != Py_None && !tensor_of(a[2], at::kInt, {nr, W}, par)) || !stream_of(a[4], s))
        return not_taken();
    return call([&] { return c->api.reorder(c->ctx, r0, nr, static_cast<const int32_t*>(par), W, s); });
}

PyObject* select_beams(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r0, nr, C, W_new, depth;
    if (n != 10 || !int_of(a[0], r0) || !int_of(a[1], nr) || !int_of(a[4], C) || !int_of(a[5], W_new)) return not_taken();
    const int32_t W = width_of(c, r0, &depth), W_prev = depth >= 1 ? W : 1;
    void *bs, *lp, *par, *codes, *sc, *s;
    if (!tensor_of(a[2], at::kFloat, {nr, W_prev}, bs) || !tensor_of(a[3], at::kFloat, {nr, W_prev, C}, lp) ||
        !tensor_of(a[6], at::kInt, {nr, W_new}, par) || !tensor_of(a[7], at::kInt, {nr, W_new}, codes) ||
        !tensor_of(a[8], at::kFloat, {nr, W_new}, sc) || !stream_of(a[9], s))
        return not_taken();
    return call([&] {
        return c->api.select(c->ctx, r0, nr, static_cast<const float*>(bs), static_cast<const float*>(lp), C, W_new, static_cast<int32_t*>(par),
                             static_cast<int32_t*>(codes), static_cast<float*>(sc), s);
    });
}

struct Token {       // one decode call's records of a layer
    void *k, *v, *alpha, *beta;
};
bool token_of(const Caller* c, PyObject* const* a, int32_t nr, int32_t W, Token& t) {
    const int64_t Hk = c->cfg.num_heads;
    return tensor_of(a[0], c->rec, {nr, W, Hk, c->cfg.dk}, t.k) && tensor_of(a[1], c->rec, {nr, W, c->Hv, c->cfg.dv}, t.v) &&
           tensor_of(a[2], at::kFloat, {nr, W, c->Hv}, t.alpha) && tensor_of(a[3], at::kFloat, {nr, W, c->Hv}, t.beta);
}
bool query_of(const Caller* c, PyObject* const* a, int32_t nr, int32_t W, void*& q, void*& out) {
    return tensor_of(a[0], c->rec, {nr, W, (int64_t)c->cfg.num_heads, c->cfg.dk}, q) && tensor_of(a[1], c->out, {nr, W, c->Hv, c->cfg.dv}, out);
}

PyObject* append(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r0, nr, l;
    Token t;
    void* s;
    if (n != 8 || !int_of(a[0], r0) || !int_of(a[1], nr) || !int_of(a[2], l) || !token_of(c, a + 3, nr, width_of(c, r0), t) || !stream_of(a[7], s))
        return not_taken();
    return call([&] {
        return c->api.append(c->ctx, r0, nr, l, t.k, t.v, static_cast<const float*>(t.alpha), static_cast<const float*>(t.beta), s);
    });
}

PyObject* decode(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r0, nr, l;
    void *q, *out, *s;
    if (n != 6 || !int_of(a[0], r0) || !int_of(a[1], nr) || !int_of(a[2], l) || !query_of(c, a + 3, nr, width_of(c, r0), q, out) || !stream_of(a[5], s))
        return not_taken();
    return call([&] { return c->api.decode(c->ctx, r0, nr, l, q, out, s); });
}

PyObject* append_decode(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r0, nr, l;
    if (n != 10 || !int_of(a[0], r0) || !int_of(a[1], nr) || !int_of(a[2], l)) return not_taken();
    const int32_t W = width_of(c, r0);
    Token t;
    void *q, *out, *s;
    if (!token_of(c, a + 3, nr, W, t) || !query_of(c, a + 7, nr, W, q, out) || !stream_of(a[9], s)) return not_taken();
    return call([&] {
        return c->api.append_decode(c->ctx, r0, nr, l, t.k, t.v, static_cast<const float*>(t.alpha), static_cast<const float*>(t.beta), q, out, s);
    });
}

PyObject* export_state(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r, l;
    void *S0, *s;
    if (n != 4 || !int_of(a[0], r) || !int_of(a[1], l) || !tensor_of(a[2], at::kFloat, {c->Hv, c->cfg.dv, c->cfg.dk}, S0) || !stream_of(a[3], s))
        return not_taken();
    return call([&] { return c->api.export_state(c->ctx, r, l, static_cast<float*>(S0), s); });
}

PyObject* release(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    auto* c = reinterpret_cast<Caller*>(self);
    int32_t r;
    if (n != 1 || !int_of(a[0], r)) return not_taken();
    return PyLong_FromLong(c->api.release(c->ctx, r));
}

// ---- the type ----
// Caller(handle, config address, function addresses in the order of Api)
int caller_init(PyObject* self, PyObject* args, PyObject*) {
    auto* c = reinterpret_cast<Caller*>(self);
    unsigned long long handle, cfg;
    PyObject* fns;
    if (!PyArg_ParseTuple(args, "KKO!", &handle, &cfg, &PyTuple_Type, &fns)) return -1;
    if (PyTuple_GET_SIZE(fns) != API_FUNCTIONS) {
        PyErr_SetString(PyExc_ValueError, "wrong number of library functions");
        return -1;
    }
    void** slots = reinterpret_cast<void**>(&c->api);
    for (int i = 0; i < API_FUNCTIONS; ++i) {
        slots[i] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(fns, i));
        if (PyErr_Occurred()) return -1;
    }
    c->ctx = reinterpret_cast<onela_ctx*>(handle);
    c->cfg = *reinterpret_cast<const onela_config*>(cfg);
    c->Hv = c->cfg.num_v_heads > 0 ? c->cfg.num_v_heads : c->cfg.num_heads;
    c->rec = c->cfg.rec_dtype == ONELA_DTYPE_BF16 ? at::kBFloat16 : at::kFloat;
    c->out = c->cfg.out_dtype == ONELA_DTYPE_BF16 ? at::kBFloat16 : at::kFloat;
    return 0;
}

// a C++ exception (from torch's side of a look-up) becomes a Python one
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    try {
        return F(self, args, n);
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
#define METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<name>)), METH_FASTCALL, nullptr}
PyMethodDef caller_methods[] = {METHOD(init_state), METHOD(init_states),  METHOD(prefill), METHOD(reorder),       METHOD(select_beams),
                                METHOD(append),     METHOD(decode),       METHOD(append_decode), METHOD(export_state),  METHOD(release), {nullptr, nullptr, 0, nullptr}};
PyType_Slot caller_slots[] = {{Py_tp_init, reinterpret_cast<void*>(caller_init)},
                              {Py_tp_new, reinterpret_cast<void*>(PyType_GenericNew)},
                              {Py_tp_methods, caller_methods},
                              {0, nullptr}};
PyType_Spec caller_spec = {"_onela_pycall.Caller", sizeof(Caller), 0, Py_TPFLAGS_DEFAULT, caller_slots};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_onela_pycall", nullptr, -1, nullptr, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__onela_pycall() {
    PyObject* type = PyType_FromSpec(&caller_spec);
    if (!type) return nullptr;
    PyObject* m = PyModule_Create(&module_def);
    if (!m || PyModule_AddObjectRef(m, "Caller", type) < 0 || PyModule_AddIntConstant(m, "NOT_TAKEN", NOT_TAKEN) < 0) {
        Py_XDECREF(m);
        Py_DECREF(type);
        return nullptr;
    }
    Py_DECREF(type);
    return m;
}
