// rlm_py.cpp -- the Python binding's call path in native code.
//
// Building the C structures of one call from ctypes objects, attribute by attribute, took
// 8-20 us of Python per call on the host (a decode step runs 1.2 us on the GPU).  Host
// time of a call, before and now, on the GB300's Arm cores: decode step 12.6 -> 3.8 us,
// prefill 17.7 -> 5.5 (with a workspace from torch's allocator 27 -> 11), mixer prefill
// 31 -> 11, backward 29 -> 10; the C ABI itself takes 3.5 of them.  Each
// function here reads the tensors' attributes, fills the structures of rlm.h on the stack
// and calls the C ABI with the GIL released; it returns the call's status.  An argument
// that is not the plain case (a contiguous CUDA tensor of the expected type and rank,
// a stream handle) makes it return None, and the Python code beside it runs its own
// checks and raises its own error.
//
// No object, pointer or size is kept from one call to the next: only the interned
// attribute names, torch's dtype objects and five torch functions.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../../include/rlm.h"

namespace {

PyObject *s_dtype, *s_is_cuda, *s_is_contiguous, *s_shape, *s_data_ptr, *s_device, *s_cuda_stream;
PyObject *s_decay, *s_freq, *s_amp, *s_phase, *s_s, *s_coef, *s_conv_w, *s_scale, *s_c_raw, *s_lambda_c, *s_u, *s_index;
PyObject *g_f32, *g_bf16, *g_u8;                  // torch dtypes
PyObject *g_get_device, *g_get_stream, *g_empty, *g_raw_alloc, *g_raw_delete;  // torch functions
PyObject *g_empty_kw;                             // ("dtype", "device")
PyObject *g_numel, *g_element_size;

struct Shape {
    Py_ssize_t n;
    long long d[4];
};

bool is_true_attr(PyObject *o, PyObject *name) {
    PyObject *v = PyObject_GetAttr(o, name);
    if (!v) return false;
    const bool ok = v == Py_True;
    Py_DECREF(v);
    return ok;
}
bool is_true_call(PyObject *o, PyObject *name) {
    PyObject *v = PyObject_CallMethodNoArgs(o, name);
    if (!v) return false;
    const bool ok = v == Py_True;
    Py_DECREF(v);
    return ok;
}

// A contiguous CUDA tensor: its dtype object (borrowed, compared only), shape and pointer.
bool read_tensor(PyObject *t, PyObject **dtype, Shape *sh, void **ptr) {
    PyObject *dt = PyObject_GetAttr(t, s_dtype);
    if (!dt) return false;
    *dtype = dt;
    Py_DECREF(dt);   // torch's dtype objects live as long as torch
    if (!is_true_attr(t, s_is_cuda) || !is_true_call(t, s_is_contiguous)) return false;
    PyObject *shape = PyObject_GetAttr(t, s_shape);
    if (!shape) return false;
    bool ok = PyTuple_Check(shape) && PyTuple_GET_SIZE(shape) <= 4;
    if (ok) {
        sh->n = PyTuple_GET_SIZE(shape);
        for (Py_ssize_t i = 0; i < sh->n && ok; ++i) {
            sh->d[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(shape, i));
            ok = !(sh->d[i] == -1 && PyErr_Occurred());
        }
    }
    Py_DECREF(shape);
    if (!ok) return false;
    PyObject *p = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (!p) return false;
    *ptr = reinterpret_cast<void *>(PyLong_AsUnsignedLongLong(p));
    Py_DECREF(p);
    return !PyErr_Occurred();
}

bool field(PyObject *t, rlm_tensor *o) {
    PyObject *dt;
    Shape sh;
    if (!read_tensor(t, &dt, &sh, &o->ptr) || (dt != g_f32 && dt != g_bf16)) return false;
    o->dtype = dt == g_bf16 ? RLM_BF16 : RLM_F32;
    if (sh.n == 3) {
        o->B = sh.d[0];
        o->L = sh.d[1];
        o->D = sh.d[2];
    } else if (sh.n == 2) {   // a single token per batch row
        o->B = sh.d[0];
        o->L = 1;
        o->D = sh.d[1];
    } else {
        return false;
    }
    return true;
}

// An fp32 tensor attribute of the given rank.
bool plain(PyObject *o, PyObject *name, int rank, float **ptr, Shape *sh) {
    PyObject *t = PyObject_GetAttr(o, name);
    if (!t) return false;
    PyObject *dt;
    void *p;
    const bool ok = read_tensor(t, &dt, sh, &p) && dt == g_f32 && sh->n == rank;
    Py_DECREF(t);   // the caller's object keeps it
    *ptr = static_cast<float *>(p);
    return ok;
}
bool fits(long long v) { return v >= 0 && v <= 0x7fffffff; }

bool params(PyObject *o, rlm_params *p) {
    Shape a, b;
    float *q[4];
    if (!plain(o, s_decay, 2, &q[0], &a) || !plain(o, s_freq, 2, &q[1], &b) || !plain(o, s_amp, 2, &q[2], &b) ||
        !plain(o, s_phase, 2, &q[3], &b) || !fits(a.d[0]) || !fits(a.d[1]))
        return false;
    *p = rlm_params{q[0], q[1], q[2], q[3], (int)a.d[0], (int)a.d[1]};
    return true;
}
bool grads(PyObject *o, rlm_grads *g) {
    rlm_params p;
    if (!params(o, &p)) return false;
    *g = rlm_grads{const_cast<float *>(p.decay), const_cast<float *>(p.freq), const_cast<float *>(p.amp),
                   const_cast<float *>(p.phase), p.D, p.M};
    return true;
}
// Optional structures: *out is null for None.
bool state(PyObject *o, rlm_state *s, rlm_state **out) {
    *out = nullptr;
    if (o == Py_None) return true;
    Shape a, c;
    if (!plain(o, s_s, 4, &s->s, &a) || !plain(o, s_coef, 3, &s->coef, &c) || !fits(a.d[0]) || !fits(a.d[1]) ||
        !fits(a.d[2]))
        return false;
    s->B = (int)a.d[0];
    s->D = (int)a.d[1];
    s->M = (int)a.d[2];
    *out = s;
    return true;
}
bool opt_field(PyObject *o, rlm_tensor *t, rlm_tensor **out) {
    *out = nullptr;
    if (o == Py_None) return true;
    if (!field(o, t)) return false;
    *out = t;
    return true;
}
bool local_path(PyObject *o, rlm_local *l, rlm_local **out) {
    *out = nullptr;
    if (o == Py_None) return true;
    Shape a, b;
    float *w, *sc;
    if (!plain(o, s_conv_w, 2, &w, &a) || !plain(o, s_scale, 1, &sc, &b) || a.d[1] == 0 || !fits(a.d[0]) ||
        !fits(a.d[1]))
        return false;   // (K = 0 takes the general route)
    *l = rlm_local{w, sc, (int)a.d[0], (int)a.d[1]};
    *out = l;
    return true;
}
bool coupling(PyObject *o, rlm_coupling *c, rlm_coupling **out) {
    *out = nullptr;
    if (o == Py_None) return true;
    Shape a;
    float *p;
    if (!plain(o, s_c_raw, 2, &p, &a) || !fits(a.d[0])) return false;
    PyObject *v = PyObject_GetAttr(o, s_lambda_c);
    if (!v) return false;
    const double d = PyFloat_AsDouble(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) return false;
    *c = rlm_coupling{p, (float)d, (int)a.d[0]};
    *out = c;
    return true;
}
bool conv_state(PyObject *o, rlm_conv_state *c, rlm_conv_state **out) {
    *out = nullptr;
    if (o == Py_None) return true;
    PyObject *t = PyObject_GetAttr(o, s_u), *dt;
    if (!t) return false;
    Shape sh;
    void *p;
    const bool ok = read_tensor(t, &dt, &sh, &p) && (dt == g_f32 || dt == g_bf16) && sh.n == 3 && fits(sh.d[1] + 1) &&
                    fits(sh.d[2]);
    Py_DECREF(t);
    if (!ok) return false;
    *c = rlm_conv_state{sh.d[1] > 0 ? p : nullptr, dt == g_bf16 ? RLM_BF16 : RLM_F32, (int64_t)sh.d[0], (int)sh.d[2],
                        (int)sh.d[1] + 1};
    *out = c;
    return true;
}

// The stream handle: the current device's current stream for None.
bool stream_handle(PyObject *o, void **st) {
    PyObject *v;
    if (o == Py_None) {
        PyObject *dev = PyObject_CallNoArgs(g_get_device);
        if (!dev) return false;
        v = PyObject_CallOneArg(g_get_stream, dev);
        Py_DECREF(dev);
    } else if (PyLong_Check(o)) {
        v = o;
        Py_INCREF(v);
    } else {
        v = PyObject_GetAttr(o, s_cuda_stream);
    }
    if (!v) return false;
    *st = PyLong_Check(v) ? reinterpret_cast<void *>(PyLong_AsUnsignedLongLong(v)) : nullptr;
    const bool ok = PyLong_Check(v) && !PyErr_Occurred();
    Py_DECREF(v);
    return ok;
}

// The workspace of a call that brought none, given back once the call has been enqueued.
// torch's allocator hands a block that was freed to later work of the stream the block was
// allocated under, so it is allocated under the stream that the call runs on: by torch.empty
// when that is the current one, else by the allocator's entry that takes a stream.
struct Scratch {
    PyObject *tensor = nullptr;   // torch.empty's, or
    PyObject *raw = nullptr;      // the address from raw_alloc
    void release() {
        Py_XDECREF(tensor);
        if (raw) {
            PyObject *r = PyObject_CallOneArg(g_raw_delete, raw);
            if (!r) PyErr_WriteUnraisable(g_raw_delete);
            Py_XDECREF(r);
            Py_DECREF(raw);
        }
        tensor = raw = nullptr;
    }
};

// Whether st is the current stream of the current device, and that device's index.
bool current(void *st, long *device, bool *is) {
    PyObject *dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return false;
    *device = PyLong_AsLong(dev);
    void *now = nullptr;
    PyObject *v = PyObject_CallOneArg(g_get_stream, dev);
    Py_DECREF(dev);
    if (!v) return false;
    now = reinterpret_cast<void *>(PyLong_AsUnsignedLongLong(v));
    Py_DECREF(v);
    *is = now == st;
    return !PyErr_Occurred();
}

bool allocate(size_t need, PyObject *stream, PyObject *like, rlm_launch *ln, Scratch *own) {
    long device = 0;
    bool same = true;
    if (stream != Py_None && !current(ln->stream, &device, &same)) return false;
    PyObject *n = PyLong_FromSize_t(need), *dev = PyObject_GetAttr(like, s_device);
    bool ok = n && dev;
    if (ok && same) {
        PyObject *args[3] = {n, g_u8, dev};
        own->tensor = PyObject_Vectorcall(g_empty, args, 1, g_empty_kw);
        PyObject *p = own->tensor ? PyObject_CallMethodNoArgs(own->tensor, s_data_ptr) : nullptr;
        if (p) ln->workspace = reinterpret_cast<void *>(PyLong_AsUnsignedLongLong(p));
        Py_XDECREF(p);
        ok = p && !PyErr_Occurred();
    } else if (ok) {
        // raw_alloc takes the current device's memory: the fields' device, or not the plain case.
        PyObject *idx = PyObject_GetAttr(dev, s_index);
        ok = idx && PyLong_Check(idx) && PyLong_AsLong(idx) == device;
        Py_XDECREF(idx);
        PyObject *handle = ok ? PyLong_FromVoidPtr(ln->stream) : nullptr;
        PyObject *args[2] = {n, handle};
        own->raw = handle ? PyObject_Vectorcall(g_raw_alloc, args, 2, nullptr) : nullptr;
        Py_XDECREF(handle);
        if (own->raw) ln->workspace = PyLong_AsVoidPtr(own->raw);
        ok = own->raw && !PyErr_Occurred();
    }
    Py_XDECREF(n);
    Py_XDECREF(dev);
    if (!ok) {
        PyErr_Clear();   // the call takes the Python route, which raises its own
        own->release();
    }
    ln->workspace_bytes = need;
    return ok;
}

// The launch context: the caller's workspace, or a fresh one of `need` bytes.
bool launch(PyObject *stream, PyObject *ws, size_t need, PyObject *like, rlm_launch *ln, Scratch *own) {
    ln->workspace = nullptr;
    ln->workspace_bytes = 0;
    if (!stream_handle(stream, &ln->stream)) return false;
    if (ws == Py_None) return need == 0 || allocate(need, stream, like, ln, own);
    PyObject *p = PyObject_CallMethodNoArgs(ws, s_data_ptr);
    PyObject *n = p ? PyObject_CallMethodNoArgs(ws, g_numel) : nullptr;
    PyObject *e = n ? PyObject_CallMethodNoArgs(ws, g_element_size) : nullptr;
    if (e) {
        ln->workspace = reinterpret_cast<void *>(PyLong_AsUnsignedLongLong(p));
        ln->workspace_bytes = PyLong_AsSize_t(n) * PyLong_AsSize_t(e);
    }
    Py_XDECREF(p);
    Py_XDECREF(n);
    Py_XDECREF(e);
    return e && !PyErr_Occurred();
}

// Not the plain case: the Python code beside the call decides.
PyObject *other() {
    PyErr_Clear();
    Py_RETURN_NONE;
}

template <typename F>
PyObject *finish(Scratch &own, F call) {
    rlm_status s;
    Py_BEGIN_ALLOW_THREADS
    s = call();
    Py_END_ALLOW_THREADS
    own.release();
    return PyLong_FromLong((long)s);
}

// (x, params, state_in, y, state_out, workspace, stream)
PyObject *mix_prefill(PyObject *, PyObject *const *a, Py_ssize_t n) {
    rlm_tensor x, y;
    rlm_params p;
    rlm_state si, so, *psi, *pso;
    rlm_launch ln;
    Scratch own;
    if (n != 7 || !field(a[0], &x) || !params(a[1], &p) || !state(a[2], &si, &psi) || !field(a[3], &y) ||
        !state(a[4], &so, &pso) || x.D > 0x7fffffff)
        return other();
    const size_t need = a[5] == Py_None ? rlm_prefill_workspace_size(x.B, x.L, (int)x.D, p.M, x.dtype) : 0;
    if (!launch(a[6], a[5], need, a[0], &ln, &own)) return other();
    return finish(own, [&] { return rlm_mix_prefill_from(&x, &p, psi, &y, pso, &ln); });
}

// (x_t, state, y_t, stream)
PyObject *mix_decode(PyObject *, PyObject *const *a, Py_ssize_t n) {
    rlm_tensor x, y;
    rlm_state s, *ps;
    rlm_launch ln;
    Scratch own;
    if (n != 4 || !field(a[0], &x) || !state(a[1], &s, &ps) || !ps || !field(a[2], &y) ||
        !launch(a[3], Py_None, 0, a[0], &ln, &own))
        return other();
    return finish(own, [&] { return rlm_mix_decode(&x, ps, &y, &ln); });
}

// (dy, x, params, state_in, d_state_out, dx, dparams, d_state_in, workspace, stream)
PyObject *mix_backward(PyObject *, PyObject *const *a, Py_ssize_t n) {
    rlm_tensor dy, x, dx;
    rlm_params p;
    rlm_state si, go, ds, *psi, *pgo, *pds;
    rlm_grads g;
    rlm_launch ln;
    Scratch own;
    if (n != 10 || !field(a[0], &dy) || !field(a[1], &x) || !params(a[2], &p) || !state(a[3], &si, &psi) ||
        !state(a[4], &go, &pgo) || !field(a[5], &dx) || !grads(a[6], &g) || !state(a[7], &ds, &pds) ||
        x.D > 0x7fffffff)
        return other();
    const size_t need = a[8] == Py_None ? rlm_backward_workspace_size(x.B, x.L, (int)x.D, p.M, x.dtype) : 0;
    if (!launch(a[9], a[8], need, a[1], &ln, &own)) return other();
    return finish(own, [&] { return rlm_mix_backward_from(&dy, &x, &p, psi, pgo, &dx, &g, pds, &ln); });
}

// (x, g, params, local, coupling, state_in, conv_in, z, state_out, conv_out, workspace, stream)
PyObject *mixer_prefill(PyObject *, PyObject *const *a, Py_ssize_t n) {
    rlm_tensor x, g, z, *pg;
    rlm_params p;
    rlm_local l, *pl;
    rlm_coupling c, *pc;
    rlm_state si, so, *psi, *pso;
    rlm_conv_state ci, co, *pci, *pco;
    rlm_launch ln;
    Scratch own;
    if (n != 12 || !field(a[0], &x) || !opt_field(a[1], &g, &pg) || !params(a[2], &p) ||
        !local_path(a[3], &l, &pl) || !coupling(a[4], &c, &pc) || !state(a[5], &si, &psi) ||
        !conv_state(a[6], &ci, &pci) || !field(a[7], &z) || !state(a[8], &so, &pso) ||
        !conv_state(a[9], &co, &pco) || x.D > 0x7fffffff)
        return other();
    const size_t need = a[10] == Py_None ? rlm_prefill_workspace_size(x.B, x.L, (int)x.D, p.M, x.dtype) : 0;
    if (!launch(a[11], a[10], need, a[0], &ln, &own)) return other();
    return finish(own, [&] { return rlm_mixer_prefill(&x, pg, &p, pl, pc, psi, pci, &z, pso, pco, &ln); });
}

// (x_t, g_t, state, local, coupling, conv, z_t, stream)
PyObject *mixer_decode(PyObject *, PyObject *const *a, Py_ssize_t n) {
    rlm_tensor x, g, z, *pg;
    rlm_state s, *ps;
    rlm_local l, *pl;
    rlm_coupling c, *pc;
    rlm_conv_state cv, *pcv;
    rlm_launch ln;
    Scratch own;
    if (n != 8 || !field(a[0], &x) || !opt_field(a[1], &g, &pg) || !state(a[2], &s, &ps) || !ps ||
        !local_path(a[3], &l, &pl) || !coupling(a[4], &c, &pc) || !conv_state(a[5], &cv, &pcv) || !field(a[6], &z) ||
        !launch(a[7], Py_None, 0, a[0], &ln, &own))
        return other();
    return finish(own, [&] { return rlm_mixer_decode(&x, pg, ps, pl, pc, pcv, &z, &ln); });
}

#define RLM_FN(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {RLM_FN(mix_prefill),   RLM_FN(mix_decode),   RLM_FN(mix_backward),
                          RLM_FN(mixer_prefill), RLM_FN(mixer_decode), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_rlm_py", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__rlm_py(void) {
    struct {
        PyObject **to;
        const char *name;
    } names[] = {{&s_dtype, "dtype"},     {&s_is_cuda, "is_cuda"},   {&s_is_contiguous, "is_contiguous"},
                 {&s_shape, "shape"},     {&s_data_ptr, "data_ptr"}, {&s_device, "device"},
                 {&s_cuda_stream, "cuda_stream"}, {&s_decay, "decay"}, {&s_freq, "freq"},
                 {&s_amp, "amp"},         {&s_phase, "phase"},       {&s_s, "s"},
                 {&s_coef, "coef"},       {&s_conv_w, "conv_w"},     {&s_scale, "scale"},
                 {&s_c_raw, "c_raw"},     {&s_lambda_c, "lambda_c"}, {&s_u, "u"},               {&s_index, "index"},
                 {&g_numel, "numel"},     {&g_element_size, "element_size"}};
    for (auto &v : names)
        if (!(*v.to = PyUnicode_InternFromString(v.name))) return nullptr;
    PyObject *torch = PyImport_ImportModule("torch"), *c = PyImport_ImportModule("torch._C");
    if (!torch || !c) return nullptr;
    if (!(g_f32 = PyObject_GetAttrString(torch, "float32")) || !(g_bf16 = PyObject_GetAttrString(torch, "bfloat16")) ||
        !(g_u8 = PyObject_GetAttrString(torch, "uint8")) || !(g_empty = PyObject_GetAttrString(torch, "empty")) ||
        !(g_get_device = PyObject_GetAttrString(c, "_cuda_getDevice")) ||
        !(g_get_stream = PyObject_GetAttrString(c, "_cuda_getCurrentRawStream")) ||
        !(g_raw_alloc = PyObject_GetAttrString(c, "_cuda_cudaCachingAllocator_raw_alloc")) ||
        !(g_raw_delete = PyObject_GetAttrString(c, "_cuda_cudaCachingAllocator_raw_delete")) ||
        !(g_empty_kw = Py_BuildValue("(ss)", "dtype", "device")))
        return nullptr;
    Py_DECREF(torch);
    Py_DECREF(c);
    return PyModule_Create(&kModule);
}
