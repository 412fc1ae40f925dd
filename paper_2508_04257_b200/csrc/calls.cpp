// The calls a program makes once per layer and step (prediction, appends, attention), from Python objects to the C entry points without
// ctypes: checks, records of device addresses, result tensors, the call with the interpreter released.
//
// Why: a decode step is two calls, and their argument marshalling in Python took longer than the kernels of a short sequence.  CPU time
// of a call, ctypes and here: append of one token 9.3 and 3.3 us, decode attention (three tensors allocated) 14.1 and 7.0.
//
// The module knows nothing of where the library came from: bind() gets the entry points' addresses from binding.py, which loads it.
// Objects are read anew at every call; of a subclass, whatever its c() returns is taken.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "../../include/kvsink.h"

namespace {

decltype(&kvsink_cache_sizes) f_cache_sizes;
decltype(&kvsink_predict_sinks) f_predict_sinks;
decltype(&kvsink_quantize_append) f_quantize_append;
decltype(&kvsink_quantize_append_calibrated) f_quantize_append_calibrated;
decltype(&kvsink_quantize_append_pertoken) f_quantize_append_pertoken;
decltype(&kvsink_decode_attention) f_decode_attention;
decltype(&kvsink_decode_attention_calibrated) f_decode_attention_calibrated;
decltype(&kvsink_decode_attention_pertoken) f_decode_attention_pertoken;
decltype(&kvsink_prefill_attention) f_prefill_attention;
PyObject *config_type, *cache_type, *params_type, *error_type;

// attribute names, interned once
enum Name { BATCH, N_Q_HEADS, N_KV_HEADS, HEAD_DIM, HIDDEN, BITS, GROUP, MAX_SEQ, TOPK, PFN_N, CHANNELS, K_CODES, V_CODES, K_SCALE, K_ZERO, V_SCALE,
            V_ZERO, K_TAIL, SINK_K, SINK_V, SINKS, BITMASK, POS, COUNT, STATUS, SEQ_LEN, SIZES, DECODE_WORKSPACE, DATA_PTR, C_RECORD, NUMEL, NAMES };
const char *const NAME[NAMES] = {"batch", "n_q_heads", "n_kv_heads", "head_dim", "hidden", "bits", "group", "max_seq", "topk", "pfn_n", "channels", "k_codes",
                                 "v_codes", "k_scale", "k_zero", "v_scale", "v_zero", "k_tail", "sink_k", "sink_v", "sinks", "bitmask", "pos", "count", "status",
                                 "seq_len", "sizes", "decode_workspace_bytes", "data_ptr", "c", "numel"};
PyObject *name[NAMES];

struct Ref {      // an owned reference
    PyObject *o;
    explicit Ref(PyObject *x = nullptr) : o(x) {}
    ~Ref() { Py_XDECREF(o); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
};

// As ctypes converts: whole numbers only, their low 32 bits.
bool as_int32(PyObject *o, int32_t *out)
{
    if (!o) return false;
    if (!PyLong_Check(o)) {
        PyErr_Format(PyExc_TypeError, "int expected instead of %s instance", Py_TYPE(o)->tp_name);
        return false;
    }
    *out = (int32_t)PyLong_AsUnsignedLongLongMask(o);
    return !PyErr_Occurred();
}

bool int_attr(PyObject *o, Name n, int32_t *out)
{
    Ref v(PyObject_GetAttr(o, name[n]));
    return as_int32(v.o, out);
}

// What an object's own c() gives: a ctypes record of `size` bytes.
bool record(PyObject *o, void *out, size_t size)
{
    Ref r(PyObject_CallMethodNoArgs(o, name[C_RECORD]));
    if (!r.o) return false;
    Py_buffer view;
    if (PyObject_GetBuffer(r.o, &view, PyBUF_SIMPLE)) return false;
    const bool fits = (size_t)view.len == size;
    if (fits) memcpy(out, view.buf, size);
    PyBuffer_Release(&view);
    if (!fits) PyErr_SetString(PyExc_TypeError, "c() gave a record of another size");
    return fits;
}

bool read_config(PyObject *o, kvsink_config *c)
{
    if ((PyObject *)Py_TYPE(o) != config_type) return record(o, c, sizeof(*c));
    memset(c, 0, sizeof(*c));
    if (!int_attr(o, BATCH, &c->batch) || !int_attr(o, N_Q_HEADS, &c->n_q_heads) || !int_attr(o, N_KV_HEADS, &c->n_kv_heads) ||
        !int_attr(o, HEAD_DIM, &c->head_dim) || !int_attr(o, HIDDEN, &c->hidden) || !int_attr(o, BITS, &c->bits) || !int_attr(o, GROUP, &c->group) ||
        !int_attr(o, MAX_SEQ, &c->max_seq) || !int_attr(o, TOPK, &c->topk) || !int_attr(o, PFN_N, &c->pfn_n))
        return false;
    Ref given(PyObject_GetAttr(o, name[CHANNELS]));
    if (!given.o) return false;
    Ref list(PySequence_Tuple(given.o));
    if (!list.o) return false;
    const Py_ssize_t n = PyObject_Size(given.o);
    if (n < 0) return false;
    c->n_channels = (int32_t)n;
    for (Py_ssize_t i = 0; i < PyTuple_GET_SIZE(list.o) && i < 8; ++i)
        if (!as_int32(PyTuple_GET_ITEM(list.o, i), &c->channels[i])) return false;
    return true;
}

// Device address of a tensor; null for None.
bool address(PyObject *o, void **out)
{
    if (!o) return false;
    if (THPVariable_CheckExact(o)) {
        *out = THPVariable_Unpack(o).data_ptr();
        return true;
    }
    if (o == Py_None) {
        *out = nullptr;
        return true;
    }
    Ref v(PyObject_CallMethodNoArgs(o, name[DATA_PTR]));
    if (!v.o) return false;
    *out = PyLong_AsVoidPtr(v.o);
    return !PyErr_Occurred();
}

template <typename T>
bool address_attr(PyObject *o, Name n, T **out)
{
    Ref v(PyObject_GetAttr(o, name[n]));
    void *p = nullptr;
    if (!address(v.o, &p)) return false;
    *out = (T *)p;
    return true;
}

bool read_cache(PyObject *o, kvsink_cache *c)
{
    if ((PyObject *)Py_TYPE(o) != cache_type) return record(o, c, sizeof(*c));
    memset(c, 0, sizeof(*c));
    Ref sinks(PyObject_GetAttr(o, name[SINKS]));
    return sinks.o && address_attr(o, K_CODES, &c->k_codes) && address_attr(o, V_CODES, &c->v_codes) && address_attr(o, K_SCALE, &c->k_scale) &&
           address_attr(o, K_ZERO, &c->k_zero) && address_attr(o, V_SCALE, &c->v_scale) && address_attr(o, V_ZERO, &c->v_zero) &&
           address_attr(o, K_TAIL, &c->k_tail) && address_attr(o, SINK_K, &c->sink_k) && address_attr(o, SINK_V, &c->sink_v) &&
           address_attr(sinks.o, BITMASK, &c->sink_bitmask) && address_attr(sinks.o, POS, &c->sink_pos) && address_attr(sinks.o, COUNT, &c->sink_count) &&
           address_attr(o, STATUS, &c->status) && int_attr(o, SEQ_LEN, &c->seq_len);
}

bool read_params(PyObject *o, kvsink_static_params *p)
{
    if ((PyObject *)Py_TYPE(o) != params_type) return record(o, p, sizeof(*p));
    memset(p, 0, sizeof(*p));
    return address_attr(o, K_SCALE, (float **)&p->k_scale) && address_attr(o, K_ZERO, (float **)&p->k_zero) &&
           address_attr(o, V_SCALE, (float **)&p->v_scale) && address_attr(o, V_ZERO, (float **)&p->v_zero);
}

const at::Tensor *tensor(PyObject *o)
{
    if (THPVariable_Check(o)) return &THPVariable_Unpack(o);
    PyErr_Format(PyExc_AttributeError, "'%s' object is not a tensor", Py_TYPE(o)->tp_name);
    return nullptr;
}

bool require(bool ok, const char *what)
{
    if (!ok) PyErr_SetString(PyExc_AssertionError, what);
    return ok;
}

// A status of the library as the binding raises it.
bool done(int rc, const char *what)
{
    if (!rc) return true;
    Ref e(PyObject_CallFunction(error_type, "is", rc, what));
    if (e.o) PyErr_SetObject(error_type, e.o);
    return false;
}

void *stream() { return (void *)c10::cuda::getCurrentCUDAStream().stream(); }

// Without the interpreter for its life: a launch can wait for room in the queue, an allocation for the allocator's lock.
struct NoInterpreter {
    PyThreadState *s = PyEval_SaveThread();
    ~NoInterpreter() { PyEval_RestoreThread(s); }
};

template <typename F>
int released(F call)
{
    NoInterpreter none;
    return call();
}

bool arguments(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, n);
    return false;
}

// The tensor passed for a result, or a new one on q's device.
PyObject *result(PyObject *given, const at::Tensor &q, at::IntArrayRef shape, at::ScalarType type)
{
    if (given != Py_None) return Py_NewRef(given);
    at::Tensor made;
    {
        NoInterpreter none;
        made = q.new_empty(shape, q.options().dtype(type));
    }
    return THPVariable_Wrap(made);
}

bool workspace_of(PyObject *w, void **at, size_t *bytes)
{
    if (!address(w, at)) return false;
    if (THPVariable_CheckExact(w)) {
        *bytes = (size_t)THPVariable_Unpack(w).numel();
        return true;
    }
    Ref n(PyObject_CallMethodNoArgs(w, name[NUMEL]));
    if (!n.o) return false;
    *bytes = PyLong_AsSize_t(n.o);
    return !PyErr_Occurred();
}

PyObject *predict_sinks(PyObject *, PyObject *const *a, Py_ssize_t n)      // cfg, hidden, sinks, workspace
{
    HANDLE_TH_ERRORS
    if (!arguments(n, 4)) return nullptr;
    const at::Tensor *hidden = tensor(a[1]);
    if (!hidden || !require(hidden->is_cuda() && hidden->scalar_type() == at::kHalf && hidden->dim() == 3 && hidden->stride(2) == 1,
                            "hidden: fp16 [B, S, d] on the device, last axis contiguous"))
        return nullptr;
    kvsink_config c;
    if (!read_config(a[0], &c)) return nullptr;
    int64_t need = 0;
    if (a[3] == Py_None) {
        kvsink_sizes s;
        if (!done(f_cache_sizes(&c, &s), "kvsink_cache_sizes")) return nullptr;
        need = s.predict_workspace_bytes;
    }
    Ref ws(result(a[3], *hidden, {need}, at::kByte));
    void *w, *mask, *pos, *count;
    size_t bytes;
    if (!ws.o || !workspace_of(ws.o, &w, &bytes) || !address_attr(a[2], BITMASK, &mask) || !address_attr(a[2], POS, &pos) || !address_attr(a[2], COUNT, &count)) return nullptr;
    const void *at = hidden->data_ptr();
    const int64_t S = hidden->size(1), sb = hidden->stride(0), ss = hidden->stride(1);
    void *st = stream();
    if (!done(released([&] { return f_predict_sinks(&c, at, (int32_t)S, sb, ss, (uint32_t *)mask, (int32_t *)pos, (int32_t *)count, w, bytes, st); }), "kvsink_predict_sinks")) return nullptr;
    return Py_NewRef(a[2]);
    END_HANDLE_TH_ERRORS
}

PyObject *quantize_append(PyObject *, PyObject *const *a, Py_ssize_t n)      // mode, cfg, cache, params, k_new, v_new
{
    HANDLE_TH_ERRORS
    int32_t mode;
    if (!arguments(n, 6) || !as_int32(a[0], &mode)) return nullptr;
    const at::Tensor *k = tensor(a[4]), *v = k ? tensor(a[5]) : nullptr;
    if (!v || !require(k->is_cuda() && k->scalar_type() == at::kHalf && k->dim() == 4 && k->stride(3) == 1, "k_new: fp16 [B, Hkv, T, D] on the device, last axis contiguous") ||
        !require(v->sizes() == k->sizes() && v->strides() == k->strides() && v->scalar_type() == at::kHalf, "v_new: the shape, strides and type of k_new"))
        return nullptr;
    kvsink_config c;
    kvsink_cache cache;
    kvsink_static_params sp;
    if (!read_cache(a[2], &cache) || (mode == 1 && !read_params(a[3], &sp)) || !read_config(a[1], &c)) return nullptr;
    const void *kp = k->data_ptr(), *vp = v->data_ptr();
    const int32_t T = (int32_t)k->size(2);
    const int64_t sb = k->stride(0), sh = k->stride(1), stt = k->stride(2);
    void *st = stream();
    const int rc = released([&] {
        return mode == 1   ? f_quantize_append_calibrated(&c, &cache, &sp, kp, vp, T, sb, sh, stt, st)
               : mode == 2 ? f_quantize_append_pertoken(&c, &cache, kp, vp, T, sb, sh, stt, st)
                           : f_quantize_append(&c, &cache, kp, vp, T, sb, sh, stt, st);
    });
    if (!done(rc, mode == 1 ? "kvsink_quantize_append_calibrated" : (mode == 2 ? "kvsink_quantize_append_pertoken" : "kvsink_quantize_append"))) return nullptr;
    Ref len(PyLong_FromLong(cache.seq_len));
    if (!len.o || PyObject_SetAttr(a[2], name[SEQ_LEN], len.o)) return nullptr;
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

// out and lse (None where it is not wanted), as given or new; an allocation that throws leaves what was made before it to its owner
bool results(PyObject *out, PyObject *lse, PyObject *want_lse, const at::Tensor &q, const kvsink_config &c, int64_t T, Ref *o, Ref *l)
{
    const int want = lse == Py_None ? PyObject_IsTrue(want_lse) : 0;
    if (want < 0) return false;
    const int64_t shape[4] = {c.batch, c.n_q_heads, T < 0 ? (int64_t)c.head_dim : T, c.head_dim};
    o->o = result(out, q, at::IntArrayRef(shape, T < 0 ? 3 : 4), at::kFloat);
    if (!o->o) return false;
    l->o = want ? result(lse, q, at::IntArrayRef(shape, T < 0 ? 2 : 3), at::kFloat) : Py_NewRef(lse);
    return l->o != nullptr;
}

PyObject *decode_attention(PyObject *, PyObject *const *a, Py_ssize_t n)      // mode, cfg, cache, params, q, out, lse, workspace, want_lse
{
    HANDLE_TH_ERRORS
    int32_t mode;
    if (!arguments(n, 9) || !as_int32(a[0], &mode)) return nullptr;
    const at::Tensor *q = tensor(a[4]);
    if (!q || !require(q->is_cuda() && q->scalar_type() == at::kHalf && q->is_contiguous(), "q: fp16 [B, Hq, D] on the device, contiguous")) return nullptr;
    kvsink_config c;
    kvsink_cache cache;
    kvsink_static_params sp;
    if (!read_config(a[1], &c)) return nullptr;
    Ref out, lse;
    if (!results(a[5], a[6], a[8], *q, c, -1, &out, &lse)) return nullptr;
    int64_t need = 0;
    if (a[7] == Py_None) {
        Ref sizes(PyObject_GetAttr(a[2], name[SIZES]));
        if (!sizes.o) return nullptr;
        Ref bytes(PyObject_GetItem(sizes.o, name[DECODE_WORKSPACE]));
        if (!bytes.o) return nullptr;
        need = PyLong_AsLongLong(bytes.o);
        if (PyErr_Occurred()) return nullptr;
    }
    Ref ws(result(a[7], *q, {need}, at::kByte));
    void *w, *o, *l;
    size_t bytes;
    if (!ws.o || !workspace_of(ws.o, &w, &bytes) || !address(out.o, &o) || !address(lse.o, &l) || !read_cache(a[2], &cache) || (mode == 1 && !read_params(a[3], &sp))) return nullptr;
    const void *qp = q->data_ptr();
    void *st = stream();
    const int rc = released([&] {
        return mode == 1   ? f_decode_attention_calibrated(&c, &cache, &sp, qp, (float *)o, (float *)l, w, bytes, st)
               : mode == 2 ? f_decode_attention_pertoken(&c, &cache, qp, (float *)o, (float *)l, w, bytes, st)
                           : f_decode_attention(&c, &cache, qp, (float *)o, (float *)l, w, bytes, st);
    });
    if (!done(rc, mode == 1 ? "kvsink_decode_attention_calibrated" : (mode == 2 ? "kvsink_decode_attention_pertoken" : "kvsink_decode_attention"))) return nullptr;
    return PyTuple_Pack(2, out.o, lse.o);
    END_HANDLE_TH_ERRORS
}

PyObject *prefill_attention(PyObject *, PyObject *const *a, Py_ssize_t n)      // cfg, cache, q, q_pos0, out, lse, want_lse
{
    HANDLE_TH_ERRORS
    int32_t pos0;
    if (!arguments(n, 7)) return nullptr;
    const at::Tensor *q = tensor(a[2]);
    if (!q || !require(q->is_cuda() && q->scalar_type() == at::kHalf && q->dim() == 4 && q->stride(3) == 1, "q: fp16 [B, Hq, T, D] on the device, last axis contiguous") ||
        !as_int32(a[3], &pos0))
        return nullptr;
    kvsink_config c;
    kvsink_cache cache;
    if (!read_config(a[0], &c)) return nullptr;
    const int64_t T = q->size(2), sb = q->stride(0), sh = q->stride(1), stt = q->stride(2);
    Ref out, lse;
    void *o, *l;
    if (!results(a[4], a[5], a[6], *q, c, T, &out, &lse) || !address(out.o, &o) || !address(lse.o, &l) || !read_cache(a[1], &cache)) return nullptr;
    const void *qp = q->data_ptr();
    void *st = stream();
    if (!done(released([&] { return f_prefill_attention(&c, &cache, qp, (int32_t)T, pos0, sb, sh, stt, (float *)o, (float *)l, st); }), "kvsink_prefill_attention")) return nullptr;
    return PyTuple_Pack(2, out.o, lse.o);
    END_HANDLE_TH_ERRORS
}

// bind(addresses of the entry points by name, Config, KVCache, StaticParams, KvsinkError)
PyObject *bind(PyObject *, PyObject *args)
{
    PyObject *at, *types[4];
    if (!PyArg_ParseTuple(args, "O!OOOO", &PyDict_Type, &at, &types[0], &types[1], &types[2], &types[3])) return nullptr;
    const struct { const char *name; void **to; } all[] = {
        {"kvsink_cache_sizes", (void **)&f_cache_sizes}, {"kvsink_predict_sinks", (void **)&f_predict_sinks},
        {"kvsink_quantize_append", (void **)&f_quantize_append}, {"kvsink_quantize_append_calibrated", (void **)&f_quantize_append_calibrated},
        {"kvsink_quantize_append_pertoken", (void **)&f_quantize_append_pertoken}, {"kvsink_decode_attention", (void **)&f_decode_attention},
        {"kvsink_decode_attention_calibrated", (void **)&f_decode_attention_calibrated},
        {"kvsink_decode_attention_pertoken", (void **)&f_decode_attention_pertoken}, {"kvsink_prefill_attention", (void **)&f_prefill_attention}};
    for (const auto &f : all) {
        PyObject *v = PyDict_GetItemString(at, f.name);
        *f.to = v ? PyLong_AsVoidPtr(v) : nullptr;
        if (!*f.to) {
            if (!PyErr_Occurred()) PyErr_Format(PyExc_ImportError, "no address for %s", f.name);
            return nullptr;
        }
    }
    for (PyObject *t : types) Py_INCREF(t);      // kept for the life of the process
    config_type = types[0]; cache_type = types[1]; params_type = types[2]; error_type = types[3];
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {{"bind", (PyCFunction)bind, METH_VARARGS, nullptr},
                         {"predict_sinks", (PyCFunction)(void (*)(void))predict_sinks, METH_FASTCALL, nullptr},
                         {"quantize_append", (PyCFunction)(void (*)(void))quantize_append, METH_FASTCALL, nullptr},
                         {"decode_attention", (PyCFunction)(void (*)(void))decode_attention, METH_FASTCALL, nullptr},
                         {"prefill_attention", (PyCFunction)(void (*)(void))prefill_attention, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void)
{
    for (int i = 0; i < NAMES; ++i)
        if (!(name[i] = PyUnicode_InternFromString(NAME[i]))) return nullptr;
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "abi", KVSINK_CALLS_ABI)) {      // what it was built for, compared by binding.py
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
