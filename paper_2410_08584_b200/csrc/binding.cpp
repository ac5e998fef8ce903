// Native half of binding.py: turns torch tensors into the C ABI's pointers.
//
// A decode step on a short cache takes about 10 us on the GPU, and a Python loop over ctypes
// calls took 14 us per call to marshal it (a c_void_p object per argument, several Python-level
// tensor queries per tensor, two Python objects for the stream), so it set the pace of
// single-request decoding.  Here a call reads the tensors' fields directly.  Checks, exceptions and default
// allocations are those that binding.py documents; nothing is cached between calls.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/autograd/utils/wrap_outputs.h>

#include "../../include/zipvl.h"

namespace {

PyObject *g_error_class = nullptr;   // binding.ZipvlError

struct Failed {};                    // a Python exception is set

[[noreturn]] void raise(PyObject *type, const std::string &text) {
    PyErr_SetString(type, text.c_str());
    throw Failed{};
}

// The library call itself runs without the interpreter lock (a launch may wait for room in the queue).
template <typename... P, typename... A>
void check(zipvl_status (*call)(P...), const A &...args) {
    PyThreadState *thread = PyEval_SaveThread();
    const zipvl_status s = call(static_cast<P>(args)...);
    PyEval_RestoreThread(thread);
    if (s == ZIPVL_OK) return;
    PyObject *e = PyObject_CallFunction(g_error_class, "is", (int)s, zipvl_last_error());
    if (e) {
        PyErr_SetObject(g_error_class, e);
        Py_DECREF(e);
    }
    throw Failed{};
}

const at::Tensor &tensor(PyObject *o, const char *name) {
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string("zipvl: ") + name + " must be a tensor");
    return THPVariable_Unpack(o);
}

void *ptr(PyObject *o, const char *name) { return o == Py_None ? nullptr : tensor(o, name).data_ptr(); }

// [L, H, d] with contiguous (H, d) rows and any token stride >= H*d
bool token_strided(const at::Tensor &t) {
    return t.dim() == 3 && t.stride(2) == 1 && t.stride(1) == t.size(2) && t.stride(0) >= t.size(1) * t.size(2);
}

const at::Tensor &dev(PyObject *o, const char *name, bool strided = false) {
    const at::Tensor &t = tensor(o, name);
    if (!t.is_cuda() || !(t.is_contiguous() || (strided && token_strided(t))))
        raise(PyExc_ValueError, std::string("zipvl: ") + name + " must be a contiguous CUDA tensor" +
                                    (strided ? " (or [L, H, d] rows with a token stride)" : ""));
    return t;
}

const at::Tensor &dev(PyObject *o, const char *name, at::ScalarType type) {
    const at::Tensor &t = dev(o, name);
    if (t.scalar_type() != type)
        raise(PyExc_TypeError, std::string("zipvl: ") + name + " must be torch." +
                                   (type == at::kFloat ? "float32" : type == at::kInt ? "int32" : "int64"));
    return t;
}

void same_stride(const at::Tensor &k, const at::Tensor &v) {
    if (k.stride(0) != v.stride(0) || !k.sizes().equals(v.sizes()))
        raise(PyExc_ValueError, "zipvl: k and v must have the same shape and token stride");
}

int dtype_code(const at::Tensor &t) {
    switch (t.scalar_type()) {
        case at::kBFloat16: return ZIPVL_BF16;
        case at::kFloat: return ZIPVL_F32;
        case at::kHalf: return ZIPVL_F16;
        default: raise(PyExc_TypeError, std::string("zipvl: dtype ") + c10::toString(t.scalar_type()) +
                                            " (bfloat16, float16 or float32)");
    }
}

// a ctypes structure of the C ABI, copied out of its buffer
template <typename T>
T structure(PyObject *o, const char *name) {
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE)) throw Failed{};
    const bool fits = view.len == (Py_ssize_t)sizeof(T);
    T out{};
    if (fits) memcpy(&out, view.buf, sizeof(T));
    PyBuffer_Release(&view);
    if (!fits) raise(PyExc_TypeError, std::string("zipvl: ") + name + " is not the structure this call takes");
    return out;
}

void *stream(PyObject *o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) throw Failed{};
    void *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (!p && PyErr_Occurred()) throw Failed{};
    return p;
}

long long integer(PyObject *o) {
    PyObject *i = PyLong_Check(o) ? Py_NewRef(o) : PyNumber_Long(o);
    if (!i) throw Failed{};
    const long long v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw Failed{};
    return v;
}
int32_t int_arg(PyObject *o) { return (int32_t)integer(o); }
float real(PyObject *o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Failed{};
    return (float)v;
}

// an argument the caller gave, or a fresh tensor on the device of `like`
at::Tensor given_or_empty(PyObject *o, const char *name, at::IntArrayRef shape, at::ScalarType type, const at::Tensor &like) {
    return o == Py_None ? at::empty(shape, like.options().dtype(type)) : tensor(o, name);
}
at::Tensor workspace(PyObject *o, size_t bytes, const at::Tensor &like) {
    const int64_t n = bytes > 256 ? (int64_t)bytes : 256;
    return given_or_empty(o, "ws", {n}, at::kByte, like);
}
template <typename F>
at::Tensor lazy_workspace(PyObject *o, const at::Tensor &like, F bytes) {
    return o == Py_None ? workspace(o, bytes(), like) : tensor(o, "ws");
}
int32_t *status(PyObject *o) { return (int32_t *)ptr(o, "status"); }

PyObject *wrap(const at::Tensor &t) { return THPVariable_Wrap(t); }
PyObject *wrap(const at::Tensor &a, const at::Tensor &b) { return Py_BuildValue("NN", wrap(a), wrap(b)); }

zipvl_layer plain_layer(int L, int Hq, int Hkv, int d, int dtype) {
    zipvl_layer l{};
    l.L = L; l.n_q_heads = Hq; l.n_kv_heads = Hkv; l.head_dim = d; l.dtype = dtype;
    return l;
}
size_t decode_bytes(const zipvl_decode_desc &d, int max_len, int batch) {
    const zipvl_layer l = plain_layer(max_len, d.n_q_heads, d.n_kv_heads, d.head_dim, d.dtype);
    return zipvl_workspace_bytes(ZIPVL_OP_DECODE, &l, 0, batch);
}
at::Tensor out_like(PyObject *o, const at::Tensor &q) { return o == Py_None ? at::empty_like(q) : tensor(o, "out"); }

// Stacked Q [n_seq, L, Hq, d] and K [n_seq, L, Hkv, d], contiguous
void batch_desc(const at::Tensor &q, const at::Tensor &k, zipvl_layer *l, zipvl_batch *b) {
    if (q.dim() != 4 || k.dim() != 4 || !q.is_contiguous() || !k.is_contiguous())
        raise(PyExc_ValueError, "zipvl: batched calls take contiguous [n_seq, L, H, d] tensors");
    *l = plain_layer((int)q.size(1), (int)q.size(2), (int)k.size(2), (int)q.size(3), dtype_code(q));
    *b = zipvl_batch{(int32_t)q.size(0), 0, 0, 0};
}

using Args = PyObject *const *;

// (layer, q, k, probe_pos, acc, norm, total, ws, status, stream)
PyObject *score(Args a) {
    const zipvl_layer l = structure<zipvl_layer>(a[0], "layer");
    const at::Tensor &q = dev(a[1], "q", true), &k = dev(a[2], "k", true), &probe = dev(a[3], "probe_pos", at::kInt);
    const at::Tensor acc = given_or_empty(a[4], "acc", {l.L}, at::kFloat, q);
    const at::Tensor norm = given_or_empty(a[5], "norm", {l.L}, at::kFloat, q);
    const int P = (int)probe.numel();
    const at::Tensor ws = lazy_workspace(a[7], q, [&] { return zipvl_workspace_bytes(ZIPVL_OP_SCORE, &l, P, 1); });
    check(zipvl_score, &l, q.data_ptr(), k.data_ptr(), (const int32_t *)probe.data_ptr(), P, (float *)acc.data_ptr(),
                      (float *)norm.data_ptr(), (double *)ptr(a[6], "total"), ws.data_ptr(), (size_t)ws.numel(),
                      status(a[8]), stream(a[9]));
    return wrap(acc, norm);
}

// (acc, norm, tau, mode, fixed_k, k_out, idx, kept_mass, ws, status, stream)
PyObject *select(Args a) {
    const at::Tensor &acc = dev(a[0], "acc", at::kFloat), &norm = dev(a[1], "norm", at::kFloat);
    const int L = (int)acc.numel();
    const at::Tensor k_out = given_or_empty(a[5], "k_out", {1}, at::kInt, acc);
    const at::Tensor idx = given_or_empty(a[6], "idx", {L}, at::kInt, acc);
    const at::Tensor ws = lazy_workspace(a[8], acc, [&] {
        const zipvl_layer l = plain_layer(L, 1, 1, 64, ZIPVL_F32);
        return zipvl_workspace_bytes(ZIPVL_OP_SELECT, &l, 0, 1);
    });
    check(zipvl_select, L, (const float *)acc.data_ptr(), (const float *)norm.data_ptr(), real(a[2]),
                       (uint32_t)integer(a[3]), int_arg(a[4]), (int32_t *)k_out.data_ptr(), (int32_t *)idx.data_ptr(),
                       (float *)ptr(a[7], "kept_mass"), ws.data_ptr(), (size_t)ws.numel(), status(a[9]), stream(a[10]));
    return wrap(k_out, idx);
}

struct PrefillArgs {
    zipvl_layer l;
    const at::Tensor &q, &k, &v, &idx, &k_dev;
    int k_max, mode;
    at::Tensor out, ws;
};
PrefillArgs prefill_args(PyObject *layer, Args t, PyObject *k_max, PyObject *out, PyObject *mode, PyObject *ws) {
    PrefillArgs p{structure<zipvl_layer>(layer, "layer"), dev(t[0], "q", true), dev(t[1], "k", true), dev(t[2], "v", true),
                  dev(t[3], "idx", at::kInt), dev(t[4], "k_dev", at::kInt), int_arg(k_max), int_arg(mode), {}, {}};
    same_stride(p.k, p.v);
    p.out = out != Py_None ? tensor(out, "out")
                           : at::empty({p.mode == ZIPVL_OUT_PADDED ? p.l.L : p.k_max, p.l.n_q_heads, p.l.head_dim}, p.q.options());
    p.ws = lazy_workspace(ws, p.q, [&] { return zipvl_workspace_bytes(ZIPVL_OP_SPARSE_PREFILL, &p.l, 0, 1); });
    return p;
}

// (layer, q, k, v, idx, k_dev, k_max, out, out_mode, ws, status, stream)
PyObject *sparse_prefill(Args a) {
    const PrefillArgs p = prefill_args(a[0], a + 1, a[6], a[7], a[8], a[9]);
    check(zipvl_sparse_prefill, &p.l, p.q.data_ptr(), p.k.data_ptr(), p.v.data_ptr(), (const int32_t *)p.idx.data_ptr(),
                               (const int32_t *)p.k_dev.data_ptr(), p.k_max, p.out.data_ptr(), p.mode, p.ws.data_ptr(),
                               (size_t)p.ws.numel(), status(a[10]), stream(a[11]));
    return wrap(p.out);
}

// (layer, q, k, v, idx, k_dev, k_max, k_cache, v_cache, capacity, out, out_mode, len_out, ws, status, stream)
PyObject *sparse_prefill_compact(Args a) {
    const PrefillArgs p = prefill_args(a[0], a + 1, a[6], a[10], a[11], a[13]);
    const at::Tensor &kc = dev(a[7], "k_cache"), &vc = dev(a[8], "v_cache");
    const at::Tensor len = given_or_empty(a[12], "len_out", {1}, at::kInt, p.k);
    check(zipvl_sparse_prefill_compact, &p.l, p.q.data_ptr(), p.k.data_ptr(), p.v.data_ptr(),
                                       (const int32_t *)p.idx.data_ptr(), (const int32_t *)p.k_dev.data_ptr(), p.k_max,
                                       p.out.data_ptr(), p.mode, kc.data_ptr(), vc.data_ptr(), int_arg(a[9]),
                                       (int32_t *)len.data_ptr(), p.ws.data_ptr(), (size_t)p.ws.numel(), status(a[14]),
                                       stream(a[15]));
    return wrap(p.out, len);
}

// (q, k, probe_pos, acc, norm, ws, status, stream)
PyObject *score_batch(Args a) {
    const at::Tensor &q = dev(a[0], "q"), &k = dev(a[1], "k"), &probe = dev(a[2], "probe_pos", at::kInt);
    zipvl_layer l;
    zipvl_batch b;
    batch_desc(q, k, &l, &b);
    const int P = (int)probe.size(1);
    const at::Tensor acc = given_or_empty(a[3], "acc", {b.n_seq, l.L}, at::kFloat, q);
    const at::Tensor norm = given_or_empty(a[4], "norm", {b.n_seq, l.L}, at::kFloat, q);
    const at::Tensor ws = lazy_workspace(a[5], q, [&] { return zipvl_workspace_bytes_batch(ZIPVL_OP_SCORE, &l, P, b.n_seq); });
    check(zipvl_score_batch, &l, &b, q.data_ptr(), k.data_ptr(), (const int32_t *)probe.data_ptr(), P,
                            (float *)acc.data_ptr(), (float *)norm.data_ptr(), nullptr, ws.data_ptr(), (size_t)ws.numel(),
                            status(a[6]), stream(a[7]));
    return wrap(acc, norm);
}

// (acc, norm, tau, mode, fixed_k, k_out, idx, ws, status, stream)
PyObject *select_batch(Args a) {
    const at::Tensor &acc = dev(a[0], "acc", at::kFloat), &norm = dev(a[1], "norm", at::kFloat);
    if (acc.dim() != 2) raise(PyExc_ValueError, "zipvl: acc must be [n_seq, L]");
    const int n = (int)acc.size(0), L = (int)acc.size(1);
    const at::Tensor k_out = given_or_empty(a[5], "k_out", {n}, at::kInt, acc);
    const at::Tensor idx = given_or_empty(a[6], "idx", {n, L}, at::kInt, acc);
    const at::Tensor ws = lazy_workspace(a[7], acc, [&] {
        const zipvl_layer l = plain_layer(L, 1, 1, 64, ZIPVL_F32);
        return zipvl_workspace_bytes(ZIPVL_OP_SELECT, &l, 0, 1);
    });
    check(zipvl_select_batch, L, n, (const float *)acc.data_ptr(), (const float *)norm.data_ptr(), real(a[2]),
                             (uint32_t)integer(a[3]), int_arg(a[4]), (int32_t *)k_out.data_ptr(),
                             (int32_t *)idx.data_ptr(), nullptr, ws.data_ptr(), (size_t)ws.numel(), status(a[8]),
                             stream(a[9]));
    return wrap(k_out, idx);
}

// (q, k, v, idx, k_dev, k_max, k_cache, v_cache, capacity, out, out_mode, len_out, ws, status, stream)
PyObject *sparse_prefill_batch(Args a) {
    const at::Tensor &q = dev(a[0], "q"), &k = dev(a[1], "k"), &v = dev(a[2], "v");
    const at::Tensor &idx = dev(a[3], "idx", at::kInt), &k_dev = dev(a[4], "k_dev", at::kInt);
    zipvl_layer l;
    zipvl_batch b;
    batch_desc(q, k, &l, &b);
    const int k_max = int_arg(a[5]), mode = int_arg(a[10]);
    const at::Tensor out = a[9] != Py_None ? tensor(a[9], "out")
                                           : at::empty({b.n_seq, mode == ZIPVL_OUT_PADDED ? l.L : k_max, l.n_q_heads, l.head_dim}, q.options());
    const at::Tensor ws = lazy_workspace(a[12], q, [&] { return zipvl_workspace_bytes(ZIPVL_OP_SPARSE_PREFILL, &l, 0, 1); });
    at::Tensor len;
    if (a[11] != Py_None) len = tensor(a[11], "len_out");
    else if (a[6] != Py_None) len = at::empty({b.n_seq}, q.options().dtype(at::kInt));
    check(zipvl_sparse_prefill_batch, &l, &b, q.data_ptr(), k.data_ptr(), v.data_ptr(), (const int32_t *)idx.data_ptr(),
                                     (const int32_t *)k_dev.data_ptr(), k_max, out.data_ptr(), mode,
                                     ptr(a[6], "k_cache"), ptr(a[7], "v_cache"), int_arg(a[8]),
                                     len.defined() ? (int32_t *)len.data_ptr() : nullptr, ws.data_ptr(),
                                     (size_t)ws.numel(), status(a[13]), stream(a[14]));
    return Py_BuildValue("NN", wrap(out), len.defined() ? wrap(len) : Py_NewRef(Py_None));
}

// (layer, k, v, idx, k_dev, k_max, k_cache, v_cache, capacity, len_out, status, stream)
PyObject *compact_kv(Args a) {
    const zipvl_layer l = structure<zipvl_layer>(a[0], "layer");
    const at::Tensor &k = dev(a[1], "k", true), &v = dev(a[2], "v", true), &kc = dev(a[6], "k_cache"), &vc = dev(a[7], "v_cache");
    same_stride(k, v);
    const at::Tensor len = given_or_empty(a[9], "len_out", {1}, at::kInt, k);
    check(zipvl_compact_kv, &l, k.data_ptr(), v.data_ptr(), (const int32_t *)ptr(a[3], "idx"),
                           (const int32_t *)ptr(a[4], "k_dev"), int_arg(a[5]), kc.data_ptr(), vc.data_ptr(), int_arg(a[8]),
                           (int32_t *)len.data_ptr(), status(a[10]), stream(a[11]));
    return wrap(len);
}

// (desc, q, k_new, v_new, k_cache, v_cache, cache_off, capacity, seq_lens, max_len, out, ws, status, stream)
PyObject *decode(Args a) {
    const at::Tensor &q = dev(a[1], "q"), &kc = dev(a[4], "k_cache"), &vc = dev(a[5], "v_cache");
    const at::Tensor &off = dev(a[6], "cache_off", at::kLong), &cap = dev(a[7], "capacity", at::kInt);
    const at::Tensor &lens = dev(a[8], "seq_lens", at::kInt);
    const zipvl_decode_desc d = structure<zipvl_decode_desc>(a[0], "desc");
    const int max_len = int_arg(a[9]);
    const at::Tensor out = out_like(a[10], q);
    const at::Tensor ws = lazy_workspace(a[11], q, [&] { return decode_bytes(d, max_len, d.batch); });
    check(zipvl_decode, &d, q.data_ptr(), ptr(a[2], "k_new"), ptr(a[3], "v_new"), kc.data_ptr(), vc.data_ptr(),
                       (const int64_t *)off.data_ptr(), (const int32_t *)cap.data_ptr(), (int32_t *)lens.data_ptr(),
                       max_len, out.data_ptr(), ws.data_ptr(), (size_t)ws.numel(), status(a[12]), stream(a[13]));
    return wrap(out);
}

// (desc, q, k_new, v_new, k_pages, v_pages, block_table, capacity, seq_lens, max_len, out, ws, status, stream)
PyObject *decode_paged(Args a) {
    const at::Tensor &q = dev(a[1], "q"), &kp = dev(a[4], "k_pages"), &vp = dev(a[5], "v_pages");
    const at::Tensor &table = dev(a[6], "block_table", at::kInt), &cap = dev(a[7], "capacity", at::kInt);
    const at::Tensor &lens = dev(a[8], "seq_lens", at::kInt);
    if (table.dim() != 2 || kp.dim() < 2) raise(PyExc_ValueError, "zipvl: block_table [B, max_pages], pages [n_pages, page_rows, Hkv, d]");
    const zipvl_decode_desc d = structure<zipvl_decode_desc>(a[0], "desc");
    const int max_len = int_arg(a[9]);
    const at::Tensor out = out_like(a[10], q);
    const at::Tensor ws = lazy_workspace(a[11], q, [&] { return decode_bytes(d, max_len, d.batch); });
    check(zipvl_decode_paged, &d, q.data_ptr(), ptr(a[2], "k_new"), ptr(a[3], "v_new"), kp.data_ptr(), vp.data_ptr(),
                             (const int32_t *)table.data_ptr(), (int32_t)table.size(1), (int32_t)kp.size(1),
                             (int32_t)kp.size(0), (const int32_t *)cap.data_ptr(), (int32_t *)lens.data_ptr(), max_len,
                             out.data_ptr(), ws.data_ptr(), (size_t)ws.numel(), status(a[12]), stream(a[13]));
    return wrap(out);
}

// (desc, q, k_new, v_new, k_cache, v_cache, cache_off, capacity, seq_lens, max_len, out, status, stream)
PyObject *decode_noalloc(Args a) {
    const at::Tensor &q = dev(a[1], "q"), &kc = dev(a[4], "k_cache"), &vc = dev(a[5], "v_cache"), &out = dev(a[10], "out");
    const at::Tensor &off = dev(a[6], "cache_off", at::kLong), &cap = dev(a[7], "capacity", at::kInt);
    const at::Tensor &lens = dev(a[8], "seq_lens", at::kInt);
    const zipvl_decode_desc d = structure<zipvl_decode_desc>(a[0], "desc");
    check(zipvl_decode_noalloc, &d, q.data_ptr(), ptr(a[2], "k_new"), ptr(a[3], "v_new"), kc.data_ptr(), vc.data_ptr(),
                               (const int64_t *)off.data_ptr(), (const int32_t *)cap.data_ptr(),
                               (int32_t *)lens.data_ptr(), int_arg(a[9]), out.data_ptr(), status(a[11]), stream(a[12]));
    return Py_NewRef(a[10]);
}

// attributes of a QuantCache
struct Cache {
    PyObject *o;
    at::Tensor get(const char *name) const {
        PyObject *v = PyObject_GetAttrString(o, name);
        if (!v) throw Failed{};
        if (!THPVariable_Check(v)) {
            Py_DECREF(v);
            raise(PyExc_TypeError, std::string("zipvl: cache.") + name + " must be a tensor");
        }
        at::Tensor t = THPVariable_Unpack(v);
        Py_DECREF(v);
        return t;
    }
    void *p(const char *name) const { return get(name).data_ptr(); }
    int32_t cap(const char *name) const {
        PyObject *v = PyObject_GetAttrString(o, name);
        if (!v) throw Failed{};
        const long long n = PyLong_AsLongLong(v);   // QuantCache makes them int
        Py_DECREF(v);
        if (n == -1 && PyErr_Occurred()) throw Failed{};
        return (int32_t)n;
    }
};

// (layer, k, v, idx, k_dev, k_max, cache, status, stream)
PyObject *quantize_kv(Args a) {
    const zipvl_layer l = structure<zipvl_layer>(a[0], "layer");
    const at::Tensor &k = dev(a[1], "k", true), &v = dev(a[2], "v", true), &idx = dev(a[3], "idx", at::kInt);
    same_stride(k, v);
    const Cache c{a[6]};
    const at::Tensor lens = c.get("lens");
    check(zipvl_quantize_kv, &l, k.data_ptr(), v.data_ptr(), (const int32_t *)idx.data_ptr(),
                            (const int32_t *)ptr(a[4], "k_dev"), int_arg(a[5]), c.p("k_hi"), c.p("v_hi"), c.p("p_hi"),
                            c.cap("cap_hi"), c.p("k_lo"), c.p("v_lo"), c.p("p_lo"), c.cap("cap_lo"),
                            (int32_t *)lens.data_ptr(), status(a[7]), stream(a[8]));
    return wrap(lens);
}

// (desc, q, k_new, v_new, cache, max_len, out, ws, status, stream)
PyObject *decode_quant(Args a) {
    const at::Tensor &q = dev(a[1], "q");
    const zipvl_decode_desc d = structure<zipvl_decode_desc>(a[0], "desc");
    const int max_len = int_arg(a[5]);
    const at::Tensor out = out_like(a[6], q);
    const at::Tensor ws = lazy_workspace(a[7], q, [&] { return decode_bytes(d, max_len, 1); });
    const Cache c{a[4]};
    check(zipvl_decode_quant, &d, q.data_ptr(), ptr(a[2], "k_new"), ptr(a[3], "v_new"), c.p("k_hi"), c.p("v_hi"),
                             c.p("p_hi"), c.cap("cap_hi"), c.p("k_lo"), c.p("v_lo"), c.p("p_lo"), c.cap("cap_lo"),
                             (int32_t *)c.p("lens"), max_len, out.data_ptr(), ws.data_ptr(), (size_t)ws.numel(),
                             status(a[8]), stream(a[9]));
    return wrap(out);
}

// (desc, q, k_new, v_new, table, max_len, out, ws, status, stream)
PyObject *decode_quant_batch(Args a) {
    const at::Tensor &q = dev(a[1], "q"), &table = dev(a[4], "table", at::kLong);
    const zipvl_decode_desc d = structure<zipvl_decode_desc>(a[0], "desc");
    if (table.dim() != 2 || table.size(0) != d.batch || table.size(1) != 8)
        raise(PyExc_ValueError, "table must be int64 [batch, 8]");
    const int max_len = int_arg(a[5]);
    const at::Tensor out = out_like(a[6], q);
    const at::Tensor ws = lazy_workspace(a[7], q, [&] { return decode_bytes(d, max_len, d.batch); });
    check(zipvl_decode_quant_batch, &d, q.data_ptr(), ptr(a[2], "k_new"), ptr(a[3], "v_new"),
                                   (const zipvl_quant_cache *)table.data_ptr(), max_len, out.data_ptr(), ws.data_ptr(),
                                   (size_t)ws.numel(), status(a[8]), stream(a[9]));
    return wrap(out);
}

template <PyObject *(*F)(Args), int N>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "zipvl native call: %d arguments wanted, %zd given", N, n);
        return nullptr;
    }
    try {
        return F(args);
    } catch (const Failed &) {
        return nullptr;
    } catch (const c10::Error &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

PyObject *set_error_class(PyObject *, PyObject *cls) {
    Py_XDECREF(g_error_class);
    g_error_class = Py_NewRef(cls);
    Py_RETURN_NONE;
}

#define ZIPVL_ENTRY(name, n) {#name, (PyCFunction)(void (*)(void))entry<name, n>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ZIPVL_ENTRY(score, 10),
                         ZIPVL_ENTRY(select, 11),
                         ZIPVL_ENTRY(sparse_prefill, 12),
                         ZIPVL_ENTRY(sparse_prefill_compact, 16),
                         ZIPVL_ENTRY(score_batch, 8),
                         ZIPVL_ENTRY(select_batch, 10),
                         ZIPVL_ENTRY(sparse_prefill_batch, 15),
                         ZIPVL_ENTRY(compact_kv, 12),
                         ZIPVL_ENTRY(decode, 14),
                         ZIPVL_ENTRY(decode_paged, 14),
                         ZIPVL_ENTRY(decode_noalloc, 13),
                         ZIPVL_ENTRY(quantize_kv, 9),
                         ZIPVL_ENTRY(decode_quant, 10),
                         ZIPVL_ENTRY(decode_quant_batch, 10),
                         {"set_error_class", set_error_class, METH_O, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
