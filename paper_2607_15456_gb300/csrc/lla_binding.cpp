// lla_binding.cpp -- native marshalling of the Python binding's calls (paper_2607_15456_gb300/lla.py).
//
// Each function takes the arguments of the Python function of the same name (with a stream handle or
// None for the current stream), fills the structs of include/lla.h straight from the objects and calls
// liblla with the GIL released.  It handles the ordinary call and nothing else: plain CUDA tensors
// (torch.nn.Parameter among them) that are contiguous, or None, Python ints in range, bf16 or fp32 data.
// Anything else (integer addresses,
// tensor subclasses, host or strided tensors, other types, wrong lengths) returns None, and the caller
// goes through its Python marshalling, which accepts or refuses it as it always did.  No reference is
// kept to any argument.
//
// A call is bound by this on the host: marshalling 24 layers in Python took 95 us beside 25 us of
// kernel, a decode call 13 us; here 5 and 2 us.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <cstdint>
#include <limits>
#include <vector>

#include "lla.h"

namespace {

struct Names {
    PyObject *T, *H, *d, *r_k, *r_v, *storage, *scale;
    PyObject *codec[6];
    PyObject *pool, *num_blocks, *block_table, *max_blocks;
} names;

struct Unusual {};  // thrown to leave for the Python path

// A new reference that is dropped at the end of its scope.
struct Ref {
    PyObject *o;
    explicit Ref(PyObject *p) : o(p) {
        if (!o) throw Unusual();
    }
    ~Ref() { Py_XDECREF(o); }
    Ref(const Ref &) = delete;
    Ref &operator=(const Ref &) = delete;
};

int64_t integer(PyObject *o) {
    if (!PyLong_CheckExact(o)) throw Unusual();
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    if (over) throw Unusual();
    return v;
}
int32_t integer32(PyObject *o) {
    const int64_t v = integer(o);
    if (v < std::numeric_limits<int32_t>::min() || v > std::numeric_limits<int32_t>::max()) throw Unusual();
    return static_cast<int32_t>(v);
}
int32_t attr32(PyObject *o, PyObject *name) {
    const Ref r(PyObject_GetAttr(o, name));
    return integer32(r.o);
}
double real(PyObject *o) {
    if (!PyFloat_CheckExact(o)) throw Unusual();
    return PyFloat_AS_DOUBLE(o);
}

const at::Tensor &tensor(PyObject *o) {
    if (!THPVariable_CheckExact(o)) throw Unusual();
    const at::Tensor &t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || !t.is_contiguous()) throw Unusual();
    return t;
}
void *address(PyObject *o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
void *attr_address(PyObject *o, PyObject *name) {
    const Ref r(PyObject_GetAttr(o, name));  // the object keeps the tensor alive
    return address(r.o);
}
lla_dtype dtype(const at::Tensor &t) {
    if (t.scalar_type() == at::kBFloat16) return LLA_BF16;
    if (t.scalar_type() == at::kFloat) return LLA_F32;
    throw Unusual();
}
size_t nbytes(const at::Tensor &t) { return static_cast<size_t>(t.numel()) * t.element_size(); }

lla_geometry geometry(PyObject *o) {
    lla_geometry g;
    g.T = attr32(o, names.T);
    g.H = attr32(o, names.H);
    g.d = attr32(o, names.d);
    g.r_k = attr32(o, names.r_k);
    g.r_v = attr32(o, names.r_v);
    g.block_size = LLA_BLOCK_TOKENS;
    const Ref st(PyObject_GetAttr(o, names.storage)), sc(PyObject_GetAttr(o, names.scale));
    if (!PyUnicode_CheckExact(st.o)) throw Unusual();
    g.storage = PyUnicode_CompareWithASCIIString(st.o, "bf16") == 0 ? LLA_BF16 : LLA_F32;
    if (sc.o == Py_None && g.d <= 0) throw Unusual();
    g.scale = static_cast<float>(sc.o == Py_None ? 1.0 / std::sqrt(static_cast<double>(g.d)) : real(sc.o));
    return g;
}
lla_codec codec(PyObject *o) {
    void *p[6];
    for (int i = 0; i < 6; ++i) p[i] = attr_address(o, names.codec[i]);
    return lla_codec{p[0], p[1], p[2], p[3], static_cast<const float *>(p[4]), static_cast<const float *>(p[5])};
}
lla_cache cache(PyObject *o) {
    lla_cache c;
    c.pool = attr_address(o, names.pool);
    const Ref nb(PyObject_GetAttr(o, names.num_blocks));
    c.num_blocks = integer(nb.o);
    c.block_table = static_cast<const int32_t *>(attr_address(o, names.block_table));
    c.max_blocks_per_seq = attr32(o, names.max_blocks);
    return c;
}
lla_rope rope(PyObject *base, PyObject *pairing) {
    return lla_rope{real(base), static_cast<lla_rope_pairing>(integer32(pairing))};
}
void *stream_of(PyObject *o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    return reinterpret_cast<void *>(static_cast<intptr_t>(integer(o)));
}

// Runs `body` (which marshals, then calls liblla): its status as an int, or None for the Python path.
template <typename F>
PyObject *guarded(Py_ssize_t nargs, Py_ssize_t want, F body) {
    if (nargs != want) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return nullptr;
    }
    int status = 0;
    try {
        status = body();
    } catch (...) {  // Unusual, or an exception of torch (a tensor without storage)
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    return PyLong_FromLong(status);
}

// Releases the GIL for its scope.
struct NoGil {
    PyThreadState *s = PyEval_SaveThread();
    ~NoGil() { PyEval_RestoreThread(s); }
};

using DecodeFn = decltype(&lla_decode_attn);
PyObject *decode(DecodeFn fn, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 12, [&] {
        const lla_geometry g = geometry(a[0]);
        const lla_codec cd = codec(a[1]);
        const lla_cache ch = cache(a[2]);
        const at::Tensor &q = tensor(a[6]), &ws = tensor(a[10]);
        if (q.dim() < 1) throw Unusual();
        const auto *ctx = static_cast<const int32_t *>(address(a[3]));
        const int32_t max_ctx = integer32(a[4]), loop = integer32(a[5]), B = static_cast<int32_t>(q.size(0));
        void *ck = address(a[7]), *cv = address(a[8]), *out = address(a[9]), *w = ws.data_ptr(), *qp = q.data_ptr();
        const lla_dtype io = dtype(q);
        const size_t wb = nbytes(ws);
        void *st = stream_of(a[11]);
        NoGil nogil;
        return fn(&g, &cd, &ch, ctx, B, max_ctx, loop, qp, ck, cv, io, out, w, wb, st);
    });
}
PyObject *decode_attn(PyObject *, PyObject *const *a, Py_ssize_t n) { return decode(&lla_decode_attn, a, n); }
PyObject *decode_attn_2d(PyObject *, PyObject *const *a, Py_ssize_t n) { return decode(&lla_decode_attn_2d, a, n); }

PyObject *decode_attn_loops(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 11, [&] {
        const lla_geometry g = geometry(a[0]);
        const lla_codec cd = codec(a[1]);
        const lla_cache ch = cache(a[2]);
        const at::Tensor &q = tensor(a[5]), &ws = tensor(a[9]);
        if (q.dim() < 2) throw Unusual();
        const auto *ctx = static_cast<const int32_t *>(address(a[3]));
        const int32_t max_ctx = integer32(a[4]), B = static_cast<int32_t>(q.size(1));
        void *ck = address(a[6]), *cv = address(a[7]), *out = address(a[8]), *w = ws.data_ptr(), *qp = q.data_ptr();
        const lla_dtype io = dtype(q);
        const size_t wb = nbytes(ws);
        void *st = stream_of(a[10]);
        NoGil nogil;
        return lla_decode_attn_loops(&g, &cd, &ch, ctx, B, max_ctx, qp, ck, cv, io, out, w, wb, st);
    });
}

PyObject *decode_attn_rope(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 14, [&] {
        const lla_geometry g = geometry(a[0]);
        const lla_codec cd = codec(a[1]);
        const lla_cache ch = cache(a[2]);
        const lla_rope rp = rope(a[3], a[4]);
        const at::Tensor &q = tensor(a[8]), &ws = tensor(a[12]);
        if (q.dim() < 1) throw Unusual();
        const auto *ctx = static_cast<const int32_t *>(address(a[5]));
        const int32_t max_ctx = integer32(a[6]), loop = integer32(a[7]), B = static_cast<int32_t>(q.size(0));
        void *ck = address(a[9]), *cv = address(a[10]), *out = address(a[11]), *w = ws.data_ptr(), *qp = q.data_ptr();
        const lla_dtype io = dtype(q);
        const size_t wb = nbytes(ws);
        void *st = stream_of(a[13]);
        NoGil nogil;
        return lla_decode_attn_rope(&g, &cd, &ch, &rp, ctx, B, max_ctx, loop, qp, ck, cv, io, out, w, wb, st);
    });
}

PyObject *decode_attn_decoupled(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 18, [&] {
        const lla_geometry g = geometry(a[0]);
        const lla_codec cd = codec(a[1]);
        const lla_cache ch = cache(a[2]);
        void *pool = address(a[3]);
        const int32_t dr = integer32(a[4]);
        const lla_rope rp = rope(a[5], a[6]);
        const at::Tensor &q = tensor(a[10]), &ws = tensor(a[16]);
        if (q.dim() < 1) throw Unusual();
        const auto *ctx = static_cast<const int32_t *>(address(a[7]));
        const int32_t max_ctx = integer32(a[8]), loop = integer32(a[9]), B = static_cast<int32_t>(q.size(0));
        void *qr = address(a[11]), *ck = address(a[12]), *cv = address(a[13]), *ckr = address(a[14]), *out = address(a[15]);
        void *w = ws.data_ptr(), *qp = q.data_ptr();
        const lla_dtype io = dtype(q);
        const size_t wb = nbytes(ws);
        void *st = stream_of(a[17]);
        NoGil nogil;
        return lla_decode_attn_decoupled(&g, &cd, &ch, pool, dr, &rp, ctx, B, max_ctx, loop, qp, qr, ck, cv, ckr, io, out, w,
                                         wb, st);
    });
}

using EncodeFn = decltype(&lla_encode);
PyObject *encode_with(EncodeFn fn, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 7, [&] {
        const lla_geometry g = geometry(a[0]);
        const lla_codec cd = codec(a[1]);
        const lla_cache ch = cache(a[2]);
        const at::Tensor &x = tensor(a[3]);
        void *xk = x.data_ptr(), *xv = address(a[4]);
        const auto *slots = static_cast<const int64_t *>(address(a[5]));
        const int32_t N = x.dim() == 4 ? static_cast<int32_t>(x.size(1)) : 0;
        const lla_dtype xd = dtype(x);
        void *st = stream_of(a[6]);
        NoGil nogil;
        return fn(&g, &cd, &ch, xk, xv, xd, slots, N, st);
    });
}
PyObject *encode(PyObject *, PyObject *const *a, Py_ssize_t n) { return encode_with(&lla_encode, a, n); }
PyObject *encode_2d(PyObject *, PyObject *const *a, Py_ssize_t n) { return encode_with(&lla_encode_2d, a, n); }

PyObject *encode_layers(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 7, [&] {
        const lla_geometry g = geometry(a[0]);
        for (int i = 1; i < 5; ++i)
            if (!PyList_CheckExact(a[i]) && !PyTuple_CheckExact(a[i])) throw Unusual();
        const Py_ssize_t L = PySequence_Fast_GET_SIZE(a[1]);
        if (L < 1 || L > 4096) throw Unusual();
        for (int i = 2; i < 5; ++i)
            if (PySequence_Fast_GET_SIZE(a[i]) != L) throw Unusual();
        std::vector<lla_codec> cds(L);
        std::vector<lla_cache> chs(L);
        std::vector<const void *> xk(L), xv(L);
        // an attribute could run Python code that changes a list, so each item is held while it is read
        auto item = [&](int i, Py_ssize_t l) {
            if (PySequence_Fast_GET_SIZE(a[i]) != L) throw Unusual();
            PyObject *o = PySequence_Fast_GET_ITEM(a[i], l);
            Py_INCREF(o);
            return o;
        };
        for (Py_ssize_t l = 0; l < L; ++l) {
            const Ref c(item(1, l)), h(item(2, l)), k(item(3, l)), v(item(4, l));
            cds[l] = codec(c.o);
            chs[l] = cache(h.o);
            xk[l] = address(k.o);
            xv[l] = address(v.o);
        }
        const Ref first(item(3, 0));
        const at::Tensor &x = tensor(first.o);
        const auto *slots = static_cast<const int64_t *>(address(a[5]));
        const int32_t N = x.dim() == 4 ? static_cast<int32_t>(x.size(1)) : 0;
        const lla_dtype xd = dtype(x);
        void *st = stream_of(a[6]);
        NoGil nogil;
        return lla_encode_layers(&g, static_cast<int32_t>(L), cds.data(), chs.data(), xk.data(), xv.data(), xd, slots, N, st);
    });
}

PyObject *prefill_attn(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 9, [&] {
        const lla_geometry g = geometry(a[0]);
        const lla_codec cd = codec(a[1]);
        const lla_cache ch = cache(a[2]);
        const at::Tensor &cu = tensor(a[3]), &q = tensor(a[6]);
        if (cu.dim() < 1) throw Unusual();
        const int32_t max_len = integer32(a[4]), loop = integer32(a[5]), B = static_cast<int32_t>(cu.size(0)) - 1;
        const auto *cp = static_cast<const int32_t *>(cu.data_ptr());
        void *qp = q.data_ptr(), *out = address(a[7]);
        const lla_dtype io = dtype(q);
        void *st = stream_of(a[8]);
        NoGil nogil;
        return lla_prefill_attn(&g, &cd, &ch, cp, B, max_len, loop, qp, io, out, st);
    });
}

PyObject *prefill_attn_rope(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 12, [&] {
        const lla_geometry g = geometry(a[0]);
        const lla_codec cd = codec(a[1]);
        const lla_cache ch = cache(a[2]);
        const lla_rope rp = rope(a[3], a[4]);
        const at::Tensor &cu = tensor(a[5]), &q = tensor(a[8]), &ws = tensor(a[10]);
        if (cu.dim() < 1) throw Unusual();
        const int32_t max_len = integer32(a[6]), loop = integer32(a[7]), B = static_cast<int32_t>(cu.size(0)) - 1;
        const auto *cp = static_cast<const int32_t *>(cu.data_ptr());
        void *qp = q.data_ptr(), *out = address(a[9]), *w = ws.data_ptr();
        const lla_dtype io = dtype(q);
        const size_t wb = nbytes(ws);
        void *st = stream_of(a[11]);
        NoGil nogil;
        return lla_prefill_attn_rope(&g, &cd, &ch, &rp, cp, B, max_len, loop, qp, io, out, w, wb, st);
    });
}

#define LLA_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    LLA_METHOD(decode_attn), LLA_METHOD(decode_attn_2d), LLA_METHOD(decode_attn_loops), LLA_METHOD(decode_attn_rope),
    LLA_METHOD(decode_attn_decoupled), LLA_METHOD(encode), LLA_METHOD(encode_2d), LLA_METHOD(encode_layers),
    LLA_METHOD(prefill_attn), LLA_METHOD(prefill_attn_rope), {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_lla_native", "Native marshalling of the calls of lla.py.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__lla_native() {
    auto s = [](const char *t) { return PyUnicode_InternFromString(t); };
    names = Names{s("T"), s("H"), s("d"), s("r_k"), s("r_v"), s("storage"), s("scale"),
                  {s("w_down_k"), s("w_down_v"), s("w_up_k"), s("w_up_v"), s("mu_k"), s("mu_v")},
                  s("pool"), s("num_blocks"), s("block_table"), s("max_blocks_per_seq")};
    return PyModule_Create(&module);
}
