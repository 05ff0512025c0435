// The hot calls of the Python binding (pvq.py), as a CPython extension: tensor checks, output
// allocation and the C-ABI call without leaving native code.  A call on a small matrix is bound by the host:
// through ctypes it cost 6 to 14 us of Python (attribute look-ups, torch.empty, argument conversion)
// around a C call of a few us.
//
// The entry points of the library are handed over as addresses (init), so that the library stays the one
// pvq.py loaded.  Same checks and errors as before; no arithmetic of the codec happens here.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <vector>

#include "pvq.h"

namespace {

// ---- the library, as pvq.py found it
struct Entries {
    decltype(&pvq_encode) encode;
    decltype(&pvq_encode_amp) encode_amp;
    decltype(&pvq_decode) decode;
    decltype(&pvq_roundtrip) roundtrip;
    decltype(&pvq_rotate_encode) rotate_encode;
    decltype(&pvq_rotate_roundtrip) rotate_roundtrip;
    decltype(&pvq_encode_batched) encode_batched;
    decltype(&pvq_decode_batched) decode_batched;
    decltype(&pvq_code_words) code_words;
    decltype(&pvq_scale_row_stride) scale_row_stride;
} lib;
PyObject* raise_error = nullptr;  // raise_error(status, where) raises PvqError
PyObject *k_get, *k_x, *k_out, *k_codes, *k_scale_idx, *k_row_norm, *k_edges, *k_levels, *k_cols;

bool failed(int status, const char* where) {
    if (status == PVQ_OK) return false;
    PyObject* r = PyObject_CallFunction(raise_error, "is", status, where);
    Py_XDECREF(r);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, where);
    return true;
}

// A C-ABI call with the interpreter lock released (it may wait when the launch queue is full).
template <class F>
int unlocked(F&& f) {
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = f();
    Py_END_ALLOW_THREADS
    return status;
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

const at::Tensor* tensor_of(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a tensor");
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}

bool row_major(const at::Tensor& t) {
    if (!t.is_cuda()) {
        PyErr_SetString(PyExc_ValueError, "expected a CUDA tensor");
        return false;
    }
    if (!t.is_contiguous() && !(t.dim() == 2 && t.stride(1) == 1)) {
        PyErr_SetString(PyExc_ValueError, "expected a row-major tensor");
        return false;
    }
    return true;
}

// Data pointer of a tensor of the given type, or null for None.
bool pointer(PyObject* o, at::ScalarType type, void** out) {
    *out = nullptr;
    if (o == Py_None) return true;
    const at::Tensor* t = tensor_of(o);
    if (!t) return false;
    if (!t->is_cuda()) {
        PyErr_SetString(PyExc_ValueError, "expected a CUDA tensor");
        return false;
    }
    if (t->scalar_type() != type) {
        PyErr_Format(PyExc_TypeError, "expected dtype %s, got %s", c10::toString(type), c10::toString(t->scalar_type()));
        return false;
    }
    if (!row_major(*t)) return false;
    *out = t->data_ptr();
    return true;
}

bool integer(PyObject* o, long long* out) {
    *out = PyLong_AsLongLong(o);
    return !(*out == -1 && PyErr_Occurred());
}

bool want_args(Py_ssize_t got, Py_ssize_t want) {
    if (got == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
    return false;
}

// The input matrix of the encode-side calls.
struct Input {
    const at::Tensor* t;
    int dtype;
    long long rows, cols, ld;
};
bool input(PyObject* o, Input* in) {
    in->t = tensor_of(o);
    if (!in->t) return false;
    if (in->t->dim() != 2) {
        PyErr_SetString(PyExc_ValueError, "expected a matrix");
        return false;
    }
    if (!row_major(*in->t)) return false;
    if (in->t->scalar_type() == at::kFloat)
        in->dtype = PVQ_DTYPE_F32;
    else if (in->t->scalar_type() == at::kBFloat16)
        in->dtype = PVQ_DTYPE_BF16;
    else {
        PyErr_SetString(PyExc_TypeError, "input must be float32 or bfloat16");
        return false;
    }
    in->rows = in->t->size(0);
    in->cols = in->t->size(1);
    in->ld = in->t->stride(0);
    return true;
}

struct Params {
    long long N, K, b;
};
bool params(PyObject* const* a, Params* p) {
    if (!integer(a[0], &p->N) || !integer(a[1], &p->K) || !integer(a[2], &p->b)) return false;
    if (p->N == 0) {
        PyErr_SetString(PyExc_ZeroDivisionError, "group size 0");
        return false;
    }
    return true;
}

// codes, scale_idx and row_norm of the encode calls: the caller's (a tuple of three), or new ones
struct Encoded {
    PyObject* result = nullptr;  // the tuple to return
    void *codes, *sidx, *rnorm;
};
bool encoded(PyObject* out, const Input& in, const Params& p, Encoded* e) {
    if (out != Py_None) {
        PyObject* seq = PySequence_Tuple(out);
        if (!seq) return false;
        if (PyTuple_GET_SIZE(seq) != 3) {
            Py_DECREF(seq);
            PyErr_SetString(PyExc_ValueError, "expected three output tensors");
            return false;
        }
        e->result = seq;
        return pointer(PyTuple_GET_ITEM(seq, 0), at::kInt, &e->codes) && pointer(PyTuple_GET_ITEM(seq, 1), at::kByte, &e->sidx) &&
               pointer(PyTuple_GET_ITEM(seq, 2), at::kFloat, &e->rnorm);
    }
    int W = 0;
    if (failed(lib.code_words(static_cast<int>(p.N), static_cast<int>(p.K), &W), "pvq_code_words")) return false;
    const long long G = in.cols / p.N;
    const auto dev = in.t->device();
    at::Tensor codes = at::detail::empty_cuda({in.rows, G, W}, at::kInt, dev, std::nullopt);
    at::Tensor sidx = at::detail::empty_cuda({in.rows, static_cast<int64_t>(lib.scale_row_stride(G, static_cast<int>(p.b)))}, at::kByte, dev, std::nullopt);
    at::Tensor rnorm = at::detail::empty_cuda({in.rows}, at::kFloat, dev, std::nullopt);
    e->codes = codes.data_ptr();
    e->sidx = sidx.data_ptr();
    e->rnorm = rnorm.data_ptr();
    e->result = PyTuple_New(3);
    if (!e->result) return false;
    PyTuple_SET_ITEM(e->result, 0, THPVariable_Wrap(std::move(codes)));
    PyTuple_SET_ITEM(e->result, 1, THPVariable_Wrap(std::move(sidx)));
    PyTuple_SET_ITEM(e->result, 2, THPVariable_Wrap(std::move(rnorm)));
    return true;
}

// the bf16 output of the decode calls: the caller's, or a new one
struct Output {
    PyObject* result = nullptr;
    void* p;
    long long ld;
};
bool output(PyObject* out, long long rows, long long cols, c10::Device dev, Output* o) {
    if (out != Py_None) {
        const at::Tensor* t = tensor_of(out);
        if (!t || !pointer(out, at::kBFloat16, &o->p)) return false;
        o->ld = t->dim() > 0 ? t->stride(0) : 0;
        Py_INCREF(out);
        o->result = out;
        return true;
    }
    at::Tensor t = at::detail::empty_cuda({rows, cols}, at::kBFloat16, dev, std::nullopt);
    o->p = t.data_ptr();
    o->ld = cols;
    o->result = THPVariable_Wrap(std::move(t));
    return o->result != nullptr;
}

PyObject* finish(PyObject* result, bool bad) {
    if (!bad) return result;
    Py_XDECREF(result);
    return nullptr;
}

// encode(x, N, K, scale_bits, table, edges, out, amp_mode)
PyObject* bind_encode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Input in;
    Params p;
    Encoded e;
    void *table, *edges;
    long long amp = -1;
    if (!want_args(n, 8) || !input(a[0], &in) || !params(a + 1, &p) || !pointer(a[4], at::kInt, &table) || !pointer(a[5], at::kFloat, &edges))
        return nullptr;
    if (a[7] != Py_None && !integer(a[7], &amp)) return nullptr;
    if (!encoded(a[6], in, p, &e)) return finish(e.result, true);
    void* s = stream();
    const void* x = in.t->data_ptr();
    const bool plain = a[7] == Py_None;
    const int st = unlocked([&] {
        if (plain)
            return lib.encode(x, in.dtype, in.rows, in.cols, in.ld, p.N, p.K, p.b, static_cast<uint32_t*>(table), static_cast<float*>(edges),
                              static_cast<uint32_t*>(e.codes), static_cast<uint8_t*>(e.sidx), static_cast<float*>(e.rnorm), s);
        return lib.encode_amp(x, in.dtype, in.rows, in.cols, in.ld, p.N, p.K, p.b, static_cast<int>(amp), static_cast<uint32_t*>(table),
                              static_cast<float*>(edges), static_cast<uint32_t*>(e.codes), static_cast<uint8_t*>(e.sidx),
                              static_cast<float*>(e.rnorm), s);
    });
    return finish(e.result, failed(st, plain ? "pvq_encode" : "pvq_encode_amp"));
    END_HANDLE_TH_ERRORS
}

// rotate_encode(x, block, signs, N, K, scale_bits, table, edges, out)
PyObject* bind_rotate_encode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Input in;
    Params p;
    Encoded e;
    void *signs, *table, *edges;
    long long block;
    if (!want_args(n, 9) || !input(a[0], &in) || !integer(a[1], &block) || !pointer(a[2], at::kFloat, &signs) || !params(a + 3, &p) ||
        !pointer(a[6], at::kInt, &table) || !pointer(a[7], at::kFloat, &edges))
        return nullptr;
    if (!encoded(a[8], in, p, &e)) return finish(e.result, true);
    void* s = stream();
    const void* x = in.t->data_ptr();
    const int st = unlocked([&] {
        return lib.rotate_encode(x, in.dtype, in.rows, in.cols, in.ld, static_cast<int>(block), static_cast<float*>(signs), p.N, p.K, p.b,
                                 static_cast<uint32_t*>(table), static_cast<float*>(edges), static_cast<uint32_t*>(e.codes),
                                 static_cast<uint8_t*>(e.sidx), static_cast<float*>(e.rnorm), s);
    });
    return finish(e.result, failed(st, "pvq_rotate_encode"));
    END_HANDLE_TH_ERRORS
}

// decode(codes, scale_idx, row_norm, N, K, scale_bits, table, levels, out, status)
PyObject* bind_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Params p;
    Output o;
    void *codes, *sidx, *rnorm, *table, *levels, *status;
    if (!want_args(n, 10)) return nullptr;
    const at::Tensor* ct = tensor_of(a[0]);
    if (!ct) return nullptr;
    if (ct->dim() != 3) {
        PyErr_SetString(PyExc_ValueError, "expected codes of three dimensions");
        return nullptr;
    }
    if (!pointer(a[0], at::kInt, &codes) || !pointer(a[1], at::kByte, &sidx) || !pointer(a[2], at::kFloat, &rnorm) || !params(a + 3, &p) ||
        !pointer(a[6], at::kInt, &table) || !pointer(a[7], at::kFloat, &levels) || !pointer(a[9], at::kInt, &status))
        return nullptr;
    const long long rows = ct->size(0), cols = ct->size(1) * p.N;
    if (!output(a[8], rows, cols, ct->device(), &o)) return finish(o.result, true);
    void* s = stream();
    const int st = unlocked([&] {
        return lib.decode(static_cast<uint32_t*>(codes), static_cast<uint8_t*>(sidx), static_cast<float*>(rnorm), rows, cols, p.N, p.K, p.b,
                          static_cast<uint32_t*>(table), static_cast<float*>(levels), o.p, o.ld, static_cast<uint32_t*>(status), s);
    });
    return finish(o.result, failed(st, "pvq_decode"));
    END_HANDLE_TH_ERRORS
}

// roundtrip(x, N, K, scale_bits, table, edges, levels, out)
PyObject* bind_roundtrip(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Input in;
    Params p;
    Output o;
    void *table, *edges, *levels;
    if (!want_args(n, 8) || !input(a[0], &in) || !params(a + 1, &p) || !pointer(a[4], at::kInt, &table) || !pointer(a[5], at::kFloat, &edges) ||
        !pointer(a[6], at::kFloat, &levels))
        return nullptr;
    if (!output(a[7], in.rows, in.cols, in.t->device(), &o)) return finish(o.result, true);
    void* s = stream();
    const void* x = in.t->data_ptr();
    const int st = unlocked([&] {
        return lib.roundtrip(x, in.dtype, in.rows, in.cols, in.ld, p.N, p.K, p.b, static_cast<uint32_t*>(table), static_cast<float*>(edges),
                             static_cast<float*>(levels), o.p, o.ld, s);
    });
    return finish(o.result, failed(st, "pvq_roundtrip"));
    END_HANDLE_TH_ERRORS
}

// rotate_roundtrip(x, block, signs, N, K, scale_bits, table, edges, levels, out)
PyObject* bind_rotate_roundtrip(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Input in;
    Params p;
    Output o;
    void *signs, *table, *edges, *levels;
    long long block;
    if (!want_args(n, 10) || !input(a[0], &in) || !integer(a[1], &block) || !pointer(a[2], at::kFloat, &signs) || !params(a + 3, &p) ||
        !pointer(a[6], at::kInt, &table) || !pointer(a[7], at::kFloat, &edges) || !pointer(a[8], at::kFloat, &levels))
        return nullptr;
    if (!output(a[9], in.rows, in.cols, in.t->device(), &o)) return finish(o.result, true);
    void* s = stream();
    const void* x = in.t->data_ptr();
    const int st = unlocked([&] {
        return lib.rotate_roundtrip(x, in.dtype, in.rows, in.cols, in.ld, static_cast<int>(block), static_cast<float*>(signs), p.N, p.K, p.b,
                                    static_cast<uint32_t*>(table), static_cast<float*>(edges), static_cast<float*>(levels), o.p, o.ld, s);
    });
    return finish(o.result, failed(st, "pvq_rotate_roundtrip"));
    END_HANDLE_TH_ERRORS
}

// Entries of one item of a batched call: a dict, or any mapping with get().
struct Held {  // references to what a mapping returned, as long as it is looked at
    std::vector<PyObject*> refs;
    ~Held() {
        for (PyObject* o : refs) Py_DECREF(o);
    }
};
PyObject* item_value(PyObject* d, PyObject* key, bool needed, Held* held) {  // null: not there, or an error
    PyObject* v;
    if (PyDict_CheckExact(d)) {
        v = PyDict_GetItemWithError(d, key);
        Py_XINCREF(v);
        if (!v && needed && !PyErr_Occurred()) PyErr_SetObject(PyExc_KeyError, key);
    } else {
        v = needed ? PyObject_GetItem(d, key) : PyObject_CallMethodOneArg(d, k_get, key);
    }
    if (v) held->refs.push_back(v);
    return v;
}
const at::Tensor* item_tensor(PyObject* d, PyObject* key, bool needed, Held* held, bool* bad) {
    if (*bad) return nullptr;
    PyObject* v = item_value(d, key, needed, held);
    if (!v) {
        *bad = PyErr_Occurred() != nullptr;
        return nullptr;
    }
    if (v == Py_None && !needed) return nullptr;
    const at::Tensor* t = tensor_of(v);
    *bad = !t;
    return t;
}

bool describe(PyObject* items, std::vector<pvq_matrix_desc>* descs) {
    if (PyObject_Length(items) < 0) return false;  // (anything that has a length and can be gone through)
    PyObject* seq = PySequence_Fast(items, "expected a sequence of matrices");
    if (!seq) return false;
    const Py_ssize_t count = PySequence_Fast_GET_SIZE(seq);
    descs->resize(static_cast<size_t>(count));
    bool bad = false;
    for (Py_ssize_t i = 0; i < count && !bad; ++i) {
        PyObject* it = PySequence_Fast_GET_ITEM(seq, i);
        pvq_matrix_desc& d = (*descs)[static_cast<size_t>(i)];
        Held held;
        const at::Tensor* x = item_tensor(it, k_x, false, &held, &bad);
        const at::Tensor* out = item_tensor(it, k_out, false, &held, &bad);
        const at::Tensor* codes = item_tensor(it, k_codes, true, &held, &bad);
        const at::Tensor* sidx = item_tensor(it, k_scale_idx, true, &held, &bad);
        const at::Tensor* rnorm = item_tensor(it, k_row_norm, true, &held, &bad);
        const at::Tensor* edges = item_tensor(it, k_edges, false, &held, &bad);
        const at::Tensor* levels = item_tensor(it, k_levels, false, &held, &bad);
        if (bad) break;
        PyObject* cols_o = item_value(it, k_cols, true, &held);
        long long cols = 0;
        bad = !cols_o || !integer(cols_o, &cols);
        if (!bad && codes->dim() != 3) {
            PyErr_SetString(PyExc_ValueError, "expected codes of three dimensions");
            bad = true;
        }
        if (bad) break;
        d.d_x = x ? x->data_ptr() : nullptr;
        d.d_out = out ? out->data_ptr() : nullptr;
        d.d_codes = static_cast<uint32_t*>(codes->data_ptr());
        d.d_scale_idx = static_cast<uint8_t*>(sidx->data_ptr());
        d.d_row_norm = static_cast<float*>(rnorm->data_ptr());
        d.d_edges = edges ? static_cast<const float*>(edges->data_ptr()) : nullptr;
        d.d_levels = levels ? static_cast<const float*>(levels->data_ptr()) : nullptr;
        d.rows = codes->size(0);
        d.cols = cols;
        d.ld = x ? x->stride(0) : cols;
        d.ld_out = out ? out->stride(0) : cols;
    }
    Py_DECREF(seq);
    return !bad;
}

// encode_batched(items, dtype code, N, K, scale_bits, table)
PyObject* bind_encode_batched(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Params p;
    void* table;
    long long dtype;
    std::vector<pvq_matrix_desc> descs;
    if (!want_args(n, 6) || !describe(a[0], &descs) || !integer(a[1], &dtype) || !params(a + 2, &p) || !pointer(a[5], at::kInt, &table)) return nullptr;
    void* s = stream();
    const int st = unlocked([&] {
        return lib.encode_batched(descs.data(), static_cast<int>(descs.size()), static_cast<int>(dtype), p.N, p.K, p.b, static_cast<uint32_t*>(table), s);
    });
    if (failed(st, "pvq_encode_batched")) return nullptr;
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

// decode_batched(items, N, K, scale_bits, table, status)
PyObject* bind_decode_batched(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Params p;
    void *table, *status;
    std::vector<pvq_matrix_desc> descs;
    if (!want_args(n, 6) || !describe(a[0], &descs) || !params(a + 1, &p) || !pointer(a[4], at::kInt, &table) || !pointer(a[5], at::kInt, &status)) return nullptr;
    void* s = stream();
    const int st = unlocked([&] {
        return lib.decode_batched(descs.data(), static_cast<int>(descs.size()), p.N, p.K, p.b, static_cast<uint32_t*>(table), static_cast<uint32_t*>(status), s);
    });
    if (failed(st, "pvq_decode_batched")) return nullptr;
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

// init(raise_error, address of every entry of `Entries`, in its order)
PyObject* bind_init(PyObject*, PyObject* const* a, Py_ssize_t n) {
    constexpr Py_ssize_t count = sizeof(Entries) / sizeof(void*);
    if (!want_args(n, count + 1)) return nullptr;
    void* addr[count];
    for (Py_ssize_t i = 0; i < count; ++i) {
        addr[i] = PyLong_AsVoidPtr(a[i + 1]);
        if (PyErr_Occurred()) return nullptr;
    }
    std::memcpy(&lib, addr, sizeof lib);
    Py_INCREF(a[0]);
    Py_XSETREF(raise_error, a[0]);
    Py_RETURN_NONE;
}

template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyMethodDef method(const char* name) {
    return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(F)), METH_FASTCALL, nullptr};
}
PyMethodDef methods[] = {method<bind_init>("init"),
                         method<bind_encode>("encode"),
                         method<bind_decode>("decode"),
                         method<bind_roundtrip>("roundtrip"),
                         method<bind_rotate_encode>("rotate_encode"),
                         method<bind_rotate_roundtrip>("rotate_roundtrip"),
                         method<bind_encode_batched>("encode_batched"),
                         method<bind_decode_batched>("decode_batched"),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_bind", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__bind() {
    k_get = PyUnicode_InternFromString("get");
    k_x = PyUnicode_InternFromString("x");
    k_out = PyUnicode_InternFromString("out");
    k_codes = PyUnicode_InternFromString("codes");
    k_scale_idx = PyUnicode_InternFromString("scale_idx");
    k_row_norm = PyUnicode_InternFromString("row_norm");
    k_edges = PyUnicode_InternFromString("edges");
    k_levels = PyUnicode_InternFromString("levels");
    k_cols = PyUnicode_InternFromString("cols");
    return PyModule_Create(&module);
}
