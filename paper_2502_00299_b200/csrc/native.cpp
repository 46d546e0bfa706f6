// The per-call part of the Python binding: argument checks, output allocation and the C ABI call of the entry points that a program
// calls per layer or per model, in one native function each.
//
// A layer call of a short prompt takes 12 to 17 us on the device, and marshalling it through ctypes took about 20 us on the
// host: sizes asked of the library, three allocations and a stream object through Python, sixteen converted arguments.
// These functions do the same work in 5 to 7.
//
// They take what programs normally pass - plain tensors and plain ints - and answer None for everything else (subclasses,
// other number types, tensors that fail a check, a scratch buffer that has to grow, an active torch-function mode), before
// anything is queued: the Python function then goes its general way, which raises the errors. A status of the C ABI other
// than 0 is returned as an int. Nothing is kept between calls but the dict in which the binding keeps its scratch tensors.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>
#include <memory>
#include <vector>

#include "../../include/chunkkv.h"

namespace {

PyObject* g_scratch = nullptr;           // the binding's dict of the scratch tensors handed to the library, by device

// What a call cannot take: the caller returns None.
struct Decline {};

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_CheckExact(o)) throw Decline{};
    return THPVariable_Unpack(o);
}
const at::Tensor& checked(PyObject* o, at::ScalarType type) {
    const at::Tensor& t = tensor(o);
    if (!t.is_cuda() || t.scalar_type() != type || !t.is_contiguous()) throw Decline{};
    return t;
}
// The same with at least `need` elements.
const at::Tensor& sized(PyObject* o, at::ScalarType type, long long need) {
    const at::Tensor& t = checked(o, type);
    if (t.numel() < need) throw Decline{};
    return t;
}
int narrow(long long v) {
    if (v < INT_MIN || v > INT_MAX) throw Decline{};
    return static_cast<int>(v);
}
int integer(PyObject* o) {
    if (!PyLong_CheckExact(o)) throw Decline{};
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    if (over != 0) throw Decline{};
    return narrow(v);
}
// None: the current stream of the current device; else a torch.cuda.Stream.
void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
    if (v == nullptr) { PyErr_Clear(); throw Decline{}; }
    void* s = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) { PyErr_Clear(); throw Decline{}; }
    return s;
}
void room(size_t need) {
    PyObject* dev = g_scratch != nullptr && need > 0 ? PyLong_FromLong(c10::cuda::current_device()) : nullptr;
    if (dev == nullptr) throw Decline{};
    PyObject* buf = PyDict_GetItemWithError(g_scratch, dev);       // (borrowed)
    Py_DECREF(dev);
    if (buf == nullptr || !THPVariable_Check(buf) || THPVariable_Unpack(buf).numel() < static_cast<long long>(need)) throw Decline{};
}
at::Tensor rows(const at::Tensor& like, long long heads, long long n, long long d) {
    return at::empty({heads, n, d}, at::TensorOptions().dtype(at::kBFloat16).device(like.device()));
}
at::Tensor ids(const at::Tensor& like, long long heads, long long n) {
    return at::empty({heads, n}, at::TensorOptions().dtype(at::kInt).device(like.device()));
}
struct Ref {                             // an owned reference
    PyObject* p = nullptr;
    Ref() = default;
    Ref(const Ref&) = delete;
    Ref& operator=(const Ref&) = delete;
    ~Ref() { Py_XDECREF(p); }
    template <class Make>
    void* set(PyObject* given, at::ScalarType type, long long n, Make make) {      // the given output (n elements of `type`) or a new one; its address
        if (given != Py_None) {
            sized(given, type, n);
            p = given;
            Py_INCREF(p);
        } else {
            p = THPVariable_Wrap(make());
            if (p == nullptr) { PyErr_Clear(); throw Decline{}; }
        }
        return tensor(p).data_ptr();
    }
};

// Runs `call` without the interpreter lock, which is held again however it ends.
template <class Call>
int unlocked(Call call) {
    struct Unlock {
        PyThreadState* save = PyEval_SaveThread();
        ~Unlock() { PyEval_RestoreThread(save); }
    } unlock;
    return call();
}

// Runs `body`, which returns a new reference; None for what it declines. (A C++ exception is one of torch's about a tensor: the
// general way meets and raises it as well.)
template <class Body>
PyObject* guarded(Py_ssize_t n, Py_ssize_t want, Body body) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments expected", want);
        return nullptr;
    }
    try {
        if (at::impl::torch_function_mode_enabled()) throw Decline{};
        return body();
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

// scratch(dict): the dict in which the binding keeps the scratch tensors; returns the one in use
PyObject* scratch(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n > 1 || (n == 1 && !PyDict_CheckExact(a[0]))) { PyErr_SetString(PyExc_TypeError, "a dict expected"); return nullptr; }
    if (n == 1) {
        Py_INCREF(a[0]);
        Py_XSETREF(g_scratch, a[0]);
    }
    PyObject* r = g_scratch != nullptr ? g_scratch : Py_None;
    Py_INCREF(r);
    return r;
}

// layer(q_obs, K, V, Hq, w, c, budget, reuse_idx, out_K, out_V, out_idx, stream) -> (out_K, out_V, out_idx)
PyObject* layer(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 12, [&]() -> PyObject* {
        const at::Tensor& K = checked(a[1], at::kBFloat16);
        if (K.dim() != 3) throw Decline{};
        const at::Tensor& V = sized(a[2], at::kBFloat16, K.numel());
        const int Hkv = narrow(K.size(0)), L = narrow(K.size(1)), d = narrow(K.size(2));
        const int Hq = integer(a[3]), w = integer(a[4]), c = integer(a[5]), budget = integer(a[6]);
        const int n_max = chunkkv_out_len(L, w, c, budget);
        if (n_max < 0) throw Decline{};
        const long long n_row = static_cast<long long>(Hkv) * n_max;
        const void* q = a[0] == Py_None ? nullptr : sized(a[0], at::kBFloat16, static_cast<long long>(Hq) * w * d).data_ptr();
        const int32_t* reuse = a[7] == Py_None ? nullptr : static_cast<const int32_t*>(sized(a[7], at::kInt, n_row).data_ptr());
        if (reuse == nullptr) room(chunkkv_workspace_bytes(L, Hq, Hkv, d, w, c));
        void* s = stream_of(a[11]);
        Ref oK, oV, oI;
        void* pK = oK.set(a[8], at::kBFloat16, n_row * d, [&] { return rows(K, Hkv, n_max, d); });
        void* pV = oV.set(a[9], at::kBFloat16, n_row * d, [&] { return rows(K, Hkv, n_max, d); });
        int32_t* pI = static_cast<int32_t*>(oI.set(a[10], at::kInt, n_row, [&] { return ids(K, Hkv, n_max); }));
        const void *k = K.data_ptr(), *v = V.data_ptr();
        const int st = unlocked([&] { return chunkkv_compress_layer(q, k, v, L, Hq, Hkv, d, w, c, budget, reuse, pK, pV, pI, s); });
        if (st != 0) return PyLong_FromLong(st);
        return PyTuple_Pack(3, oK.p, oV.p, oI.p);
    });
}

// layer_strided: as layer, K and V [Hkv, L, d] views with a contiguous last dimension
PyObject* layer_strided(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 12, [&]() -> PyObject* {
        const at::Tensor &K = tensor(a[1]), &V = tensor(a[2]);
        for (const at::Tensor* t : {&K, &V})
            if (!t->is_cuda() || t->scalar_type() != at::kBFloat16 || t->dim() != 3 || t->stride(2) != 1) throw Decline{};
        for (int i = 0; i < 3; ++i)
            if (V.size(i) < K.size(i)) throw Decline{};
        const int Hkv = narrow(K.size(0)), L = narrow(K.size(1)), d = narrow(K.size(2));
        const int Hq = integer(a[3]), w = integer(a[4]), c = integer(a[5]), budget = integer(a[6]);
        const int n_max = chunkkv_out_len(L, w, c, budget);
        if (n_max < 0) throw Decline{};
        const long long n_row = static_cast<long long>(Hkv) * n_max;
        const void* q = a[0] == Py_None ? nullptr : sized(a[0], at::kBFloat16, static_cast<long long>(Hq) * w * d).data_ptr();
        const int32_t* reuse = a[7] == Py_None ? nullptr : static_cast<const int32_t*>(sized(a[7], at::kInt, n_row).data_ptr());
        if (reuse == nullptr) room(chunkkv_workspace_bytes(L, Hq, Hkv, d, w, c));
        void* s = stream_of(a[11]);
        Ref oK, oV, oI;
        void* pK = oK.set(a[8], at::kBFloat16, n_row * d, [&] { return rows(K, Hkv, n_max, d); });
        void* pV = oV.set(a[9], at::kBFloat16, n_row * d, [&] { return rows(K, Hkv, n_max, d); });
        int32_t* pI = static_cast<int32_t*>(oI.set(a[10], at::kInt, n_row, [&] { return ids(K, Hkv, n_max); }));
        const void *k = K.data_ptr(), *v = V.data_ptr();
        const long long kt = K.stride(1), kh = K.stride(0), vt = V.stride(1), vh = V.stride(0);
        const int st = unlocked([&] {
            return chunkkv_compress_layer_strided(q, k, v, L, Hq, Hkv, d, w, c, budget, kt, kh, vt, vh, reuse, pK, pV, pI, s);
        });
        if (st != 0) return PyLong_FromLong(st);
        return PyTuple_Pack(3, oK.p, oV.p, oI.p);
    });
}

// layer_alg1(q_obs, K, V, Hq, w, c, budget, out_K, out_V, out_idx, stream) -> (out_K, out_V, out_idx)
PyObject* layer_alg1(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 11, [&]() -> PyObject* {
        const at::Tensor& K = checked(a[1], at::kBFloat16);
        if (K.dim() != 3) throw Decline{};
        const at::Tensor& V = sized(a[2], at::kBFloat16, K.numel());
        const int Hkv = narrow(K.size(0)), L = narrow(K.size(1)), d = narrow(K.size(2));
        const int Hq = integer(a[3]), w = integer(a[4]), c = integer(a[5]), budget = integer(a[6]);
        const int n_max = chunkkv_out_len_alg1(L, w, c, budget);
        if (n_max < 0) throw Decline{};
        const long long n_row = static_cast<long long>(Hkv) * n_max;
        const at::Tensor& q = sized(a[0], at::kBFloat16, static_cast<long long>(Hq) * w * d);
        room(chunkkv_workspace_bytes(L, Hq, Hkv, d, w, c));
        void* s = stream_of(a[10]);
        Ref oK, oV, oI;
        void* pK = oK.set(a[7], at::kBFloat16, n_row * d, [&] { return rows(K, Hkv, n_max, d); });
        void* pV = oV.set(a[8], at::kBFloat16, n_row * d, [&] { return rows(K, Hkv, n_max, d); });
        int32_t* pI = static_cast<int32_t*>(oI.set(a[9], at::kInt, n_row, [&] { return ids(K, Hkv, n_max); }));
        const void *pq = q.data_ptr(), *k = K.data_ptr(), *v = V.data_ptr();
        const int st = unlocked([&] { return chunkkv_compress_layer_alg1(pq, k, v, L, Hq, Hkv, d, w, c, budget, pK, pV, pI, s); });
        if (st != 0) return PyLong_FromLong(st);
        return PyTuple_Pack(3, oK.p, oV.p, oI.p);
    });
}

// layer_paged(q_obs, K, V, Hq, w, c, budget, block_table, cache_K, cache_V, reuse_idx, out_idx, stream) -> idx
PyObject* layer_paged(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 13, [&]() -> PyObject* {
        const at::Tensor &K = checked(a[1], at::kBFloat16), &cK = checked(a[8], at::kBFloat16);
        if (K.dim() != 3 || cK.dim() < 2) throw Decline{};
        const int Hkv = narrow(K.size(0)), L = narrow(K.size(1)), d = narrow(K.size(2));
        const int Hq = integer(a[3]), w = integer(a[4]), c = integer(a[5]), budget = integer(a[6]);
        const int n_max = chunkkv_out_len(L, w, c, budget);
        if (n_max < 0) throw Decline{};
        const long long page = narrow(cK.size(1)), pages = narrow(cK.size(0)), n_row = static_cast<long long>(Hkv) * n_max;
        if (page < 1) throw Decline{};
        const at::Tensor &V = sized(a[2], at::kBFloat16, K.numel()), &bt = sized(a[7], at::kInt, (n_max + page - 1) / page);
        const at::Tensor& cV = sized(a[9], at::kBFloat16, pages * page * Hkv * d);
        if (cK.numel() < pages * page * Hkv * d) throw Decline{};
        const void* q = a[0] == Py_None ? nullptr : sized(a[0], at::kBFloat16, static_cast<long long>(Hq) * w * d).data_ptr();
        const int32_t* reuse = a[10] == Py_None ? nullptr : static_cast<const int32_t*>(sized(a[10], at::kInt, n_row).data_ptr());
        if (reuse == nullptr) room(chunkkv_workspace_bytes(L, Hq, Hkv, d, w, c));
        void* s = stream_of(a[12]);
        Ref oI;
        int32_t* pI = static_cast<int32_t*>(oI.set(a[11], at::kInt, n_row, [&] { return ids(K, Hkv, n_max); }));
        const void *k = K.data_ptr(), *v = V.data_ptr();
        const int32_t* table = static_cast<const int32_t*>(bt.data_ptr());
        void *pK = cK.data_ptr(), *pV = cV.data_ptr();
        const int st = unlocked([&] {
            return chunkkv_compress_layer_paged(q, k, v, L, Hq, Hkv, d, w, c, budget, reuse, table, static_cast<int>(page),
                                                static_cast<int>(pages), pK, pV, pI, s);
        });
        if (st != 0) return PyLong_FromLong(st);
        Py_INCREF(oI.p);
        return oI.p;
    });
}

// window_queries(qkv, Hq, Hkv, d, w, cos_rows, sin_rows, stream) -> q_obs
PyObject* window_queries(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 8, [&]() -> PyObject* {
        const at::Tensor &x = checked(a[0], at::kBFloat16), &co = checked(a[5], at::kFloat), &si = checked(a[6], at::kFloat);
        if (x.dim() != 2) throw Decline{};
        const int T = narrow(x.size(0)), Hq = integer(a[1]), Hkv = integer(a[2]), d = integer(a[3]), w = integer(a[4]);
        if (Hq < 0 || w < 0 || d < 0 || co.numel() < static_cast<long long>(w) * (d / 2) || si.numel() < static_cast<long long>(w) * (d / 2)) throw Decline{};
        const long long row = x.size(1);
        void* s = stream_of(a[7]);
        Ref out;
        void* p = out.set(Py_None, at::kBFloat16, 0, [&] { return rows(x, Hq, w, d); });
        const void* px = x.data_ptr();
        const float *pc = static_cast<const float*>(co.data_ptr()), *ps = static_cast<const float*>(si.data_ptr());
        const int st = unlocked([&] { return chunkkv_window_queries(px, row, T, Hq, Hkv, d, w, pc, ps, p, s); });
        if (st != 0) return PyLong_FromLong(st);
        Py_INCREF(out.p);
        return out.p;
    });
}

// score(q_obs, K, w, c, want_token_scores, stream) -> (chunk scores, token scores or None)
PyObject* score(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 6, [&]() -> PyObject* {
        const at::Tensor &q = checked(a[0], at::kBFloat16), &K = checked(a[1], at::kBFloat16);
        if (q.dim() < 3 || K.dim() < 2) throw Decline{};
        const int Hq = narrow(q.size(0)), d = narrow(q.size(2)), Hkv = narrow(K.size(0)), L = narrow(K.size(1));
        const int w = integer(a[2]), c = integer(a[3]), C = chunkkv_num_chunks(L, w, c);
        if (C < 0 || !PyBool_Check(a[4])) throw Decline{};
        if (q.numel() < static_cast<long long>(Hq) * w * d || K.numel() < static_cast<long long>(Hkv) * L * d) throw Decline{};
        const bool tokens = a[4] == Py_True;
        room(chunkkv_workspace_bytes(L, Hq, Hkv, d, w, c));
        if (tokens) room(chunkkv_workspace_bytes(L, Hq, Hkv, d, w, 1));
        void* s = stream_of(a[5]);
        const auto f32 = at::TensorOptions().dtype(at::kFloat).device(K.device());
        Ref cs, ts;
        float* pc = static_cast<float*>(cs.set(Py_None, at::kFloat, 0, [&] { return at::empty({Hkv, C}, f32); }));
        float* pt = nullptr;
        if (tokens) pt = static_cast<float*>(ts.set(Py_None, at::kFloat, 0, [&] { return at::empty({Hkv, L - w}, f32); }));
        const void *pq = q.data_ptr(), *pk = K.data_ptr();
        const int st = unlocked([&] { return chunkkv_score(pq, pk, L, Hq, Hkv, d, w, c, pt, pc, s); });
        if (st != 0) return PyLong_FromLong(st);
        return PyTuple_Pack(2, cs.p, tokens ? ts.p : Py_None);
    });
}

// The items of a list or tuple as they are now, with a reference to each: an allocation can run Python code (a dispatch mode, a
// finalizer), which may change the list.
struct Items {
    Ref own;
    PyObject** p;
    Py_ssize_t n;
    explicit Items(PyObject* o) {
        if (!PyList_CheckExact(o) && !PyTuple_CheckExact(o)) throw Decline{};
        own.p = PySequence_Tuple(o);
        if (own.p == nullptr) throw Decline{};
        p = PySequence_Fast_ITEMS(own.p);
        n = PySequence_Fast_GET_SIZE(own.p);
    }
};

// model(layers, Hq, w, c, budget, n_reuse, stream, outs, strided) -> list of (out_K, out_V, out_idx); `outs` None or a list of tuples
PyObject* model(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 9, [&]() -> PyObject* {
        const Items layers(a[0]);
        const bool strided = a[8] == Py_True;
        if (layers.n < 1) throw Decline{};
        const int Hq = integer(a[1]), w = integer(a[2]);
        std::vector<const void*> q(layers.n), k(layers.n), v(layers.n);
        std::vector<void*> oK(layers.n), oV(layers.n);
        std::vector<int32_t*> oI(layers.n);
        int Hkv = 0, L = 0, d = 0;
        long long st[4] = {0, 0, 0, 0};
        std::vector<std::unique_ptr<Items>> held;       // the layers' and the outputs' tensors, until the call has been queued
        for (Py_ssize_t i = 0; i < layers.n; ++i) {
            const Items& t = *held.emplace_back(std::make_unique<Items>(layers.p[i]));
            if (t.n != 3) throw Decline{};
            for (int j = 1; j < 3; ++j) {
                const at::Tensor& x = strided ? tensor(t.p[j]) : checked(t.p[j], at::kBFloat16);
                if (x.dim() != 3) throw Decline{};
                if (i == 0 && j == 1) { Hkv = narrow(x.size(0)); L = narrow(x.size(1)); d = narrow(x.size(2)); }
                if (x.size(0) != Hkv || x.size(1) != L || x.size(2) != d) throw Decline{};
                if (strided) {
                    long long* w = st + 2 * (j - 1);
                    if (i == 0) { w[0] = x.stride(1); w[1] = x.stride(0); }
                    if (!x.is_cuda() || x.scalar_type() != at::kBFloat16 || x.stride(2) != 1 || x.stride(1) != w[0] || x.stride(0) != w[1])
                        throw Decline{};
                }
                (j == 1 ? k : v)[i] = x.data_ptr();
            }
            q[i] = t.p[0] == Py_None ? nullptr : sized(t.p[0], at::kBFloat16, static_cast<long long>(Hq) * w * d).data_ptr();
        }
        const int c = integer(a[3]), budget = integer(a[4]), n_reuse = integer(a[5]);
        const int n_max = chunkkv_out_len(L, w, c, budget);
        if (n_max < 0) throw Decline{};
        const long long n_row = static_cast<long long>(Hkv) * n_max;
        const int nl = narrow(layers.n);
        const size_t need = chunkkv_model_workspace_bytes(nl, L, Hq, Hkv, d, w, c, budget, n_reuse);
        room(need > 0 ? need : 1);
        if (strided) room(chunkkv_workspace_bytes(L, Hq, Hkv, d, w, c));
        void* s = stream_of(a[6]);
        Ref res;
        res.p = PyList_New(layers.n);
        if (res.p == nullptr) throw Decline{};
        if (a[7] == Py_None) {
            const at::Tensor& like = tensor(held[0]->p[1]);
            for (Py_ssize_t i = 0; i < layers.n; ++i) {
                Ref x, y, z;
                oK[i] = x.set(Py_None, at::kBFloat16, 0, [&] { return rows(like, Hkv, n_max, d); });
                oV[i] = y.set(Py_None, at::kBFloat16, 0, [&] { return rows(like, Hkv, n_max, d); });
                oI[i] = static_cast<int32_t*>(z.set(Py_None, at::kInt, 0, [&] { return ids(like, Hkv, n_max); }));
                PyObject* t = PyTuple_Pack(3, x.p, y.p, z.p);
                if (t == nullptr) throw Decline{};
                PyList_SET_ITEM(res.p, i, t);
            }
        } else {
            const Items outs(a[7]);
            if (outs.n != layers.n) throw Decline{};
            for (Py_ssize_t i = 0; i < layers.n; ++i) {
                if (!PyTuple_CheckExact(outs.p[i])) throw Decline{};
                const Items& o = *held.emplace_back(std::make_unique<Items>(outs.p[i]));
                if (o.n != 3) throw Decline{};
                oK[i] = sized(o.p[0], at::kBFloat16, n_row * d).data_ptr();
                oV[i] = sized(o.p[1], at::kBFloat16, n_row * d).data_ptr();
                oI[i] = static_cast<int32_t*>(sized(o.p[2], at::kInt, n_row).data_ptr());
                Py_INCREF(outs.p[i]);
                PyList_SET_ITEM(res.p, i, outs.p[i]);
            }
        }
        const int status = unlocked([&] {
            return strided ? chunkkv_compress_model_strided(nl, q.data(), k.data(), v.data(), L, Hq, Hkv, d, w, c, budget, n_reuse, st[0], st[1], st[2],
                                                            st[3], oK.data(), oV.data(), oI.data(), s)
                           : chunkkv_compress_model(nl, q.data(), k.data(), v.data(), L, Hq, Hkv, d, w, c, budget, n_reuse, oK.data(), oV.data(),
                                                    oI.data(), s);
        });
        if (status != 0) return PyLong_FromLong(status);
        Py_INCREF(res.p);
        return res.p;
    });
}

PyMethodDef kMethods[] = {
#define CKV_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
    CKV_METHOD(scratch), CKV_METHOD(layer), CKV_METHOD(layer_strided), CKV_METHOD(layer_alg1), CKV_METHOD(layer_paged),
    CKV_METHOD(window_queries), CKV_METHOD(score), CKV_METHOD(model), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", "Per-call part of the binding (see binding.py).", -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&kModule); }
