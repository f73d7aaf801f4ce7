// Argument marshalling of the hot calls in native code: the CPython face of the C ABI that binding.py's methods use.
//
// What bounds it: a decoding cycle makes one to three calls per layer, each a few microseconds of device work, so the
// host time per call decides whether the stream ever runs dry.  Through ctypes a call cost 8.5 - 10 us (conversion of
// 8 to 17 arguments, a c_void_p object for each pointer, the stream looked up through three Python layers) of which
// the launch itself is 2 - 3; here the tensors' device pointers and torch's current stream are read directly.
//
// Every function takes the context handle as an integer first and returns the vispec_status; tensors must be
// contiguous CUDA tensors (AssertionError otherwise), None stands for NULL.  The interpreter lock is released around
// the C call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <c10/util/Exception.h>
#include <torch/csrc/autograd/python_variable.h>

#include "vispec.h"

namespace {

// One call's arguments, read from left to right.  After a failed conversion `ok` is false and an exception is set.
struct Args {
    PyObject* const* a;
    Py_ssize_t n;
    Py_ssize_t i = 0;
    bool ok = true;

    Args(PyObject* const* args, Py_ssize_t nargs, Py_ssize_t want) : a(args), n(nargs) {
        if (nargs != want) {
            PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, nargs);
            ok = false;
        }
    }
    vispec_ctx* ctx() {
        if (!ok) return nullptr;
        void* p = PyLong_AsVoidPtr(a[i++]);
        if (!p && PyErr_Occurred()) ok = false;
        return static_cast<vispec_ctx*>(p);
    }
    int num() {
        if (!ok) return 0;
        const long v = PyLong_AsLong(a[i++]);
        if (v == -1 && PyErr_Occurred()) ok = false;
        return static_cast<int>(v);
    }
    float real() {
        if (!ok) return 0.f;
        const double v = PyFloat_AsDouble(a[i++]);
        if (v == -1.0 && PyErr_Occurred()) ok = false;
        return static_cast<float>(v);
    }
    // The tensor whose sizes the call needs (at least / exactly `dims` of them); nullptr with an exception otherwise.
    const at::Tensor* tensor(int dims, bool exact = true) {
        if (!ok) return nullptr;
        PyObject* o = a[i];
        if (!THPVariable_Check(o)) {
            PyErr_SetString(PyExc_TypeError, "a CUDA tensor is expected");
            ok = false;
            return nullptr;
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (exact ? t.dim() != dims : t.dim() < dims) {
            PyErr_Format(PyExc_ValueError, "a tensor of %d dimensions is expected, got %d", dims, (int)t.dim());
            ok = false;
            return nullptr;
        }
        return &t;
    }
    template <typename T = void>
    T* ptr() {
        if (!ok) return nullptr;
        PyObject* o = a[i++];
        if (o == Py_None) return nullptr;
        if (!THPVariable_Check(o)) {
            PyErr_SetString(PyExc_TypeError, "a CUDA tensor or None is expected");
            ok = false;
            return nullptr;
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, "device pointers must come from contiguous CUDA tensors");
            ok = false;
            return nullptr;
        }
        return static_cast<T*>(t.data_ptr());
    }
};

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// The interpreter lock is given up for as long as this lives.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};

// The call itself, without the interpreter lock.
template <typename F>
PyObject* finish(const Args& g, F&& call) {
    if (!g.ok) return nullptr;
    void* const st = stream();
    int rc;
    {
        Unlocked unlocked;
        rc = call(st);
    }
    return PyLong_FromLong(rc);
}

// What the interpreter calls: an exception that torch throws on the way - a tensor without storage (a fake or wrapped one) has
// no data pointer, a process without a usable device has no current stream - becomes a RuntimeError; past this frame it would
// end the process.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
    try {
        return F(self, args, nargs);
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    } catch (...) {
        PyErr_SetString(PyExc_RuntimeError, "unknown C++ exception");
    }
    return nullptr;
}

int size(const at::Tensor* t, int d) { return t ? static_cast<int>(t->size(d)) : 0; }

#define NATIVE(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs)

NATIVE(tree_mask_build) {   // handle, parents, tree_mask, depth
    Args g(args, nargs, 4);
    vispec_ctx* c = g.ctx();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* parents = g.ptr<int32_t>(); auto* mask = g.ptr<uint64_t>(); auto* depth = g.ptr<int32_t>();
    return finish(g, [&](void* st) { return vispec_tree_mask_build(c, parents, B, N, mask, depth, st); });
}

NATIVE(tree_verify_attn) {  // handle, layer, q, k_cache, v_cache, kv_len, tree_mask, positions, scale, out, lse
    Args g(args, nargs, 11);
    vispec_ctx* c = g.ctx();
    const int layer = g.num();
    const at::Tensor* t = g.tensor(2, false);
    const int B = size(t, 0), N = size(t, 1);
    auto* q = g.ptr(); auto* k = g.ptr(); auto* v = g.ptr();
    auto* kv_len = g.ptr<int32_t>(); auto* mask = g.ptr<uint64_t>(); auto* pos = g.ptr<int32_t>();
    const float scale = g.real();
    auto* out = g.ptr(); auto* lse = g.ptr<float>();
    return finish(g, [&](void* st) { return vispec_tree_verify_attn(c, layer, q, k, v, kv_len, mask, pos, B, N, scale, out, lse, st); });
}

NATIVE(tree_verify_attn_rope) {  // handle, layer, q, k_new, v_new, rope_table, kv_len, tree_mask, scale, out, lse
    Args g(args, nargs, 11);
    vispec_ctx* c = g.ctx();
    const int layer = g.num();
    const at::Tensor* t = g.tensor(2, false);
    const int B = size(t, 0), N = size(t, 1);
    auto* q = g.ptr(); auto* k = g.ptr(); auto* v = g.ptr(); auto* table = g.ptr();
    auto* kv_len = g.ptr<int32_t>(); auto* mask = g.ptr<uint64_t>();
    const float scale = g.real();
    auto* out = g.ptr(); auto* lse = g.ptr<float>();
    return finish(g, [&](void* st) { return vispec_tree_verify_attn_rope(c, layer, q, k, v, table, kv_len, mask, B, N, scale, out, lse, st); });
}

NATIVE(tree_verify_attn_paged) {  // handle, layer, q, kv_len, block_table, tree_mask, scale, out, lse
    Args g(args, nargs, 9);
    vispec_ctx* c = g.ctx();
    const int layer = g.num();
    const at::Tensor* t = g.tensor(2, false);
    const int B = size(t, 0), N = size(t, 1);
    auto* q = g.ptr(); auto* kv_len = g.ptr<int32_t>();
    const int stride = size(g.tensor(2), 1);
    auto* table = g.ptr<int32_t>(); auto* mask = g.ptr<uint64_t>();
    const float scale = g.real();
    auto* out = g.ptr(); auto* lse = g.ptr<float>();
    return finish(g, [&](void* st) { return vispec_tree_verify_attn_paged(c, layer, q, kv_len, table, stride, mask, B, N, scale, out, lse, st); });
}

NATIVE(tree_verify_attn_static) {  // q, k_cache, v_cache, kv_len, tree_mask, scale, out, lse, status_word
    Args g(args, nargs, 9);
    const at::Tensor* t = g.tensor(4);
    const int B = size(t, 0), N = size(t, 1), Hq = size(t, 2), D = size(t, 3);
    auto* q = g.ptr();
    const at::Tensor* tk = g.tensor(4);
    const int Hkv = size(tk, 1), S_max = size(tk, 2);
    auto* k = g.ptr(); auto* v = g.ptr(); auto* kv_len = g.ptr<int32_t>(); auto* mask = g.ptr<uint64_t>();
    const float scale = g.real();
    auto* out = g.ptr(); auto* lse = g.ptr<float>(); auto* status = g.ptr<int>();
    return finish(g, [&](void* st) { return vispec_tree_verify_attn_static(q, k, v, kv_len, mask, B, N, Hq, Hkv, D, S_max, scale, out, lse, status, st); });
}

NATIVE(rope_table_build) {  // handle, positions, theta, table
    Args g(args, nargs, 4);
    vispec_ctx* c = g.ctx();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* pos = g.ptr<int32_t>();
    const float theta = g.real();
    auto* table = g.ptr();
    return finish(g, [&](void* st) { return vispec_rope_table_build(c, pos, B, N, theta, table, st); });
}

NATIVE(rope_tree_rows) {  // handle, layer, q, k_new, v_new, positions, kv_len, theta
    Args g(args, nargs, 8);
    vispec_ctx* c = g.ctx();
    const int layer = g.num();
    auto* q = g.ptr(); auto* k = g.ptr(); auto* v = g.ptr();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* pos = g.ptr<int32_t>(); auto* kv_len = g.ptr<int32_t>();
    const float theta = g.real();
    return finish(g, [&](void* st) { return vispec_rope_tree_rows(c, layer, q, k, v, pos, kv_len, B, N, theta, st); });
}

NATIVE(rope_tree_rows_paged) {  // handle, layer, q, k_new, v_new, positions, kv_len, block_table, theta
    Args g(args, nargs, 9);
    vispec_ctx* c = g.ctx();
    const int layer = g.num();
    auto* q = g.ptr(); auto* k = g.ptr(); auto* v = g.ptr();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* pos = g.ptr<int32_t>(); auto* kv_len = g.ptr<int32_t>();
    const int stride = size(g.tensor(2), 1);
    auto* table = g.ptr<int32_t>();
    const float theta = g.real();
    return finish(g, [&](void* st) { return vispec_rope_tree_rows_paged(c, layer, q, k, v, pos, kv_len, table, stride, B, N, theta, st); });
}

NATIVE(accept) {  // handle, draft_ids, target_ids, parents, path, accept_len, bonus
    Args g(args, nargs, 7);
    vispec_ctx* c = g.ctx();
    auto* draft = g.ptr<int32_t>(); auto* target = g.ptr<int32_t>();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* parents = g.ptr<int32_t>(); auto* path = g.ptr<int32_t>(); auto* alen = g.ptr<int32_t>(); auto* bonus = g.ptr<int32_t>();
    return finish(g, [&](void* st) { return vispec_accept(c, draft, target, parents, B, N, path, alen, bonus, st); });
}

NATIVE(accept_commit) {  // handle, layer_begin, layer_end, draft_ids, target_ids, parents, kv_len, path, accept_len, bonus, kv_len_out
    Args g(args, nargs, 11);
    vispec_ctx* c = g.ctx();
    const int lb = g.num(), le = g.num();
    auto* draft = g.ptr<int32_t>(); auto* target = g.ptr<int32_t>();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* parents = g.ptr<int32_t>(); auto* kv_len = g.ptr<int32_t>(); auto* path = g.ptr<int32_t>();
    auto* alen = g.ptr<int32_t>(); auto* bonus = g.ptr<int32_t>(); auto* out = g.ptr<int32_t>();
    return finish(g, [&](void* st) { return vispec_accept_commit(c, lb, le, draft, target, parents, kv_len, B, N, path, alen, bonus, out, st); });
}

NATIVE(accept_commit_paged) {  // ... kv_len, block_table, path, accept_len, bonus, kv_len_out
    Args g(args, nargs, 12);
    vispec_ctx* c = g.ctx();
    const int lb = g.num(), le = g.num();
    auto* draft = g.ptr<int32_t>(); auto* target = g.ptr<int32_t>();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* parents = g.ptr<int32_t>(); auto* kv_len = g.ptr<int32_t>();
    const int stride = size(g.tensor(2), 1);
    auto* table = g.ptr<int32_t>(); auto* path = g.ptr<int32_t>();
    auto* alen = g.ptr<int32_t>(); auto* bonus = g.ptr<int32_t>(); auto* out = g.ptr<int32_t>();
    return finish(g, [&](void* st) { return vispec_accept_commit_paged(c, lb, le, draft, target, parents, kv_len, table, stride, B, N, path, alen, bonus, out, st); });
}

NATIVE(kv_compact) {  // handle, layer_begin, layer_end, path, accept_len, kv_len, kv_len_out
    Args g(args, nargs, 7);
    vispec_ctx* c = g.ctx();
    const int lb = g.num(), le = g.num();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* path = g.ptr<int32_t>(); auto* alen = g.ptr<int32_t>(); auto* kv_len = g.ptr<int32_t>(); auto* out = g.ptr<int32_t>();
    return finish(g, [&](void* st) { return vispec_kv_compact(c, lb, le, path, alen, kv_len, out, B, N, st); });
}

NATIVE(kv_compact_paged) {  // handle, layer_begin, layer_end, path, accept_len, kv_len, block_table, kv_len_out
    Args g(args, nargs, 8);
    vispec_ctx* c = g.ctx();
    const int lb = g.num(), le = g.num();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), N = size(t, 1);
    auto* path = g.ptr<int32_t>(); auto* alen = g.ptr<int32_t>(); auto* kv_len = g.ptr<int32_t>();
    const int stride = size(g.tensor(2), 1);
    auto* table = g.ptr<int32_t>(); auto* out = g.ptr<int32_t>();
    return finish(g, [&](void* st) { return vispec_kv_compact_paged(c, lb, le, path, alen, kv_len, table, stride, out, B, N, st); });
}

NATIVE(accept_sampled) {  // handle, draft_ids, parents, p_target, p_draft, u_accept, u_bonus, path, accept_len, bonus
    Args g(args, nargs, 10);
    vispec_ctx* c = g.ctx();
    auto* draft = g.ptr<int32_t>(); auto* parents = g.ptr<int32_t>();
    const at::Tensor* t = g.tensor(3);
    const int B = size(t, 0), N = size(t, 1), V = size(t, 2);
    auto* p = g.ptr<float>(); auto* ph = g.ptr<float>(); auto* ua = g.ptr<float>(); auto* ub = g.ptr<float>();
    auto* path = g.ptr<int32_t>(); auto* alen = g.ptr<int32_t>(); auto* bonus = g.ptr<int32_t>();
    return finish(g, [&](void* st) { return vispec_accept_sampled(c, draft, parents, p, ph, ua, ub, B, N, V, path, alen, bonus, st); });
}

NATIVE(tree_rerank) {  // handle, cand_parent, cand_token, cand_score, K, parents, draft_ids, selected
    Args g(args, nargs, 8);
    vispec_ctx* c = g.ctx();
    const at::Tensor* t = g.tensor(2);
    const int B = size(t, 0), M = size(t, 1);
    auto* cp = g.ptr<int32_t>(); auto* ct = g.ptr<int32_t>(); auto* cs = g.ptr<float>();
    const int K = g.num();
    auto* parents = g.ptr<int32_t>(); auto* ids = g.ptr<int32_t>(); auto* sel = g.ptr<int32_t>();
    return finish(g, [&](void* st) { return vispec_tree_rerank(c, cp, ct, cs, B, M, K, parents, ids, sel, st); });
}

#define ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<name>)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    ENTRY(tree_mask_build), ENTRY(tree_verify_attn), ENTRY(tree_verify_attn_rope), ENTRY(tree_verify_attn_paged),
    ENTRY(tree_verify_attn_static), ENTRY(rope_table_build), ENTRY(rope_tree_rows), ENTRY(rope_tree_rows_paged),
    ENTRY(accept), ENTRY(accept_commit), ENTRY(accept_commit_paged), ENTRY(kv_compact), ENTRY(kv_compact_paged),
    ENTRY(accept_sampled), ENTRY(tree_rerank), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", "Hot calls of libvispec without ctypes", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&kModule); }
