// Native marshalling for the calls a program makes eagerly, once per layer or step: the attention, acceptance, compaction and
// LM-head entry points.  Checks and pointers are the same as in s4c.py's ctypes calls; what differs is the price of a call -- a
// dozen attribute look-ups, conversions and allocations through the interpreter took 12 us of host time around a kernel of
// 8 us.  Everything else stays with ctypes.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "s4c.h"

namespace {

struct BadArgument {};  // a Python error is set

constexpr at::ScalarType kAny = at::ScalarType::Undefined;

const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
        throw BadArgument();
    }
    return THPVariable_Unpack(o);
}
void* ptr(const at::Tensor& t, at::ScalarType dtype, const char* name) {
    if (!t.is_cuda()) {
        PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor (the library has no CPU path)", name);
        throw BadArgument();
    }
    if (!t.is_contiguous()) {
        PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
        throw BadArgument();
    }
    if (dtype != kAny && t.scalar_type() != dtype) {
        PyErr_Format(PyExc_TypeError, "%s must be %s, got %s", name, c10::toString(dtype), c10::toString(t.scalar_type()));
        throw BadArgument();
    }
    return t.data_ptr();
}
void* ptr(PyObject* o, at::ScalarType dtype, const char* name) { return o == Py_None ? nullptr : ptr(tensor(o, name), dtype, name); }
template <typename T = int32_t>
T* i32(PyObject* o, const char* name) {
    return static_cast<T*>(ptr(o, at::kInt, name));
}
float* f32(PyObject* o, const char* name) { return static_cast<float*>(ptr(o, at::kFloat, name)); }

long integer(PyObject* o) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw BadArgument();
    return v;
}
double real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw BadArgument();
    return v;
}
void* stream_of(PyObject* o) {  // None: the current stream; else an object with `cuda_stream`
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw BadArgument();
    void* s = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!s && PyErr_Occurred()) throw BadArgument();
    return s;
}
s4c_dtype dtype_of(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return S4C_F32;
    if (t.scalar_type() == at::kBFloat16) return S4C_BF16;
    PyErr_Format(PyExc_TypeError, "unsupported dtype %s: the library takes float32 or bfloat16", c10::toString(t.scalar_type()));
    throw BadArgument();
}
struct Scratch {
    void* p;
    size_t bytes;
    explicit Scratch(PyObject* o) : p(ptr(o, kAny, "workspace")), bytes(o == Py_None ? 0 : (size_t)THPVariable_Unpack(o).nbytes()) {}
};
void count(Py_ssize_t n, Py_ssize_t want) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n);
        throw BadArgument();
    }
}
// (return code, result)
PyObject* answer(int rc, PyObject* result) {
    PyObject* t = PyTuple_New(2);
    PyTuple_SET_ITEM(t, 0, PyLong_FromLong(rc));
    PyTuple_SET_ITEM(t, 1, result);
    return t;
}
template <typename F>
PyObject* guarded(F f) {
    try {
        return f();
    } catch (const BadArgument&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// attention(q, k_cache, v_cache, cache_len, parent, n_nodes, out, scale, status, workspace, stream, max_cache_len, rows, scratch_fn)
// -> (rc, out); scratch_fn(nbytes, device) gives a workspace where one is needed and none was passed
PyObject* attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        count(n, 14);
        const at::Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k_cache"), &v = tensor(a[2], "v_cache");
        if (q.dim() != 4 || k.dim() != 4 || v.dim() != 4 || k.size(0) != q.size(0) || k.size(3) != q.size(3) || v.sizes() != k.sizes()) {
            PyErr_SetString(PyExc_ValueError, "k_cache / v_cache must be [B,Hkv,C,d]");
            throw BadArgument();
        }
        if (k.scalar_type() != q.scalar_type() || v.scalar_type() != q.scalar_type()) {
            PyErr_SetString(PyExc_TypeError, "q, k_cache and v_cache must share one dtype");
            throw BadArgument();
        }
        const int B = (int)q.size(0), Hq = (int)q.size(1), T = (int)q.size(2), d = (int)q.size(3), Hkv = (int)k.size(1), C = (int)k.size(2);
        const bool rows = PyObject_IsTrue(a[12]) == 1;
        const s4c_dtype dt = dtype_of(q);
        PyObject* out = a[6];
        if (out == Py_None)
            out = THPVariable_Wrap(rows ? at::empty({B, T, Hq, d}, q.options()) : at::empty_like(q));
        else
            Py_INCREF(out);
        PyObject* ws = nullptr;
        try {
            const size_t need = a[9] == Py_None ? s4c_tree_attention_workspace_bytes(B, T, Hq, Hkv, d, C, dt) : 0;
            if (need) {
                ws = PyObject_CallFunction(a[13], "nO", (Py_ssize_t)need, a[0]);
                if (!ws) throw BadArgument();
            }
            const Scratch scratch(ws ? ws : a[9]);
            const int rc = (rows ? s4c_tree_attention_rows : s4c_tree_attention)(
                ptr(q, kAny, "q"), ptr(k, kAny, "k_cache"), ptr(v, kAny, "v_cache"), i32(a[3], "cache_len"), i32(a[4], "parent"),
                i32(a[5], "n_nodes"), ptr(out, q.scalar_type(), "out"), B, T, Hq, Hkv, d, C, (int)integer(a[11]), dt, (float)real(a[7]),
                i32(a[8], "status"), scratch.p, scratch.bytes, stream_of(a[10]));
            Py_XDECREF(ws);
            return answer(rc, out);
        } catch (...) {
            Py_XDECREF(ws);
            Py_DECREF(out);
            throw;
        }
    });
}

// accept(target_logits, draft_probs, tokens, parent, temperature, uniforms, n_nodes, max_depth, accept_len, path, next_token, near_tie,
//        status, workspace, stream) -> rc
PyObject* accept(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        count(n, 15);
        const at::Tensor& logits = tensor(a[0], "target_logits");
        const Scratch scratch(a[13]);
        return PyLong_FromLong(s4c_tree_accept(
            static_cast<const float*>(ptr(logits, at::kFloat, "target_logits")), f32(a[1], "draft_probs"), i32(a[2], "tokens"), i32(a[3], "parent"),
            i32(a[6], "n_nodes"), (float)real(a[4]), f32(a[5], "uniforms"), (int)logits.size(0), (int)logits.size(1), (int)logits.size(2),
            (int)integer(a[7]), i32(a[8], "accept_len"), i32(a[9], "path"), i32(a[10], "next_token"),
            static_cast<uint8_t*>(ptr(a[11], at::kByte, "near_tie")), i32(a[12], "status"), scratch.p, scratch.bytes, stream_of(a[14])));
    });
}

// compact(k_ptrs, v_ptrs, n_layers, B, Hkv, C, d, is_f32, cache_len, path, accept_len, T, feat_in, feat_out, hid, status, stream) -> rc
PyObject* compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        count(n, 17);
        const int layers = (int)integer(a[2]);
        const at::Tensor& path = tensor(a[9], "path");
        return PyLong_FromLong(s4c_kv_compact(
            layers ? static_cast<void* const*>(ptr(a[0], at::kLong, "k_ptrs")) : nullptr,
            layers ? static_cast<void* const*>(ptr(a[1], at::kLong, "v_ptrs")) : nullptr, layers, i32(a[8], "cache_len"),
            static_cast<const int32_t*>(ptr(path, at::kInt, "path")), i32(a[10], "accept_len"), (int)path.size(1) - 1, ptr(a[12], kAny, "feat_in"),
            ptr(a[13], kAny, "feat_out"), (int)integer(a[3]), (int)integer(a[11]), (int)integer(a[4]), (int)integer(a[6]), (int)integer(a[5]),
            (int)integer(a[14]), integer(a[7]) ? S4C_F32 : S4C_BF16, i32(a[15], "status"), stream_of(a[16])));
    });
}

// lm_head(hidden, weight, k, token, logit, status, workspace, stream, scratch_fn) -> (rc, (token, logit, status)); what is None is made:
// token and logit are [R] for k = 0 (the greedy call), else [R, k]
PyObject* lm_head(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        count(n, 9);
        const at::Tensor &h = tensor(a[0], "hidden"), &w = tensor(a[1], "weight");
        if (h.dim() != 2 || w.dim() != 2) {
            PyErr_SetString(PyExc_ValueError, "hidden must be [R,H] and weight [V,H]");
            throw BadArgument();
        }
        const int R = (int)h.size(0), H = (int)h.size(1), V = (int)w.size(0), k = (int)integer(a[2]);
        PyObject* made[3] = {};
        PyObject* ws = nullptr;
        try {
            for (int i = 0; i < 3; ++i) {
                if (a[3 + i] != Py_None) {
                    Py_INCREF(made[i] = a[3 + i]);
                    continue;
                }
                const auto opt = h.options().dtype(i == 1 ? at::kFloat : at::kInt);
                made[i] = THPVariable_Wrap(i == 2 ? at::empty({1}, opt) : k ? at::empty({R, k}, opt) : at::empty({R}, opt));
            }
            if (a[6] == Py_None) {
                ws = PyObject_CallFunction(a[8], "nO", (Py_ssize_t)s4c_lm_head_topk_workspace_bytes(R, V, H, k ? k : 1), a[0]);
                if (!ws) throw BadArgument();
            }
            const Scratch scratch(ws ? ws : a[6]);
            const int rc = s4c_lm_head_topk(ptr(h, at::kBFloat16, "hidden"), ptr(w, at::kBFloat16, "weight"), R, V, H, k ? k : 1, i32(made[0], "token"),
                                            f32(made[1], k ? "logit" : "max_logit"), i32(made[2], "status"), scratch.p, scratch.bytes, stream_of(a[7]));
            Py_XDECREF(ws);
            PyObject* t = PyTuple_New(3);
            for (int i = 0; i < 3; ++i) PyTuple_SET_ITEM(t, i, made[i]);
            return answer(rc, t);
        } catch (...) {
            Py_XDECREF(ws);
            for (PyObject* o : made) Py_XDECREF(o);
            throw;
        }
    });
}

// accept_tokens(target_token, tokens, parent, V, n_nodes, max_depth, accept_len, path, next_token, status, stream)
// -> (rc, (accept_len, path, next_token, status)); outputs that are None are made
PyObject* accept_tokens(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        count(n, 11);
        const at::Tensor& t = tensor(a[0], "target_token");
        if (t.dim() != 2) {
            PyErr_SetString(PyExc_ValueError, "target_token must be [B,T]");
            throw BadArgument();
        }
        const int B = (int)t.size(0), T = (int)t.size(1), max_depth = a[5] == Py_None ? T - 1 : (int)integer(a[5]);
        PyObject* made[4] = {};
        try {
            for (int i = 0; i < 4; ++i) {
                if (a[6 + i] != Py_None)
                    Py_INCREF(made[i] = a[6 + i]);
                else
                    made[i] = THPVariable_Wrap(i == 1 ? at::empty({B, max_depth + 1}, t.options().dtype(at::kInt)) : at::empty({B}, t.options().dtype(at::kInt)));
            }
            const int rc = s4c_tree_accept_tokens(static_cast<const int32_t*>(ptr(t, at::kInt, "target_token")), i32(a[1], "tokens"), i32(a[2], "parent"),
                                                  i32(a[4], "n_nodes"), B, T, (int)integer(a[3]), max_depth, i32(made[0], "accept_len"),
                                                  i32(made[1], "path"), i32(made[2], "next_token"), i32(made[3], "status"), stream_of(a[10]));
            PyObject* r = PyTuple_New(4);
            for (int i = 0; i < 4; ++i) PyTuple_SET_ITEM(r, i, made[i]);
            return answer(rc, r);
        } catch (...) {
            for (PyObject* o : made) Py_XDECREF(o);
            throw;
        }
    });
}

PyMethodDef methods[] = {
    {"attention", (PyCFunction)(void (*)())attention, METH_FASTCALL, nullptr},
    {"accept", (PyCFunction)(void (*)())accept, METH_FASTCALL, nullptr},
    {"compact", (PyCFunction)(void (*)())compact, METH_FASTCALL, nullptr},
    {"lm_head", (PyCFunction)(void (*)())lm_head, METH_FASTCALL, nullptr},
    {"accept_tokens", (PyCFunction)(void (*)())accept_tokens, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_bind", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__bind() { return PyModule_Create(&module_def); }
