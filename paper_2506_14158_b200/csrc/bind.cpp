// Native marshalling for the calls a program makes eagerly, once per layer or step: the attention, acceptance, compaction and
// LM-head entry points.  What is accepted, and what is raised for the rest, is the same as with s4c.py's ctypes calls; what differs
// is the price of a call -- a dozen attribute look-ups, conversions and allocations through the interpreter took 12 us of host time around a kernel of
// 8 us.  Everything else stays with ctypes.
#include <Python.h>

#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
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

int integer(PyObject* o) {  // an int or what stands for one (`__index__`); a float is refused
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw BadArgument();
    return (int)v;
}
int to_integer(PyObject* o) {  // int(o)
    if (PyLong_Check(o)) return integer(o);
    PyObject* i = PyNumber_Long(o);
    if (!i) throw BadArgument();
    const long v = PyLong_AsLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw BadArgument();
    return (int)v;
}
float to_real(PyObject* o) {  // float(o)
    if (PyFloat_Check(o)) return (float)PyFloat_AS_DOUBLE(o);
    PyObject* f = PyNumber_Float(o);
    if (!f) throw BadArgument();
    const double v = PyFloat_AsDouble(f);
    Py_DECREF(f);
    return (float)v;
}
bool truth(PyObject* o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw BadArgument();
    return v == 1;
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
// The interpreter lock is given up around allocations and the library's calls, as torch and ctypes do: a launch that finds the
// stream's queue full waits there for as long as the GPU takes, and the program's other threads go on meanwhile.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};
template <typename F>
auto unlocked(F f) {
    const Unlocked u;
    return f();
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
// Exceptions leave as the Python exceptions that torch's own functions raise for them (out of memory, index, type ...).
template <typename F>
PyObject* guarded(F f) {
    HANDLE_TH_ERRORS
    try {
        return f();
    } catch (const BadArgument&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}
// The arguments are taken one by one in the order of the call (the order in which a compiler evaluates the arguments of a C++ call
// is its own): of several wrong ones the first is named, and no CUDA call is made before all of them have passed.

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
        const bool rows = truth(a[12]);
        const s4c_dtype dt = dtype_of(q);
        PyObject* out = a[6];
        if (out == Py_None)
            out = THPVariable_Wrap(unlocked([&] { return rows ? at::empty({B, T, Hq, d}, q.options()) : at::empty_like(q); }));
        else
            Py_INCREF(out);
        PyObject* ws = nullptr;
        try {
            const size_t need = a[9] == Py_None ? s4c_tree_attention_workspace_bytes(B, T, Hq, Hkv, d, C, dt) : 0;
            if (need) {
                ws = PyObject_CallFunction(a[13], "nO", (Py_ssize_t)need, a[0]);
                if (!ws) throw BadArgument();
            }
            const void *qp = ptr(q, kAny, "q"), *kp = ptr(k, kAny, "k_cache"), *vp = ptr(v, kAny, "v_cache");
            const int32_t *len = i32(a[3], "cache_len"), *parent = i32(a[4], "parent"), *n_nodes = i32(a[5], "n_nodes");
            void* op = ptr(out, q.scalar_type(), "out");
            const int max_len = to_integer(a[11]);
            const float scale = to_real(a[7]);
            int32_t* status = i32(a[8], "status");
            const Scratch scratch(ws ? ws : a[9]);
            void* stream = stream_of(a[10]);
            const int rc = unlocked([&] {
                return (rows ? s4c_tree_attention_rows : s4c_tree_attention)(qp, kp, vp, len, parent, n_nodes, op, B, T, Hq, Hkv, d, C, max_len, dt,
                                                                             scale, status, scratch.p, scratch.bytes, stream);
            });
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
        const at::Tensor& t = tensor(a[0], "target_logits");
        const float *logits = static_cast<const float*>(ptr(t, at::kFloat, "target_logits")), *probs = f32(a[1], "draft_probs");
        const int32_t *tokens = i32(a[2], "tokens"), *parent = i32(a[3], "parent"), *n_nodes = i32(a[6], "n_nodes");
        const float temperature = to_real(a[4]);
        const float* uniforms = f32(a[5], "uniforms");
        const int max_depth = to_integer(a[7]);
        int32_t *accept_len = i32(a[8], "accept_len"), *path = i32(a[9], "path"), *next_token = i32(a[10], "next_token");
        uint8_t* near_tie = static_cast<uint8_t*>(ptr(a[11], at::kByte, "near_tie"));
        int32_t* status = i32(a[12], "status");
        const Scratch scratch(a[13]);
        void* stream = stream_of(a[14]);
        const int B = (int)t.size(0), T = (int)t.size(1), V = (int)t.size(2);
        const int rc = unlocked([&] {
            return s4c_tree_accept(logits, probs, tokens, parent, n_nodes, temperature, uniforms, B, T, V, max_depth, accept_len, path, next_token,
                                   near_tie, status, scratch.p, scratch.bytes, stream);
        });
        return PyLong_FromLong(rc);
    });
}

// compact(k_ptrs, v_ptrs, n_layers, B, Hkv, C, d, is_f32, cache_len, path, accept_len, T, feat_in, feat_out, hid, status, stream) -> rc
PyObject* compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        count(n, 17);
        const at::Tensor& p = tensor(a[9], "path");
        const int max_depth = (int)p.size(1) - 1, layers = to_integer(a[2]);
        void* const* k_ptrs = layers ? static_cast<void* const*>(ptr(a[0], at::kLong, "k_ptrs")) : nullptr;
        void* const* v_ptrs = layers ? static_cast<void* const*>(ptr(a[1], at::kLong, "v_ptrs")) : nullptr;
        int32_t* len = i32(a[8], "cache_len");
        const int32_t *path = static_cast<const int32_t*>(ptr(p, at::kInt, "path")), *accept_len = i32(a[10], "accept_len");
        const void* feat_in = ptr(a[12], kAny, "feat_in");
        void* feat_out = ptr(a[13], kAny, "feat_out");
        const int B = integer(a[3]), T = integer(a[11]), Hkv = integer(a[4]), d = integer(a[6]), C = integer(a[5]), hid = integer(a[14]);
        const s4c_dtype dt = truth(a[7]) ? S4C_F32 : S4C_BF16;
        int32_t* status = i32(a[15], "status");
        void* stream = stream_of(a[16]);
        const int rc = unlocked([&] {
            return s4c_kv_compact(k_ptrs, v_ptrs, layers, len, path, accept_len, max_depth, feat_in, feat_out, B, T, Hkv, d, C, hid, dt, status, stream);
        });
        return PyLong_FromLong(rc);
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
        const int R = (int)h.size(0), H = (int)h.size(1), V = (int)w.size(0), k = integer(a[2]);
        PyObject* made[3] = {};
        PyObject* ws = nullptr;
        try {
            for (int i = 0; i < 3; ++i) {
                if (a[3 + i] != Py_None) {
                    Py_INCREF(made[i] = a[3 + i]);
                    continue;
                }
                const auto opt = h.options().dtype(i == 1 ? at::kFloat : at::kInt);
                made[i] = THPVariable_Wrap(unlocked([&] { return i == 2 ? at::empty({1}, opt) : k ? at::empty({R, k}, opt) : at::empty({R}, opt); }));
            }
            if (a[6] == Py_None) {
                ws = PyObject_CallFunction(a[8], "nO", (Py_ssize_t)s4c_lm_head_topk_workspace_bytes(R, V, H, k ? k : 1), a[0]);
                if (!ws) throw BadArgument();
            }
            const void *hidden = ptr(h, at::kBFloat16, "hidden"), *weight = ptr(w, at::kBFloat16, "weight");
            int32_t* token = i32(made[0], "token");
            float* logit = f32(made[1], k ? "logit" : "max_logit");
            int32_t* status = i32(made[2], "status");
            const Scratch scratch(ws ? ws : a[6]);
            void* stream = stream_of(a[7]);
            const int rc = unlocked(
                [&] { return s4c_lm_head_topk(hidden, weight, R, V, H, k ? k : 1, token, logit, status, scratch.p, scratch.bytes, stream); });
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
        const int B = (int)t.size(0), T = (int)t.size(1), max_depth = a[5] == Py_None ? T - 1 : to_integer(a[5]);
        PyObject* made[4] = {};
        try {
            for (int i = 0; i < 4; ++i) {
                if (a[6 + i] != Py_None)
                    Py_INCREF(made[i] = a[6 + i]);
                else
                    made[i] = THPVariable_Wrap(unlocked([&] {
                        const auto opt = t.options().dtype(at::kInt);
                        return i == 1 ? at::empty({B, max_depth + 1}, opt) : at::empty({B}, opt);
                    }));
            }
            const int32_t* target = static_cast<const int32_t*>(ptr(t, at::kInt, "target_token"));
            const int32_t *tokens = i32(a[1], "tokens"), *parent = i32(a[2], "parent"), *n_nodes = i32(a[4], "n_nodes");
            const int V = to_integer(a[3]);
            int32_t *accept_len = i32(made[0], "accept_len"), *path = i32(made[1], "path"), *next_token = i32(made[2], "next_token");
            int32_t* status = i32(made[3], "status");
            void* stream = stream_of(a[10]);
            const int rc = unlocked([&] {
                return s4c_tree_accept_tokens(target, tokens, parent, n_nodes, B, T, V, max_depth, accept_len, path, next_token, status, stream);
            });
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
