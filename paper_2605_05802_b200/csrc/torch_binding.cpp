// Native half of binding.py: takes the tensors of a call apart and calls the C ABI.
//
// A gate call on a handful of groups lasts a few microseconds on the device; marshalled in
// Python (attribute look-ups, dtype comparisons and numel() per tensor, ctypes conversions)
// it cost 7-10 us of host time and the GPU waited for it.  Here a call is a few dozen plain
// loads.  The checks are those the C side cannot make: a tensor must live where the call
// dereferences it, have the declared element type, be contiguous and hold at least the
// elements the call reads or writes.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <string>

#include "sr_gate.h"
#include "sr_probe.h"

namespace {

struct Raised {};                        // a Python exception has been set

[[noreturn]] void raise(PyObject* type, const std::string& text) {
    PyErr_SetString(type, text.c_str());
    throw Raised();
}

const char* dtype_name(c10::ScalarType t) {
    switch (t) {
        case c10::ScalarType::Int: return "torch.int32";
        case c10::ScalarType::Long: return "torch.int64";
        case c10::ScalarType::Byte: return "torch.uint8";
        case c10::ScalarType::Float: return "torch.float32";
        case c10::ScalarType::Double: return "torch.float64";
        default: return c10::toString(t);
    }
}

constexpr int64_t kAnySize = -1;
constexpr c10::ScalarType kAnyType = c10::ScalarType::Undefined;
PyObject* g_cuda_stream = nullptr;       // interned "cuda_stream"

// The positional arguments of one call, read one after the other.
struct Args {
    PyObject* const* at;

    const at::Tensor* tensor(const char* name) {
        PyObject* o = *at++;
        if (o == Py_None) return nullptr;
        if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string(name) + " must be a tensor or None");
        return &THPVariable_Unpack(o);
    }
    static void* address(const at::Tensor* t, c10::ScalarType type, int64_t need, bool host, const char* name) {
        if (t == nullptr) return nullptr;
        if (type != kAnyType && t->scalar_type() != type)
            raise(PyExc_TypeError, std::string(name) + ": expected " + dtype_name(type) + ", got " + dtype_name(t->scalar_type()));
        if (!t->is_contiguous()) raise(PyExc_ValueError, std::string(name) + " must be contiguous");
        if (t->is_cuda() == host)
            raise(PyExc_ValueError, std::string(name) + " must be a " + (host ? "host" : "CUDA") + " tensor");
        if (need != kAnySize && t->numel() < need)
            raise(PyExc_ValueError, std::string(name) + " holds " + std::to_string(t->numel()) +
                                        " elements, the call writes or reads " + std::to_string(need));
        return t->data_ptr();
    }
    template <typename T>
    T* buffer(c10::ScalarType type, int64_t need, const char* name, bool host = false) {
        return static_cast<T*>(address(tensor(name), type, need, host, name));
    }
    // workspace / state / arena: any element type, its size in bytes
    void* scratch(const char* name, size_t& bytes) {
        const at::Tensor* t = tensor(name);
        bytes = t ? (size_t)t->numel() * t->element_size() : 0;
        return address(t, kAnyType, kAnySize, false, name);
    }
    int32_t integer() {                  // modulo 2^32, as a C caller's conversion
        PyObject* o = PyNumber_Index(*at++);
        if (o == nullptr) throw Raised();
        const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
        Py_DECREF(o);
        if (v == (unsigned long long)-1 && PyErr_Occurred()) throw Raised();
        return (int32_t)v;
    }
    double real() {                      // whatever float() takes
        PyObject* o = *at++;
        if (PyFloat_Check(o)) return PyFloat_AS_DOUBLE(o);
        PyObject* f = PyNumber_Float(o);
        if (f == nullptr) throw Raised();
        const double v = PyFloat_AS_DOUBLE(f);
        Py_DECREF(f);
        return v;
    }
    static void* handle(PyObject* stream) {
        PyObject* v = PyObject_GetAttr(stream, g_cuda_stream);
        if (v == nullptr) throw Raised();
        void* h = PyLong_AsVoidPtr(v);
        Py_DECREF(v);
        if (h == nullptr && PyErr_Occurred()) throw Raised();
        return h;
    }
    void* stream() {                     // None: the current stream of the current device
        PyObject* o = *at++;
        return o == Py_None ? c10::cuda::getCurrentCUDAStream().stream() : handle(o);
    }
    void* copy_stream() {
        PyObject* o = *at++;
        return o == Py_None ? nullptr : handle(o);
    }
};

struct Shape3 { int32_t G, N, stride; int64_t P; };
Shape3 group_shape(const at::Tensor* t, const char* name) {
    if (t == nullptr || t->dim() != 3) raise(PyExc_ValueError, std::string(name) + " must be [groups, N, stride]");
    Shape3 s{(int32_t)t->size(0), (int32_t)t->size(1), (int32_t)t->size(2), 0};
    s.P = (int64_t)s.N * (s.N - 1) / 2;
    return s;
}
void two_dims(const at::Tensor* t, const char* name, int32_t& G, int32_t& N) {
    if (t == nullptr || t->dim() != 2) raise(PyExc_ValueError, std::string(name) + " must be [groups, N]");
    G = (int32_t)t->size(0);
    N = (int32_t)t->size(1);
}

// Runs `body(args)` -> return code, without the GIL around the library call itself.
template <typename Body>
PyObject* guarded(PyObject* const* argv, Py_ssize_t argc, Py_ssize_t want, Body body) {
    if (argc != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, argc);
        return nullptr;
    }
    try {
        Args a{argv};
        const int rc = body(a);
        if (rc == SR_OK) Py_RETURN_NONE;
        return PyLong_FromLong(rc);
    } catch (const Raised&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <typename Call>
int unlocked(Call call) {
    PyThreadState* st = PyEval_SaveThread();
    const int rc = call();
    PyEval_RestoreThread(st);
    return rc;
}

constexpr auto kI32 = c10::ScalarType::Int;
constexpr auto kI64 = c10::ScalarType::Long;
constexpr auto kU8 = c10::ScalarType::Byte;
constexpr auto kF32 = c10::ScalarType::Float;
constexpr auto kF64 = c10::ScalarType::Double;

// What every gate call has in common: inputs, threshold and the outputs of a batch.
struct GateCall {
    Shape3 d;
    int32_t *seqs, *lens, K, norm, *pair_dist, *pair_sum, *status;
    double threshold, *mean;
    uint8_t* stop;

    void inputs(Args& a, bool host) {
        const at::Tensor* s = a.tensor("seqs");
        d = group_shape(s, "seqs");
        seqs = static_cast<int32_t*>(Args::address(s, kI32, kAnySize, host, "seqs"));
        lens = a.buffer<int32_t>(kI32, (int64_t)d.G * d.N, "lens", host);
    }
    void setting(Args& a) {
        K = a.integer();
        threshold = a.real();
        norm = a.integer();
    }
    void outputs(Args& a, bool host) {
        pair_dist = a.buffer<int32_t>(kI32, d.G * d.P, "pair_dist", host);
        pair_sum = a.buffer<int32_t>(kI32, d.G, "pair_sum", host);
        mean = a.buffer<double>(kF64, d.G, "mean", host);
        stop = a.buffer<uint8_t>(kU8, d.G, "stop", host);
    }
};

PyObject* py_gate(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 12, [](Args& a) {
        GateCall c;
        c.inputs(a, false); c.setting(a); c.outputs(a, false);
        c.status = a.buffer<int32_t>(kI32, 1, "status");
        size_t bytes;
        void* ws = a.scratch("workspace", bytes);
        void* s = a.stream();
        return unlocked([&] { return sr_gate(c.seqs, c.lens, c.d.G, c.d.N, c.d.stride, c.K, c.threshold, c.norm, c.pair_dist, c.pair_sum, c.mean, c.stop, c.status, ws, bytes, s); });
    });
}

PyObject* py_gate_noalloc(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 11, [](Args& a) {
        GateCall c;
        c.inputs(a, false); c.setting(a); c.outputs(a, false);
        c.status = a.buffer<int32_t>(kI32, 1, "status");
        void* s = a.stream();
        return unlocked([&] { return sr_gate_noalloc(c.seqs, c.lens, c.d.G, c.d.N, c.d.stride, c.K, c.threshold, c.norm, c.pair_dist, c.pair_sum, c.mean, c.stop, c.status, s); });
    });
}

PyObject* py_gate_decide(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 13, [](Args& a) {
        GateCall c;
        c.inputs(a, false); c.setting(a); c.outputs(a, false);
        uint8_t* exact = a.buffer<uint8_t>(kU8, c.d.G, "exact");
        c.status = a.buffer<int32_t>(kI32, 1, "status");
        size_t bytes;
        void* ws = a.scratch("workspace", bytes);
        void* s = a.stream();
        return unlocked([&] { return sr_gate_decide(c.seqs, c.lens, c.d.G, c.d.N, c.d.stride, c.K, c.threshold, c.norm, c.pair_dist, c.pair_sum, c.mean, c.stop, exact, c.status, ws, bytes, s); });
    });
}

PyObject* py_gate_host(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 13, [](Args& a) {
        GateCall c;
        c.inputs(a, true); c.setting(a); c.outputs(a, true);
        c.status = a.buffer<int32_t>(kI32, 1, "status", true);
        size_t bytes;
        void* arena = a.scratch("arena", bytes);
        void* s = a.stream();
        void* cs = a.copy_stream();
        return unlocked([&] { return sr_gate_host(c.seqs, c.lens, c.d.G, c.d.N, c.d.stride, c.K, c.threshold, c.norm, c.pair_dist, c.pair_sum, c.mean, c.stop, c.status, arena, bytes, s, cs); });
    });
}

PyObject* py_gate_host_packed(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 15, [](Args& a) {
        GateCall c;
        int32_t* symbols = a.buffer<int32_t>(kI32, kAnySize, "symbols", true);
        const at::Tensor* rs = a.tensor("row_start");
        c.d.N = a.integer();
        c.d.stride = a.integer();
        const int64_t rows = rs ? rs->numel() - 1 : -1;
        if (rows < 0 || c.d.N == 0 || rows % c.d.N) raise(PyExc_ValueError, "row_start needs n_groups * N + 1 entries");
        c.d.G = (int32_t)(rows / c.d.N);
        c.d.P = (int64_t)c.d.N * (c.d.N - 1) / 2;
        int64_t* start = static_cast<int64_t*>(Args::address(rs, kI64, kAnySize, true, "row_start"));
        c.setting(a); c.outputs(a, true);
        c.status = a.buffer<int32_t>(kI32, 1, "status", true);
        size_t bytes;
        void* arena = a.scratch("arena", bytes);
        void* s = a.stream();
        void* cs = a.copy_stream();
        return unlocked([&] { return sr_gate_host_packed(symbols, start, c.d.G, c.d.N, c.d.stride, c.K, c.threshold, c.norm, c.pair_dist, c.pair_sum, c.mean, c.stop, c.status, arena, bytes, s, cs); });
    });
}

PyObject* py_incr_init(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 5, [](Args& a) {
        size_t bytes;
        void* state = a.scratch("state", bytes);
        const int32_t G = a.integer(), N = a.integer(), steps = a.integer();
        void* s = a.stream();
        return unlocked([&] { return sr_incr_init(state, bytes, G, N, steps, s); });
    });
}

PyObject* py_gate_step_incremental(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 10, [](Args& a) {
        GateCall c;
        size_t bytes;
        void* state = a.scratch("state", bytes);
        const at::Tensor* na = a.tensor("new_actions");
        two_dims(na, "new_actions", c.d.G, c.d.N);
        c.d.P = (int64_t)c.d.N * (c.d.N - 1) / 2;
        int32_t* actions = static_cast<int32_t*>(Args::address(na, kI32, kAnySize, false, "new_actions"));
        c.threshold = a.real();
        c.norm = a.integer();
        c.outputs(a, false);
        c.status = a.buffer<int32_t>(kI32, 1, "status");
        void* s = a.stream();
        return unlocked([&] { return sr_gate_step_incremental(state, bytes, actions, c.d.G, c.d.N, c.threshold, c.norm, c.pair_dist, c.pair_sum, c.mean, c.stop, c.status, s); });
    });
}

PyObject* py_gate_or_rule(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 10, [](Args& a) {
        const at::Tensor *mt = a.tensor("mean"), *lt = a.tensor("lens"), *dt = a.tensor("done");
        const int32_t N = a.integer(), K = a.integer();
        const double threshold = a.real(), tau_high = a.real();
        if (mt == nullptr || mt->dim() < 1) raise(PyExc_ValueError, "mean must be [groups]");
        const int32_t G = (int32_t)mt->size(0);
        const double* mean = static_cast<double*>(Args::address(mt, kF64, kAnySize, false, "mean"));
        const int32_t* lens = static_cast<int32_t*>(Args::address(lt, kI32, (int64_t)G * N, false, "lens"));
        const uint8_t* done = static_cast<uint8_t*>(Args::address(dt, kU8, (int64_t)G * N, false, "done"));
        double* tau = a.buffer<double>(kF64, G, "tau");
        uint8_t* stop = a.buffer<uint8_t>(kU8, G, "stop");
        void* s = a.stream();
        return unlocked([&] { return sr_gate_or_rule(mean, lens, done, G, N, K, threshold, tau_high, tau, stop, s); });
    });
}

PyObject* py_group_signals(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 8, [](Args& a) {
        GateCall c;
        c.inputs(a, false);
        const int32_t K = a.integer();
        double* upr = a.buffer<double>(kF64, c.d.G, "unique_prefix_ratio");
        double* uar = a.buffer<double>(kF64, c.d.G, "unique_action_ratio");
        double* ent = a.buffer<double>(kF64, c.d.G, "action_entropy");
        double* jac = a.buffer<double>(kF64, c.d.G, "bigram_jaccard_mean");
        void* s = a.stream();
        return unlocked([&] { return sr_group_signals(c.seqs, c.lens, c.d.G, c.d.N, c.d.stride, K, upr, uar, ent, jac, s); });
    });
}

PyObject* py_batch_stats(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 5, [](Args& a) {
        const at::Tensor* t = a.tensor("adv");
        int32_t G, N;
        two_dims(t, "adv", G, N);
        const float* adv = static_cast<float*>(Args::address(t, kF32, kAnySize, false, "adv"));
        const uint8_t* stop = a.buffer<uint8_t>(kU8, G, "stop");
        int64_t* counts = a.buffer<int64_t>(kI64, 3, "counts");
        double* sumsq = a.buffer<double>(kF64, 2, "sumsq");
        void* s = a.stream();
        return unlocked([&] { return sr_batch_stats(adv, stop, G, N, counts, sumsq, s); });
    });
}

PyObject* py_kept_groups(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 7, [](Args& a) {
        const at::Tensor *st = a.tensor("stop"), *zt = a.tensor("zero_var"), *it = a.tensor("index"), *ct = a.tensor("count");
        size_t bytes;
        void* ws = a.scratch("workspace", bytes);
        PyObject* g = *a.at++;
        int32_t G;
        if (g == Py_None) {
            const at::Tensor* from = st ? st : (zt ? zt : it);
            if (from == nullptr || from->dim() < 1) raise(PyExc_ValueError, "n_groups is not given and no tensor tells it");
            G = (int32_t)from->size(0);
        } else {
            Args one{&g};
            G = one.integer();
        }
        const uint8_t* stop = static_cast<uint8_t*>(Args::address(st, kU8, G, false, "stop"));
        const uint8_t* zero_var = static_cast<uint8_t*>(Args::address(zt, kU8, G, false, "zero_var"));
        int32_t* index = static_cast<int32_t*>(Args::address(it, kI32, G, false, "index"));
        int32_t* count = static_cast<int32_t*>(Args::address(ct, kI32, 1, false, "count"));
        void* s = a.stream();
        return unlocked([&] { return sr_kept_groups(stop, zero_var, G, index, count, ws, bytes, s); });
    });
}

PyObject* py_grpo_advantage(PyObject*, PyObject* const* argv, Py_ssize_t argc) {
    return guarded(argv, argc, 6, [](Args& a) {
        const at::Tensor* t = a.tensor("rewards");
        int32_t G, N;
        two_dims(t, "rewards", G, N);
        const float* rewards = static_cast<float*>(Args::address(t, kF32, kAnySize, false, "rewards"));
        const uint8_t* drop = a.buffer<uint8_t>(kU8, G, "drop_mask");
        const float eps = (float)a.real();
        float* adv = a.buffer<float>(kF32, (int64_t)G * N, "adv");
        uint8_t* zero_var = a.buffer<uint8_t>(kU8, G, "zero_var");
        void* s = a.stream();
        return unlocked([&] { return sr_grpo_advantage(rewards, drop, G, N, eps, adv, zero_var, s); });
    });
}

#define SR_METHOD(name) {"sr_" #name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    SR_METHOD(gate), SR_METHOD(gate_noalloc), SR_METHOD(gate_decide), SR_METHOD(gate_host),
    SR_METHOD(gate_host_packed), SR_METHOD(incr_init), SR_METHOD(gate_step_incremental),
    SR_METHOD(gate_or_rule), SR_METHOD(group_signals), SR_METHOD(batch_stats),
    SR_METHOD(kept_groups), SR_METHOD(grpo_advantage), {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (g_cuda_stream == nullptr) return nullptr;
    return PyModule_Create(&g_module);
}
