// Argument marshalling of the hot calls: torch tensors to the plain pointers and sizes of the C-ABI
// (include/picospec.h), with the checks a caller relies on (CUDA tensor, dtype, shape, contiguity).
// A call has 10 to 20 tensors; done in Python the checks, the ctypes objects and the foreign call
// cost 8 to 14 us of host time, as much as the kernel launches behind them.  The library itself stays
// free of torch and Python: it is opened here by path.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include <initializer_list>
#include <string>

#include "../../include/picospec.h"

namespace {

struct Refused {
    std::string why;
};

struct Api {
    decltype(&picospec_compress) compress;
    decltype(&picospec_verify) verify;
    decltype(&picospec_verify_range) verify_range;
    decltype(&picospec_residual_sample) residual_sample;
    decltype(&picospec_target_topk) target_topk;
    decltype(&picospec_edge_resample) edge_resample;
    decltype(&picospec_wire_pack) wire_pack;
    decltype(&picospec_wire_unpack) wire_unpack;
    void* handle;
} api;

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) throw Refused{"expected a tensor"};
    return THPVariable_Unpack(o);
}

// data pointer of a contiguous CUDA tensor of the given type (and shape, if given); None is null
void* ptr(PyObject* o, at::ScalarType type, const std::initializer_list<int64_t>* shape) {
    if (o == Py_None) return nullptr;
    const at::Tensor& t = tensor(o);
    if (!t.is_cuda()) throw Refused{"picospec takes CUDA tensors only (there is no CPU path)"};
    if (t.scalar_type() != type)
        throw Refused{std::string("expected dtype ") + c10::toString(type) + ", got " + c10::toString(t.scalar_type())};
    if (shape && !t.sizes().equals(at::IntArrayRef(shape->begin(), shape->size()))) {
        std::string want;
        for (int64_t d : *shape) want += (want.empty() ? "" : ", ") + std::to_string(d);
        std::string got;
        for (int64_t d : t.sizes()) got += (got.empty() ? "" : ", ") + std::to_string(d);
        throw Refused{"expected shape (" + want + "), got (" + got + ")"};
    }
    if (!t.is_contiguous()) throw Refused{"expected a contiguous tensor"};
    return t.data_ptr();
}
int* i32(PyObject* o, std::initializer_list<int64_t> shape) { return (int*)ptr(o, at::kInt, &shape); }
float* f32(PyObject* o, std::initializer_list<int64_t> shape) { return (float*)ptr(o, at::kFloat, &shape); }

// [B, R, V] logits with a contiguous vocabulary and uniformly pitched rows
struct Logits {
    const void* p;
    picospec_dtype dtype;
    int64_t B, R, V, pitch;
    explicit Logits(PyObject* o) {
        const at::Tensor& t = tensor(o);
        if (!t.is_cuda() || t.dim() != 3 || t.stride(2) != 1)
            throw Refused{"logits must be a CUDA tensor [B, R, V] with contiguous vocabulary"};
        B = t.size(0); R = t.size(1); V = t.size(2);
        pitch = R > 1 ? t.stride(1) : (B > 1 ? t.stride(0) : V);
        if ((R > 1 && B > 1 && t.stride(0) != R * pitch) || pitch < V) throw Refused{"rows must be uniformly pitched"};
        if (t.scalar_type() == at::kFloat) dtype = PICOSPEC_F32;
        else if (t.scalar_type() == at::kBFloat16) dtype = PICOSPEC_BF16;
        else throw Refused{"logits must be float32 or bfloat16"};
        p = t.data_ptr();
    }
};

long long integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Refused{""};
    return v;
}
double real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Refused{""};
    return v;
}
picospec_ctx* context(PyObject* o) { return (picospec_ctx*)(uintptr_t)PyLong_AsVoidPtr(o); }
void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }
int64_t last_size(PyObject* o) {
    const at::Tensor& t = tensor(o);
    if (t.dim() < 1) throw Refused{"expected a tensor with at least one dimension"};
    return t.size(-1);
}

// Runs `body(args)` (which returns the library's code) without the interpreter lock around the call
// itself; a refused argument becomes a ValueError.
template <typename F> PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F&& body) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
        return nullptr;
    }
    try {
        return PyLong_FromLong(body());
    } catch (const Refused& r) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, r.why.c_str());
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}
template <typename F> int unlocked(F&& call) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return rc;
}

// context, logits, temperature, top_k, top_p, k_max, u_draft, q_idx, q_prob, q_count, draft_tok
PyObject* py_compress(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 11, [&] {
        picospec_ctx* ctx = context(a[0]);
        const Logits l(a[1]);
        const int64_t B = l.B, G = l.R, K = integer(a[5]);
        const float* T = f32(a[2], {B});
        const int top_k = (int)integer(a[3]);
        const float top_p = (float)real(a[4]);
        int* idx = i32(a[7], {B, G, K});
        float* prob = f32(a[8], {B, G, K});
        int* count = i32(a[9], {B, G});
        const float* u = f32(a[6], {B, G});
        int* tok = i32(a[10], {B, G});
        void* s = stream();
        return unlocked([&] {
            return api.compress(ctx, l.p, l.dtype, (int)B, (int)G, (int)l.V, l.pitch, T, top_k, top_p, (int)K, idx, prob, count,
                                u, tok, s);
        });
    });
}

// context, logits, temperature, draft_tok, q_idx, q_prob, q_count, u_accept, u_resample, accept_len, p_draft,
// resid_mass, borderline_count, token
PyObject* py_verify(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 14, [&] {
        picospec_ctx* ctx = context(a[0]);
        const Logits l(a[1]);
        const int64_t B = l.B, G = l.R - 1, K = last_size(a[4]);
        const float* T = f32(a[2], {B});
        const int* dt = i32(a[3], {B, G});
        const int* idx = i32(a[4], {B, G, K});
        const float* prob = f32(a[5], {B, G, K});
        const int* count = i32(a[6], {B, G});
        const float* ua = f32(a[7], {B, G});
        int* alen = i32(a[9], {B});
        float* pd = f32(a[10], {B, G});
        float* rm = f32(a[11], {B, G});
        int* bc = i32(a[12], {1});
        const float* ur = f32(a[8], {B, 2});
        int* tok = i32(a[13], {B});
        void* s = stream();
        return unlocked([&] {
            return api.verify(ctx, l.p, l.dtype, (int)B, (int)G, (int)l.V, l.pitch, T, dt, idx, prob, count, (int)K, ua, alen, pd,
                              rm, bc, ur, tok, s);
        });
    });
}

// context, logits, temperature, gamma, r0, r1, state_in, draft_tok, q_idx, q_prob, q_count, u_accept, u_resample,
// accept_len, p_draft, resid_mass, borderline_count, token, state
PyObject* py_verify_range(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 19, [&] {
        picospec_ctx* ctx = context(a[0]);
        const Logits l(a[1]);
        const int64_t B = l.B, G = l.R - 1, K = last_size(a[8]);
        const float* T = f32(a[2], {B});
        const int* gamma = i32(a[3], {B});
        const int r0 = (int)integer(a[4]), r1 = (int)integer(a[5]);
        const int* state_in = i32(a[6], {B});
        const int* dt = i32(a[7], {B, G});
        const int* idx = i32(a[8], {B, G, K});
        const float* prob = f32(a[9], {B, G, K});
        const int* count = i32(a[10], {B, G});
        const float* ua = f32(a[11], {B, G});
        int* alen = i32(a[13], {B});
        float* pd = f32(a[14], {B, G});
        float* rm = f32(a[15], {B, G});
        int* bc = i32(a[16], {1});
        const float* ur = f32(a[12], {B, 2});
        int* tok = i32(a[17], {B});
        int* state = i32(a[18], {B});
        void* s = stream();
        return unlocked([&] {
            return api.verify_range(ctx, l.p, l.dtype, (int)B, (int)G, (int)l.V, l.pitch, T, gamma, r0, r1, state_in, dt, idx,
                                    prob, count, (int)K, ua, alen, pd, rm, bc, ur, tok, state, s);
        });
    });
}

// context, logits, temperature, pos, q_idx, q_prob, q_count, u_resample, token, mass
PyObject* py_residual_sample(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&] {
        picospec_ctx* ctx = context(a[0]);
        const Logits l(a[1]);
        const int64_t B = l.B, G = l.R - 1, K = G > 0 ? last_size(a[4]) : 1;
        const float* T = f32(a[2], {B});
        const int* pos = i32(a[3], {B});
        const int* idx = (const int*)ptr(a[4], at::kInt, nullptr);
        const float* prob = (const float*)ptr(a[5], at::kFloat, nullptr);
        const int* count = (const int*)ptr(a[6], at::kInt, nullptr);
        const float* ur = f32(a[7], {B, 2});
        int* tok = i32(a[8], {B});
        float* mass = f32(a[9], {B});
        void* s = stream();
        return unlocked([&] {
            return api.residual_sample(ctx, l.p, l.dtype, (int)B, (int)G, (int)l.V, l.pitch, T, pos, idx, prob, count, (int)K, ur,
                                       tok, mass, s);
        });
    });
}

// context, logits, temperature, pos, k, p_idx, p_prob, p_count
PyObject* py_target_topk(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 8, [&] {
        picospec_ctx* ctx = context(a[0]);
        const Logits l(a[1]);
        const int64_t B = l.B, K = integer(a[4]);
        int* idx = i32(a[5], {B, K});
        float* prob = f32(a[6], {B, K});
        int* count = i32(a[7], {B});
        const float* T = f32(a[2], {B});
        const int* pos = i32(a[3], {B});
        void* s = stream();
        return unlocked([&] {
            return api.target_topk(ctx, l.p, l.dtype, (int)B, (int)l.R, (int)l.V, l.pitch, T, pos, (int)K, idx, prob, count, s);
        });
    });
}

// context, logits, temperature, pos, p_idx, p_prob, p_count, u, token, mass
PyObject* py_edge_resample(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&] {
        picospec_ctx* ctx = context(a[0]);
        const Logits l(a[1]);
        const int64_t B = l.B, K = last_size(a[4]);
        int* tok = i32(a[8], {B});
        float* mass = f32(a[9], {B});
        const float* T = f32(a[2], {B});
        const int* pos = i32(a[3], {B});
        const int* idx = i32(a[4], {B, K});
        const float* prob = f32(a[5], {B, K});
        const int* count = i32(a[6], {B});
        const float* u = f32(a[7], {B});
        void* s = stream();
        return unlocked([&] {
            return api.edge_resample(ctx, l.p, l.dtype, (int)B, (int)l.R, (int)l.V, l.pitch, T, pos, idx, prob, count, (int)K, u,
                                     tok, mass, s);
        });
    });
}

// context, q_idx, q_prob, q_count, rows, K, prob_type, buf, bytes_out
PyObject* py_wire_pack(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 9, [&] {
        picospec_ctx* ctx = context(a[0]);
        const int* idx = (const int*)ptr(a[1], at::kInt, nullptr);
        const float* prob = (const float*)ptr(a[2], at::kFloat, nullptr);
        const int* count = (const int*)ptr(a[3], at::kInt, nullptr);
        const int R = (int)integer(a[4]), K = (int)integer(a[5]), type = (int)integer(a[6]);
        void* buf = ptr(a[7], at::kByte, nullptr);
        const long long capacity = tensor(a[7]).numel();
        const std::initializer_list<int64_t> one = {1};
        long long* bytes = (long long*)ptr(a[8], at::kLong, &one);
        void* s = stream();
        return unlocked([&] { return api.wire_pack(ctx, idx, prob, count, R, K, type, buf, capacity, bytes, s); });
    });
}

// context, buf, nbytes, rows, K, q_idx, q_prob, q_count
PyObject* py_wire_unpack(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 8, [&] {
        picospec_ctx* ctx = context(a[0]);
        const void* buf = ptr(a[1], at::kByte, nullptr);
        const long long nbytes = integer(a[2]);
        const int64_t R = integer(a[3]), K = integer(a[4]);
        int* idx = i32(a[5], {R, K});
        float* prob = f32(a[6], {R, K});
        int* count = i32(a[7], {R});
        void* s = stream();
        return unlocked([&] { return api.wire_unpack(ctx, buf, nbytes, (int)R, (int)K, idx, prob, count, s); });
    });
}

// logits -> (B, R, V), checked: for calls that allocate their outputs from the shape
PyObject* py_logits(PyObject*, PyObject* const* a, Py_ssize_t n) {
    int64_t size[3] = {0, 0, 0};
    PyObject* ok = guarded(n, 1, [&] {
        const Logits l(a[0]);
        size[0] = l.B; size[1] = l.R; size[2] = l.V;
        return 0;
    });
    if (!ok) return nullptr;
    Py_DECREF(ok);
    return Py_BuildValue("(LLL)", (long long)size[0], (long long)size[1], (long long)size[2]);
}

// path of libpicospec.so
PyObject* py_open(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 1, [&] {
        const char* path = PyUnicode_AsUTF8(a[0]);
        if (!path) throw Refused{""};
        api.handle = dlopen(path, RTLD_NOW | RTLD_LOCAL);
        if (!api.handle) throw Refused{dlerror()};
        auto find = [&](const char* name) {
            void* f = dlsym(api.handle, name);
            if (!f) throw Refused{std::string("libpicospec.so lacks ") + name};
            return f;
        };
#define PICOSPEC_FIND(f) api.f = (decltype(api.f))find("picospec_" #f)
        PICOSPEC_FIND(compress);
        PICOSPEC_FIND(verify);
        PICOSPEC_FIND(verify_range);
        PICOSPEC_FIND(residual_sample);
        PICOSPEC_FIND(target_topk);
        PICOSPEC_FIND(edge_resample);
        PICOSPEC_FIND(wire_pack);
        PICOSPEC_FIND(wire_unpack);
#undef PICOSPEC_FIND
        return 0;
    });
}

#define PICOSPEC_METHOD(f) {#f, (PyCFunction)(void (*)())py_##f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PICOSPEC_METHOD(open),
                         PICOSPEC_METHOD(logits),
                         PICOSPEC_METHOD(compress),
                         PICOSPEC_METHOD(verify),
                         PICOSPEC_METHOD(verify_range),
                         PICOSPEC_METHOD(residual_sample),
                         PICOSPEC_METHOD(target_topk),
                         PICOSPEC_METHOD(edge_resample),
                         PICOSPEC_METHOD(wire_pack),
                         PICOSPEC_METHOD(wire_unpack),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__marshal() { return PyModule_Create(&module); }
