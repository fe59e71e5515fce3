// Python binding of libnova_attn (module paper_2608_00029_b200._binding): argument checks and marshalling only, the same
// checks and messages for every tensor as documented in nova_attn.py and nova_lmhead.py, then one call of the C ABI.
//
// Why it is native: a small problem is bound by the host.  With the checks in Python and the call through ctypes a
// forward took 11.7 us to issue and a training pass of the smallest workload (B=1, H=2, T=64) 42 us, of which the C ABI
// and the launches are about a third; reading a torch.Tensor's fields from C++ costs a few nanoseconds each.
//
// Every function returns the status of the C ABI; a wrong tensor raises TypeError or ValueError before the call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <string>

#include "../../include/nova_attn.h"
#include "../../include/nova_lmhead.h"

namespace {

struct Failed {};  // a Python exception has been set

[[noreturn]] void raise(PyObject* type, const std::string& msg) {
    PyErr_SetString(type, msg.c_str());
    throw Failed{};
}

const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string(name) + " must be a torch.Tensor");
    return THPVariable_Unpack(o);
}

std::string shape_text(at::IntArrayRef s) {
    std::string r = "(";
    for (size_t i = 0; i < s.size(); ++i) r += (i ? ", " : "") + std::to_string(s[i]);
    return r + (s.size() == 1 ? ",)" : ")");
}

void check_shape(const at::Tensor& t, const char* name, at::IntArrayRef want) {
    if (t.sizes() != want)
        raise(PyExc_ValueError, std::string(name) + " has shape " + shape_text(t.sizes()) + ", expected " + shape_text(want));
}

void* data(const at::Tensor& t) { return t.data_ptr(); }

// Contiguous bf16 tensor on the GPU, [B,H,T,D].
void* bf16(PyObject* o, const char* name, at::IntArrayRef want) {
    const at::Tensor& t = tensor(o, name);
    if (t.scalar_type() != at::kBFloat16 || !t.is_cuda() || !t.is_contiguous())
        raise(PyExc_TypeError, std::string(name) + " must be a contiguous CUDA bf16 tensor");
    if (want.empty()) {
        if (t.dim() != 4) raise(PyExc_ValueError, std::string(name) + " must have four dimensions [B,H,T,D]");
    } else {
        check_shape(t, name, want);
    }
    return data(t);
}

// [B,H,T,D]-shaped bf16 view on the GPU whose last dimension is contiguous.
void* view(PyObject* o, const char* name, at::IntArrayRef want, nova_attn_strides* st) {
    const at::Tensor& t = tensor(o, name);
    if (t.scalar_type() != at::kBFloat16 || !t.is_cuda() || t.dim() != 4 || t.stride(3) != 1)
        raise(PyExc_TypeError,
              std::string(name) + " must be a 4-D CUDA bf16 view [B,H,T,D] with a contiguous last dimension");
    if (!want.empty()) check_shape(t, name, want);
    *st = nova_attn_strides{t.stride(0), t.stride(1), t.stride(2)};
    return data(t);
}

float* f32(PyObject* o, const char* name, at::IntArrayRef want) {
    const at::Tensor& t = tensor(o, name);
    if (t.scalar_type() != at::kFloat || !t.is_cuda() || !t.is_contiguous() || t.sizes() != want)
        raise(PyExc_TypeError, std::string(name) + " must be a contiguous CUDA fp32 tensor of shape " + shape_text(want));
    return static_cast<float*>(data(t));
}

// As float(o) and int(o) read them: text and numbers of other types are fine.
float real(PyObject* o) {
    PyObject* f = PyNumber_Float(o);
    if (!f) throw Failed{};
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return static_cast<float>(v);
}

int truth(PyObject* o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw Failed{};
    return v;
}

int integer(PyObject* o) {
    PyObject* i = PyNumber_Long(o);
    if (!i) throw Failed{};
    const long v = PyLong_AsLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw Failed{};
    return static_cast<int>(v);
}

// The stream's handle; None is torch's current stream of the current device.
void* stream(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw Failed{};
    void* p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!p && PyErr_Occurred()) throw Failed{};
    return p;
}

// The caller's workspace (any type: a span of bytes on the GPU), or one of `need` bytes allocated for this call.  That one is
// given back when the call returns, before its kernels have run, so it has to come from the memory of the stream that they
// run on: what is allocated on that stream next is ordered behind them.
struct Workspace {
    at::Tensor own;
    void* ptr;
    size_t bytes;
    Workspace(PyObject* o, size_t need, PyObject* like, void* stream) {
        const at::Tensor* t = &own;
        if (o == Py_None) {
            const at::Tensor& l = tensor(like, "tensor");
            c10::cuda::CUDAStreamGuard guard(
                c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(stream), l.device().index()));
            own = at::empty({static_cast<int64_t>(need)}, l.options().dtype(at::kByte));
        } else {
            t = &tensor(o, "workspace");
        }
        if (!t->is_cuda() || !t->is_non_overlapping_and_dense())
            raise(PyExc_TypeError, "workspace must be a CUDA tensor without gaps");
        ptr = data(*t);
        bytes = t->nbytes();
    }
};

struct Dims {
    int B, H, T, D;
    explicit Dims(at::IntArrayRef s)
        : B(static_cast<int>(s[0])), H(static_cast<int>(s[1])), T(static_cast<int>(s[2])), D(static_cast<int>(s[3])) {}
};

template <typename F>
int without_gil(F&& f) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return rc;
}

using Args = PyObject* const*;

int attn_fwd(Args a) {  // Q K V O LSE scale causal stream
    void* q = bf16(a[0], "Q", {});
    const at::IntArrayRef s = THPVariable_Unpack(a[0]).sizes();
    void *k = bf16(a[1], "K", s), *v = bf16(a[2], "V", s), *o = bf16(a[3], "O", s);
    float* lse = f32(a[4], "LSE", s.slice(0, 3));
    const Dims d(s);
    const float scale = real(a[5]);
    const int causal = truth(a[6]);
    void* st = stream(a[7]);
    return without_gil([&] { return nova_attn_fwd(q, k, v, o, lse, d.B, d.H, d.T, d.D, scale, causal, st); });
}

int attn_fwd_strided(Args a) {
    nova_attn_strides sq, sk, sv, so;
    void* q = view(a[0], "Q", {}, &sq);
    const at::IntArrayRef s = THPVariable_Unpack(a[0]).sizes();
    void *k = view(a[1], "K", s, &sk), *v = view(a[2], "V", s, &sv), *o = view(a[3], "O", s, &so);
    float* lse = f32(a[4], "LSE", s.slice(0, 3));
    const Dims d(s);
    const float scale = real(a[5]);
    const int causal = truth(a[6]);
    void* st = stream(a[7]);
    return without_gil([&] {
        return nova_attn_fwd_strided(q, k, v, o, lse, d.B, d.H, d.T, d.D, &sq, &sk, &sv, &so, scale, causal, st);
    });
}

int preprocess(Args a) {  // O dO Delta stream
    void* o = bf16(a[0], "O", {});
    const at::IntArrayRef s = THPVariable_Unpack(a[0]).sizes();
    void* dO = bf16(a[1], "dO", s);
    float* delta = f32(a[2], "Delta", s.slice(0, 3));
    const Dims d(s);
    void* st = stream(a[3]);
    return without_gil([&] { return nova_attn_bwd_preprocess(o, dO, delta, d.B, d.H, d.T, d.D, st); });
}

int preprocess_strided(Args a) {
    nova_attn_strides so, sdo;
    void* o = view(a[0], "O", {}, &so);
    const at::IntArrayRef s = THPVariable_Unpack(a[0]).sizes();
    void* dO = view(a[1], "dO", s, &sdo);
    float* delta = f32(a[2], "Delta", s.slice(0, 3));
    const Dims d(s);
    void* st = stream(a[3]);
    return without_gil(
        [&] { return nova_attn_bwd_preprocess_strided(o, dO, delta, d.B, d.H, d.T, d.D, &so, &sdo, st); });
}

int preprocess_exact(Args a) {  // Q K V dO LSE Delta scale causal stream
    void* q = bf16(a[0], "Q", {});
    const at::IntArrayRef s = THPVariable_Unpack(a[0]).sizes();
    void *k = bf16(a[1], "K", s), *v = bf16(a[2], "V", s), *dO = bf16(a[3], "dO", s);
    float *lse = f32(a[4], "LSE", s.slice(0, 3)), *delta = f32(a[5], "Delta", s.slice(0, 3));
    const Dims d(s);
    const float scale = real(a[6]);
    const int causal = truth(a[7]);
    void* st = stream(a[8]);
    return without_gil([&] {
        return nova_attn_bwd_preprocess_exact(q, k, v, dO, lse, delta, d.B, d.H, d.T, d.D, scale, causal, st);
    });
}

// The tensors every contiguous backward takes: Q K V [O] dO LSE Delta dQ dK dV from a[0] on.
struct BwdTensors {
    void *q, *k, *v, *o = nullptr, *dO, *dq, *dk, *dv;
    float *lse, *delta;
    Dims d;
    int used;
    BwdTensors(Args a, bool with_o) : q(bf16(a[0], "Q", {})), d(THPVariable_Unpack(a[0]).sizes()) {
        const at::IntArrayRef s = THPVariable_Unpack(a[0]).sizes();
        k = bf16(a[1], "K", s);
        v = bf16(a[2], "V", s);
        int i = 3;
        if (with_o) o = bf16(a[i++], "O", s);
        dO = bf16(a[i], "dO", s);
        lse = f32(a[i + 1], "LSE", s.slice(0, 3));
        delta = f32(a[i + 2], "Delta", s.slice(0, 3));
        dq = bf16(a[i + 3], "dQ", s);
        dk = bf16(a[i + 4], "dK", s);
        dv = bf16(a[i + 5], "dV", s);
        used = i + 6;
    }
};

int bwd(Args a) {  // Q K V O dO LSE Delta dQ dK dV scale causal workspace stream steps
    const BwdTensors t(a, true);
    const Dims& d = t.d;
    const float scale = real(a[10]);
    const int causal = truth(a[11]);
    void* st = stream(a[13]);
    const Workspace ws(a[12], nova_attn_bwd_workspace_bytes(d.B, d.H, d.T, d.D), a[0], st);
    const int steps = integer(a[14]);
    return without_gil([&] {
        return nova_attn_bwd_steps(t.q, t.k, t.v, t.o, t.dO, t.lse, t.delta, t.dq, t.dk, t.dv, d.B, d.H, d.T, d.D, scale,
                                   causal, ws.ptr, ws.bytes, st, steps);
    });
}

int bwd_static_scratch(Args a) {  // Q K V O dO LSE Delta dQ dK dV scale causal stream
    const BwdTensors t(a, true);
    const Dims& d = t.d;
    const float scale = real(a[10]);
    const int causal = truth(a[11]);
    void* st = stream(a[12]);
    return without_gil([&] {
        return nova_attn_bwd_static_scratch(t.q, t.k, t.v, t.o, t.dO, t.lse, t.delta, t.dq, t.dk, t.dv, d.B, d.H, d.T, d.D,
                                            scale, causal, st);
    });
}

int bwd_deterministic(Args a) {  // Q K V dO LSE Delta dQ dK dV scale causal stream
    const BwdTensors t(a, false);
    const Dims& d = t.d;
    const float scale = real(a[9]);
    const int causal = truth(a[10]);
    void* st = stream(a[11]);
    return without_gil([&] {
        return nova_attn_bwd_deterministic(t.q, t.k, t.v, t.dO, t.lse, t.delta, t.dq, t.dk, t.dv, d.B, d.H, d.T, d.D, scale,
                                           causal, st);
    });
}

int bwd_strided(Args a) {  // Q K V dO LSE Delta dQ dK dV scale causal workspace stream
    nova_attn_strides sq, sk, sv, sdo, sdq, sdk, sdv;
    void* q = view(a[0], "Q", {}, &sq);
    const at::IntArrayRef s = THPVariable_Unpack(a[0]).sizes();
    void *k = view(a[1], "K", s, &sk), *v = view(a[2], "V", s, &sv), *dO = view(a[3], "dO", s, &sdo);
    void *dq = view(a[6], "dQ", s, &sdq), *dk = view(a[7], "dK", s, &sdk), *dv = view(a[8], "dV", s, &sdv);
    float *lse = f32(a[4], "LSE", s.slice(0, 3)), *delta = f32(a[5], "Delta", s.slice(0, 3));
    const Dims d(s);
    const float scale = real(a[9]);
    const int causal = truth(a[10]);
    void* st = stream(a[12]);
    const Workspace ws(a[11], nova_attn_bwd_workspace_bytes(d.B, d.H, d.T, d.D), a[0], st);
    return without_gil([&] {
        return nova_attn_bwd_strided(q, k, v, dO, lse, delta, dq, dk, dv, d.B, d.H, d.T, d.D, &sq, &sk, &sv, &sdo, &sdq, &sdk,
                                     &sdv, scale, causal, ws.ptr, ws.bytes, st);
    });
}

int lmhead_fwd(Args a) {  // X W targets logits lse loss workspace stream
    void* xw[2];
    for (int i = 0; i < 2; ++i) {
        const char* name = i ? "W" : "X";
        const at::Tensor& t = tensor(a[i], name);
        if (t.scalar_type() != at::kBFloat16 || !t.is_cuda() || !t.is_contiguous() || t.dim() != 2)
            raise(PyExc_TypeError, std::string(name) + " must be a contiguous 2-D CUDA bf16 tensor");
        xw[i] = data(t);
    }
    const at::Tensor &X = THPVariable_Unpack(a[0]), &W = THPVariable_Unpack(a[1]);
    const int64_t M = X.size(0), K = X.size(1), N = W.size(0);
    if (W.size(1) != K) raise(PyExc_ValueError, "X [M,K] and W [N,K] must agree in K");
    const at::Tensor& tg = tensor(a[2], "targets");
    if (tg.scalar_type() != at::kInt || !tg.is_cuda() || !tg.is_contiguous() || tg.sizes() != at::IntArrayRef({M}))
        raise(PyExc_TypeError, "targets must be a contiguous CUDA int32 tensor [M]");
    void* logits = nullptr;
    if (a[3] != Py_None) {
        const at::Tensor& t = tensor(a[3], "logits");
        if (t.scalar_type() != at::kBFloat16 || !t.is_cuda() || !t.is_contiguous() || t.sizes() != at::IntArrayRef({M, N}))
            raise(PyExc_TypeError, "logits must be a contiguous CUDA bf16 tensor [M,N] or None");
        logits = data(t);
    }
    float* stat[2];
    for (int i = 0; i < 2; ++i) {
        const char* name = i ? "loss" : "lse";
        const at::Tensor& t = tensor(a[4 + i], name);
        if (t.scalar_type() != at::kFloat || !t.is_cuda() || !t.is_contiguous() || t.sizes() != at::IntArrayRef({M}))
            raise(PyExc_TypeError, std::string(name) + " must be a contiguous CUDA fp32 tensor [M]");
        stat[i] = static_cast<float*>(data(t));
    }
    const int m = static_cast<int>(M), n = static_cast<int>(N), k = static_cast<int>(K);
    void* st = stream(a[7]);
    const Workspace ws(a[6], nova_lmhead_workspace_bytes(m, n, k), a[0], st);
    const int* targets = static_cast<const int*>(data(tg));
    return without_gil(
        [&] { return nova_lmhead_fwd(xw[0], xw[1], targets, logits, stat[0], stat[1], m, n, k, ws.ptr, ws.bytes, st); });
}

template <int (*F)(Args), int kCount>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != kCount) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", kCount, n);
        return nullptr;
    }
    try {
        return PyLong_FromLong(F(args));
    } catch (const Failed&) {
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

#define NOVA_ENTRY(name, f, count) \
    {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<f, count>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    NOVA_ENTRY("attn_fwd", attn_fwd, 8),
    NOVA_ENTRY("attn_fwd_strided", attn_fwd_strided, 8),
    NOVA_ENTRY("preprocess", preprocess, 4),
    NOVA_ENTRY("preprocess_strided", preprocess_strided, 4),
    NOVA_ENTRY("preprocess_exact", preprocess_exact, 9),
    NOVA_ENTRY("bwd", bwd, 15),
    NOVA_ENTRY("bwd_static_scratch", bwd_static_scratch, 13),
    NOVA_ENTRY("bwd_deterministic", bwd_deterministic, 12),
    NOVA_ENTRY("bwd_strided", bwd_strided, 13),
    NOVA_ENTRY("lmhead_fwd", lmhead_fwd, 8),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

// What this module was compiled against.  It reads tensors through torch's C++ classes, whose layout belongs to one version:
// with another it must not load (the build looks for the same text in the file to see whether it is out of date).
const char kBuiltFor[] = "nova binding for " NOVA_BUILT_FOR;

bool runs_with_what_it_was_built_for() {
    PyObject* torch = PyImport_ImportModule("torch");
    PyObject* version = torch ? PyObject_GetAttrString(torch, "__version__") : nullptr;
    PyObject* now = version ? PyUnicode_FromFormat("nova binding for torch %S, Python %d.%d", version, PY_MAJOR_VERSION,
                                                   PY_MINOR_VERSION) : nullptr;
    const bool same = now && PyUnicode_CompareWithASCIIString(now, kBuiltFor) == 0;
    if (now && !same)
        PyErr_Format(PyExc_ImportError, "this is the %s, loaded with torch %S: run python -m paper_2608_00029_b200.build",
                     kBuiltFor, version);
    Py_XDECREF(now);
    Py_XDECREF(version);
    Py_XDECREF(torch);
    return same;
}

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return runs_with_what_it_was_built_for() ? PyModule_Create(&module) : nullptr; }
