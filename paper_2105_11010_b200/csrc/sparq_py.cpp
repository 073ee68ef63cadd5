// CPython side of the binding: checks torch tensors, takes their addresses and torch's current
// stream, and calls the C ABI of sparq.h.
//
// Why native: a small layer takes 3-10 us on the device, and marshalling one call through
// ctypes (about twenty tensor attributes and sixteen converted arguments) took the host 13 us,
// which was the whole cost of a batch-1 network.  Here a call costs the host about 1 us plus
// the launch itself.
//
// Every function takes its arguments by position in the order of the wrappers in _binding.py,
// which own the keyword names and defaults, and returns the C ABI's status.
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>

#include "sparq.h"

namespace {

using at::Tensor;

// Thrown after a Python error has been set.
struct PyFail {};

[[noreturn]] void fail(const char *fmt, const char *name)
{
    PyErr_Format(PyExc_ValueError, fmt, name);
    throw PyFail();
}

// Positional arguments of one call, taken in order.
struct Args {
    PyObject *const *a;
    Py_ssize_t n, i = 0;

    Args(PyObject *const *args, Py_ssize_t nargs, Py_ssize_t want) : a(args), n(nargs)
    {
        if (nargs != want) {
            PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs);
            throw PyFail();
        }
    }
    PyObject *next() { return a[i++]; }
    // a tensor, or nullptr for None
    const Tensor *opt(const char *name)
    {
        PyObject *o = next();
        if (o == Py_None) return nullptr;
        if (!THPVariable_Check(o)) {
            PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor", name);
            throw PyFail();
        }
        return &THPVariable_Unpack(o);
    }
    const Tensor &tensor(const char *name)
    {
        const Tensor *t = opt(name);
        if (!t) {
            PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor", name);
            throw PyFail();
        }
        return *t;
    }
    int64_t integer()
    {
        const int64_t v = PyLong_AsLongLong(next());
        if (v == -1 && PyErr_Occurred()) throw PyFail();
        return v;
    }
    float real()
    {
        const double v = PyFloat_AsDouble(next());
        if (v == -1.0 && PyErr_Occurred()) throw PyFail();
        return (float)v;
    }
    bool truth()
    {
        const int v = PyObject_IsTrue(next());
        if (v < 0) throw PyFail();
        return v != 0;
    }
    // (a, b) of a two-element sequence
    void pair(int *x, int *y)
    {
        PyObject *o = next();
        for (int k = 0; k < 2; ++k) {
            PyObject *e = PySequence_GetItem(o, k);
            if (!e) throw PyFail();
            const long v = PyLong_AsLong(e);
            Py_DECREF(e);
            if (v == -1 && PyErr_Occurred()) throw PyFail();
            *(k ? y : x) = (int)v;
        }
    }
    // None: torch's current stream; an integer handle; or an object with `cuda_stream`
    void *stream()
    {
        PyObject *o = next();
        if (o == Py_None) return (void *)c10::cuda::getCurrentCUDAStream().stream();
        void *p = nullptr;
        if (PyLong_Check(o)) {
            p = PyLong_AsVoidPtr(o);
        } else {
            PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
            if (!h) throw PyFail();
            p = PyLong_AsVoidPtr(h);
            Py_DECREF(h);
        }
        if (!p && PyErr_Occurred()) throw PyFail();
        return p;
    }
};

// Attribute names of SparqParams, interned once.
PyObject *g_mode, *g_bits, *g_mask, *g_rounding;

int64_t attr(PyObject *o, PyObject *name)
{
    PyObject *v = PyObject_GetAttr(o, name);
    if (!v) throw PyFail();
    const int64_t x = PyLong_AsLongLong(v);
    Py_DECREF(v);
    if (x == -1 && PyErr_Occurred()) throw PyFail();
    return x;
}

sparq_params params_of(PyObject *o)
{
    sparq_params p;
    p.mode = (int32_t)attr(o, g_mode);
    p.window_bits = (int32_t)attr(o, g_bits);
    p.placement_mask = (uint32_t)attr(o, g_mask);
    p.rounding = (int32_t)attr(o, g_rounding);
    return p;
}

const char *dtype_text(at::ScalarType t)
{
    switch (t) {
    case at::kByte: return "torch.uint8";
    case at::kChar: return "torch.int8";
    case at::kInt: return "torch.int32";
    case at::kFloat: return "torch.float32";
    default: return "another dtype";
    }
}

// Address of a contiguous CUDA (or, with `host`, CPU) tensor of type T; nullptr for None.
template <class T>
T *data(const Tensor *t, at::ScalarType want, const char *name, bool host = false)
{
    if (!t) return nullptr;
    if (t->is_cuda() == host)
        fail(host ? "%s must be a CPU tensor (pinned for asynchronous copies)" : "%s must be a CUDA tensor", name);
    if (t->scalar_type() != want) {
        PyErr_Format(PyExc_ValueError, "%s must have dtype %s, got %s", name, dtype_text(want), c10::toString(t->scalar_type()));
        throw PyFail();
    }
    if (!t->is_contiguous()) fail("%s must be contiguous", name);
    return (T *)t->data_ptr();
}

// The epilogue arguments shared by every fused call, in the wrappers' order: scale, bias, relu,
// inv_out_scale, acc_out, f32_out, u8_out, next_transform, residual, residual_scale.
struct Epilogue {
    sparq_epilogue e = {};
    sparq_params next = {};

    Epilogue(Args &a, int64_t m, int64_t n, bool host)
    {
        const Tensor *scale = a.opt("scale"), *bias = a.opt("bias");
        if (scale && scale->numel() < n) fail("%s has fewer than N elements", "scale");
        if (bias && bias->numel() < n) fail("%s has fewer than N elements", "bias");
        e.scale = data<float>(scale, at::kFloat, "scale");
        e.bias = data<float>(bias, at::kFloat, "bias");
        e.relu = a.truth();
        e.inv_out_scale = a.real();
        const Tensor *acc = a.opt("acc_out"), *f32 = a.opt("f32_out"), *u8 = a.opt("u8_out");
        PyObject *nx = a.next();
        if (nx != Py_None) {
            next = params_of(nx);
            e.next_transform = &next;
        }
        const Tensor *res = a.opt("residual");
        e.residual_scale = a.real();
        const Tensor *all[4] = {acc, f32, u8, res};
        const char *names[4] = {"acc_out", "f32_out", "u8_out", "residual"};
        for (int i = 0; i < 4; ++i)
            if (all[i] && all[i]->numel() < m * n) fail("%s has fewer than M*N elements", names[i]);
        e.acc_out = data<int32_t>(acc, at::kInt, "acc_out", host);
        e.f32_out = data<float>(f32, at::kFloat, "f32_out", host);
        e.u8_out = data<uint8_t>(u8, at::kByte, "u8_out", host);
        e.residual = data<uint8_t>(res, at::kByte, "residual", host);
    }
};
constexpr int kEpilogueArgs = 10;

// The call itself without the interpreter lock (a full launch queue, or a host-buffer form's
// synchronization, blocks only this thread).
template <class F>
PyObject *call(F f)
{
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

template <class F>
PyObject *guarded(F f)
{
    try {
        return f();
    } catch (const PyFail &) {
    } catch (const std::exception &x) {
        PyErr_SetString(PyExc_RuntimeError, x.what());
    }
    return nullptr;
}

#define SPARQ_PY(NAME) PyObject *NAME(PyObject *, PyObject *const *args, Py_ssize_t nargs)

// rows and row length of a tensor whose rows lie along its last axis
void rows_of(const Tensor &t, size_t *rows, size_t *row_len)
{
    *row_len = t.dim() ? (size_t)t.size(-1) : 1;
    *rows = *row_len ? (size_t)t.numel() / *row_len : 0;
}

// (inp, out, rows, row_len, params, stream)
PyObject *quantize_call(PyObject *const *args, Py_ssize_t nargs, bool host)
{
    return guarded([&] {
        Args a(args, nargs, 6);
        const Tensor &in = a.tensor("inp"), &out = a.tensor("out");
        const int64_t rows = a.integer(), len = a.integer();
        int64_t count = 0;
        if (rows < 0 || len < 0) fail("%s must not be negative", "rows and row_len");
        if (__builtin_mul_overflow(rows, len, &count) || in.numel() < count || out.numel() < count)
            fail("%s smaller than rows * row_len", "tensor");
        const sparq_params p = params_of(a.next());
        const uint8_t *src = data<uint8_t>(&in, at::kByte, "inp", host);
        uint8_t *dst = data<uint8_t>(&out, at::kByte, "out", host);
        void *st = a.stream();
        return call([&] { return (host ? sparq_quantize_host : sparq_quantize)(src, dst, (size_t)rows, (size_t)len, &p, st); });
    });
}
SPARQ_PY(py_quantize) { return quantize_call(args, nargs, false); }
SPARQ_PY(py_quantize_host) { return quantize_call(args, nargs, true); }

// (A, B, params, epilogue..., stream)
PyObject *gemm_call(PyObject *const *args, Py_ssize_t nargs, bool host,
                    int (*fn)(const uint8_t *, int64_t, const int8_t *, int64_t, int64_t, int64_t, int64_t,
                              const sparq_params *, const sparq_epilogue *, void *))
{
    return guarded([&] {
        Args a(args, nargs, 3 + kEpilogueArgs + 1);
        const Tensor &A = a.tensor("A"), &B = a.tensor("B");
        if (A.dim() != 2 || B.dim() != 2) fail("%s must be matrices", "A and B");
        const int64_t M = A.size(0), K = A.size(1), N = B.size(0);
        if (B.size(1) != K) fail("%s disagree on K", "A and B");
        const sparq_params p = params_of(a.next());
        const Epilogue ep(a, M, N, host);
        const uint8_t *pa = data<uint8_t>(&A, at::kByte, "A", host);
        const int8_t *pb = data<int8_t>(&B, at::kChar, "B");
        void *st = a.stream();
        return call([&] { return fn(pa, K, pb, K, M, N, K, &p, &ep.e, st); });
    });
}
SPARQ_PY(py_gemm) { return gemm_call(args, nargs, false, sparq_gemm_s8); }
SPARQ_PY(py_gemm_static) { return gemm_call(args, nargs, false, sparq_gemm_s8_static); }
SPARQ_PY(py_gemm_host) { return gemm_call(args, nargs, true, sparq_gemm_s8_host); }

// (x, w, stride, pad, params, epilogue..., stream)
PyObject *conv_call(PyObject *const *args, Py_ssize_t nargs, bool host)
{
    return guarded([&] {
        Args a(args, nargs, 5 + kEpilogueArgs + 1);
        const Tensor &x = a.tensor("x"), &w = a.tensor("w");
        if (x.dim() != 4 || w.dim() != 4) fail("%s must be 4-dimensional", "x and w");
        const int64_t nb = x.size(0), h = x.size(1), wd = x.size(2), c = x.size(3);
        const int64_t cout = w.size(0), r = w.size(1), s = w.size(2);
        if (w.size(3) != c) fail("%s disagree on the channel count", "x and w");
        int sh, sw, ph, pw;
        a.pair(&sh, &sw);
        a.pair(&ph, &pw);
        // output pixels, for the size checks of the outputs; the library refuses bad geometry
        const int64_t ho = sh > 0 ? (h + 2 * ph - r) / sh + 1 : 0, wo = sw > 0 ? (wd + 2 * pw - s) / sw + 1 : 0;
        const sparq_params p = params_of(a.next());
        const Epilogue ep(a, nb * ho * wo, cout, host);
        const uint8_t *px = data<uint8_t>(&x, at::kByte, "x", host);
        const int8_t *pwgt = data<int8_t>(&w, at::kChar, "w");
        void *st = a.stream();
        return call([&] {
            return (host ? sparq_conv2d_nhwc_s8_host : sparq_conv2d_nhwc_s8)(px, (int)nb, (int)h, (int)wd, (int)c, pwgt, (int)cout,
                                                                             (int)r, (int)s, sh, sw, ph, pw, &p, &ep.e, st);
        });
    });
}
SPARQ_PY(py_conv2d) { return conv_call(args, nargs, false); }
SPARQ_PY(py_conv2d_host) { return conv_call(args, nargs, true); }

// (activations, params, data, ctrl, stream); `activations` is the input or, decoding, the output
PyObject *codec_call(PyObject *const *args, Py_ssize_t nargs, bool encode)
{
    return guarded([&] {
        Args a(args, nargs, 5);
        const Tensor &t = a.tensor(encode ? "inp" : "out");
        const sparq_params p = params_of(a.next());
        const Tensor &d = a.tensor("data"), &c = a.tensor("ctrl");
        const int cb = sparq_packed_ctrl_bits(&p);
        if (cb < 0) return PyLong_FromLong(cb);
        const int64_t units = t.numel() / 16;
        if (d.numel() < units * 2 * p.window_bits || c.numel() < units * cb) fail("%s plane too small", "data / ctrl");
        size_t rows, len;
        rows_of(t, &rows, &len);
        uint8_t *pt = data<uint8_t>(&t, at::kByte, encode ? "inp" : "out");
        uint8_t *pd = data<uint8_t>(&d, at::kByte, "data"), *pc = data<uint8_t>(&c, at::kByte, "ctrl");
        void *st = a.stream();
        return call([&] {
            return encode ? sparq_pack(pt, rows, len, &p, pd, pc, st) : sparq_unpack(pd, pc, rows, len, &p, pt, st);
        });
    });
}
SPARQ_PY(py_pack) { return codec_call(args, nargs, true); }
SPARQ_PY(py_unpack) { return codec_call(args, nargs, false); }

// Address and library dtype of a float32 / bfloat16 tensor.
const void *float_data(const Tensor &t, int *dtype)
{
    const bool bf16 = t.scalar_type() == at::kBFloat16;
    if (!t.is_cuda() || !t.is_contiguous() || !(bf16 || t.scalar_type() == at::kFloat))
        fail("%s must be a contiguous CUDA tensor of float32 or bfloat16", "x");
    *dtype = bf16 ? SPARQ_DTYPE_BF16 : SPARQ_DTYPE_F32;
    return t.data_ptr();
}

// (x, max_inout, stream)
SPARQ_PY(py_absmax)
{
    return guarded([&] {
        Args a(args, nargs, 3);
        const Tensor &x = a.tensor("x"), &m = a.tensor("max_inout");
        int dt;
        const void *px = float_data(x, &dt);
        float *pm = data<float>(&m, at::kFloat, "max_inout");
        void *st = a.stream();
        const size_t n = (size_t)x.numel();
        return call([&] { return sparq_absmax(px, dt, n, pm, st); });
    });
}

// (x, max_dev, out, stream)
SPARQ_PY(py_quantize_act)
{
    return guarded([&] {
        Args a(args, nargs, 4);
        const Tensor &x = a.tensor("x"), &m = a.tensor("max_dev"), &out = a.tensor("out");
        int dt;
        const void *px = float_data(x, &dt);
        if (out.numel() < x.numel()) fail("%s is smaller than x", "out");
        const float *pm = data<float>(&m, at::kFloat, "max_dev");
        uint8_t *po = data<uint8_t>(&out, at::kByte, "out");
        void *st = a.stream();
        const size_t n = (size_t)x.numel();
        return call([&] { return sparq_quantize_act_u8(px, dt, n, pm, po, st); });
    });
}

// (w, out, scale_out, stream)
SPARQ_PY(py_quantize_weight)
{
    return guarded([&] {
        Args a(args, nargs, 4);
        const Tensor &w = a.tensor("w"), &out = a.tensor("out"), &sc = a.tensor("scale_out");
        const int64_t cout = w.dim() ? w.size(0) : 1, k = cout ? w.numel() / cout : 0;
        if (out.numel() < w.numel() || sc.numel() < cout) fail("%s too small", "out / scale_out");
        const float *pw = data<float>(&w, at::kFloat, "w");
        int8_t *po = data<int8_t>(&out, at::kChar, "out");
        float *ps = data<float>(&sc, at::kFloat, "scale_out");
        void *st = a.stream();
        return call([&] { return sparq_quantize_weight_s8(pw, cout, k, po, ps, st); });
    });
}

// K' of these parameters, or an error status (< 0)
int64_t expanded_k(int64_t K, const sparq_params &p) { return sparq_sparse24_expanded_k(K, &p); }

// (A, params, a_exp, stream)
SPARQ_PY(py_expand_activations)
{
    return guarded([&] {
        Args a(args, nargs, 4);
        const Tensor &A = a.tensor("A");
        const sparq_params p = params_of(a.next());
        const Tensor &x = a.tensor("a_exp");
        size_t rows, K;
        rows_of(A, &rows, &K);
        const int64_t kx = expanded_k((int64_t)K, p);
        if (kx < 0) return PyLong_FromLongLong(kx);
        if (x.numel() < (int64_t)rows * kx) fail("%s too small", "a_exp");
        const uint8_t *pa = data<uint8_t>(&A, at::kByte, "A");
        uint8_t *px = data<uint8_t>(&x, at::kByte, "a_exp");
        void *st = a.stream();
        return call([&] { return sparq_sparse24_expand_activations(pa, rows, K, &p, px, st); });
    });
}

// (A, w_exp, params, workspace, epilogue..., stream)
SPARQ_PY(py_gemm_sparse24)
{
    return guarded([&] {
        Args a(args, nargs, 4 + kEpilogueArgs + 1);
        const Tensor &A = a.tensor("A"), &w = a.tensor("w_exp");
        if (A.dim() != 2 || w.dim() < 1) fail("%s must be matrices", "A and w_exp");
        const int64_t M = A.size(0), K = A.size(1), N = w.size(0);
        const sparq_params p = params_of(a.next());
        const int64_t kx = expanded_k(K, p);
        if (kx < 0) return PyLong_FromLongLong(kx);
        if (w.numel() != N * kx) fail("%s does not have N * K' elements", "w_exp");
        const Tensor *ws = a.opt("workspace");
        if (ws && ws->numel() < M * kx) fail("%s smaller than M * K'", "workspace");
        const Epilogue ep(a, M, N, false);
        const uint8_t *pa = data<uint8_t>(&A, at::kByte, "A");
        const int8_t *pw = data<int8_t>(&w, at::kChar, "w_exp");
        uint8_t *pws = data<uint8_t>(ws, at::kByte, "workspace");
        void *st = a.stream();
        return call([&] { return sparq_gemm_s8_sparse24(pa, pw, M, N, K, &p, &ep.e, pws, st); });
    });
}

#define SPARQ_DEF(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, nullptr}

PyMethodDef kMethods[] = {
    SPARQ_DEF("quantize", py_quantize),
    SPARQ_DEF("quantize_host", py_quantize_host),
    SPARQ_DEF("gemm", py_gemm),
    SPARQ_DEF("gemm_static", py_gemm_static),
    SPARQ_DEF("gemm_host", py_gemm_host),
    SPARQ_DEF("conv2d", py_conv2d),
    SPARQ_DEF("conv2d_host", py_conv2d_host),
    SPARQ_DEF("pack", py_pack),
    SPARQ_DEF("unpack", py_unpack),
    SPARQ_DEF("absmax", py_absmax),
    SPARQ_DEF("quantize_act", py_quantize_act),
    SPARQ_DEF("quantize_weight", py_quantize_weight),
    SPARQ_DEF("expand_activations", py_expand_activations),
    SPARQ_DEF("gemm_sparse24", py_gemm_sparse24),
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void)
{
    g_mode = PyUnicode_InternFromString("mode");
    g_bits = PyUnicode_InternFromString("window_bits");
    g_mask = PyUnicode_InternFromString("placement_mask");
    g_rounding = PyUnicode_InternFromString("rounding");
    if (!g_mode || !g_bits || !g_mask || !g_rounding) return nullptr;
    return PyModule_Create(&kModule);
}
