// Native marshalling of the runtime entry points: torch tensors in, one call of the C ABI, no arithmetic.
//
// A small layer is bounded by the host: 256 x 512 x 512 keeps the device busy for 8 us, and the same call through
// ctypes took 19 us (nine addresses boxed one by one, a slice, a stream object, seventeen converted arguments).  This
// module reads the tensors directly.  Functions check what binding.py documents (AssertionError) and return the
// status code of the entry point; linear() and calibrate() return their outputs on success.
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <memory>
#include <vector>

#include "../../include/pq.h"

namespace {

struct Failed {};  // a Python error is set

[[noreturn]] void fail(const char *what) {
    PyErr_SetString(PyExc_AssertionError, what);
    throw Failed{};
}
void require(bool ok, const char *what) {
    if (!ok) fail(what);
}

const at::Tensor &tensor(PyObject *o) {
    require(THPVariable_Check(o), "a tensor is expected");
    return THPVariable_Unpack(o);
}
void *ptr(const at::Tensor &t) {
    require(t.is_cuda(), "device tensors only");
    return t.data_ptr();
}
template <typename T>
T *ptr_as(PyObject *o) {  // None is NULL
    return o == Py_None ? nullptr : static_cast<T *>(ptr(tensor(o)));
}
template <typename T>
T *ptr_of(PyObject *o, at::ScalarType type, const char *what) {
    if (o == Py_None) return nullptr;
    const at::Tensor &t = tensor(o);
    require(t.scalar_type() == type, what);
    return static_cast<T *>(ptr(t));
}
const at::Tensor &matrix(PyObject *o) {
    const at::Tensor &t = tensor(o);
    require(t.scalar_type() == at::kBFloat16 && t.dim() == 2 && t.stride(1) == 1, "a bf16 matrix with unit column stride is expected");
    return t;
}
void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
int64_t integer(PyObject *o) {
    const int64_t v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Failed{};
    return v;
}
double number(PyObject *o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Failed{};
    return v;
}
void output(const at::Tensor &Y, int64_t M, int64_t N) {
    require(Y.scalar_type() == at::kBFloat16 && Y.dim() == 2 && Y.size(0) == M && Y.size(1) == N && Y.stride(1) == 1,
            "the output is bf16 [M, N] with unit column stride");
}
void dense_output(PyObject *o, int64_t M, int64_t K) {
    if (o == Py_None) return;
    output(tensor(o), M, K);
    require(tensor(o).is_contiguous(), "y_out is contiguous");
}

// Runs f(args) with C++ exceptions turned into Python errors; n = number of arguments.
template <typename F>
PyObject *guarded(Py_ssize_t given, Py_ssize_t n, F &&f) {
    if (given != n) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return nullptr;
    }
    try {
        return f();
    } catch (const Failed &) {
        return nullptr;
    } catch (...) {  // torch's own errors keep their Python types (an allocation that fails is torch.OutOfMemoryError)
        torch::translate_exception_to_python(std::current_exception());
        return nullptr;
    }
}
PyObject *status(pq_status s) { return PyLong_FromLong(s); }
// The call itself, without the interpreter lock: a launch waits when the stream's queue is full.
template <typename F>
pq_status unlocked(F &&call) {
    PyThreadState *state = PyEval_SaveThread();
    const pq_status s = call();
    PyEval_RestoreThread(state);
    return s;
}

// linear(X, ts_x, xq, sfx, wq, sfw, ts_w, Y or None, ws) -> Y or status
PyObject *linear(PyObject *, PyObject *const *a, Py_ssize_t given) {
    return guarded(given, 9, [&]() -> PyObject * {
        const at::Tensor &X = matrix(a[0]), &W = tensor(a[4]);
        require(W.dim() >= 1, "wq is [N, K / 2]");
        const int64_t M = X.size(0), K = X.size(1), N = W.size(0), ld = X.stride(0);
        const bool make = a[7] == Py_None;
        at::Tensor Y = make ? at::empty({M, N}, X.options()) : tensor(a[7]);
        output(Y, M, N);
        const void *x = ptr(X);
        const float *ts_x = ptr_as<float>(a[1]), *ts_w = ptr_as<float>(a[6]);
        uint8_t *xq = ptr_as<uint8_t>(a[2]), *sfx = ptr_as<uint8_t>(a[3]), *sfw = ptr_as<uint8_t>(a[5]);
        const uint8_t *wq = static_cast<const uint8_t *>(ptr(W));
        void *y = ptr(Y), *ws = ptr_as<void>(a[8]), *st = stream();
        const int64_t ldy = Y.stride(0);
        const size_t ws_bytes = ws ? static_cast<size_t>(tensor(a[8]).numel()) : 0;
        const pq_status s = unlocked([&] { return pq_linear_w4a4(x, M, K, ld, ts_x, xq, sfx, wq, sfw, ts_w, N, y, ldy, ws, ws_bytes, st); });
        if (s != PQ_OK) return status(s);
        if (make) return THPVariable_Wrap(std::move(Y));
        Py_INCREF(a[7]);
        return a[7];
    });
}

// gemm(xq, sfx, ts_x, wq, sfw, ts_w, Y, ws) -> status
PyObject *gemm(PyObject *, PyObject *const *a, Py_ssize_t given) {
    return guarded(given, 8, [&]() -> PyObject * {
        const at::Tensor &X = tensor(a[0]), &W = tensor(a[3]), &Y = tensor(a[6]);
        require(X.dim() == 2 && W.dim() >= 1, "codes are [rows, K / 2]");
        const int64_t M = X.size(0), K = X.size(1) * 2, N = W.size(0), ldy = Y.dim() == 2 ? Y.stride(0) : 0;
        output(Y, M, N);
        const uint8_t *xq = static_cast<const uint8_t *>(ptr(X)), *wq = static_cast<const uint8_t *>(ptr(W));
        const uint8_t *sfx = ptr_as<uint8_t>(a[1]), *sfw = ptr_as<uint8_t>(a[4]);
        const float *ts_x = ptr_as<float>(a[2]), *ts_w = ptr_as<float>(a[5]);
        void *y = ptr(Y), *ws = ptr_as<void>(a[7]), *st = stream();
        const size_t ws_bytes = ws ? static_cast<size_t>(tensor(a[7]).numel()) : 0;
        return status(unlocked([&] { return pq_gemm_w4a4(xq, sfx, ts_x, wq, sfw, ts_w, M, N, K, y, ldy, ws, ws_bytes, st); }));
    });
}

// norm_quant(H, kind, a, b, eps, perm, ts_x, codes, sf, sf_layout, y_out) -> status
PyObject *norm_quant(PyObject *, PyObject *const *a, Py_ssize_t given) {
    return guarded(given, 11, [&]() -> PyObject * {
        const at::Tensor &H = matrix(a[0]);
        const int64_t M = H.size(0), K = H.size(1), ld = H.stride(0);
        const float *pa = ptr_of<float>(a[2], at::kFloat, "a is fp32"), *pb = ptr_of<float>(a[3], at::kFloat, "b is fp32");
        const int32_t *perm = ptr_of<int32_t>(a[5], at::kInt, "perm is int32");
        require(pa && tensor(a[2]).numel() == K && (!pb || tensor(a[3]).numel() == K) && (!perm || tensor(a[5]).numel() == K),
                "a, b and perm hold K values");
        dense_output(a[10], M, K);
        const int kind = static_cast<int>(integer(a[1])), layout = static_cast<int>(integer(a[9]));
        const float eps = static_cast<float>(number(a[4]));
        const float *ts_x = ptr_as<float>(a[6]);
        uint8_t *codes = ptr_as<uint8_t>(a[7]), *sf = ptr_as<uint8_t>(a[8]);
        void *h = ptr(H), *y = ptr_as<void>(a[10]), *st = stream();
        return status(unlocked([&] { return pq_norm_quant_nvfp4(h, M, K, ld, kind, pa, pb, eps, perm, ts_x, codes, sf, layout, y, st); }));
    });
}

// hadamard_quant(X, perm, ts_x, codes, sf, sf_layout, y_out) -> status
PyObject *hadamard_quant(PyObject *, PyObject *const *a, Py_ssize_t given) {
    return guarded(given, 7, [&]() -> PyObject * {
        const at::Tensor &X = matrix(a[0]);
        const int64_t M = X.size(0), K = X.size(1), ld = X.stride(0);
        const int32_t *perm = ptr_of<int32_t>(a[1], at::kInt, "perm is int32");
        require(!perm || (tensor(a[1]).numel() == K && tensor(a[1]).is_contiguous()), "perm holds K contiguous values");
        require((a[3] == Py_None) == (a[4] == Py_None), "codes and sf come together");
        uint8_t *codes = ptr_of<uint8_t>(a[3], at::kByte, "codes are uint8"), *sf = ptr_of<uint8_t>(a[4], at::kByte, "sf is uint8");
        require(!codes || (a[2] != Py_None && tensor(a[2]).scalar_type() == at::kFloat), "ts_x is fp32");
        dense_output(a[6], M, K);
        const float *ts_x = ptr_as<float>(a[2]);
        const int layout = static_cast<int>(integer(a[5]));
        void *x = ptr(X), *y = ptr_as<void>(a[6]), *st = stream();
        return status(unlocked([&] { return pq_hadamard_quant_nvfp4(x, M, K, ld, perm, ts_x, codes, sf, layout, y, st); }));
    });
}

// fakequant(T, kind, bits, group, perm, out) -> status
PyObject *fakequant(PyObject *, PyObject *const *a, Py_ssize_t given) {
    return guarded(given, 6, [&]() -> PyObject * {
        const at::Tensor &T = matrix(a[0]), &out = matrix(a[5]);
        const pq_format fmt = {static_cast<int>(integer(a[1])), static_cast<int>(integer(a[2])), static_cast<int>(integer(a[3]))};
        const int64_t rows = T.size(0), K = T.size(1), ld = T.stride(0), ldo = out.stride(0);
        const int32_t *perm = ptr_as<int32_t>(a[4]);
        void *src = ptr(T), *dst = ptr(out), *st = stream();
        return status(unlocked([&] { return pq_fakequant_int(src, rows, K, ld, fmt, perm, dst, ldo, st); }));
    });
}

// calibrate(Xs, Wt, kind, bits, group, J, tau, sf_layout)
//   -> status, or (sumsq_a, sumsq_w, amax_a, ts_x, ts_w, perms, err_x, err_w, lam, E, select, wq, sfw, rows)
PyObject *calibrate(PyObject *, PyObject *const *a, Py_ssize_t given) {
    return guarded(given, 8, [&]() -> PyObject * {
        const at::Tensor &W = matrix(a[1]);
        const int64_t N = W.size(0), K = W.size(1), ldw = W.stride(0);
        const pq_format fmt = {static_cast<int>(integer(a[2])), static_cast<int>(integer(a[3])), static_cast<int>(integer(a[4]))};
        const int J = static_cast<int>(integer(a[5])), layout = static_cast<int>(integer(a[7]));
        const double tau = number(a[6]);
        std::vector<const void *> xs;
        std::vector<int64_t> rows, lds;
        int64_t total = 0;
        // a tuple of its own holds the batches: another thread may empty the caller's list while the lock is released below
        PyObject *held = PySequence_Tuple(a[0]);
        if (!held) throw Failed{};
        const std::unique_ptr<PyObject, void (*)(PyObject *)> hold(held, [](PyObject *o) { Py_DECREF(o); });
        const Py_ssize_t n = PyTuple_GET_SIZE(held);
        for (Py_ssize_t i = 0; i < n; ++i) {
            const at::Tensor &X = matrix(PyTuple_GET_ITEM(held, i));
            require(X.size(1) == K, "batches have the weight's width");
            xs.push_back(ptr(X)), rows.push_back(X.size(0)), lds.push_back(X.stride(0));
            total += X.size(0);
        }
        const void *w = ptr(W);
        void *o[13], *st = stream();
        auto call = [&](void *ws, size_t ws_bytes) {
            return pq_calibrate(static_cast<int>(n), xs.data(), rows.data(), lds.data(), w, N, K, ldw, fmt, J, tau, layout,
                                static_cast<double *>(o[0]), static_cast<double *>(o[1]), static_cast<float *>(o[2]), static_cast<float *>(o[3]),
                                static_cast<float *>(o[4]), static_cast<int32_t *>(o[5]), static_cast<double *>(o[6]),
                                static_cast<double *>(o[7]), static_cast<double *>(o[8]), static_cast<double *>(o[9]),
                                static_cast<int32_t *>(o[10]), static_cast<uint8_t *>(o[11]), static_cast<uint8_t *>(o[12]), ws, ws_bytes, st);
        };
        const size_t need = pq_calibrate_workspace_bytes(static_cast<int>(n), rows.data(), N, K, fmt, J), sf_size = pq_sf_bytes(N, K, layout);
        if (!need || !sf_size) {  // nothing is allocated for sizes the call refuses (and without a workspace it launches nothing)
            for (void *&p : o) p = nullptr;
            return status(call(nullptr, 0));
        }
        const auto like = W.options();
        const auto f64 = like.dtype(at::kDouble), f32 = like.dtype(at::kFloat), i32 = like.dtype(at::kInt), u8 = like.dtype(at::kByte);
        const int64_t Kg = K / (fmt.kind == 0 ? 16 : fmt.group);
        at::Tensor out[13] = {at::empty({K}, f64), at::empty({K}, f64), at::empty({K}, f32), at::empty({1}, f32), at::empty({1}, f32),
                              at::empty({J + 1, K}, i32), at::empty({J + 2, Kg}, f64), at::empty({J + 2, Kg}, f64), at::empty({2}, f64),
                              at::empty({J + 2}, f64), at::empty({2}, i32), at::empty({N, K / 2}, u8), at::empty({static_cast<int64_t>(sf_size)}, u8)};
        at::Tensor scratch = at::empty({static_cast<int64_t>(need)}, u8);
        void *ws = ptr(scratch);
        for (int i = 0; i < 13; ++i) o[i] = out[i].data_ptr();
        const pq_status s = unlocked([&] { return call(ws, need); });
        if (s != PQ_OK) return status(s);
        PyObject *t = PyTuple_New(14);
        if (!t) return nullptr;
        for (int i = 0; i < 13; ++i) PyTuple_SET_ITEM(t, i, THPVariable_Wrap(std::move(out[i])));
        PyTuple_SET_ITEM(t, 13, PyLong_FromLongLong(total));
        return t;
    });
}

template <typename F>
PyCFunction fast(F f) {
    return reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(f));
}
PyMethodDef methods[] = {{"linear", fast(linear), METH_FASTCALL, nullptr},
                         {"gemm", fast(gemm), METH_FASTCALL, nullptr},
                         {"norm_quant", fast(norm_quant), METH_FASTCALL, nullptr},
                         {"hadamard_quant", fast(hadamard_quant), METH_FASTCALL, nullptr},
                         {"fakequant", fast(fakequant), METH_FASTCALL, nullptr},
                         {"calibrate", fast(calibrate), METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pq_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pq_native() { return PyModule_Create(&module); }
