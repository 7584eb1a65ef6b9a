// Argument marshalling of the Python binding for the calls a program makes per layer: torch tensors in, one C-ABI
// call on torch's current stream, the output tensor back. Nothing here computes.
//
// Why native: the same marshalling in Python (ctypes argument objects, torch.cuda.current_stream, torch.empty) took
// 8 of the 13 us that a layer call cost the calling thread, more than the kernels of a few-row layer take on the GPU
// (5.8-10 us), so decoding ran at the speed of the binding. Measured per layer call with a given workspace, M = 1,
// K = N = 5120: 13.4 us before, 5.7 us with this file (2.9 with the output given; the rest is torch making it).
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/agileq.h"

namespace {

PyObject* g_error = nullptr;      // binding.AgileqError(status, what)

struct Bad {};                    // a Python exception is set

[[noreturn]] void type_error(const char* what) {
    PyErr_SetString(PyExc_TypeError, what);
    throw Bad{};
}

// The positional arguments of one call, taken in order.
class Args {
  public:
    Args(PyObject* const* v, Py_ssize_t n, Py_ssize_t want) : v_(v) {
        if (n != want) type_error("wrong number of arguments");
    }
    int integer() {
        const long r = PyLong_AsLong(v_[i_++]);
        if (r == -1 && PyErr_Occurred()) throw Bad{};
        if (r > INT_MAX || r < INT_MIN) {
            PyErr_SetString(PyExc_OverflowError, "argument does not fit an int");
            throw Bad{};
        }
        return (int)r;
    }
    aq_handle_t handle() {        // None (a closed handle) is NULL, which the library refuses
        if (v_[i_] == Py_None) {
            ++i_;
            return nullptr;
        }
        void* p = PyLong_AsVoidPtr(v_[i_++]);
        if (!p && PyErr_Occurred()) throw Bad{};
        return (aq_handle_t)p;
    }
    const at::Tensor& tensor() {
        PyObject* o = v_[i_++];
        if (!THPVariable_Check(o)) type_error("expected a torch.Tensor");
        return THPVariable_Unpack(o);
    }
    at::Tensor optional() {       // undefined for None
        if (v_[i_] == Py_None) {
            ++i_;
            return at::Tensor();
        }
        return tensor();
    }

  private:
    PyObject* const* v_;
    Py_ssize_t i_ = 0;
};

void* ptr(const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }
// a matrix's sizes
void sizes2(const at::Tensor& t, int& rows, int& cols) {
    if (t.dim() != 2) {
        PyErr_SetString(PyExc_ValueError, "expected a matrix (two dimensions)");
        throw Bad{};
    }
    rows = (int)t.size(0);
    cols = (int)t.size(1);
}
void sizes3(const at::Tensor& t, int& a, int& b, int& c) {
    if (t.dim() != 3) {
        PyErr_SetString(PyExc_ValueError, "expected three dimensions");
        throw Bad{};
    }
    a = (int)t.size(0);
    b = (int)t.size(1);
    c = (int)t.size(2);
}
at::Tensor make(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like) {
    return at::empty(sizes, at::TensorOptions().dtype(type).device(like.device()));
}
void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

void check(int status, const char* what) {
    if (status == AQ_OK) return;
    PyObject* e = PyObject_CallFunction(g_error, "is", status, what);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Bad{};
}
// The C call runs without the interpreter lock, as through ctypes. The lock comes back on every way out: a tensor without
// storage (sparse, fake) throws when f asks for its address, and that becomes a Python exception above.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    Unlocked() = default;
    Unlocked(const Unlocked&) = delete;
    ~Unlocked() { PyEval_RestoreThread(state); }
};
template <class F>
void call(const char* what, F&& f) {
    int status;
    {
        Unlocked unlocked;
        status = f();
    }
    check(status, what);
}
at::Tensor workspace_for(const at::Tensor& given, int M, int K, int N, int group, const at::Tensor& like) {
    if (given.defined()) return given;
    const size_t n = aq_workspace_bytes(M, K, N, group);
    if (n == 0) check(AQ_ERR_SHAPE, "aq_workspace_bytes");
    return make({(int64_t)n}, at::kByte, like);
}

template <PyObject* (*F)(PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject*, PyObject* const* v, Py_ssize_t n) {
    HANDLE_TH_ERRORS          // torch's own errors (out of memory, ...) as torch's Python exceptions
    try {
        return F(v, n);
    } catch (const Bad&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// linear(handle, bits, x, packed, scales, N, group, scale_mode, clip_shift_or_exp, row_idx, y, acc_dump, workspace,
//        trip, alpha, k_max): y
PyObject* linear(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 16);
    const aq_handle_t h = a.handle();
    const int bits = a.integer();
    const at::Tensor &x = a.tensor(), packed = a.optional(), scales = a.optional();
    const int N = a.integer(), group = a.integer(), mode = a.integer(), clip = a.integer();
    const at::Tensor rows = a.optional();
    at::Tensor y = a.optional();
    const at::Tensor acc = a.optional();
    at::Tensor ws = a.optional();
    const int trip = a.integer();
    const at::Tensor alpha = a.optional();
    const int k_max = a.integer();
    int M, K;
    sizes2(x, M, K);
    if (rows.defined()) M = (int)rows.size(0);
    if (!y.defined()) y = make({M, N}, at::kHalf, x);
    ws = workspace_for(ws, M, K, N, group, x);
    void* s = stream();
    if (trip)
        call("aq_linear_w4a4_trip", [&] {
            return aq_linear_w4a4_trip(h, ptr(x), M, K, ptr(packed), ptr(scales), N, group, (const uint8_t*)ptr(alpha), k_max,
                                       mode, clip, (const int32_t*)ptr(rows), ptr(y), (int32_t*)ptr(acc), ptr(ws), (size_t)ws.numel(), s);
        });
    else
        call(bits == 8 ? "aq_linear_w4a8" : "aq_linear_w4a4", [&] {
            return (bits == 8 ? aq_linear_w4a8 : aq_linear_w4a4)(h, ptr(x), M, K, ptr(packed), ptr(scales), N, group, mode, clip,
                                                                 (const int32_t*)ptr(rows), ptr(y), (int32_t*)ptr(acc), ptr(ws),
                                                                 (size_t)ws.numel(), s);
        });
    return THPVariable_Wrap(std::move(y));
}

// linear_asym(handle, bits, x, packed, scales, offsets, N, group, row_idx, y, acc_dump, workspace): y
PyObject* linear_asym(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 12);
    const aq_handle_t h = a.handle();
    const int bits = a.integer();
    const at::Tensor &x = a.tensor(), packed = a.optional(), scales = a.optional(), offsets = a.optional();
    const int N = a.integer(), group = a.integer();
    const at::Tensor rows = a.optional();
    at::Tensor y = a.optional();
    const at::Tensor acc = a.optional();
    at::Tensor ws = a.optional();
    int M, K;
    sizes2(x, M, K);
    if (rows.defined()) M = (int)rows.size(0);
    if (!y.defined()) y = make({M, N}, at::kHalf, x);
    ws = workspace_for(ws, M, K, N, group, x);
    void* s = stream();
    call("aq_linear_asym", [&] {
        return (bits == 8 ? aq_linear_w4a8_asym : aq_linear_w4a4_asym)(h, ptr(x), M, K, ptr(packed), ptr(scales), (const float*)ptr(offsets),
                                                                       N, group, (const int32_t*)ptr(rows), ptr(y), (int32_t*)ptr(acc),
                                                                       ptr(ws), (size_t)ws.numel(), s);
    });
    return THPVariable_Wrap(std::move(y));
}

// linear_chain(handle, bits, packed_codes, x, packed, scales, N, group, next_bits, next_exp, scale_mode,
//              clip_shift_or_exp, row_idx, q_next, acc_dump, workspace): q_next
PyObject* linear_chain(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 16);
    const aq_handle_t h = a.handle();
    const int bits = a.integer(), packed_codes = a.integer();
    const at::Tensor &x = a.tensor(), packed = a.optional(), scales = a.optional();
    const int N = a.integer(), group = a.integer(), next_bits = a.integer(), next_exp = a.integer(), mode = a.integer(), clip = a.integer();
    const at::Tensor rows = a.optional();
    at::Tensor q = a.optional();
    const at::Tensor acc = a.optional();
    at::Tensor ws = a.optional();
    int M, K;
    sizes2(x, M, K);
    if (rows.defined()) M = (int)rows.size(0);
    if (!q.defined()) q = packed_codes ? make({M, N / 2}, at::kByte, x) : make({M, N}, at::kChar, x);
    ws = workspace_for(ws, M, K, N, group, x);
    void* s = stream();
    if (packed_codes)
        call("aq_linear_chain_act4", [&] {
            return (bits == 8 ? aq_linear_w4a8_chain_act4 : aq_linear_w4a4_chain_act4)(
                h, ptr(x), M, K, ptr(packed), ptr(scales), N, group, mode, clip, (const int32_t*)ptr(rows), ptr(q), next_exp,
                (int32_t*)ptr(acc), ptr(ws), (size_t)ws.numel(), s);
        });
    else
        call("aq_linear_chain", [&] {
            return (bits == 8 ? aq_linear_w4a8_chain : aq_linear_w4a4_chain)(
                h, ptr(x), M, K, ptr(packed), ptr(scales), N, group, mode, clip, (const int32_t*)ptr(rows), (int8_t*)ptr(q), next_bits,
                next_exp, (int32_t*)ptr(acc), ptr(ws), (size_t)ws.numel(), s);
        });
    return THPVariable_Wrap(std::move(q));
}

// gemm(handle, packed_codes, q, packed, scales, N, group, scale_exp, y, acc_dump, workspace): y
PyObject* gemm(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 11);
    const aq_handle_t h = a.handle();
    const int packed_codes = a.integer();
    const at::Tensor &q = a.tensor(), packed = a.optional(), scales = a.optional();
    const int N = a.integer(), group = a.integer();
    const at::Tensor e = a.optional();
    at::Tensor y = a.optional();
    const at::Tensor acc = a.optional();
    at::Tensor ws = a.optional();
    int M, K;
    sizes2(q, M, K);
    if (packed_codes) K *= 2;
    if (!y.defined()) y = make({M, N}, at::kHalf, q);
    ws = workspace_for(ws, M, K, N, group, q);
    void* s = stream();
    if (packed_codes)
        call("aq_gemm_w4_act4", [&] {
            return aq_gemm_w4_act4(h, ptr(q), M, K, ptr(packed), ptr(scales), N, group, (const int32_t*)ptr(e), ptr(y),
                                   (int32_t*)ptr(acc), ptr(ws), (size_t)ws.numel(), s);
        });
    else
        call("aq_gemm_w4", [&] {
            return aq_gemm_w4(h, (const int8_t*)ptr(q), M, K, ptr(packed), ptr(scales), N, group, (const int32_t*)ptr(e), ptr(y),
                              (int32_t*)ptr(acc), ptr(ws), (size_t)ws.numel(), s);
        });
    return THPVariable_Wrap(std::move(y));
}

// quantize_act(handle, x, bits, scale_mode, clip_shift_or_exp, row_idx, workspace): (q, e)
PyObject* quantize_act(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 7);
    const aq_handle_t h = a.handle();
    const at::Tensor& x = a.tensor();
    const int bits = a.integer(), mode = a.integer(), clip = a.integer();
    const at::Tensor rows = a.optional();
    at::Tensor ws = a.optional();
    int M, K;
    sizes2(x, M, K);
    if (rows.defined()) M = (int)rows.size(0);
    at::Tensor q = make({M, K}, at::kChar, x), e = make({1}, at::kInt, x);
    if (!ws.defined()) ws = make({256}, at::kByte, x);
    void* s = stream();
    call("aq_quantize_act", [&] {
        return aq_quantize_act(h, ptr(x), M, K, bits, mode, clip, (const int32_t*)ptr(rows), (int8_t*)ptr(q), (int32_t*)ptr(e), ptr(ws),
                               (size_t)ws.numel(), s);
    });
    return Py_BuildValue("(NN)", THPVariable_Wrap(std::move(q)), THPVariable_Wrap(std::move(e)));
}

// token_select(handle, scores, n_keep, workspace): idx
PyObject* token_select(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 4);
    const aq_handle_t h = a.handle();
    const at::Tensor& scores = a.tensor();
    const int n_keep = a.integer();
    at::Tensor ws = a.optional();
    const int M = (int)scores.size(0);
    at::Tensor idx = make({n_keep > 1 ? n_keep : 1}, at::kInt, scores);
    if (n_keep < 1) idx = idx.slice(0, 0, n_keep);
    if (!ws.defined()) ws = make({256 + (M + 255) / 256 * 256}, at::kByte, scores);
    void* s = stream();
    call("aq_token_select", [&] {
        return aq_token_select(h, (const float*)ptr(scores), M, n_keep, (int32_t*)ptr(idx), ptr(ws), (size_t)ws.numel(), s);
    });
    return THPVariable_Wrap(std::move(idx));
}

// log2_factors(handle, x, factors, workspace): (factors, max bits, workspace)
PyObject* log2_factors(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 4);
    const aq_handle_t h = a.handle();
    const at::Tensor& x = a.tensor();
    at::Tensor f = a.optional(), ws = a.optional();
    if (!f.defined()) f = make(x.sizes(), at::kByte, x);
    at::Tensor mx = make({1}, at::kInt, x);
    if (!ws.defined()) ws = make({256}, at::kByte, x);
    void* s = stream();
    call("aq_log2_quantize_factors", [&] {
        return aq_log2_quantize_factors(h, ptr(x), (long long)x.numel(), (uint8_t*)ptr(f), (uint32_t*)ptr(mx), ptr(ws),
                                        (size_t)ws.numel(), s);
    });
    return Py_BuildValue("(NNN)", THPVariable_Wrap(std::move(f)), THPVariable_Wrap(std::move(mx)), THPVariable_Wrap(std::move(ws)));
}

// attn_v(handle, on_factors, p, p_max_bits, v_codes, v_scale_exp, y, workspace): (y, workspace)
PyObject* attn_v(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 8);
    const aq_handle_t h = a.handle();
    const int on_factors = a.integer();
    const at::Tensor &p = a.tensor(), mx = a.optional(), &vc = a.tensor(), ve = a.optional();
    at::Tensor y = a.optional(), ws = a.optional();
    int H, M, J;
    sizes3(p, H, M, J);
    const int D = (int)vc.size(2);
    if (!y.defined()) y = make({H, M, D}, at::kHalf, p);
    if (!ws.defined()) ws = make({(int64_t)aq_attn_workspace_bytes(H, M, J, D)}, at::kByte, p);
    void* s = stream();
    if (on_factors)
        call("aq_attn_v_factors_tc", [&] {
            return aq_attn_v_factors_tc(h, (const uint8_t*)ptr(p), (const uint32_t*)ptr(mx), (const int8_t*)ptr(vc), (const int32_t*)ptr(ve),
                                        H, M, J, D, ptr(y), ptr(ws), (size_t)ws.numel(), s);
        });
    else
        call("aq_attn_v_log2_tc", [&] {
            return aq_attn_v_log2_tc(h, (const int8_t*)ptr(p), (const uint32_t*)ptr(mx), (const int8_t*)ptr(vc), (const int32_t*)ptr(ve), H,
                                     M, J, D, ptr(y), ptr(ws), (size_t)ws.numel(), s);
        });
    return Py_BuildValue("(NN)", THPVariable_Wrap(std::move(y)), THPVariable_Wrap(std::move(ws)));
}

// attn_qk(handle, q, q_exp, k, k_exp, s, workspace): (s, workspace)
PyObject* attn_qk(PyObject* const* v, Py_ssize_t n) {
    Args a(v, n, 7);
    const aq_handle_t h = a.handle();
    const at::Tensor &q = a.tensor(), qe = a.optional(), &k = a.tensor(), ke = a.optional();
    at::Tensor sc = a.optional(), ws = a.optional();
    int H, M, D;
    sizes3(q, H, M, D);
    const int J = (int)k.size(1);
    if (!sc.defined()) sc = make({H, M, J}, at::kHalf, q);
    if (!ws.defined()) ws = make({256}, at::kByte, q);
    void* s = stream();
    call("aq_attn_qk_tc", [&] {
        return aq_attn_qk_tc(h, (const int8_t*)ptr(q), (const int32_t*)ptr(qe), (const int8_t*)ptr(k), (const int32_t*)ptr(ke), H, M, J, D,
                             ptr(sc), ptr(ws), (size_t)ws.numel(), s);
    });
    return Py_BuildValue("(NN)", THPVariable_Wrap(std::move(sc)), THPVariable_Wrap(std::move(ws)));
}

// set_error(AgileqError)
PyObject* set_error(PyObject*, PyObject* cls) {
    Py_INCREF(cls);
    Py_XSETREF(g_error, cls);
    Py_RETURN_NONE;
}

#define AQ_FAST(name) {#name, (PyCFunction)(void (*)(void))guarded<name>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    AQ_FAST(linear), AQ_FAST(linear_asym), AQ_FAST(linear_chain), AQ_FAST(gemm), AQ_FAST(quantize_act), AQ_FAST(token_select),
    AQ_FAST(log2_factors), AQ_FAST(attn_v), AQ_FAST(attn_qk), {"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_aq_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__aq_host(void) { return PyModule_Create(&module); }
