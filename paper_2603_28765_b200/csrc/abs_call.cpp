// The calls of binding.py that allocate their outputs and enqueue kernels, without the interpreter in between: argument
// unpacking, output allocation, device guard, current stream, and the call through the C ABI of
// include/abs_b200.h, whose addresses binding.py passes in.  A quantize call is two kernels of a few microseconds on small
// tensors, and marshalling it from Python took 31 us, with a fill kernel for the one float of the tensor scale.
#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <ATen/record_function.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/abs_b200.h"

namespace {

struct Entry {
    decltype(&abs_quantize_ex) quantize;
    decltype(&abs_quantize_transposed) quantize_transposed;
    decltype(&abs_quantize_dequantize) quantize_dequantize;
    decltype(&abs_dequantize_ex) dequantize;
    decltype(&abs_matmul) matmul;
    decltype(&abs_matmul_bf16) matmul_bf16;
    decltype(&abs_matmul_bf16_scaled) matmul_bf16_scaled;
    decltype(&abs_matmul_workspace_bytes) matmul_workspace_bytes;
    decltype(&abs_scales_bytes_swizzled) scales_bytes_swizzled;
} entry;

// A Python exception is set.
struct Raised {};

at::Tensor tensor(PyObject* o, const char* what) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s: a tensor was expected", what);
        throw Raised();
    }
    return THPVariable_Unpack(o);
}
int64_t integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised();
    return v;
}
void require(bool ok, const char* what) {
    if (ok) return;
    PyErr_SetString(PyExc_AssertionError, what);
    throw Raised();
}
// The ctypes structure AbsOpts, or None.
struct Opts {
    abs_opts_t value = {0, 0, 0, 0, 0};
    const abs_opts_t* ptr = nullptr;
    explicit Opts(PyObject* o) {
        if (o == Py_None) return;
        Py_buffer view;
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Raised();
        const bool fits = view.len == (Py_ssize_t)sizeof(value);
        if (fits) memcpy(&value, view.buf, sizeof(value));
        PyBuffer_Release(&view);
        if (!fits) {
            PyErr_SetString(PyExc_TypeError, "opts: not an AbsOpts structure");
            throw Raised();
        }
        ptr = &value;
    }
};
// The stream a call's kernels run on, with the guard of the tensor's device in force.  What a call allocates comes from the
// current stream's pool.  Where the caller names another stream, the allocator is told that it is used there (a workspace that is
// released when the call returns, or an output that is dropped, must not be handed out again while the kernels are pending), and
// fills run there too, before the kernels.
class Work {
    // Whether the call's outputs are allocated through the dispatcher, which is a third of the 0.9 us that at::empty takes (a quantize call allocates three tensors): where
    // somebody listens there (dispatch modes, fake tensors, transforms and tracers put a key of their own into the thread's set; profilers
    // record the operator), or deterministic algorithms are asked for, with which at::empty fills what it allocates.
    static bool dispatched() {
        const c10::DispatchKeySet keys = c10::impl::tls_local_dispatch_key_set().included_;
        return !(keys - c10::default_included_set).empty() || at::hasCallbacks() || at::globalContext().deterministicAlgorithms();
    }
    c10::Device device;
    bool other = false;                  // not the current stream
    const bool dispatch = dispatched();

    c10::cuda::CUDAStream torch_stream() const { return c10::cuda::getStreamFromExternal((cudaStream_t)stream, device.index()); }

  public:
    void* stream;
    Work(PyObject* o, c10::Device d) : device(d) {
        void* const current = (void*)c10::cuda::getCurrentCUDAStream(device.index()).stream();
        stream = current;
        if (o == Py_None) return;
        PyObject* s = PyObject_GetAttrString(o, "cuda_stream");
        if (!s) throw Raised();
        stream = PyLong_AsVoidPtr(s);
        Py_DECREF(s);
        if (!stream && PyErr_Occurred()) throw Raised();
        other = stream != current;
    }
    at::Tensor empty(at::IntArrayRef sizes, at::ScalarType type) const {
        at::Tensor t = dispatch ? at::empty(sizes, at::TensorOptions().dtype(type).device(device))
                                : at::Tensor(at::detail::empty_cuda(sizes, type, device, std::nullopt));
        if (other && t.numel() > 0) c10::cuda::CUDACachingAllocator::recordStream(t.storage().data_ptr(), torch_stream());
        return t;
    }
    at::Tensor zeros(at::IntArrayRef sizes, at::ScalarType type) const {
        at::Tensor t = empty(sizes, type);
        if (!other) return t.zero_();
        const c10::cuda::CUDAStreamGuard on(torch_stream());
        return t.zero_();
    }
    at::Tensor bytes(int64_t n) const { return empty({n}, at::kByte); }
    // One float: the kernels always write the tensor scale of a tensor that has elements, unless it is an input.
    at::Tensor tensor_scale(PyObject* o, bool written) const {
        if (o != Py_None) return tensor(o, "tensor_scale");
        return written ? empty({1}, at::kFloat) : zeros({1}, at::kFloat);
    }
};
at::Tensor given_or(PyObject* o, const char* what, const std::function<at::Tensor()>& make) { return o == Py_None ? make() : tensor(o, what); }
int bits_of(int64_t fmt) {
    switch (fmt) {
        case ABS_FMT_NVFP4: case ABS_FMT_IF4: case ABS_FMT_NVFP4_BS8: case ABS_FMT_IF4_BS8: return 4;
        case ABS_FMT_IF3: case ABS_FMT_IF3_BS8: return 3;
        case ABS_FMT_IF6_E2M3: case ABS_FMT_IF6_E3M2: return 6;
        default: return 0;
    }
}
int group_of(int64_t fmt) { return fmt >= ABS_FMT_NVFP4_BS8 ? 8 : 16; }
int known_bits(int64_t fmt) {
    const int b = bits_of(fmt);
    if (!b) {
        PyErr_Format(PyExc_KeyError, "%lld", (long long)fmt);
        throw Raised();
    }
    return b;
}
at::Tensor input_matrix(PyObject* o) {
    at::Tensor x = tensor(o, "x");
    require(x.is_cuda() && x.scalar_type() == at::kBFloat16 && x.dim() == 2 && x.is_contiguous(),
            "x: a contiguous two-dimensional bfloat16 CUDA tensor");
    return x;
}
template <typename F> abs_status_t unlocked(F call) {
    abs_status_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return rc;
}
PyObject* result(abs_status_t rc, std::initializer_list<at::Tensor> tensors) {
    PyObject* t = PyTuple_New(1 + (Py_ssize_t)tensors.size());
    if (!t) throw Raised();
    PyTuple_SET_ITEM(t, 0, PyLong_FromLong((long)rc));
    Py_ssize_t i = 1;
    for (const at::Tensor& x : tensors) PyTuple_SET_ITEM(t, i++, THPVariable_Wrap(x));
    return t;
}
bool count(Py_ssize_t have, Py_ssize_t want) {
    if (have == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, have);
    return false;
}

// Every function body: C++ exceptions (an allocation that fails, say) become Python exceptions.
#define ABS_CALL_BEGIN(N)          \
    if (!count(n, N)) return nullptr; \
    HANDLE_TH_ERRORS               \
    try {
#define ABS_CALL_END               \
    } catch (const Raised&) {      \
        return nullptr;            \
    }                              \
    END_HANDLE_TH_ERRORS

// (addresses of the nine functions of Entry, in its order)
PyObject* init(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ABS_CALL_BEGIN(9)
    void** f = reinterpret_cast<void**>(&entry);
    static_assert(sizeof(Entry) == 9 * sizeof(void*), "nine addresses");
    for (int i = 0; i < 9; ++i) {
        f[i] = PyLong_AsVoidPtr(a[i]);
        if (!f[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null address");
            throw Raised();
        }
    }
    Py_RETURN_NONE;
    ABS_CALL_END
}

// (fmt, x, codes, scales, tensor_scale, opts, stream) -> (status, codes, scales, tensor_scale)
PyObject* quantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ABS_CALL_BEGIN(7)
    const int64_t fmt = integer(a[0]);
    const at::Tensor x = input_matrix(a[1]);
    const Opts opts(a[5]);
    const int64_t rows = x.size(0), cols = x.size(1);
    const c10::Device dev = x.device();
    const c10::cuda::CUDAGuard guard(dev);
    const Work work(a[6], dev);
    const at::Tensor codes = given_or(a[2], "codes", [&] { return work.bytes(std::max<int64_t>(cols % 16 == 0 ? rows * cols / 16 * (2 * bits_of(fmt)) : 0, 1)); });
    const at::Tensor scales = given_or(a[3], "scales", [&] {
        if (opts.value.flags & ABS_F_SCALES_SWIZZLED)
            return work.zeros({std::max<int64_t>((int64_t)entry.scales_bytes_swizzled((abs_fmt_t)fmt, rows, cols), 1)}, at::kByte);
        known_bits(fmt);
        return work.bytes(std::max<int64_t>(rows * cols / group_of(fmt), 1));
    });
    const bool written = rows * cols > 0 && cols % 16 == 0 && bits_of(fmt) && !(opts.value.flags & ABS_F_ALPHA_GIVEN);
    const at::Tensor ts = work.tensor_scale(a[4], written);
    void *px = x.data_ptr(), *pc = codes.data_ptr(), *ps = scales.data_ptr(), *s = work.stream;
    float* pt = (float*)ts.data_ptr();
    return result(unlocked([&] { return entry.quantize((abs_fmt_t)fmt, px, rows, cols, pc, ps, pt, opts.ptr, s); }), {codes, scales, ts});
    ABS_CALL_END
}

// The same arguments and result.
PyObject* quantize_transposed(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ABS_CALL_BEGIN(7)
    const int64_t fmt = integer(a[0]);
    const at::Tensor x = input_matrix(a[1]);
    const Opts opts(a[5]);
    const int64_t rows = x.size(0), cols = x.size(1);
    const c10::Device dev = x.device();
    const c10::cuda::CUDAGuard guard(dev);
    const Work work(a[6], dev);
    const at::Tensor codes = given_or(a[2], "codes_t", [&] { return work.bytes(std::max<int64_t>(rows * cols * known_bits(fmt) / 8, 1)); });
    const at::Tensor scales = given_or(a[3], "scales_t", [&] { return work.bytes(std::max<int64_t>(rows * cols / 16, 1)); });
    const bool written = rows * cols > 0 && rows % 16 == 0 && cols % 16 == 0 && !(opts.value.flags & ABS_F_ALPHA_GIVEN);
    const at::Tensor ts = work.tensor_scale(a[4], written);
    void *px = x.data_ptr(), *pc = codes.data_ptr(), *ps = scales.data_ptr(), *s = work.stream;
    float* pt = (float*)ts.data_ptr();
    return result(unlocked([&] { return entry.quantize_transposed((abs_fmt_t)fmt, px, rows, cols, pc, ps, pt, opts.ptr, s); }),
                  {codes, scales, ts});
    ABS_CALL_END
}

// (fmt, x, out, codes, scales, tensor_scale, opts, stream) -> (status, out, tensor_scale); codes and scales optional outputs
PyObject* quantize_dequantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ABS_CALL_BEGIN(8)
    const int64_t fmt = integer(a[0]);
    const at::Tensor x = input_matrix(a[1]);
    const Opts opts(a[6]);
    const int64_t rows = x.size(0), cols = x.size(1);
    const c10::Device dev = x.device();
    const c10::cuda::CUDAGuard guard(dev);
    const Work work(a[7], dev);
    const at::Tensor out = given_or(a[2], "out", [&] { return work.empty({rows, cols}, at::kBFloat16); });
    void* pc = a[3] == Py_None ? nullptr : tensor(a[3], "codes").data_ptr();
    void* ps = a[4] == Py_None ? nullptr : tensor(a[4], "scales").data_ptr();
    const bool written = rows * cols > 0 && cols % 16 == 0 && bits_of(fmt) && !(opts.value.flags & ABS_F_ALPHA_GIVEN);
    const at::Tensor ts = work.tensor_scale(a[5], written);
    void *px = x.data_ptr(), *po = out.data_ptr(), *s = work.stream;
    float* pt = (float*)ts.data_ptr();
    return result(unlocked([&] { return entry.quantize_dequantize((abs_fmt_t)fmt, px, rows, cols, po, pc, ps, pt, opts.ptr, s); }), {out, ts});
    ABS_CALL_END
}

// (fmt, codes, scales, tensor_scale, rows, cols, out, opts, stream) -> (status, out)
PyObject* dequantize(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ABS_CALL_BEGIN(9)
    const int64_t fmt = integer(a[0]), rows = integer(a[4]), cols = integer(a[5]);
    const at::Tensor codes = tensor(a[1], "codes"), scales = tensor(a[2], "scales"), ts = tensor(a[3], "tensor_scale");
    const Opts opts(a[7]);
    const c10::Device dev = codes.device();
    const c10::cuda::OptionalCUDAGuard guard(dev);      // a tensor that is not on a GPU raises
    const Work work(a[8], dev);
    const at::Tensor out = given_or(a[6], "out", [&] { return work.empty({rows, cols}, opts.value.flags & ABS_F_OUT_FP32 ? at::kFloat : at::kBFloat16); });
    void *pc = codes.data_ptr(), *ps = scales.data_ptr(), *po = out.data_ptr(), *s = work.stream;
    const float* pt = (const float*)ts.data_ptr();
    return result(unlocked([&] { return entry.dequantize((abs_fmt_t)fmt, pc, ps, pt, rows, cols, po, opts.ptr, s); }), {out});
    ABS_CALL_END
}

// (fmt, qa, qb, m, n, k, out, workspace, stream, bf16, next_fmt or None, next_alpha)
//   -> (status, out, workspace[, next_alpha]); status -1 where the shape or format has no workspace size
PyObject* matmul(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ABS_CALL_BEGIN(12)
    const int64_t fmt = integer(a[0]), M = integer(a[3]), N = integer(a[4]), K = integer(a[5]);
    at::Tensor q[6];
    for (int op = 0; op < 2; ++op) {
        PyObject* t = PySequence_Fast(a[1 + op], "a quantized operand is (codes, scales, alpha)");
        if (!t) throw Raised();
        const bool three = PySequence_Fast_GET_SIZE(t) >= 3;
        try {
            for (int i = 0; three && i < 3; ++i) q[3 * op + i] = tensor(PySequence_Fast_GET_ITEM(t, i), "a quantized operand");
        } catch (...) {
            Py_DECREF(t);
            throw;
        }
        Py_DECREF(t);
        if (!three) {
            PyErr_SetString(PyExc_IndexError, "a quantized operand is (codes, scales, alpha)");
            throw Raised();
        }
    }
    const int64_t need = (int64_t)entry.matmul_workspace_bytes((abs_fmt_t)fmt, M, N, K);
    if (need == 0) return result((abs_status_t)-1, {});
    const int bf16 = PyObject_IsTrue(a[9]);
    if (bf16 < 0) throw Raised();
    const c10::Device dev = q[0].device();
    const c10::cuda::OptionalCUDAGuard guard(dev);
    const Work work(a[8], dev);
    const at::Tensor ws = given_or(a[7], "workspace", [&] { return work.bytes(need + 1024); });
    const at::Tensor out = given_or(a[6], "out", [&] { return work.empty({M, N}, bf16 ? at::kBFloat16 : at::kFloat); });
    require(out.scalar_type() == (bf16 ? at::kBFloat16 : at::kFloat), "out: float32, or bfloat16 with bf16");
    const int64_t off = (int64_t)((0 - (uintptr_t)ws.data_ptr()) & 1023u);
    void *pw = (uint8_t*)ws.data_ptr() + off, *po = out.data_ptr(), *s = work.stream;
    const size_t ws_bytes = (size_t)std::max<int64_t>(ws.numel() - off, 0);
    void* p[6];
    for (int i = 0; i < 6; ++i) p[i] = q[i].data_ptr();
    if (a[10] != Py_None) {
        require(bf16, "next_fmt: bf16 output only");
        const int64_t next_fmt = integer(a[10]);
        const at::Tensor next = work.tensor_scale(a[11], true);
        float* pn = (float*)next.data_ptr();
        return result(unlocked([&] {
                          return entry.matmul_bf16_scaled((abs_fmt_t)fmt, p[0], p[1], (const float*)p[2], p[3], p[4], (const float*)p[5], M, N, K,
                                                          po, (abs_fmt_t)next_fmt, pn, pw, ws_bytes, s);
                      }), {out, ws, next});
    }
    return result(unlocked([&] {
                      return bf16 ? entry.matmul_bf16((abs_fmt_t)fmt, p[0], p[1], (const float*)p[2], p[3], p[4], (const float*)p[5], M, N, K, po, pw,
                                                      ws_bytes, s)
                                  : entry.matmul((abs_fmt_t)fmt, p[0], p[1], (const float*)p[2], p[3], p[4], (const float*)p[5], M, N, K, (float*)po,
                                                 pw, ws_bytes, s);
                  }), {out, ws});
    ABS_CALL_END
}

#define ABS_METHOD(F) {#F, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(F)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {ABS_METHOD(init), ABS_METHOD(quantize), ABS_METHOD(quantize_transposed), ABS_METHOD(quantize_dequantize),
                         ABS_METHOD(dequantize), ABS_METHOD(matmul), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_abs_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__abs_call() { return PyModule_Create(&module); }
