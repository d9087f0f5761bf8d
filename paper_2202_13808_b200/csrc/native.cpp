// Python binding of the calls that a training step makes, as a native module: argument checks, output and scratch tensors,
// stream lookup and the autograd node of GELU + Linear in C++, on top of the C ABI in include/dropit.h.  A layer call is tens
// of microseconds of GPU time, less than what marshalling the same calls through ctypes takes on the host.
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/extension.h>

#include <mutex>
#include <tuple>
#include <vector>

#include "dropit.h"
#include "layer_ops.h"

namespace {

using at::Tensor;

py::object* g_error_class = nullptr;

// A status that is not OK becomes the package's DropITError.  It travels as a python_error, which is a std::exception: the autograd
// engine hands those from the thread of a backward pass to the caller, anything else that leaves a node ends the process.
void check(dropit_status s, const char* where) {
    if (s == DROPIT_OK) return;
    py::gil_scoped_acquire gil;
    PyErr_SetObject(g_error_class ? g_error_class->ptr() : PyExc_RuntimeError, py::make_tuple((int)s, where).ptr());
    python_error error;
    error.persist();
    throw error;
}

std::string type_name(const Tensor& t) { return "torch." + c10::getDtypeNames(t.scalar_type()).first; }
dropit_dtype dtype_code(const Tensor& t, const char* name) {
    if (t.scalar_type() == at::kBFloat16) return DROPIT_BF16;
    if (t.scalar_type() == at::kFloat) return DROPIT_F32;
    throw py::type_error(std::string(name) + ": dtype " + type_name(t) + " is not supported (bf16 or fp32)");
}
dropit_dtype require_cuda(const Tensor& t, const char* name) {
    if (!t.is_cuda()) throw py::value_error(std::string(name) + " must be a CUDA tensor (there is no CPU path)");
    if (!t.is_contiguous()) throw py::value_error(std::string(name) + " must be contiguous");
    return dtype_code(t, name);
}
void require_bf16(const Tensor& t, const char* where) {
    if (t.scalar_type() != at::kBFloat16) throw py::type_error(std::string(where) + " takes bf16 tensors");
}

Tensor empty1(int64_t n, at::ScalarType type, const Tensor& like) {
    return at::detail::empty_cuda({n}, type, like.device(), c10::nullopt);
}
void* ptr(const Tensor& t) { return t.defined() && t.numel() ? t.data_ptr() : nullptr; }
void* table_ptr(const c10::optional<Tensor>& t) { return t.has_value() ? ptr(*t) : nullptr; }
void* current_stream(const Tensor& t) { return c10::cuda::getCurrentCUDAStream(t.device().index()).stream(); }

// One status word per device, which every kernel's bounded waits report to.
Tensor status_word(int64_t device) {
    static std::mutex lock;
    static auto* words = new std::vector<Tensor>();      // never destroyed: the CUDA context may be gone by then
    std::lock_guard<std::mutex> guard(lock);
    if ((int64_t)words->size() <= device) words->resize(device + 1);
    Tensor& w = (*words)[device];
    if (!w.defined()) w = at::zeros({4}, at::TensorOptions().dtype(at::kInt).device(at::kCUDA, (c10::DeviceIndex)device));
    return w;
}
int32_t* status_ptr(const Tensor& like) { return status_word(like.device().index()).data_ptr<int32_t>(); }

// The caller's scratch if it is large enough, else a new one.
Tensor scratch(const c10::optional<Tensor>& given, size_t bytes, const Tensor& like) {
    if (given.has_value() && given->defined() && (size_t)given->numel() >= bytes) return *given;
    return empty1(bytes > 16 ? (int64_t)bytes : 16, at::kByte, like);
}

struct CacheParts {
    Tensor values, meta, offsets;
    int64_t k;
    size_t workspace;
};
CacheParts make_cache(const Tensor& x, dropit_dtype dt, double gamma, int fmt) {
    size_t vb, mb, ob, wb;
    const int64_t n = x.numel();
    check(dropit_cache_sizes(n, gamma, dt, (dropit_format)fmt, &vb, &mb, &ob, &wb), "dropit_cache_sizes");
    CacheParts c;
    c.k = dropit_keep_count(n, gamma);
    c.values = empty1((int64_t)(vb / (dt == DROPIT_BF16 ? 2 : 4)), x.scalar_type(), x);
    c.meta = empty1((int64_t)(mb / 4), at::kInt, x);
    c.offsets = empty1((int64_t)(ob / 4), at::kInt, x);
    c.workspace = wb;
    return c;
}

using CacheTuple = std::tuple<Tensor, Tensor, Tensor, int64_t>;

CacheTuple compress(const Tensor& x, double gamma, int fmt, const c10::optional<Tensor>& workspace) {
    const dropit_dtype dt = require_cuda(x, "x");
    c10::cuda::CUDAGuard guard(x.device());
    CacheParts c = make_cache(x, dt, gamma, fmt);
    const Tensor ws = scratch(workspace, c.workspace, x);
    check(dropit_compress(ptr(x), x.numel(), gamma, dt, (dropit_format)fmt, ptr(c.values), ptr(c.meta), (uint32_t*)ptr(c.offsets),
                          ptr(ws), (size_t)ws.numel(), status_ptr(x), current_stream(x)), "dropit_compress");
    return {c.values, c.meta, c.offsets, c.k};
}

std::tuple<Tensor, Tensor> produce(const Tensor& x, double gamma, int act, const c10::optional<Tensor>& table, bool want_y) {
    require_cuda(x, "x");
    require_bf16(x, "dropit_produce");
    c10::cuda::CUDAGuard guard(x.device());
    size_t bytes;
    check(dropit_produce_workspace(x.numel(), &bytes), "dropit_produce_workspace");
    Tensor y;
    if (want_y) y = at::empty_like(x);
    Tensor prep = empty1(bytes > 16 ? (int64_t)bytes : 16, at::kByte, x);
    check(dropit_produce(ptr(x), x.numel(), gamma, (dropit_activation)act, table.has_value() ? (const uint16_t*)ptr(*table) : nullptr,
                         ptr(y), ptr(prep), (size_t)prep.numel(), current_stream(x)), "dropit_produce");
    return {y, prep};
}

CacheTuple compress_prepared(const Tensor& y, double gamma, const Tensor& prep, int fmt, const c10::optional<Tensor>& workspace) {
    require_cuda(y, "y");
    require_bf16(y, "dropit_compress_prepared");
    c10::cuda::CUDAGuard guard(y.device());
    CacheParts c = make_cache(y, DROPIT_BF16, gamma, fmt);
    const Tensor ws = scratch(workspace, c.workspace, y);
    check(dropit_compress_prepared(ptr(y), y.numel(), gamma, (dropit_format)fmt, ptr(c.values), ptr(c.meta), (uint32_t*)ptr(c.offsets),
                                   ptr(prep), (size_t)prep.numel(), ptr(ws), (size_t)ws.numel(), status_ptr(y), current_stream(y)),
          "dropit_compress_prepared");
    return {c.values, c.meta, c.offsets, c.k};
}

std::string mismatch(const Tensor& dy, const Tensor& values) {
    return "dy dtype " + type_name(dy) + " != cache dtype " + type_name(values);
}

// `offsets` may be absent: a coordinate cache can do without its seek table.
Tensor weight_grad(const Tensor& dy, const Tensor& values, const Tensor& meta, const c10::optional<Tensor>& offsets, int64_t n, int64_t Ca,
                   int64_t k, int fmt, const c10::optional<Tensor>& out, bool accumulate, const c10::optional<Tensor>& workspace, bool no_scratch) {
    const dropit_dtype dt = require_cuda(dy, "dy");
    if (dy.scalar_type() != values.scalar_type()) throw py::type_error(mismatch(dy, values));
    const int64_t M = Ca ? n / Ca : 0, Cz = dy.size(-1);
    if (dy.numel() != M * Cz)
        throw py::value_error("dy has " + std::to_string(dy.numel()) + " elements, expected " + std::to_string(M) + " x " + std::to_string(Cz));
    if (!out.has_value() && accumulate) throw py::value_error("accumulate=True needs out");
    c10::cuda::CUDAGuard guard(dy.device());
    const Tensor dw = out.has_value() ? *out : Tensor(at::detail::empty_cuda({Cz, Ca}, at::kFloat, dy.device(), c10::nullopt));
    size_t bytes;
    check(dropit_weight_grad_workspace(M, Ca, Cz, dt, (dropit_format)fmt, &bytes), "dropit_weight_grad_workspace");
    const Tensor ws = scratch(workspace, bytes, dy);
    auto fn = no_scratch ? dropit_weight_grad_fused : dropit_weight_grad;
    check(fn(ptr(dy), ptr(values), ptr(meta), (const uint32_t*)table_ptr(offsets), M, Ca, Cz, k, dt, (dropit_format)fmt, (float*)ptr(dw),
             accumulate ? 1 : 0, ptr(ws), (size_t)ws.numel(), status_ptr(dy), current_stream(dy)),
          no_scratch ? "dropit_weight_grad_fused" : "dropit_weight_grad");
    return dw;
}

Tensor conv_weight_grad(const Tensor& dy, const Tensor& values, const Tensor& meta, const c10::optional<Tensor>& offsets, int B, int Ca, int H,
                        int W, int R, int S, int stride, int pad, int dilation, int64_t k, int fmt, const c10::optional<Tensor>& out,
                        bool accumulate, const c10::optional<Tensor>& workspace) {
    const dropit_dtype dt = require_cuda(dy, "dy");
    if (dy.scalar_type() != values.scalar_type()) throw py::type_error(mismatch(dy, values));
    const int Cz = (int)dy.size(1);
    if (!out.has_value() && accumulate) throw py::value_error("accumulate=True needs out");
    c10::cuda::CUDAGuard guard(dy.device());
    const Tensor dw = out.has_value() ? *out : Tensor(at::detail::empty_cuda({Cz, Ca, R, S}, at::kFloat, dy.device(), c10::nullopt));
    size_t bytes;
    check(dropit_conv_weight_grad_workspace(B, Ca, H, W, Cz, R, S, stride, pad, dt, (dropit_format)fmt, &bytes),
          "dropit_conv_weight_grad_workspace");
    const Tensor ws = scratch(workspace, bytes, dy);
    check(dropit_conv_weight_grad(ptr(dy), ptr(values), ptr(meta), (const uint32_t*)table_ptr(offsets), B, Ca, H, W, Cz, R, S, stride, pad,
                                  dilation, k, dt, (dropit_format)fmt, (float*)ptr(dw), accumulate ? 1 : 0, ptr(ws),
                                  (size_t)ws.numel(), status_ptr(dy), current_stream(dy)), "dropit_conv_weight_grad");
    return dw;
}

// z = GELU(x) W^T + b for bf16 tensors, with the GELU written by the library's producer kernel so that the selection statistics
// of GELU(x), the tensor the Linear caches, are taken while it is written (Sec. 3.5: the activation keeps its own cache x; only
// the Linear's cache is replaced by D(GELU(x))).
struct GeluLinear : public torch::autograd::Function<GeluLinear> {
    static Tensor forward(torch::autograd::AutogradContext* ctx, const Tensor& x, const Tensor& weight, const c10::optional<Tensor>& bias,
                          double gamma, int64_t fmt, const Tensor& table) {
        const Tensor x2 = x.reshape({-1, x.size(-1)}).contiguous();
        Tensor y, prep;
        std::tie(y, prep) = produce(x2, gamma, DROPIT_ACT_TABLE, table, true);
        std::vector<int64_t> shape = x.sizes().vec();
        shape.back() = weight.size(0);
        Tensor z = at::linear(y, weight, bias).reshape(shape);
        Tensor values, meta, offsets;
        int64_t k;
        std::tie(values, meta, offsets, k) = compress_prepared(y, gamma, prep, (int)fmt, c10::nullopt);
        ctx->save_for_backward({x2, weight, values, meta, offsets});
        ctx->saved_data["cache"] = std::vector<int64_t>{y.numel(), y.size(1), k, fmt};
        ctx->saved_data["shape"] = x.sizes().vec();
        ctx->saved_data["bias"] = bias.has_value() && bias->defined();
        return z;
    }
    static torch::autograd::variable_list backward(torch::autograd::AutogradContext* ctx, torch::autograd::variable_list grads) {
        const auto saved = ctx->get_saved_variables();
        const Tensor &x2 = saved[0], &weight = saved[1], &values = saved[2];
        const auto cache = ctx->saved_data["cache"].toIntVector();
        const Tensor dz2 = grads[0].reshape({-1, grads[0].size(-1)}).contiguous();
        const bool bias = ctx->saved_data["bias"].toBool() && ctx->needs_input_grad(2);
        // With create_graph the gradients are to be differentiated again: what can be is then formed by operations that autograd knows.
        const bool graph = at::GradMode::is_enabled();
        Tensor dx, dw, db;
        if (ctx->needs_input_grad(0)) {                                  // Eq. 3: exact, needs theta only; the activation's cache is x
            const Tensor dy = at::matmul(dz2, weight);
            if (!graph && dy.scalar_type() == at::kBFloat16 && x2.scalar_type() == at::kBFloat16 && dy.is_contiguous() &&
                reinterpret_cast<uintptr_t>(x2.data_ptr()) % 16 == 0) {
                c10::cuda::CUDAGuard guard(dy.device());
                dx = at::empty_like(x2);
                check(dropit::gelu_backward_bf16(ptr(dy), ptr(x2), ptr(dx), x2.numel(), current_stream(dy)), "gelu_backward");
            } else {
                dx = at::gelu_backward(dy, x2);
            }
            dx = dx.reshape(ctx->saved_data["shape"].toIntVector());
        }
        const bool own = !graph && weight.scalar_type() == at::kBFloat16 && dz2.scalar_type() == at::kBFloat16 && dz2.size(1) % 8 == 0 &&
                         dz2.numel() != 0 && reinterpret_cast<uintptr_t>(dz2.data_ptr()) % 16 == 0;
        if (ctx->needs_input_grad(1)) {                                  // Eq. 6
            const Tensor full = weight_grad(dz2.to(values.scalar_type()), values, saved[3], saved[4], cache[0], cache[1], cache[2],
                                            (int)cache[3], c10::nullopt, false, c10::nullopt, false);
            if (own) {                                                   // rounded to the parameter's type together with the bias gradient
                c10::cuda::CUDAGuard guard(dz2.device());
                dw = at::detail::empty_cuda(full.sizes(), at::kBFloat16, full.device(), c10::nullopt);
                if (bias) db = empty1(dz2.size(1), at::kBFloat16, dz2);
                check(dropit::finish_linear_backward((const float*)ptr(full), ptr(dw), full.numel(), ptr(dz2), dz2.size(0), dz2.size(1),
                                                     bias ? ptr(db) : nullptr, current_stream(dz2)), "finish_linear_backward");
            } else {
                dw = full.to(weight.scalar_type());
            }
        }
        if (bias && !db.defined()) db = dz2.sum(0);
        return {dx, dw, db, Tensor(), Tensor(), Tensor()};
    }
};

Tensor gelu_linear(const Tensor& x, const Tensor& weight, const c10::optional<Tensor>& bias, double gamma, int64_t fmt, const Tensor& table) {
    return GeluLinear::apply(x, weight, bias, gamma, fmt, table);
}

}  // namespace

PYBIND11_MODULE(_native, m) {
    py::register_exception_translator([](std::exception_ptr p) {
        try {
            if (p) std::rethrow_exception(p);
        } catch (python_error& e) {
            e.restore();
        }
    });
    m.def("set_error_class", [](py::object cls) { g_error_class = new py::object(cls); });
    // Without the interpreter's lock, as a call through ctypes is: a launch can wait for room in the stream's queue.
    m.def("status_word", torch::wrap_pybind_function_no_gil(status_word));
    m.def("compress", torch::wrap_pybind_function_no_gil(compress));
    m.def("produce", torch::wrap_pybind_function_no_gil(produce));
    m.def("compress_prepared", torch::wrap_pybind_function_no_gil(compress_prepared));
    m.def("weight_grad", torch::wrap_pybind_function_no_gil(weight_grad));
    m.def("conv_weight_grad", torch::wrap_pybind_function_no_gil(conv_weight_grad));
    m.def("gelu_linear", torch::wrap_pybind_function_no_gil(gelu_linear));
}
