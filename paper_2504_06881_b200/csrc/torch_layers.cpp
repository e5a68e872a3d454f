// The layers' autograd path in native code: one call from Python runs a layer's forward (allocation, argument
// checks, library call) and records a C++ autograd node whose backward does the same for the gradients.  A
// small layer's pass is host time: with a Python autograd Function the two RGB images of the small training
// configuration took 155 us for 26 us of kernels.
#include <ATen/TracerMode.h>
#include <ATen/cuda/CUDAContext.h>
#include <c10/cuda/CUDAGuard.h>
#include <torch/csrc/Exceptions.h>
#include <torch/extension.h>

#include <array>
#include <optional>
#include <string>
#include <vector>

#include "tconv.h"
#include "tconv3d.h"

namespace {

using at::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::Variable;
using torch::autograd::variable_list;

PyObject* g_error = nullptr;   // the binding's TconvError(status, where)

// Raises TconvError; callable without the GIL (the autograd engine's threads).
[[noreturn]] void fail(int rc, const char* where) {
    pybind11::gil_scoped_acquire gil;
    pybind11::object e = pybind11::reinterpret_borrow<pybind11::object>(g_error)(rc, where);
    PyErr_SetObject(g_error, e.ptr());
    python_error err;
    err.persist();
    throw std::move(err);
}

enum Kind { kDense = 0, kDepthwise = 1, kVolume = 2 };

// What a layer module fixes: kind, mode, channel combine, type, and stride / padding / dilation per axis.
struct Geom {
    int kind, mode, chan, dtype;
    std::array<int, 3> stride, pad, dil;     // dense, depthwise: [height, width]
};

struct Desc {
    tconv_desc_t d2;
    tconv3d_desc_t d3;
    std::array<int64_t, 5> y;                // output shape
    int dims;
    at::IntArrayRef out() const { return at::IntArrayRef(y.data(), dims); }
};

at::ScalarType type_of(const Geom& g) { return g.dtype == TCONV_F32 ? at::kFloat : at::kBFloat16; }

Desc make_desc(const Geom& g, const Tensor& x, const Tensor& w) {
    Desc d;
    const int nd = g.kind == kVolume ? 5 : 4;
    TORCH_CHECK_VALUE(x.dim() == nd, "x: need a tensor of ", nd, " dimensions, got ", x.dim());
    const auto i = [](int64_t v) {
        TORCH_CHECK_VALUE(v <= INT32_MAX, "a size exceeds 31 bits");
        return (int32_t)v;
    };
    d.dims = nd;
    if (g.kind == kVolume) {
        d.d3 = tconv3d_desc_t{i(x.size(0)), i(x.size(1)), i(x.size(2)), i(x.size(3)), i(x.size(4)), i(w.size(0)), i(w.size(2)),
                              i(w.size(3)), i(w.size(4)), g.stride[0], g.stride[1], g.stride[2], g.pad[0], g.pad[1], g.pad[2],
                              g.dil[0], g.dil[1], g.dil[2], g.mode, g.chan, g.dtype};
        int32_t od, oh, ow;
        if (const int rc = tconv3d_output_shape(&d.d3, &od, &oh, &ow)) fail(rc, "tconv3d_output_shape");
        d.y = {x.size(0), w.size(0), od, oh, ow};
    } else {
        const bool dw = g.kind == kDepthwise;
        d.d2 = tconv_desc_t{i(x.size(0)), i(x.size(1)), i(x.size(2)), i(x.size(3)), i(dw ? x.size(1) : w.size(0)),
                            i(w.size(dw ? 1 : 2)), i(w.size(dw ? 2 : 3)), g.stride[0], g.stride[1], g.pad[0], g.pad[1],
                            g.dil[0], g.dil[1], g.mode, g.chan, g.dtype, TCONV_PAD_ZERO, TCONV_X_SAME};
        int32_t oh, ow;
        if (const int rc = tconv_output_shape(&d.d2, &oh, &ow)) fail(rc, "tconv_output_shape");
        d.y = {x.size(0), d.d2.K, oh, ow, 0};
    }
    return d;
}

Tensor as(const Tensor& t, at::ScalarType type) {
    if (!t.defined()) return t;
    return (t.scalar_type() == type ? t : t.to(type)).contiguous();
}
void check(const Tensor& t, at::IntArrayRef shape, const char* name) {
    if (!t.defined()) return;
    TORCH_CHECK_VALUE(t.is_cuda() && t.sizes() == shape, name, ": need a contiguous CUDA tensor of shape ", shape, ", got ",
                      t.sizes(), " on ", t.device());
}
// A tensor of the backward: saved-tensor hooks may hand back another one than the forward kept.
void check_saved(const Tensor& t, const at::Device& dev, at::ScalarType type, at::IntArrayRef shape, const char* name) {
    if (!t.defined()) return;
    TORCH_CHECK_VALUE(t.is_cuda() && t.device() == dev && t.scalar_type() == type && t.is_contiguous() && t.sizes() == shape, name,
                      ": need the contiguous ", type, " tensor of shape ", shape, " on ", dev, " that the forward saved, got ",
                      t.scalar_type(), " ", t.sizes(), " on ", t.device());
}
void* ptr(const Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }
float* fptr(const Tensor& t) { return t.defined() ? t.data_ptr<float>() : nullptr; }
void* stream() { return (void*)at::cuda::getCurrentCUDAStream().stream(); }

Tensor given(const std::optional<Tensor>& t) { return t ? *t : Tensor(); }

struct Saved {
    Tensor x, w, w2, alpha, beta, winners;
};

// The layer's forward.  want: leave the winners for a backward.  Fills the tensors the backward needs.
Tensor run_forward(const Geom& g, const Tensor& x, const Tensor& w, const Tensor& w2, const Tensor& alpha, const Tensor& beta,
                   const Tensor& bias, bool want, Saved& s) {
    const auto dt = type_of(g);
    const Desc d = make_desc(g, x, w);
    TORCH_CHECK_VALUE(x.is_cuda(), "x: need a CUDA tensor, got one on ", x.device());
    c10::cuda::CUDAGuard guard(x.device());
    s.x = as(x, dt);
    s.w = as(w, dt);
    s.w2 = as(w2, dt);
    s.alpha = as(alpha, at::kFloat);
    s.beta = as(beta, at::kFloat);
    const Tensor b = as(bias, at::kFloat);
    const int64_t K = d.y[1], C = x.size(1);
    if (g.kind == kDepthwise) {
        const int64_t ws[3] = {C, w.size(1), w.size(2)}, ks[1] = {C};
        check(s.w, ws, "w"); check(s.w2, ws, "w2"); check(s.alpha, ks, "alpha"); check(s.beta, ks, "beta"); check(b, ks, "bias");
    } else {
        const int64_t ws[5] = {K, C, w.size(2), w.size(3), g.kind == kVolume ? w.size(4) : 0}, kc[2] = {K, C}, ks[1] = {K};
        const at::IntArrayRef wshape(ws, g.kind == kVolume ? 5 : 4);
        check(s.w, wshape, "w"); check(s.w2, wshape, "w2"); check(s.alpha, kc, "alpha"); check(s.beta, kc, "beta"); check(b, ks, "bias");
    }
    const auto opt = s.x.options();
    Tensor y = at::empty(d.out(), opt);
    int rc;
    const char* where;
    if (g.kind == kVolume) {
        if (want) s.winners = at::empty({(int64_t)tconv3d_winner_bytes(&d.d3)}, opt.dtype(at::kByte));
        where = "tconv3d_forward";
        rc = tconv3d_forward(&d.d3, ptr(s.x), ptr(s.w), ptr(s.w2), fptr(s.alpha), fptr(s.beta), fptr(b), ptr(y), ptr(s.winners), stream());
    } else if (g.kind == kDepthwise) {
        if (want) s.winners = at::empty({(int64_t)tconv_dw_winner_bytes(&d.d2)}, opt.dtype(at::kByte));
        where = "tconv_dw_forward";
        rc = tconv_dw_forward(&d.d2, ptr(s.x), ptr(s.w), ptr(s.w2), fptr(s.alpha), fptr(s.beta), fptr(b), ptr(y), ptr(s.winners), stream());
    } else {
        if (want) s.winners = at::empty({(int64_t)tconv_winner_bytes(&d.d2)}, opt.dtype(at::kByte));
        const size_t nws = tconv_workspace_bytes(&d.d2, 0);
        Tensor ws;
        if (nws) ws = at::empty({(int64_t)nws}, opt.dtype(at::kByte));
        where = "tconv_forward";
        rc = tconv_forward(&d.d2, ptr(s.x), ptr(s.w), ptr(s.w2), fptr(s.alpha), fptr(s.beta), fptr(b), ptr(y), ptr(s.winners), ptr(ws),
                           nws, stream());
    }
    if (rc) fail(rc, where);
    return y;
}

struct Grads {
    Tensor x, w, w2, alpha, beta, bias;
};

Grads run_backward(const Geom& g, const Saved& s, const Tensor& gy_in, bool need_x) {
    const at::Device dev = s.x.device();
    const auto dt = type_of(g);
    const int wd = g.kind == kVolume ? 5 : g.kind == kDense ? 4 : 3;
    TORCH_CHECK_VALUE(dev.is_cuda(), "x: need the CUDA tensor that the forward saved, got one on ", dev);
    TORCH_CHECK_VALUE(s.w.dim() == wd, "w: need the tensor of ", wd, " dimensions that the forward saved, got ", s.w.dim());
    c10::cuda::CUDAGuard guard(dev);
    const Desc d = make_desc(g, s.x, s.w);
    const Tensor gy = as(gy_in, dt);
    check_saved(gy, dev, dt, d.out(), "grad_y");
    const bool two = g.mode == TCONV_COMPOUND || g.mode == TCONV_PARALLEL, par = g.mode == TCONV_PARALLEL;
    const auto opt = s.x.options(), f32 = opt.dtype(at::kFloat);
    const int64_t K = d.y[1], C = s.x.size(1);
    const int64_t kc[2] = {K, C};
    const at::IntArrayRef scalars = g.kind == kDepthwise ? at::IntArrayRef(kc, 1) : at::IntArrayRef(kc, 2);
    {
        std::vector<int64_t> ws = s.w.sizes().vec();
        ws[0] = K;
        if (g.kind != kDepthwise) ws[1] = C;
        const int64_t wb[1] = {(int64_t)(g.kind == kVolume      ? tconv3d_winner_bytes(&d.d3)
                                         : g.kind == kDepthwise ? tconv_dw_winner_bytes(&d.d2)
                                                                : tconv_winner_bytes(&d.d2))};
        check_saved(s.x, dev, dt, s.x.sizes(), "x");
        check_saved(s.w, dev, dt, ws, "w");
        check_saved(s.w2, dev, dt, ws, "w2");
        check_saved(s.alpha, dev, at::kFloat, scalars, "alpha");
        check_saved(s.beta, dev, at::kFloat, scalars, "beta");
        TORCH_CHECK_VALUE(s.winners.defined(), "winners: need the tensor that the forward saved");
        check_saved(s.winners, dev, at::kByte, wb, "winners");
    }
    Grads r;
    if (need_x || g.kind == kDepthwise) r.x = at::empty(s.x.sizes(), opt);
    r.w = at::empty(s.w.sizes(), f32);
    if (par) r.w2 = at::empty(s.w.sizes(), f32);
    if (two) {
        r.alpha = at::empty(scalars, f32);
        r.beta = at::empty(scalars, f32);
    }
    r.bias = at::empty({K}, f32);
    const auto scratch = [&](size_t n) { return n ? at::empty({(int64_t)n}, opt.dtype(at::kByte)) : Tensor(); };
    int rc;
    const char* where;
    if (g.kind == kVolume) {
        const size_t n = tconv3d_workspace_bytes(&d.d3, 1);
        const Tensor ws = scratch(n);
        where = "tconv3d_backward";
        rc = tconv3d_backward(&d.d3, ptr(s.x), ptr(s.w), ptr(s.w2), fptr(s.alpha), fptr(s.beta), ptr(gy), ptr(s.winners), ptr(r.x),
                              fptr(r.w), fptr(r.w2), fptr(r.alpha), fptr(r.beta), fptr(r.bias), ptr(ws), n, stream());
    } else if (g.kind == kDepthwise) {
        const size_t n = tconv_dw_workspace_bytes(&d.d2, 1);
        const Tensor ws = scratch(n);
        where = "tconv_dw_backward";
        rc = tconv_dw_backward(&d.d2, ptr(s.x), ptr(s.w), ptr(s.w2), fptr(s.alpha), fptr(s.beta), ptr(gy), ptr(s.winners), ptr(r.x),
                               fptr(r.w), fptr(r.w2), fptr(r.alpha), fptr(r.beta), fptr(r.bias), ptr(ws), n, stream());
    } else {
        // the figure includes room for recomputed winners, which are passed here
        size_t n = tconv_workspace_bytes(&d.d2, 1);
        const size_t kept = ((size_t)s.winners.numel() + 255) / 256 * 256;
        n = n > kept ? n - kept : 0;
        const Tensor ws = scratch(n);
        where = "tconv_backward";
        rc = tconv_backward(&d.d2, ptr(s.x), ptr(s.w), ptr(s.w2), fptr(s.alpha), fptr(s.beta), ptr(gy), ptr(s.winners), ptr(r.x),
                            fptr(r.w), fptr(r.w2), fptr(r.alpha), fptr(r.beta), fptr(r.bias), ptr(ws), n, stream());
    }
    if (rc) fail(rc, where);
    return r;
}

class TropicalLayer : public torch::autograd::Function<TropicalLayer> {
public:
    // (missing tensors as empty optionals: an undefined tensor argument is not a variable to the engine)
    static Variable forward(AutogradContext* ctx, const Variable& x, const Variable& w, const std::optional<Variable>& w2_,
                            const std::optional<Variable>& alpha_, const std::optional<Variable>& beta_,
                            const std::optional<Variable>& bias_, const Geom& g) {
        const Tensor w2 = given(w2_), alpha = given(alpha_), beta = given(beta_), bias = given(bias_);
        Saved s;
        Tensor y = run_forward(g, x, w, w2, alpha, beta, bias, true, s);
        ctx->saved_data["in_type"] = (int64_t)x.scalar_type();
        ctx->saved_data["geom"] = std::vector<int64_t>{g.kind, g.mode, g.chan, g.dtype, g.stride[0], g.stride[1], g.stride[2],
                                                       g.pad[0], g.pad[1], g.pad[2], g.dil[0], g.dil[1], g.dil[2]};
        ctx->saved_data["given"] = (int64_t)((w2.defined() ? 1 : 0) | (alpha.defined() ? 2 : 0) | (beta.defined() ? 4 : 0) |
                                             (bias.defined() ? 8 : 0));
        ctx->save_for_backward({s.x, s.w, s.w2, s.alpha, s.beta, s.winners});
        return y.scalar_type() == x.scalar_type() ? y : y.to(x.scalar_type());
    }
    static variable_list backward(AutogradContext* ctx, variable_list gys) {
        const auto v = ctx->get_saved_variables();
        const Saved s{v[0], v[1], v[2], v[3], v[4], v[5]};
        const auto q = ctx->saved_data["geom"].toIntVector();
        const auto n = [&](int i) { return (int)q[i]; };
        const Geom g{n(0), n(1), n(2), n(3), {n(4), n(5), n(6)}, {n(7), n(8), n(9)}, {n(10), n(11), n(12)}};
        const int64_t has = ctx->saved_data["given"].toInt();
        if (!gys[0].defined()) return variable_list(7);
        Grads r = run_backward(g, s, gys[0], ctx->needs_input_grad(0));
        const auto in_type = (at::ScalarType)ctx->saved_data["in_type"].toInt();
        if (r.x.defined() && r.x.scalar_type() != in_type) r.x = r.x.to(in_type);
        const auto if_given = [&](const Tensor& t, int bit) { return (has & bit) ? t : Tensor(); };
        return {r.x, r.w, if_given(r.w2, 1), if_given(r.alpha, 2), if_given(r.beta, 4), if_given(r.bias, 8), Tensor()};
    }
};

// Nothing while a trace is recorded: the tracer would see the allocations alone.
std::optional<Tensor> layer(const Geom& g, const Tensor& x, const Tensor& w, const std::optional<Tensor>& w2_, const std::optional<Tensor>& alpha_,
             const std::optional<Tensor>& beta_, const std::optional<Tensor>& bias_) {
    if (at::tracer::impl::is_dispatch_enabled()) return std::nullopt;
    const Tensor w2 = given(w2_), alpha = given(alpha_), beta = given(beta_), bias = given(bias_);
    // (a tangent would be dropped without a word where nothing is recorded)
    for (const Tensor* t : {&x, &w, &w2, &alpha, &beta, &bias})
        TORCH_CHECK_NOT_IMPLEMENTED(!t->defined() || !t->_fw_grad(0).defined(), "tropical layers have no forward-mode derivative");
    bool record = false;
    if (at::GradMode::is_enabled())
        for (const Tensor* t : {&x, &w, &w2, &alpha, &beta, &bias}) record = record || (t->defined() && t->requires_grad());
    if (record) return TropicalLayer::apply(x, w, w2_, alpha_, beta_, bias_, g);
    Saved s;     // without recording the winner-free kernels run
    Tensor y = run_forward(g, x, w, w2, alpha, beta, bias, false, s);
    return y.scalar_type() == x.scalar_type() ? y : y.to(x.scalar_type());
}

}  // namespace

PYBIND11_MODULE(_tconv_torch, m) {
    pybind11::class_<Geom>(m, "Geom").def(pybind11::init([](int kind, int mode, int chan, int dtype, std::vector<int> stride,
                                                           std::vector<int> pad, std::vector<int> dil) {
        const size_t n = kind == kVolume ? 3 : 2;
        if (stride.size() != n || pad.size() != n || dil.size() != n) throw pybind11::value_error("stride, padding, dilation: one value per axis");
        Geom g{kind, mode, chan, dtype, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
        for (size_t i = 0; i < n; ++i) { g.stride[i] = stride[i]; g.pad[i] = pad[i]; g.dil[i] = dil[i]; }
        return g;
    }));
    m.def("set_error", [](pybind11::object e) { g_error = e.release().ptr(); });
    m.def("layer", &layer, pybind11::call_guard<pybind11::gil_scoped_release>());
}
