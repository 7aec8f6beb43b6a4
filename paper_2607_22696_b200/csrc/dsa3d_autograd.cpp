// The torch.autograd functions of autograd.py, compiled: the same calls into the library in the same order, without
// the interpreter.  A training step of a small problem is bound by the host - a Python autograd function costs it a
// hand-over of the interpreter lock to the engine's device thread and back, argument marshalling through ctypes and the
// bookkeeping of its context.  512 items, window (3,3,3), forward + backward back to back on a B200: 153 -> 81 us in
// fp32, 175 -> 102 us in bf16, 147 -> 80 us for the fixed window; a forward alone 28 -> 10 us.
//
// Each entry point returns None for arguments it does not take as they are (another device, dtype or layout, sizes that
// do not fit together): autograd.py then goes through its Python function, which converts them or raises.
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/extension.h>

#include <climits>

#include "../../include/dsa3d.h"

namespace {

using at::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::variable_list;

void check(int status) {
    if (status == DSA3D_OK) return;
    pybind11::gil_scoped_acquire gil;                         // the exception binding.py raises for this status
    try {
        pybind11::module_::import("paper_2607_22696_b200.binding").attr("_check")(status);
    } catch (pybind11::error_already_set& e) {
        e.restore();
    }
    python_error raised;
    raised.persist();
    throw raised;
}

bool taken(const Tensor& t, const Tensor& like) {
    return t.defined() && t.is_cuda() && t.device() == like.device() && t.scalar_type() == like.scalar_type() && t.is_contiguous();
}

// q, k, v [T, H, W, heads, d] of one supported type and device
bool taken_qkv(const Tensor& q, const Tensor& k, const Tensor& v) {
    if (!taken(q, q) || q.dim() != 5 || (q.scalar_type() != at::kFloat && q.scalar_type() != at::kBFloat16)) return false;
    for (int64_t s : q.sizes()) if (s < 1 || s > INT_MAX) return false;
    return taken(k, q) && taken(v, q) && k.numel() == q.numel() && v.numel() == q.numel();
}

int code_of(const Tensor& t) { return t.scalar_type() == at::kBFloat16 ? DSA3D_BF16 : DSA3D_F32; }

struct Shape {
    int T, H, W, heads, d, window[3], code;
    Shape(const Tensor& q, const int64_t* w)
        : T(static_cast<int>(q.size(0))), H(static_cast<int>(q.size(1))), W(static_cast<int>(q.size(2))),
          heads(static_cast<int>(q.size(3))), d(static_cast<int>(q.size(4))),
          window{static_cast<int>(w[0]), static_cast<int>(w[1]), static_cast<int>(w[2])},
          code(code_of(q)) {}
};

Tensor new_lse(const Tensor& q) {
    return at::empty({q.size(0), q.size(1), q.size(2), q.size(3)}, q.options().dtype(at::kFloat));
}

Tensor new_workspace(const Tensor& q, size_t bytes) {
    return at::empty({static_cast<int64_t>(bytes < 16 ? 16 : bytes)}, q.options().dtype(at::kByte));
}

// fp32 runs with any workspace or none: on a card too full for the sort's room it goes without, as it did before there was one.
Tensor new_backward_workspace(const Tensor& q, const Shape& s) {
    const size_t bytes = dsa3d_backward_workspace_bytes(s.T, s.H, s.W, s.heads, s.d, s.window, s.code);
    if (s.code != DSA3D_F32) return new_workspace(q, bytes);
    try {
        return new_workspace(q, bytes);
    } catch (const c10::OutOfMemoryError&) {
        return Tensor();
    }
}

struct Window { int64_t w[3]; };

void save_window(AutogradContext* ctx, const int64_t* w) {
    ctx->saved_data["window"] = std::vector<int64_t>{w[0], w[1], w[2]};
}
Window saved_window(AutogradContext* ctx) {
    const auto w = ctx->saved_data["window"].toIntVector();
    return {{w[0], w[1], w[2]}};
}

struct Dsa3d : torch::autograd::Function<Dsa3d> {
    static Tensor forward(AutogradContext* ctx, const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& offsets,
                          const std::optional<Tensor>& residual, int64_t kt, int64_t kh, int64_t kw) {
        const c10::cuda::CUDAGuard guard(q.device());
        const int64_t w[3] = {kt, kh, kw};
        const Shape s(q, w);
        Tensor out = at::empty_like(q), lse = new_lse(q);
        void* stream = c10::cuda::getCurrentCUDAStream().stream();
        check(residual
                  ? dsa3d_forward_residual(q.data_ptr(), k.data_ptr(), v.data_ptr(), offsets.data_ptr<float>(), residual->data_ptr(),
                                           s.T, s.H, s.W, s.heads, s.d, s.window, out.data_ptr(), lse.data_ptr<float>(), s.code, stream)
                  : dsa3d_forward(q.data_ptr(), k.data_ptr(), v.data_ptr(), offsets.data_ptr<float>(), s.T, s.H, s.W, s.heads, s.d,
                                  s.window, out.data_ptr(), lse.data_ptr<float>(), s.code, stream));
        ctx->save_for_backward({q, k, v, offsets, lse});
        save_window(ctx, w);
        ctx->saved_data["residual"] = residual.has_value();
        return out;
    }
    static variable_list backward(AutogradContext* ctx, const variable_list& grads) {
        const variable_list saved = ctx->get_saved_variables();
        const Tensor &q = saved[0], &k = saved[1], &v = saved[2], &offsets = saved[3], &lse = saved[4];
        const c10::cuda::CUDAGuard guard(q.device());
        const Window w = saved_window(ctx);
        const Shape s(q, w.w);
        const Tensor dout = grads[0].contiguous();
        Tensor dq = at::empty_like(q), dk = at::empty_like(q), dv = at::empty_like(q), doffsets = at::empty_like(offsets);
        const Tensor ws = new_backward_workspace(q, s);
        check(dsa3d_backward(q.data_ptr(), k.data_ptr(), v.data_ptr(), offsets.data_ptr<float>(), lse.data_ptr<float>(),
                             dout.data_ptr(), s.T, s.H, s.W, s.heads, s.d, s.window, dq.data_ptr(), dk.data_ptr(), dv.data_ptr(),
                             doffsets.data_ptr<float>(), ws.defined() ? ws.data_ptr() : nullptr,
                             ws.defined() ? static_cast<size_t>(ws.numel()) : 0, s.code, c10::cuda::getCurrentCUDAStream().stream()));
        return {dq, dk, dv, doffsets, ctx->saved_data["residual"].toBool() ? dout : Tensor(), Tensor(), Tensor(), Tensor()};
    }
};

struct Dsa3dFixedWindow : torch::autograd::Function<Dsa3dFixedWindow> {
    static Tensor forward(AutogradContext* ctx, const Tensor& q, const Tensor& k, const Tensor& v, int64_t kt, int64_t kh, int64_t kw) {
        const c10::cuda::CUDAGuard guard(q.device());
        const int64_t w[3] = {kt, kh, kw};
        const Shape s(q, w);
        Tensor out = at::empty_like(q), lse = new_lse(q);
        check(dsa3d_forward_fixed_window(q.data_ptr(), k.data_ptr(), v.data_ptr(), s.T, s.H, s.W, s.heads, s.d, s.window,
                                         out.data_ptr(), lse.data_ptr<float>(), s.code, c10::cuda::getCurrentCUDAStream().stream()));
        ctx->save_for_backward({q, k, v, lse});
        save_window(ctx, w);
        return out;
    }
    static variable_list backward(AutogradContext* ctx, const variable_list& grads) {
        const variable_list saved = ctx->get_saved_variables();
        const Tensor &q = saved[0], &k = saved[1], &v = saved[2], &lse = saved[3];
        const c10::cuda::CUDAGuard guard(q.device());
        const Window w = saved_window(ctx);
        const Shape s(q, w.w);
        const Tensor dout = grads[0].contiguous();
        Tensor dq = at::empty_like(q), dk = at::empty_like(q), dv = at::empty_like(q);
        const Tensor ws = new_workspace(q, dsa3d_backward_fixed_window_workspace_bytes(s.T, s.H, s.W, s.heads, s.d, s.window, s.code));
        check(dsa3d_backward_fixed_window(q.data_ptr(), k.data_ptr(), v.data_ptr(), lse.data_ptr<float>(), dout.data_ptr(), s.T, s.H,
                                          s.W, s.heads, s.d, s.window, dq.data_ptr(), dk.data_ptr(), dv.data_ptr(), nullptr,
                                          ws.data_ptr(), static_cast<size_t>(ws.numel()), s.code,
                                          c10::cuda::getCurrentCUDAStream().stream()));
        return {dq, dk, dv, Tensor(), Tensor(), Tensor()};
    }
};

// x [T, H, W, C], weight fp32 [taps, C], bias fp32 [C] or none
struct DwConv3d : torch::autograd::Function<DwConv3d> {
    static Tensor forward(AutogradContext* ctx, const Tensor& x, const Tensor& weight, const std::optional<Tensor>& bias, int64_t kt,
                          int64_t kh, int64_t kw) {
        const c10::cuda::CUDAGuard guard(x.device());
        const int kernel[3] = {static_cast<int>(kt), static_cast<int>(kh), static_cast<int>(kw)};
        Tensor y = at::empty_like(x);
        check(dsa3d_dwconv3d_forward(x.data_ptr(), weight.data_ptr<float>(), bias ? bias->data_ptr<float>() : nullptr,
                                     static_cast<int>(x.size(0)), static_cast<int>(x.size(1)), static_cast<int>(x.size(2)),
                                     static_cast<int>(x.size(3)), kernel, y.data_ptr(), code_of(x),
                                     c10::cuda::getCurrentCUDAStream().stream()));
        ctx->save_for_backward({x, weight});
        const int64_t w[3] = {kt, kh, kw};
        save_window(ctx, w);
        ctx->saved_data["bias"] = bias.has_value();
        return y;
    }
    static variable_list backward(AutogradContext* ctx, const variable_list& grads) {
        const variable_list saved = ctx->get_saved_variables();
        const Tensor &x = saved[0], &weight = saved[1];
        const c10::cuda::CUDAGuard guard(x.device());
        const Window w = saved_window(ctx);
        const int kernel[3] = {static_cast<int>(w.w[0]), static_cast<int>(w.w[1]), static_cast<int>(w.w[2])};
        const bool need_x = ctx->needs_input_grad(0), need_w = ctx->needs_input_grad(1);
        const bool need_b = ctx->saved_data["bias"].toBool() && ctx->needs_input_grad(2);
        const Tensor dy = grads[0].contiguous();
        const Tensor dx = need_x ? at::empty_like(x) : Tensor(), dw = need_w || need_b ? at::empty_like(weight) : Tensor();
        const Tensor db = need_b ? at::empty({x.size(3)}, x.options().dtype(at::kFloat)) : Tensor();
        const Tensor ws = need_x ? new_workspace(x, dsa3d_dwconv3d_backward_workspace_bytes(static_cast<int>(x.size(3)), kernel)) : Tensor();
        check(dsa3d_dwconv3d_backward(x.data_ptr(), weight.data_ptr<float>(), dy.data_ptr(), static_cast<int>(x.size(0)),
                                      static_cast<int>(x.size(1)), static_cast<int>(x.size(2)), static_cast<int>(x.size(3)), kernel,
                                      need_x ? dx.data_ptr() : nullptr, dw.defined() ? dw.data_ptr<float>() : nullptr,
                                      need_b ? db.data_ptr<float>() : nullptr, need_x ? ws.data_ptr() : nullptr,
                                      need_x ? static_cast<size_t>(ws.numel()) : 0, code_of(x),
                                      c10::cuda::getCurrentCUDAStream().stream()));
        return {dx, need_w ? dw : Tensor(), db, Tensor(), Tensor(), Tensor()};
    }
};

// u [tokens, C], w [O, C] of one type, bias fp32 [O]
struct OffsetsLinear : torch::autograd::Function<OffsetsLinear> {
    static Tensor forward(AutogradContext* ctx, const Tensor& u, const Tensor& w, const Tensor& bias) {
        const c10::cuda::CUDAGuard guard(u.device());
        Tensor out = at::empty({u.size(0), w.size(0)}, u.options().dtype(at::kFloat));
        check(dsa3d_offsets_linear_forward(u.data_ptr(), w.data_ptr(), bias.data_ptr<float>(), u.size(0), static_cast<int>(u.size(1)),
                                           static_cast<int>(w.size(0)), out.data_ptr<float>(), code_of(u),
                                           c10::cuda::getCurrentCUDAStream().stream()));
        ctx->save_for_backward({u, w});
        return out;
    }
    static variable_list backward(AutogradContext* ctx, const variable_list& grads) {
        const variable_list saved = ctx->get_saved_variables();
        const Tensor &u = saved[0], &w = saved[1];
        const c10::cuda::CUDAGuard guard(u.device());
        const int C = static_cast<int>(u.size(1)), O = static_cast<int>(w.size(0));
        const bool need_u = ctx->needs_input_grad(0), need_w = ctx->needs_input_grad(1), need_b = ctx->needs_input_grad(2);
        const Tensor g = grads[0].contiguous();
        const auto f32 = u.options().dtype(at::kFloat);
        const Tensor du = need_u ? at::empty_like(u) : Tensor(), dw = need_w ? at::empty({O, C}, f32) : Tensor();
        const Tensor db = need_b ? at::empty({O}, f32) : Tensor();
        const Tensor ws = new_workspace(u, dsa3d_offsets_linear_backward_workspace_bytes(u.size(0), C, O, code_of(u)));
        check(dsa3d_offsets_linear_backward(u.data_ptr(), w.data_ptr(), g.data_ptr<float>(), u.size(0), C, O,
                                            need_u ? du.data_ptr() : nullptr, need_w ? dw.data_ptr<float>() : nullptr,
                                            need_b ? db.data_ptr<float>() : nullptr, ws.data_ptr(), static_cast<size_t>(ws.numel()),
                                            code_of(u), c10::cuda::getCurrentCUDAStream().stream()));
        return {du, need_w ? dw.to(w.scalar_type()) : Tensor(), db};
    }
};

// Runs `call` without the interpreter lock; a Python exception that came up in it is raised where Python called.
template <typename F> Tensor run(F call) {
    try {
        const pybind11::gil_scoped_release released;
        return call();
    } catch (python_error& e) {
        e.restore();
        throw pybind11::error_already_set();
    }
}

bool taken_window(int64_t kt, int64_t kh, int64_t kw) {
    return kt > 0 && kh > 0 && kw > 0 && kt <= 1024 && kh <= 1024 && kw <= 1024;
}

std::optional<Tensor> dsa3d(const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& offsets,
                            const std::optional<Tensor>& residual, int64_t kt, int64_t kh, int64_t kw) {
    if (!taken_qkv(q, k, v) || !taken_window(kt, kh, kw)) return std::nullopt;
    if (!offsets.is_cuda() || offsets.device() != q.device() || offsets.scalar_type() != at::kFloat || !offsets.is_contiguous() ||
        offsets.numel() != q.numel() / q.size(4) * kt * kh * kw * 3)
        return std::nullopt;
    if (residual && (!taken(*residual, q) || residual->numel() != q.numel())) return std::nullopt;
    return run([&] { return Dsa3d::apply(q, k, v, offsets, residual, kt, kh, kw); });
}

std::optional<Tensor> dsa3d_fixed_window(const Tensor& q, const Tensor& k, const Tensor& v, int64_t kt, int64_t kh, int64_t kw) {
    if (!taken_qkv(q, k, v) || !taken_window(kt, kh, kw)) return std::nullopt;
    return run([&] { return Dsa3dFixedWindow::apply(q, k, v, kt, kh, kw); });
}

bool taken_f32(const Tensor& t, const Tensor& like, int64_t numel) {
    return t.is_cuda() && t.device() == like.device() && t.scalar_type() == at::kFloat && t.is_contiguous() && t.numel() == numel;
}

bool taken_storage(const Tensor& t, int64_t dims) {
    if (!taken(t, t) || t.dim() != dims || (t.scalar_type() != at::kFloat && t.scalar_type() != at::kBFloat16)) return false;
    for (int64_t s : t.sizes()) if (s < 1 || s > INT_MAX) return false;
    return true;
}

std::optional<Tensor> dwconv3d(const Tensor& x, const Tensor& weight, const std::optional<Tensor>& bias, int64_t kt, int64_t kh, int64_t kw) {
    if (!taken_storage(x, 4) || !taken_window(kt, kh, kw) || weight.dim() != 2 || !taken_f32(weight, x, kt * kh * kw * x.size(3)) ||
        (bias && !taken_f32(*bias, x, x.size(3))))
        return std::nullopt;
    return run([&] { return DwConv3d::apply(x, weight, bias, kt, kh, kw); });
}

std::optional<Tensor> offsets_linear(const Tensor& u, const Tensor& w, const Tensor& bias) {
    if (!taken_storage(u, 2) || !taken_storage(w, 2) || !taken(w, u) || w.size(1) != u.size(1) || !taken_f32(bias, u, w.size(0)))
        return std::nullopt;
    return run([&] { return OffsetsLinear::apply(u, w, bias); });
}

}  // namespace

PYBIND11_MODULE(_autograd_native, m) {
    m.def("dsa3d", &dsa3d);
    m.def("dsa3d_fixed_window", &dsa3d_fixed_window);
    m.def("dwconv3d", &dwconv3d);
    m.def("offsets_linear", &offsets_linear);
}
