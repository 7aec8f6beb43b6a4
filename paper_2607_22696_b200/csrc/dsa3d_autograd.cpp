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

struct Shape {
    int T, H, W, heads, d, window[3], code;
    Shape(const Tensor& q, const int64_t* w)
        : T(static_cast<int>(q.size(0))), H(static_cast<int>(q.size(1))), W(static_cast<int>(q.size(2))),
          heads(static_cast<int>(q.size(3))), d(static_cast<int>(q.size(4))),
          window{static_cast<int>(w[0]), static_cast<int>(w[1]), static_cast<int>(w[2])},
          code(q.scalar_type() == at::kBFloat16 ? DSA3D_BF16 : DSA3D_F32) {}
};

Tensor new_lse(const Tensor& q) {
    return at::empty({q.size(0), q.size(1), q.size(2), q.size(3)}, q.options().dtype(at::kFloat));
}

Tensor new_workspace(const Tensor& q, size_t bytes) {
    return at::empty({static_cast<int64_t>(bytes < 16 ? 16 : bytes)}, q.options().dtype(at::kByte));
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
        const Tensor ws = new_workspace(q, dsa3d_backward_workspace_bytes(s.T, s.H, s.W, s.heads, s.d, s.window, s.code));
        check(dsa3d_backward(q.data_ptr(), k.data_ptr(), v.data_ptr(), offsets.data_ptr<float>(), lse.data_ptr<float>(),
                             dout.data_ptr(), s.T, s.H, s.W, s.heads, s.d, s.window, dq.data_ptr(), dk.data_ptr(), dv.data_ptr(),
                             doffsets.data_ptr<float>(), ws.data_ptr(), static_cast<size_t>(ws.numel()), s.code,
                             c10::cuda::getCurrentCUDAStream().stream()));
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

}  // namespace

PYBIND11_MODULE(_autograd_native, m) {
    m.def("dsa3d", &dsa3d);
    m.def("dsa3d_fixed_window", &dsa3d_fixed_window);
}
