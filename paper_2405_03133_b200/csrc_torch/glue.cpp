// The torch side of the layer in C++: allocation of outputs and workspaces, autograd nodes and pointer marshalling around
// the C ABI calls.  Every step of the computation is in the CUDA library; this file is what layer.py would otherwise do in
// Python.  A training step of a small layer is bound by the host: 180 us in Python (autograd functions, a ctypes object and
// an allocation per argument) around 53 us of C ABI calls, most of them launches.
#include <ATen/cuda/CUDAContext.h>
#include <c10/cuda/CUDAGuard.h>
#include <dlfcn.h>
#include <torch/extension.h>

#include "lory.h"

namespace {

namespace py = pybind11;
using at::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::Variable;
using torch::autograd::variable_list;

struct Api {
  decltype(&lory_moe_workspace_bytes) workspace_bytes;
  decltype(&lory_moe_forward) forward;
  decltype(&lory_moe_backward) backward;
  decltype(&lory_moe_ffn) ffn;
  decltype(&lory_block_workspace_bytes) block_workspace_bytes;
  decltype(&lory_block_forward) block_forward;
  decltype(&lory_block_backward) block_backward;
  PyObject* check;  // binding._check: raises LoryError for a status
};
Api api = {};

// The library the binding has loaded (an environment variable may select another build of it), and its error check.
void bind(const std::string& path, py::object check) {
  void* lib = dlopen(path.c_str(), RTLD_NOW | RTLD_LOCAL);
  TORCH_CHECK(lib, "cannot load ", path, ": ", dlerror());
  auto find = [&](auto& fn, const char* name) {
    fn = reinterpret_cast<std::decay_t<decltype(fn)>>(dlsym(lib, name));
    TORCH_CHECK(fn, path, " has no ", name);
  };
  find(api.workspace_bytes, "lory_moe_workspace_bytes");
  find(api.forward, "lory_moe_forward");
  find(api.backward, "lory_moe_backward");
  find(api.ffn, "lory_moe_ffn");
  find(api.block_workspace_bytes, "lory_block_workspace_bytes");
  find(api.block_forward, "lory_block_forward");
  find(api.block_backward, "lory_block_backward");
  api.check = check.release().ptr();
}

void ok(int status) {
  if (status == LORY_OK) return;
  py::gil_scoped_acquire gil;
  py::reinterpret_borrow<py::object>(api.check)(status);  // raises
}

void* ptr(const Tensor& t) {
  TORCH_CHECK_VALUE(t.is_contiguous(), "tensors passed to the Lory library must be contiguous");
  return t.data_ptr();
}

lory_dims dims_of(const Tensor& x, const Tensor& W1, int64_t T, int64_t flags) {
  TORCH_CHECK_VALUE(x.dim() == 3, "x must be [B, L, d]");
  const auto t = x.scalar_type();
  TORCH_CHECK_TYPE(t == at::kBFloat16 || t == at::kFloat, "LoryMoE supports torch.bfloat16 and torch.float32");
  lory_dims d;
  d.B = (int)x.size(0);
  d.L = (int)x.size(1);
  d.T = (int)T;
  d.d = (int)x.size(2);
  d.f = (int)W1.size(1);
  d.E = (int)W1.size(0);
  d.dtype = t == at::kFloat ? LORY_FP32 : LORY_BF16;
  d.flags = (int)flags;
  return d;
}

Tensor bytes_like(const Tensor& x, size_t n) { return at::empty({(int64_t)n}, x.options().dtype(at::kByte)); }
void* stream_of(const Tensor& x) { return (void*)at::cuda::getCurrentCUDAStream(x.get_device()).stream(); }

// gamma undefined: the layer alone; else the layer inside the pre-norm residual block
struct Forward {
  Tensor y, route_w, ws;
};
Forward run_forward(const lory_dims& d, const Tensor& x, const Tensor& gamma, const Tensor& w_r, const Tensor& W1,
                    const Tensor& W2, const Tensor& W3, double eps, bool keep) {
  size_t fwd = 0, bwd = 0;
  ok(gamma.defined() ? api.block_workspace_bytes(&d, &fwd, &bwd) : api.workspace_bytes(&d, &fwd, &bwd));
  Forward r;
  r.ws = bytes_like(x, keep ? bwd : fwd);
  r.y = at::empty_like(x);
  r.route_w = at::empty({(int64_t)d.B * (d.L / d.T), d.E}, x.options().dtype(at::kFloat));
  const size_t n = (size_t)r.ws.numel();
  if (gamma.defined())
    ok(api.block_forward(&d, ptr(x), ptr(gamma), (float)eps, ptr(w_r), ptr(W1), ptr(W2), ptr(W3), ptr(r.y),
                         (float*)ptr(r.route_w), nullptr, ptr(r.ws), n, stream_of(x)));
  else
    ok(api.forward(&d, ptr(x), ptr(w_r), ptr(W1), ptr(W2), ptr(W3), ptr(r.y), (float*)ptr(r.route_w), nullptr, ptr(r.ws),
                   n, stream_of(x)));
  return r;
}

struct Grads {
  Tensor dx, dgamma, dw_r, dW1, dW2, dW3;
};
Grads run_backward(const lory_dims& d, const Tensor& x, const Tensor& gamma, const Tensor& w_r, const Tensor& W1,
                   const Tensor& W2, const Tensor& W3, const Tensor& ws, const Tensor& dy) {
  Grads g;
  g.dx = at::empty_like(x);
  g.dw_r = at::empty_like(w_r);
  g.dW1 = at::empty_like(W1);
  g.dW2 = at::empty_like(W2);
  g.dW3 = at::empty_like(W3);
  const size_t n = (size_t)ws.numel();
  if (gamma.defined()) {
    g.dgamma = at::empty_like(gamma);
    ok(api.block_backward(&d, ptr(x), ptr(gamma), ptr(w_r), ptr(W1), ptr(W2), ptr(W3), ptr(dy), ptr(g.dx), ptr(g.dgamma),
                          ptr(g.dw_r), ptr(g.dW1), ptr(g.dW2), ptr(g.dW3), nullptr, ptr(ws), n, stream_of(x)));
  } else {
    ok(api.backward(&d, ptr(x), ptr(w_r), ptr(W1), ptr(W2), ptr(W3), ptr(dy), ptr(g.dx), ptr(g.dw_r), ptr(g.dW1), ptr(g.dW2),
                    ptr(g.dW3), nullptr, ptr(ws), n, stream_of(x)));
  }
  return g;
}

struct LoryFunction : torch::autograd::Function<LoryFunction> {
  static variable_list forward(AutogradContext* ctx, const Variable& x_in, const c10::optional<Tensor>& gamma_in,
                               const Variable& w_r, const Variable& W1, const Variable& W2, const Variable& W3, int64_t T,
                               double eps, int64_t flags) {
    const Tensor gamma = gamma_in.value_or(Tensor());
    c10::cuda::CUDAGuard guard(x_in.device());
    const lory_dims d = dims_of(x_in, W1, T, flags);
    const Tensor x = x_in.contiguous();
    Forward r = run_forward(d, x, gamma, w_r, W1, W2, W3, eps, true);
    ctx->save_for_backward({x, gamma, w_r, W1, W2, W3});
    ctx->saved_data["ws"] = r.ws;   // merged weights and activations, until the backward has run
    ctx->saved_data["T"] = T;
    ctx->saved_data["flags"] = flags;
    ctx->mark_non_differentiable({r.route_w});
    return {r.y, r.route_w};
  }
  static variable_list backward(AutogradContext* ctx, variable_list grads) {
    const auto saved = ctx->get_saved_variables();
    const Tensor &x = saved[0], &gamma = saved[1], &w_r = saved[2], &W1 = saved[3], &W2 = saved[4], &W3 = saved[5];
    c10::cuda::CUDAGuard guard(x.device());
    TORCH_CHECK(ctx->saved_data.count("ws"), "the layer's saved activations have been used by an earlier backward");
    const Tensor ws = ctx->saved_data["ws"].toTensor();
    const lory_dims d = dims_of(x, W1, ctx->saved_data["T"].toInt(), ctx->saved_data["flags"].toInt());
    const Grads g = run_backward(d, x, gamma, w_r, W1, W2, W3, ws, grads[0].contiguous());
    ctx->saved_data.erase("ws");
    return {g.dx, g.dgamma, g.dw_r, g.dW1, g.dW2, g.dW3, Tensor(), Tensor(), Tensor()};
  }
};

std::tuple<Tensor, Tensor> moe(const Tensor& x, const c10::optional<Tensor>& gamma, const Tensor& w_r, const Tensor& W1,
                               const Tensor& W2, const Tensor& W3, int64_t T, double eps, int64_t flags) {
  py::gil_scoped_release no_gil;
  // with or without gradients: a tangent must not get lost
  bool dual = gamma.has_value() && gamma->_fw_grad(0).defined();
  for (const Tensor* t : {&x, &w_r, &W1, &W2, &W3}) dual = dual || t->_fw_grad(0).defined();
  TORCH_CHECK_NOT_IMPLEMENTED(!dual, "the Lory layer has no forward-mode derivative");
  const bool grad = at::GradMode::is_enabled() &&
                    (x.requires_grad() || w_r.requires_grad() || W1.requires_grad() || W2.requires_grad() ||
                     W3.requires_grad() || (gamma.has_value() && gamma->requires_grad()));
  if (!grad) {
    at::NoGradGuard no_grad;
    c10::cuda::CUDAGuard guard(x.device());
    Forward r = run_forward(dims_of(x, W1, T, flags), x.contiguous(), gamma.value_or(Tensor()), w_r, W1, W2, W3, eps, false);
    return {r.y, r.route_w};
  }
  auto out = LoryFunction::apply(x, gamma, w_r, W1, W2, W3, T, eps, flags);
  return {out[0], out[1]};
}

// The two halves without a node of their own, for a node in Python (see layer.py): x and dy contiguous; the workspace is the
// backward's if `keep`.
std::tuple<Tensor, Tensor, Tensor> forward(const Tensor& x, const c10::optional<Tensor>& gamma, const Tensor& w_r,
                                           const Tensor& W1, const Tensor& W2, const Tensor& W3, int64_t T, double eps,
                                           int64_t flags, bool keep) {
  py::gil_scoped_release no_gil;
  c10::cuda::CUDAGuard guard(x.device());
  Forward r = run_forward(dims_of(x, W1, T, flags), x, gamma.value_or(Tensor()), w_r, W1, W2, W3, eps, keep);
  return {r.y, r.route_w, r.ws};
}
std::vector<c10::optional<Tensor>> backward(const Tensor& x, const c10::optional<Tensor>& gamma, const Tensor& w_r,
                                            const Tensor& W1, const Tensor& W2, const Tensor& W3, const Tensor& ws,
                                            const Tensor& dy, int64_t T, int64_t flags) {
  py::gil_scoped_release no_gil;
  c10::cuda::CUDAGuard guard(x.device());
  const Grads g = run_backward(dims_of(x, W1, T, flags), x, gamma.value_or(Tensor()), w_r, W1, W2, W3, ws, dy);
  return {g.dx, gamma.has_value() ? c10::optional<Tensor>(g.dgamma) : c10::nullopt, g.dw_r, g.dW1, g.dW2, g.dW3};
}

// Prompt-only routing: one segment per sequence; the workspace keeps the merged weights.
std::tuple<Tensor, Tensor, Tensor> prefill(const Tensor& x, const Tensor& w_r, const Tensor& W1, const Tensor& W2,
                                           const Tensor& W3, int64_t flags) {
  py::gil_scoped_release no_gil;
  at::NoGradGuard no_grad;
  c10::cuda::CUDAGuard guard(x.device());
  TORCH_CHECK_VALUE(x.dim() == 3, "x must be [B, L, d]");
  Forward r = run_forward(dims_of(x, W1, x.size(1), flags), x.contiguous(), Tensor(), w_r, W1, W2, W3, 0.0, false);
  return {r.y, r.route_w, r.ws};
}

Tensor decode(const Tensor& x_in, const Tensor& W1, const Tensor& W2, const Tensor& W3, const Tensor& ws, int64_t flags) {
  py::gil_scoped_release no_gil;
  at::NoGradGuard no_grad;
  c10::cuda::CUDAGuard guard(x_in.device());
  TORCH_CHECK_VALUE(x_in.dim() == 3, "x must be [B, n, d]");
  const lory_dims d = dims_of(x_in, W1, x_in.size(1), flags | LORY_FLAG_REUSE_MERGED);
  size_t need = 0;
  ok(api.workspace_bytes(&d, &need, nullptr));
  TORCH_CHECK_VALUE(need <= (size_t)ws.numel(),
                    "more new tokens per sequence than the prompt had: the cached workspace is too small");
  const Tensor x = x_in.contiguous();
  Tensor y = at::empty_like(x);
  ok(api.ffn(&d, ptr(x), nullptr, ptr(W1), ptr(W2), ptr(W3), ptr(y), ptr(ws), (size_t)ws.numel(), stream_of(x)));
  return y;
}

}  // namespace

PYBIND11_MODULE(_torch_glue, m) {
  m.attr("tag") = LORY_GLUE_TAG;
  m.def("bind", &bind);
  m.def("moe", &moe);
  m.def("forward", &forward);
  m.def("backward", &backward);
  m.def("prefill", &prefill);
  m.def("decode", &decode);
}
