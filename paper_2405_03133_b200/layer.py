"""The layer as a torch.nn.Module: autograd over the C-ABI calls (csrc_torch/glue.cpp).

    layer = LoryMoE(d=1024, f=2752, E=32, T=256, dtype=torch.bfloat16, device="cuda")
    y = layer(x)                 # x [B, L, d], L % T == 0
    y.sum().backward()           # x.grad, layer.w_r.grad, layer.W1.grad, layer.W2.grad, layer.W3.grad

Every step of the computation runs in the CUDA library (lory_moe_forward / lory_moe_backward); the glue only allocates
the outputs and the workspace and hands pointers over.  Each forward that needs gradients keeps its own
workspace (the merged weights and activations saved for the backward) until its backward has run, so several
calls may be in flight (gradient checkpointing, several micro-batches).  Without gradients the workspace is the
smaller forward-only one and is dropped at once.
"""
from __future__ import annotations

import importlib
import threading

import torch

from . import binding as _lory


_module = None
_lock = threading.Lock()


def _glue():
    """The C++ side of this file (autograd nodes, allocations, argument marshalling): loaded by the first call that needs it,
    and built before that if it is missing or its sources have changed."""
    if _module is None:
        _load()
    return _module


def _load():
    global _module
    with _lock:
        if _module is not None:
            return
        from . import build
        _lory.load()
        build.build_glue()
        try:
            glue = importlib.import_module("._torch_glue", __package__)
        except ImportError:     # built for another interpreter
            build.build_glue(force=True)
            glue = importlib.import_module("._torch_glue", __package__)
        glue.bind(_lory.LIB_PATH, _lory._check)
        _module = glue


class _TracedFunction(torch.autograd.Function):
    """The same node in Python, for torch.jit.trace: it records a Python function as one operation, while of the C++ one it
    would record the allocation of the outputs and not what fills them."""

    @staticmethod
    def forward(ctx, x, gamma, w_r, W1, W2, W3, T, eps, flags):
        x = x.contiguous()
        keep = any(ctx.needs_input_grad)
        y, route_w, ws = _glue().forward(x, gamma, w_r, W1, W2, W3, T, eps, flags, keep)
        if keep:
            ctx.save_for_backward(x, gamma, w_r, W1, W2, W3)
            ctx.ws, ctx.T, ctx.flags = ws, T, flags
        ctx.mark_non_differentiable(route_w)
        return y, route_w

    @staticmethod
    def backward(ctx, dy, _d_route_w):
        grads = _glue().backward(*ctx.saved_tensors, ctx.ws, dy.contiguous(), ctx.T, ctx.flags)
        ctx.ws = None
        return *grads, None, None, None


def _moe(*args):
    return _TracedFunction.apply(*args) if torch.jit.is_tracing() else _glue().moe(*args)


class LoryMoE(torch.nn.Module):
    """Lory mixture-of-experts FFN layer (causal segment routing + expert merging, Sections 3 and 3.1).

    Parameters: w_r [E, d] (router), W1, W3 [E, f, d] (gate, up), W2 [E, d, f] (down), initialised N(0, std).
    forward(x) returns y [B, L, d]; `last_route_w` holds the routing weights [B*L/T, E] of the last call.
    `flags`: LORY_FLAG_* of the binding (prefix routing, first-segment gradient, ...).
    """

    def __init__(self, d: int, f: int, E: int, T: int, dtype=torch.bfloat16, device="cuda", std: float = 0.02,
                 flags: int = 0, generator: torch.Generator | None = None):
        super().__init__()
        self.T, self.flags = int(T), int(flags)

        def init(*shape):
            w = torch.randn(*shape, dtype=torch.float32, device=device, generator=generator) * std
            return torch.nn.Parameter(w.to(dtype))

        self.w_r = init(E, d)
        self.W1 = init(E, f, d)
        self.W2 = init(E, d, f)
        self.W3 = init(E, f, d)
        self.last_route_w = None

    def forward(self, x: torch.Tensor) -> torch.Tensor:
        if not x.is_cuda:
            raise RuntimeError("LoryMoE runs on a CUDA device only (there is no CPU path)")
        y, self.last_route_w = _moe(x, None, self.w_r, self.W1, self.W2, self.W3, self.T, 0.0, self.flags)
        return y


class LoryBlock(LoryMoE):
    """The layer inside a pre-norm residual block (the LLaMA block the paper's models use, Section 4.1):
    y = x + LoryMoE(RMSNorm(x; gamma, eps)).  Adds the parameter gamma [d], initialised to one."""

    def __init__(self, d: int, f: int, E: int, T: int, eps: float = 1e-5, dtype=torch.bfloat16, device="cuda",
                 std: float = 0.02, flags: int = 0, generator: torch.Generator | None = None):
        super().__init__(d, f, E, T, dtype=dtype, device=device, std=std, flags=flags, generator=generator)
        self.eps = float(eps)
        self.gamma = torch.nn.Parameter(torch.ones(d, dtype=dtype, device=device))

    def forward(self, x: torch.Tensor) -> torch.Tensor:
        if not x.is_cuda:
            raise RuntimeError("LoryBlock runs on a CUDA device only (there is no CPU path)")
        y, self.last_route_w = _moe(x, self.gamma, self.w_r, self.W1, self.W2, self.W3, self.T, self.eps, self.flags)
        return y


class LoryPromptRoutedFFN:
    """Prompt-only routing at inference (Section 3.1): `prefill` routes each sequence once from its whole prompt
    and leaves the merged FFN of every sequence in a workspace; `decode` then applies that cached FFN to new
    tokens like a dense FFN, with no routing and no merging."""

    def __init__(self, layer: LoryMoE):
        self.layer = layer
        self.ws = None
        self.batch = None

    def prefill(self, x_prompt: torch.Tensor) -> torch.Tensor:
        m = self.layer
        # on the stream torch is issuing this tensor's work on, so that the call is ordered with its producers and
        # consumers (and with later decode() calls, which share the cached workspace)
        y, self.route_w, self.ws = _glue().prefill(x_prompt, m.w_r, m.W1, m.W2, m.W3, m.flags)
        self.batch = x_prompt.shape[0]
        return y

    def decode(self, x_new: torch.Tensor) -> torch.Tensor:
        if self.ws is None:
            raise RuntimeError("call prefill() first")
        if x_new.shape[0] != self.batch:
            raise ValueError("decode() needs the batch of the prefill() whose merged FFNs are cached")
        m = self.layer
        return _glue().decode(x_new, m.W1, m.W2, m.W3, self.ws, m.flags)
