"""The work a user has this framework do, as cases that can be timed.

Every case goes through the public entry points (the torch modules, or the C ABI through its binding) with what such
a program has in hand: the layer's parameters, a batch on the GPU and, where the program keeps one, a workspace.
Sizes are those of `paper_2405_03133_b200.workloads`, of the decode measurement of bench.py, and ragged ones between.
"""
import torch

import paper_2405_03133_b200 as lory
from paper_2405_03133_b200.layer import LoryBlock, LoryMoE, LoryPromptRoutedFFN

_TORCH = {"bf16": torch.bfloat16, "fp32": torch.float32}


def listed():
    return [
        # one user's chat: one new token through the cached merged FFN, the smallest call there is
        dict(name="decode_one", kind="decode", B=1, n=1, d=1024, f=2752, E=8, dtype="bf16"),
        # a serving batch: one new token for each of eight sequences, each with a merged FFN of its own
        dict(name="decode_batch", kind="decode", B=8, n=1, d=1024, f=2752, E=8, dtype="bf16"),
        # several new tokens per sequence at once (drafted tokens, chunks of a turn), the wide model
        dict(name="decode_chunk", kind="decode", B=4, n=48, d=2048, f=5504, E=8, dtype="bf16"),
        # two prompts of a length nobody chose: routed once from the whole prompt, merged, run
        dict(name="prefill_ragged", kind="prefill", B=2, L=1000, d=1024, f=2752, E=32, dtype="bf16"),
        # evaluation: a forward with per-segment routing and no gradients, the wide model
        dict(name="eval_wide", kind="infer", B=1, L=4096, T=256, d=2048, f=5504, E=16, dtype="bf16"),
        # fine-tuning on one short document: a training step with few segments
        dict(name="train_one_document", kind="train", B=1, L=2048, T=256, d=1024, f=2752, E=8, dtype="bf16"),
        # the pre-training step: 8 instances of 4096 tokens, 32 experts (the benchmark's default workload)
        dict(name="train_pretrain", kind="train", B=8, L=4096, T=256, d=1024, f=2752, E=32, dtype="bf16"),
        # the wide model with long segments, one optimiser step of two micro-batches (gradients accumulated)
        dict(name="train_micro_batches", kind="micro", B=2, L=4096, T=1024, d=2048, f=5504, E=32, dtype="bf16"),
        # the wide model with the shortest segments: the largest amount of merged weights
        dict(name="train_short_segments", kind="train", B=4, L=4096, T=64, d=2048, f=5504, E=32, dtype="bf16"),
        # the pre-norm residual block inside a model whose sizes fill no tile
        dict(name="train_block_ragged", kind="block", B=3, L=1400, T=100, d=1000, f=2696, E=12, dtype="bf16"),
        # full precision, the tiny layer of a debugging or ablation run
        dict(name="train_fp32_tiny", kind="train", B=2, L=512, T=128, d=256, f=688, E=4, dtype="fp32"),
        # full precision at sizes that are no multiple of anything, the reference run a bf16 model is held against
        dict(name="train_fp32_ragged", kind="train", B=2, L=1125, T=125, d=500, f=1340, E=6, dtype="fp32"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _width(rng, lo, hi, step):
    """A hidden size and an FFN hidden size of 2 to 3 times it, in multiples of `step`."""
    d = max(lo, _log_int(rng, lo, hi) // step * step)
    return d, max(step, int(d * rng.uniform(2.0, 2.7)) // step * step)


def draw(rng):
    kind = rng.choice(["decode", "decode", "prefill", "infer", "train", "train", "train", "micro", "block", "fp32"])
    if kind == "fp32":
        d, f = _width(rng, 96, 768, rng.choice([1, 4, 8]))
        T = _log_int(rng, 16, 256)
        N = max(1, _log_int(rng, 256, 2048) // T)
        return dict(kind="train", B=rng.randint(1, 3), L=N * T, T=T, d=d, f=f, E=_log_int(rng, 2, 16), dtype="fp32")
    d, f = _width(rng, 256, 2048, 8)
    if kind == "decode":
        return dict(kind=kind, B=_log_int(rng, 1, 32), n=_log_int(rng, 1, 64), d=d, f=f, E=8, dtype="bf16")
    E = _log_int(rng, 4, 48)
    if kind == "prefill":
        return dict(kind=kind, B=_log_int(rng, 1, 16), L=_log_int(rng, 64, 2048), d=d, f=f, E=min(E, 32), dtype="bf16")
    T = _log_int(rng, 48, 1024)
    N = max(1, _log_int(rng, 1024, 4096) // T)
    B = _log_int(rng, 1, 2 if kind == "micro" else 4)
    return dict(kind=kind, B=B, L=N * T, T=T, d=d, f=f, E=min(E, 32) if d > 1448 else E, dtype="bf16")


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dtype, kind = _TORCH[case["dtype"]], case["kind"]
    B, d, f, E = case["B"], case["d"], case["f"], case["E"]

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32).to(dtype)

    cls = LoryBlock if kind == "block" else LoryMoE
    layer = cls(d, f, E, T=case.get("T", 1), dtype=dtype, generator=gen)
    with torch.no_grad():
        layer.w_r.mul_(25.0)  # a router that has learnt something: logits of about one, not nearly equal weights
    state = dict(kind=kind, layer=layer)
    if kind == "decode":
        state["ffn"] = LoryPromptRoutedFFN(layer)
        state["ffn"].prefill(normal(B, max(64, case["n"]), d))
        state["x"] = normal(B, case["n"], d)
        return state
    L = case["L"]
    if kind == "prefill":
        state["ffn"] = LoryPromptRoutedFFN(layer)
        state["x"] = normal(B, L, d)
    elif kind == "infer":
        state["x"] = normal(B, L, d)
    elif kind == "micro":
        # a program over the C ABI keeps its workspace and its gradient buffers from step to step
        dims = [lory.make_dims(B, L, case["T"], d, f, E, case["dtype"], flags) for flags in (0, lory.LORY_FLAG_ACCUMULATE_GRADS)]
        params = [p.detach() for p in (layer.w_r, layer.W1, layer.W2, layer.W3)]
        batches = []
        for _ in dims:
            x, dy = normal(B, L, d), normal(B, L, d)
            batches.append((x, dy, torch.empty_like(x), torch.empty_like(x)))
        state.update(dims=dims, params=params, batches=batches, grads=[torch.empty_like(p) for p in params],
                     route_w=torch.empty((B * (L // case["T"]), E), dtype=torch.float32, device="cuda"),
                     ws=torch.empty(lory.lory_moe_workspace_bytes(dims[0])[1], dtype=torch.uint8, device="cuda"))
    else:
        state["x"] = normal(B, L, d).requires_grad_()
        state["dy"] = normal(B, L, d)
    return state


def run(state):
    kind = state["kind"]
    if kind == "decode":
        return state["ffn"].decode(state["x"])
    if kind == "prefill":
        y = state["ffn"].prefill(state["x"])
        return y, state["ffn"].route_w
    layer = state["layer"]
    if kind == "infer":
        with torch.no_grad():
            y = layer(state["x"])
        return y, layer.last_route_w
    if kind == "micro":
        w_r, W1, W2, W3 = state["params"]
        for dims, (x, dy, y, dx) in zip(state["dims"], state["batches"]):
            lory.lory_moe_forward(dims, x, w_r, W1, W2, W3, y, state["route_w"], None, state["ws"])
            lory.lory_moe_backward(dims, x, w_r, W1, W2, W3, dy, dx, *state["grads"], None, state["ws"])
        return [(y, dx) for _, _, y, dx in state["batches"]], state["route_w"], state["grads"]
    y = layer(state["x"])
    grads = torch.autograd.grad(y, [state["x"], *layer.parameters()], state["dy"])
    return y.detach(), layer.last_route_w, grads


def work(case):
    """One pass: the activations and the experts read once per direction, outputs and gradients written once; the
    products of the FFN and of the merge (6 d f per token and per segment and expert forward, twice that backward)."""
    es = 2 if case["dtype"] == "bf16" else 4
    B, d, f, E = case["B"], case["d"], case["f"], case["E"]
    df = d * f
    if case["kind"] == "decode":
        tok = B * case["n"]
        return {"bytes": es * (3 * B * df + 2 * tok * d), "flops": 6 * tok * df}
    T = case["L"] if case["kind"] == "prefill" else case["T"]
    tok, S = B * case["L"], B * (case["L"] // T)
    if case["kind"] in ("prefill", "infer"):
        return {"bytes": es * (2 * tok * d + 3 * E * df), "flops": 6 * df * (tok + S * E)}
    steps = 2 if case["kind"] == "micro" else 1
    return {"bytes": es * (steps * 5 * tok * d + 9 * E * df), "flops": steps * 18 * df * (tok + S * E)}


def tolerance(case):
    # bf16 storage of inputs, merged weights, activations and results; fp32 sums everywhere in the fp32 mode
    return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 1e-4}
