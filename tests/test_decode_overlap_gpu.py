"""Decode calls queued one behind the other, with other tokens in every call: a kernel that read its predecessor's leftovers, or
overwrote what that one still reads, would show in the results (every kernel may start before the one in front has ended)."""
import numpy as np
import pytest
import torch

import paper_2405_03133_b200 as lory
from oracle import lory_oracle as O
from paper_2405_03133_b200.workloads import Workload, make_inputs, round_to_bf16

from gpu_util import max_rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d,f,n", [
    (1, 1024, 2752, 1), (8, 256, 688, 9), (4, 640, 1728, 24),   # decode_kernel
    (8, 1024, 2752, 40), (32, 520, 1376, 64),                   # decode_mma_kernel
    (64, 256, 688, 33),                                         # grouped GEMMs
])
def test_calls_in_a_row_with_other_tokens(B, d, f, n):
    wl = Workload("overlap", B=B, L=64, T=64, d=d, f=f, E=2, dtype="bf16", w_r_std=2.0, seed=31)
    inp = make_inputs(wl)
    x, w_r, W1, W2, W3 = (to_dev(inp[k], wl) for k in ("x", "w_r", "W1", "W2", "W3"))
    dims = lory.make_dims(B, wl.L, wl.L, d, f, wl.E, "bf16")
    ws = torch.empty(lory.lory_moe_workspace_bytes(dims)[0], dtype=torch.uint8, device="cuda")
    rw = torch.empty((B, wl.E), dtype=torch.float32, device="cuda")
    lory.lory_moe_forward(dims, x, w_r, W1, W2, W3, torch.empty_like(x), rw, None, ws)
    rng = np.random.default_rng(n)
    news = [round_to_bf16(rng.standard_normal((B, n, d)).astype(np.float32)) for _ in range(2)]
    refs = [O.prompt_only_inference(inp["x"], new, inp["w_r"], inp["W1"], inp["W2"], inp["W3"])[1] for new in news]
    xs = [to_dev(new, wl) for new in news]
    ddims = lory.make_dims(B, n, n, d, f, wl.E, "bf16", lory.LORY_FLAG_REUSE_MERGED)
    ys = [torch.full_like(xs[0], float("nan")) for _ in range(12)]
    torch.cuda.synchronize()
    for i, y in enumerate(ys):
        lory.lory_moe_ffn(ddims, xs[i & 1], None, W1, W2, W3, y, ws)
    lory.lory_check_status(ddims, ws)
    for i, y in enumerate(ys):
        assert torch.equal(y, ys[i & 1]), i        # the same tokens, the same bits
    for y, ref in zip(ys, refs):
        assert max_rel(y.double().cpu().numpy(), ref) <= 2e-2
