"""Where a decode call goes: both sides of the line between the decode kernels and the grouped GEMMs (widths up to 512, more
than 32 tokens with more gate tiles than SMs, more than 16 with more than three times as many)."""
import numpy as np
import pytest
import torch

import paper_2405_03133_b200 as lory
from oracle import lory_oracle as O
from paper_2405_03133_b200.workloads import Workload, make_inputs, round_to_bf16

from gpu_util import max_rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d,f,n", [
    (37, 64, 256, 33), (38, 64, 256, 33), (38, 64, 256, 64), (38, 64, 256, 32),   # 148 and 152 gate tiles
    (111, 64, 256, 17), (112, 64, 256, 17), (112, 64, 256, 32), (112, 64, 256, 16),   # 444 and 448
    (30, 512, 328, 48), (30, 520, 328, 48),   # 180, on both sides of the width
])
def test_decode_routes(B, d, f, n):
    wl = Workload("routes", B=B, L=64, T=64, d=d, f=f, E=2, dtype="bf16", w_r_std=2.0, seed=5)
    inp = make_inputs(wl)
    x, w_r, W1, W2, W3 = (to_dev(inp[k], wl) for k in ("x", "w_r", "W1", "W2", "W3"))
    dims = lory.make_dims(B, wl.L, wl.L, d, f, wl.E, "bf16")
    ws = torch.empty(lory.lory_moe_workspace_bytes(dims)[0], dtype=torch.uint8, device="cuda")
    rw = torch.empty((B, wl.E), dtype=torch.float32, device="cuda")
    lory.lory_moe_forward(dims, x, w_r, W1, W2, W3, torch.empty_like(x), rw, None, ws)
    new = round_to_bf16(np.random.default_rng(n).standard_normal((B, n, d)).astype(np.float32))
    _, ref, _ = O.prompt_only_inference(inp["x"], new, inp["w_r"], inp["W1"], inp["W2"], inp["W3"])
    ddims = lory.make_dims(B, n, n, d, f, wl.E, "bf16", lory.LORY_FLAG_REUSE_MERGED)
    xd = to_dev(new, wl)
    y = torch.full_like(xd, float("nan"))
    lory.lory_moe_ffn(ddims, xd, None, W1, W2, W3, y, ws)
    lory.lory_check_status(ddims, ws)
    assert max_rel(y.double().cpu().numpy(), ref) <= 2e-2


@pytest.mark.parametrize("B,n", [(1, 1), (8, 40), (38, 33)])
@pytest.mark.parametrize("which", ["x", "y"])
def test_unaligned_tokens_are_refused_whatever_the_route(B, n, which):
    """On the host: x and y start on 16-byte boundaries."""
    d, f, E = 64, 256, 2
    r = lambda *s: torch.randn(*s, device="cuda").bfloat16()  # noqa: E731
    x, w_r, W1, W2, W3 = r(B, 64, d), r(E, d), r(E, f, d), r(E, d, f), r(E, f, d)
    dims = lory.make_dims(B, 64, 64, d, f, E, "bf16")
    ws = torch.empty(lory.lory_moe_workspace_bytes(dims)[0], dtype=torch.uint8, device="cuda")
    lory.lory_moe_forward(dims, x, w_r, W1, W2, W3, torch.empty_like(x), torch.empty((B, E), device="cuda"), None, ws)
    bufs = dict(x=r(B, n, d), y=r(B, n, d))
    bufs[which] = r(B * n * d + 1)[1:].view(B, n, d)
    ddims = lory.make_dims(B, n, n, d, f, E, "bf16", lory.LORY_FLAG_REUSE_MERGED)
    with pytest.raises(lory.LoryError) as err:
        lory.lory_moe_ffn(ddims, bufs["x"], None, W1, W2, W3, bufs["y"], ws)
    assert err.value.status == -6
