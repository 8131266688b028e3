"""The decode kernels (cached merged FFN on a few new tokens) at the edges of their token groups and tilings."""
import numpy as np
import pytest
import torch

import paper_2405_03133_b200 as lory
from oracle import lory_oracle as O
from paper_2405_03133_b200.workloads import Workload, make_inputs, round_to_bf16

from gpu_util import max_rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d,f,counts", [
    (1, 64, 64, (1, 8, 9, 16, 17, 33, 64)),
    (3, 72, 136, (1, 7, 16, 31, 32, 48)),      # rows and columns that end inside a 64 x 64 block
    (2, 584, 8, (1, 12, 40)),                  # more column blocks than warps, fewer rows than a tile
    (16, 640, 1024, (3, 16, 24)),              # several tiles per CTA; the down projection on 16-row tiles
    (32, 896, 456, (8, 13, 20, 50)),           # two weight tiles at a time
    (32, 568, 456, (17, 32, 33, 64)),          # tcgen05: whole down-projection tiles, the last one half outside
    (16, 72, 328, (32, 33, 48, 49)),           # tcgen05: two column blocks in a stage of three; half-filled gate tiles
])
def test_decode_with_cached_merged_ffn(B, d, f, counts):
    wl = Workload("decode", B=B, L=64, T=64, d=d, f=f, E=3, dtype="bf16", w_r_std=2.0, seed=21)
    inp = make_inputs(wl)
    rng = np.random.default_rng(3)
    x, w_r, W1, W2, W3 = (to_dev(inp[k], wl) for k in ("x", "w_r", "W1", "W2", "W3"))
    dims = lory.make_dims(B, wl.L, wl.L, d, f, wl.E, "bf16")
    ws = torch.empty(lory.lory_moe_workspace_bytes(dims)[0], dtype=torch.uint8, device="cuda")
    rw = torch.empty((B, wl.E), dtype=torch.float32, device="cuda")
    lory.lory_moe_forward(dims, x, w_r, W1, W2, W3, torch.empty_like(x), rw, None, ws)
    for n in counts:
        new = round_to_bf16(rng.standard_normal((B, n, d)).astype(np.float32))
        _, ref, _ = O.prompt_only_inference(inp["x"], new, inp["w_r"], inp["W1"], inp["W2"], inp["W3"])
        xd = to_dev(new, wl)
        ddims = lory.make_dims(B, n, n, d, f, wl.E, "bf16", lory.LORY_FLAG_REUSE_MERGED)
        outs = []
        for _ in range(2):   # back to back: each kernel may start before the previous one has ended
            y = torch.full_like(xd, float("nan"))
            lory.lory_moe_ffn(ddims, xd, None, W1, W2, W3, y, ws)
            outs.append(y)
        lory.lory_check_status(ddims, ws)
        for y in outs:
            assert max_rel(y.double().cpu().numpy(), ref) <= 2e-2, n
