"""The streaming merge and adjoint (warp-level matrix instructions) at the edges of their groups of 16 segments and 16
experts, with rows that end inside a 64-column piece and rows off the 32-byte boundary, overwriting and accumulating."""
import pytest
import torch

import paper_2405_03133_b200 as lory
from oracle import lory_oracle as O
from paper_2405_03133_b200.workloads import Workload, make_inputs

from gpu_util import max_rel, tdtype, to_dev

pytestmark = pytest.mark.gpu

SHAPES = [  # segments, experts, d, f
    (1, 1, 64, 64), (1, 16, 72, 136), (16, 17, 64, 72), (17, 16, 136, 64), (33, 9, 72, 200), (64, 16, 64, 72),
    (65, 16, 72, 72),            # one segment past the streaming adjoint's range
    (16, 32, 200, 136), (17, 32, 64, 64), (32, 31, 72, 64), (48, 32, 64, 72), (49, 20, 64, 72),
    (5, 33, 72, 64), (32, 64, 64, 136), (33, 48, 64, 64), (300, 8, 64, 64),
]


@pytest.mark.parametrize("S,E,d,f", SHAPES)
@pytest.mark.parametrize("accumulate", [False, True])
def test_streaming_merge_and_adjoint(S, E, d, f, accumulate):
    wl = Workload("stream", B=S, L=32, T=32, d=d, f=f, E=E, dtype="bf16", w_r_std=2.0)
    if S % 4 == 0:
        wl = wl.with_(B=S // 4, L=128)
    inp = make_inputs(wl)
    a = (inp["x"], inp["w_r"], inp["W1"], inp["W2"], inp["W3"], wl.T)
    y, _, _ = O.forward(*a)
    ref = O.backward(*a, inp["dy"])
    x, w_r, W1, W2, W3, dy = (to_dev(inp[k], wl) for k in ("x", "w_r", "W1", "W2", "W3", "dy"))
    dims = lory.make_dims(wl.B, wl.L, wl.T, d, f, E, "bf16", lory.LORY_FLAG_ACCUMULATE_GRADS if accumulate else 0)
    # sized without the flag: a program that accumulates keeps one workspace for both kinds of call
    plain = lory.make_dims(wl.B, wl.L, wl.T, d, f, E, "bf16")
    ws = torch.empty(lory.lory_moe_workspace_bytes(plain)[1], dtype=torch.uint8, device="cuda")
    y_d, dx = torch.full_like(x, float("nan")), torch.full_like(x, float("nan"))
    rw = torch.empty((wl.S, E), dtype=torch.float32, device="cuda")
    drw = torch.empty_like(rw)
    grads, old = {}, {}
    for k, t in (("dw_r", w_r), ("dW1", W1), ("dW2", W2), ("dW3", W3)):
        o = (torch.randn_like(t, dtype=torch.float32) * float(abs(ref[k]).max() or 1.0)).to(tdtype(wl))
        old[k] = o.double().cpu().numpy()
        grads[k] = o.clone() if accumulate else torch.full_like(o, float("nan"))
    lory.lory_moe_forward(plain, x, w_r, W1, W2, W3, y_d, rw, None, ws)
    lory.lory_moe_backward(dims, x, w_r, W1, W2, W3, dy, dx, grads["dw_r"], grads["dW1"], grads["dW2"], grads["dW3"], drw, ws)
    lory.lory_check_status(plain, ws)
    errs = {"y": max_rel(y_d.double().cpu().numpy(), y), "dx": max_rel(dx.double().cpu().numpy(), ref["dx"]),
            "d_route_w": max_rel(drw.double().cpu().numpy(), ref["d_route_w"])}
    for k, g in grads.items():
        errs[k] = max_rel(g.double().cpu().numpy(), ref[k] + (old[k] if accumulate else 0.0))
    assert all(v <= 2e-2 for v in errs.values()), errs
