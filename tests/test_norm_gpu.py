"""The RMSNorm kernels of the block: rows that fit registers at each size, longer rows and rows that are no whole vectors."""
import pytest
import torch

import paper_2405_03133_b200 as lory

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [("bf16", 8), ("bf16", 520), ("bf16", 1032), ("bf16", 2048), ("bf16", 2056), ("fp32", 3),
                                     ("fp32", 260), ("fp32", 1028), ("fp32", 2050), ("fp32", 2052)])
def test_block_norm_against_torch(dtype, d):
    """One expert, so the layer is a dense FFN: outputs and gradients against torch in float64."""
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    B, L, T, f, E, eps = 2, 36, 18, 8, 1, 1e-5
    r = lambda *s: torch.randn(*s, generator=g, device="cuda").to(td)  # noqa: E731
    x, dy, gamma, w_r = r(B, L, d), r(B, L, d), r(d), r(E, d)
    W1, W2, W3 = (r(E, f, d) * 0.05).to(td), (r(E, d, f) * 0.2).to(td), (r(E, f, d) * 0.05).to(td)
    dims = lory.make_dims(B, L, T, d, f, E, dtype)
    ws = torch.empty(lory.lory_block_workspace_bytes(dims)[1], dtype=torch.uint8, device="cuda")
    y, dx, dgamma = torch.empty_like(x), torch.empty_like(x), torch.empty_like(gamma)
    grads = [torch.empty_like(t) for t in (w_r, W1, W2, W3)]
    rw = torch.empty(B * L // T, E, device="cuda")
    lory.lory_block_forward(dims, x, gamma, eps, w_r, W1, W2, W3, y, rw, None, ws)
    lory.lory_block_backward(dims, x, gamma, w_r, W1, W2, W3, dy, dx, dgamma, *grads, None, ws)
    xd, gd = x.double().requires_grad_(), gamma.double().requires_grad_()
    h = torch.nn.functional.rms_norm(xd, (d,), gd, eps)
    ref = xd + (torch.nn.functional.silu(h @ W1[0].double().T) * (h @ W3[0].double().T)) @ W2[0].double().T
    rx, rg = torch.autograd.grad(ref, (xd, gd), dy.double())
    tol = 2e-2 if dtype == "bf16" else 1e-4
    for a, b in ((y, ref.detach()), (dx, rx), (dgamma, rg)):
        assert ((a.double() - b).abs().max() / b.abs().max()).item() <= tol
