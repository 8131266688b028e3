"""The block's RMSNorm kernels where a warp takes several token rows (more than 2368 tokens in the backward, 9472 in the forward):
the dgamma sums carried from row to row, all 296 partial sums, token counts that are no multiple of a block's eight rows."""
import pytest
import torch

import paper_2405_03133_b200 as lory

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("dtype,tokens,d", [("bf16", 4203, 520), ("bf16", 2501, 2056), ("bf16", 9999, 24), ("fp32", 4203, 260),
                                            ("fp32", 2501, 301), ("fp32", 9999, 5)])
def test_many_rows_against_torch(dtype, tokens, d, accumulate):
    """One expert, so the layer is a dense FFN: outputs and gradients against torch in float64."""
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    f, E, eps = 8, 1, 1e-5
    r = lambda *s: torch.randn(*s, generator=g, device="cuda").to(td)  # noqa: E731
    x, dy, gamma, w_r = r(1, tokens, d), r(1, tokens, d), r(d), r(E, d)
    W1, W2, W3 = (r(E, f, d) * 0.05).to(td), (r(E, d, f) * 0.2).to(td), (r(E, f, d) * 0.05).to(td)
    fwd, bwd = (lory.make_dims(1, tokens, tokens, d, f, E, dtype, flags)
                for flags in (0, lory.LORY_FLAG_ACCUMULATE_GRADS if accumulate else 0))
    ws = torch.empty(lory.lory_block_workspace_bytes(fwd)[1], dtype=torch.uint8, device="cuda")
    y, dx = torch.empty_like(x), torch.empty_like(x)
    old = (r(d) * 30.0).to(td)
    dgamma = old.clone()
    grads = [torch.zeros_like(t) for t in (w_r, W1, W2, W3)]
    rw = torch.empty(1, E, device="cuda")
    lory.lory_block_forward(fwd, x, gamma, eps, w_r, W1, W2, W3, y, rw, None, ws)
    lory.lory_block_backward(bwd, x, gamma, w_r, W1, W2, W3, dy, dx, dgamma, *grads, None, ws)
    xd, gd = x.double().requires_grad_(), gamma.double().requires_grad_()
    h = torch.nn.functional.rms_norm(xd, (d,), gd, eps)
    ref = xd + (torch.nn.functional.silu(h @ W1[0].double().T) * (h @ W3[0].double().T)) @ W2[0].double().T
    rx, rg = torch.autograd.grad(ref, (xd, gd), dy.double())
    if accumulate:
        rg = rg + old.double()
    tol = 2e-2 if dtype == "bf16" else 1e-4
    for a, b in ((y, ref.detach()), (dx, rx), (dgamma, rg)):
        assert ((a.double() - b).abs().max() / b.abs().max()).item() <= tol
