"""The modules under the parts of torch that look into an autograd function: tracing, forward mode, function transforms,
saved-tensor hooks, and errors raised inside the forward and the backward node."""
import pytest
import torch
import torch.utils.checkpoint

import paper_2405_03133_b200 as lory
from paper_2405_03133_b200.layer import LoryBlock, LoryMoE

pytestmark = pytest.mark.gpu

B, L, T, d, f, E = 2, 128, 64, 64, 136, 4


def layer(cls=LoryMoE, frozen=False):
    m = cls(d, f, E, T, generator=torch.Generator(device="cuda").manual_seed(1))
    return m.requires_grad_(not frozen)


def tokens(seed):
    return torch.randn(B, L, d, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed)).bfloat16()


@pytest.mark.parametrize("cls", [LoryMoE, LoryBlock])
@pytest.mark.parametrize("grad", [True, False])
def test_traced_module_computes_for_other_inputs(cls, grad):
    m = layer(cls)
    with torch.set_grad_enabled(grad):
        traced = torch.jit.trace(m, (tokens(2),), check_trace=False)
        x = tokens(3)
        assert torch.equal(traced(x), m(x))
    if grad:
        xs = [tokens(4).requires_grad_() for _ in range(2)]
        dy = tokens(5)
        ga, gb = (torch.autograd.grad(fn(x), [x, m.W2], dy) for fn, x in zip((traced, m), xs))
        assert all(torch.equal(a, b) for a, b in zip(ga, gb))


@pytest.mark.parametrize("grad,frozen", [(True, False), (True, True), (False, False)])
def test_forward_mode_is_refused(grad, frozen):
    m = layer(frozen=frozen)
    with torch.autograd.forward_ad.dual_level(), torch.set_grad_enabled(grad):
        x = torch.autograd.forward_ad.make_dual(tokens(2), tokens(3))
        with pytest.raises(NotImplementedError):
            m(x)
        m(tokens(4))                        # no tangent, no objection


@pytest.mark.parametrize("frozen", [False, True])
def test_function_transforms_are_refused(frozen):
    m = layer(frozen=frozen)
    x = tokens(2)
    for call in (lambda: torch.vmap(m)(torch.stack([x, x])), lambda: torch.func.grad(lambda z: m(z).float().sum())(x),
                 lambda: torch.func.jvp(m, (x,), (x,))):
        with pytest.raises(RuntimeError):
            call()


def test_saved_tensor_hooks_and_checkpointing():
    m, dy = layer(LoryBlock), tokens(3)

    def grads(fn):
        x = tokens(2).requires_grad_()
        return torch.autograd.grad(fn(x), [x, *m.parameters()], dy)

    def on_cpu(x):
        with torch.autograd.graph.save_on_cpu():
            return m(x)

    ref = grads(m)
    for fn in (on_cpu, lambda x: torch.utils.checkpoint.checkpoint(m, x, use_reentrant=False)):
        assert all(torch.equal(a, b) for a, b in zip(grads(fn), ref))


def test_errors_of_the_library_surface_from_both_nodes():
    m = layer()
    for grad in (True, False):
        with torch.set_grad_enabled(grad), pytest.raises(lory.LoryError) as err:
            m(tokens(2)[:, :100].contiguous())       # no whole number of segments
        assert err.value.status == -2
    x = tokens(2).requires_grad_()
    y = m(x)
    # a gradient that does not start on a 16-byte boundary: refused on the host, before anything is launched
    dy = torch.zeros(y.numel() + 1, device="cuda", dtype=torch.bfloat16)[1:].view_as(y)
    with pytest.raises(lory.LoryError) as err:
        torch.autograd.grad(y, x, dy, retain_graph=True)
    assert err.value.status == -6
    g, = torch.autograd.grad(y, x, tokens(3))        # the saved activations are still there
    assert torch.isfinite(g).all()
