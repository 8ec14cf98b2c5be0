"""torch.jit.trace of the layer: the trace computes what the layer computes, forward and backward."""
import warnings

import pytest
import torch

from paper_2511_09323_b200.autograd import MoCFFN, moc_ffn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("options", ({}, {"recompute_up": True}, {"grouped": True}, {"post_silu": True}))
@pytest.mark.parametrize("trainable", (False, True))
def test_traced_module(options, trainable):
    torch.manual_seed(11)
    m = MoCFFN(64, 256, None if "grouped" in options else 32, **options).requires_grad_(trainable)
    x, y = (torch.randn(3, 100, 64, device="cuda").bfloat16().requires_grad_(trainable) for _ in range(2))
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")   # (sizes become constants of the trace, and torch.jit is on its way out)
        traced = torch.jit.trace(m, (x,), check_trace=False)
    got, want = traced(y), m(y)
    assert torch.equal(got, want)
    if not trainable:
        return
    leaves = [y, *m.parameters()]
    grads = [torch.autograd.grad(o, leaves, torch.ones_like(o)) for o in (got, want)]
    for a, b in zip(*grads):
        assert torch.equal(a, b)


def test_traced_function_reads_its_input():
    w = [torch.randn(96, 64, device="cuda").bfloat16() for _ in range(3)]
    x, y = (torch.randn(40, 64, device="cuda").bfloat16() for _ in range(2))
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")
        traced = torch.jit.trace(lambda a: moc_ffn(a, *w, 12, d_ff=88), (x,), check_trace=False)
    torch.testing.assert_close(traced(y).float(), moc_ffn(y, *w, 12, d_ff=88).float(), rtol=2e-2, atol=2e-2)
