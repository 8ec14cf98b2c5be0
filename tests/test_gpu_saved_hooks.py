"""Saved-tensor hooks around the layer: what they hand back is checked before the library reads it."""
import pytest
import torch

from paper_2511_09323_b200.autograd import moc_ffn

pytestmark = pytest.mark.gpu


def _grads(pack, unpack, **options):
    g = torch.Generator(device="cuda").manual_seed(5)
    leaves = [torch.randn(n, 64, generator=g, device="cuda").bfloat16().requires_grad_() for n in (40, 96, 96, 96)]
    with torch.autograd.graph.saved_tensors_hooks(pack, unpack):
        out = moc_ffn(*leaves, 12, **options)
    return torch.autograd.grad(out, leaves, torch.ones_like(out))


@pytest.mark.parametrize("options", ({}, {"recompute_up": True}))
def test_what_hooks_may_and_may_not_hand_back(options):
    def same(t):
        return t
    want = _grads(same, same, **options)
    for got in (_grads(lambda t: t.cpu(), lambda t: t.cuda(), **options), _grads(same, torch.clone, **options)):
        for a, b in zip(got, want):
            torch.testing.assert_close(a, b, rtol=2e-2, atol=2e-2)
    with pytest.raises(ValueError, match="CUDA"):                     # offloaded and not brought back
        _grads(lambda t: t.cpu(), same, **options)
    with pytest.raises(ValueError, match="contiguous"):
        _grads(same, lambda t: t.t().contiguous().t() if t.dim() == 2 else t, **options)
    with pytest.raises(ValueError, match="contiguous"):               # the compact activations alone
        _grads(same, lambda t: t.repeat_interleave(2)[::2] if t.dim() == 1 else t, **options)
    with pytest.raises(ValueError, match="another form"):
        _grads(same, lambda t: t[: t.numel() // 2].clone() if t.dim() == 1 else t, **options)
    with pytest.raises(ValueError, match="another form"):
        _grads(same, lambda t: t.short() if t.dim() == 1 else t, **options)
