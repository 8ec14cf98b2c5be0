"""The one-kernel form of the small-batch plan (csrc/small_batch_fused.cuh) on both sides of the rule for the contraction blocks of a stage
(csrc/api.cu: fused_layout): rows that are whole 128-byte lines, whole sectors or neither, 31 and 32 channels to a CTA, eight and nine tokens."""
import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tokens,d,F", [
    (8, 1032, 4340), (12, 1032, 4216), (12, 1032, 4219), (32, 1040, 3712), (12, 4104, 3400), (12, 4160, 3400), (8, 2560, 8448), (9, 2560, 8448),
    (3, 3592, 9557), (12, 2056, 16000),
])
def test_top_k(tokens, d, F):
    g = torch.Generator(device="cuda").manual_seed(tokens + F)
    k = F // 8
    x = torch.randn(tokens, d, generator=g, device="cuda").bfloat16()
    w = [(torch.randn(F, d, generator=g, device="cuda") * 0.02).bfloat16() for _ in range(3)]
    _, idx, _, _ = B.moc_ffn_forward(x, *w, k)
    out = B.moc_ffn_forward(x, *w, k, save=False)[0]
    torch.cuda.synchronize()
    assert B.moc_last_device_status() == B.MOC_OK
    gate = x.double() @ w[0].double().T
    kept = torch.zeros_like(gate).scatter_(1, idx.long(), 1)
    _check(out, gate, kept, x, w, k)


@pytest.mark.parametrize("tokens,d,F", [(6, 4104, 10944), (32, 4104, 10944), (16, 4112, 10944), (16, 4872, 4400), (16, 3336, 8896)])
def test_two_of_eight(tokens, d, F):
    g = torch.Generator(device="cuda").manual_seed(tokens + F)
    x = torch.randn(tokens, d, generator=g, device="cuda").bfloat16()
    w = [(torch.randn(F, d, generator=g, device="cuda") * 0.02).bfloat16() for _ in range(3)]
    out = B.moc_ffn_decode(x, *w, F // 4, grouped=True)
    torch.cuda.synchronize()
    assert B.moc_last_device_status() == B.MOC_OK
    gate = x.double() @ w[0].double().T
    kept = torch.zeros(tokens, F // 8, 8, device="cuda", dtype=torch.double).scatter_(2, gate.view(tokens, F // 8, 8).topk(2, dim=2).indices, 1)
    _check(out, gate, kept.view(tokens, F), x, w, F // 4)


def _check(out, gate, kept, x, w, k):
    """Z' and the sum are rounded to bf16, 2^-9 of each term and of the whole; a few picks of the call may differ where two gate values are closer
    than sums in fp32 tell: sqrt(2 / k) of their token each."""
    ref = (torch.nn.functional.silu(gate) * (x.double() @ w[1].double().T) * kept) @ w[2].double()
    off = (out.double() - ref).norm(dim=1) / ref.norm(dim=1)
    assert off.max() <= 2.0 ** -8 + (2.0 / k) ** 0.5 and (off > 2.0 ** -8).sum() <= 2, off
