"""Small batches around as many tokens as SMs, where the selector goes from one CTA per SM to two, against fp32 products."""
import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d, F, K", ((384, 1024, 128), (512, 4397, 550), (520, 9000, 600)))   # two CTAs fit an SM; just; not
@pytest.mark.parametrize("extra", (-115, -1, 0, 1, 108))
def test_decode_around_one_token_per_sm(d, F, K, extra):
    tokens = min(256, torch.cuda.get_device_properties(0).multi_processor_count + extra)
    g = torch.Generator(device="cuda").manual_seed(tokens + F)
    x = torch.randn(tokens, d, generator=g, device="cuda").bfloat16()
    w = [(torch.randn(F, d, generator=g, device="cuda") / d ** 0.5).bfloat16() for _ in range(3)]
    G, U = (x.float() @ m.float().T for m in w[:2])
    kept = torch.zeros_like(G).scatter_(1, G.topk(K, dim=1).indices, 1.0)
    want = (torch.nn.functional.silu(G) * U * kept).bfloat16().float() @ w[2].float()
    got = B.moc_ffn_decode(x, *w, K).float()
    # sums of bf16 products rounded to bf16, and a channel of nearly the same gate value kept for another here and there
    assert (got - want).norm() <= 1e-2 * want.norm()
    assert (got - want).abs().max() <= 0.05 * want.abs().max()
    assert B.moc_last_device_status() == B.MOC_OK
