"""Decode of three to five tokens on both sides of the most channels that the gathering plan's gate kernel takes in one go (csrc/decode_form.h)."""
import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tokens,d,F,share", [
    (3, 1600, 18944, 64), (3, 1600, 18945, 64), (4, 1600, 18952, 8), (5, 1024, 18950, 64), (3, 1024, 32768, 16),   # 18944 channels on 148 SMs
    (3, 4880, 18448, 64), (5, 4880, 18448, 8),                                                                     # 90 million weights of a matrix
    (3, 2504, 10000, 12), (3, 2504, 10000, 32), (3, 2504, 9976, 32),                                               # 25 million, a tenth in use
])
def test_result(tokens, d, F, share):
    g = torch.Generator(device="cuda").manual_seed(tokens + F)
    k = F // share
    x = torch.randn(tokens, d, generator=g, device="cuda").bfloat16()
    w = [(torch.randn(F, d, generator=g, device="cuda") * 0.02).bfloat16() for _ in range(3)]
    ws = B.alloc_workspace(B.make_desc(tokens, d, F, k, x.dtype), B.MOC_OP_DECODE)
    ws.fill_(0xff)    # nothing depends on what the workspace held
    out = B.moc_ffn_decode(x, *w, k, workspace=ws)
    _, idx, _, _ = B.moc_ffn_forward(x, *w, k)
    torch.cuda.synchronize()
    assert B.moc_last_device_status() == B.MOC_OK
    # against 64 bits on the forward's picks: Z' and the sum are rounded to bf16, 2^-9 of each term and of the whole; a token whose K-th and next
    # gate values are closer than sums in fp32 tell may keep the other of the two, sqrt(2 / k) of that token
    gate = x.double() @ w[0].double().T
    kept = torch.zeros_like(gate).scatter_(1, idx.long(), 1)
    ref = (torch.nn.functional.silu(gate) * (x.double() @ w[1].double().T) * kept) @ w[2].double()
    off = (out.double() - ref).norm(dim=1) / ref.norm(dim=1)
    assert off.max() <= 2.0 ** -8 + (2.0 / k) ** 0.5 and (off > 2.0 ** -8).sum() <= 1, off
