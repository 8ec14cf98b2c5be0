"""Which form of the small-batch plan a decode call takes (csrc/api.cu: decode_form, small_batch_faster_than_gathering), and that
each gives what the forward that keeps its picks gives, on both sides of the rule's sizes."""
import os

import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu
ENVIRONMENT = [v for v in ("MOC_FFN_DECODE", "MOC_FFN_SB_OVERLAP", "MOC_FFN_SB_FUSED", "MOC_FFN_SB_MIN_TOKENS") if v in os.environ]
THREE, OVERLAPPED, ONE, CHAIN = "three", "overlapped", "one", "chain"


def _form(launches):
    if "sb_fused" in launches:
        return ONE
    if "dec_down" in launches:
        return CHAIN
    return OVERLAPPED if launches["sb_gate_up"] == 2 else THREE


@pytest.mark.skipif(bool(ENVIRONMENT), reason="another form is asked for")
@pytest.mark.parametrize("tokens,d,F,k,form", [
    (6, 384, 776, 97, ONE), (6, 384, 784, 98, THREE), (32, 384, 784, 98, THREE),             # 300 thousand weights of a matrix
    (16, 2560, 7024, 878, THREE), (16, 2560, 7032, 879, OVERLAPPED),                         # 18 million
    (16, 2560, 9765, 1220, THREE), (16, 2560, 9767, 1221, ONE), (16, 2560, 9764, 1220, OVERLAPPED),   # 25 million, channels not in fours
    (32, 2560, 7032, 879, OVERLAPPED), (33, 2560, 7032, 879, THREE),
    (44, 2560, 11720, 1465, OVERLAPPED), (45, 2560, 11720, 1465, THREE),                     # 30 million
    (16, 4232, 7032, 879, ONE), (17, 4232, 7032, 879, OVERLAPPED),                           # wide layers
    (3, 1440, 3840, 480, THREE), (4, 2560, 7032, 440, OVERLAPPED), (3, 2560, 11716, 732, OVERLAPPED),   # three to five tokens: below 30 million
    (3, 2560, 11720, 732, CHAIN), (3, 2560, 11720, 1465, OVERLAPPED), (3, 4096, 9768, 1221, CHAIN),     # or 40 with 0.3 in use
    (4, 2560, 9767, 610, CHAIN),                                                             # 25 million not in fours
])
def test_form_and_result(tokens, d, F, k, form):
    g = torch.Generator(device="cuda").manual_seed(tokens + F)
    x = torch.randn(tokens, d, generator=g, device="cuda").bfloat16()
    w = [torch.zeros(F + 8, d, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
    for m in w:
        m[:F] = (torch.randn(F, d, generator=g, device="cuda") * 0.02).bfloat16()
        m[F:] = 3.0   # never selected, never read as channels
    ws = B.alloc_workspace(B.make_desc(tokens, d, F, k, x.dtype, d_ff_ld=F + 8), B.MOC_OP_DECODE)
    ws.fill_(0xff)    # nothing depends on what the workspace held
    B.moc_profile_enable(True)
    out = B.moc_ffn_decode(x, *w, k, d_ff=F, workspace=ws)
    launches = {n: v[0] for n, v in B.moc_profile_collect().items() if v[0]}
    B.moc_profile_enable(False)
    assert _form(launches) == form, launches
    _, idx, _, _ = B.moc_ffn_forward(x, *w, k, d_ff=F)
    torch.cuda.synchronize()
    assert B.moc_last_device_status() == B.MOC_OK
    # against 64 bits on the forward's picks.  Z' is rounded to bf16, the sum to bf16: each value of the sum is off by 2^-9 of its
    # term at most, the whole by 2^-9 of its norm or so and 2^-9 of itself; a token whose K-th and next gate values are closer than sums in
    # fp32 tell may keep the other of the two: sqrt(2 / k) of that token
    gate = x.double() @ w[0][:F].double().T
    kept = torch.zeros_like(gate).scatter_(1, idx.long(), 1)
    ref = (torch.nn.functional.silu(gate) * (x.double() @ w[1][:F].double().T) * kept) @ w[2][:F].double()
    off = (out.double() - ref).norm(dim=1) / ref.norm(dim=1)
    assert off.max() <= 2.0 ** -8 + (2.0 / k) ** 0.5 and (off > 2.0 ** -8).sum() <= 1, off
