"""The small batches' selector without the saved triple lists its kept channels during the search (csrc/decode_kernels.cuh): against the
forward that saves, which goes by a bitmap, where the list does not fit, the row is not in fours, or values tie."""
import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [100, 127, 128, 130, 4096, 4099, 11009, 20002])  # a sample of 128 values; fours of 1024 threads
@pytest.mark.parametrize("share", [0.0, 0.125, 0.45, 1.0])                       # the list has room for 8192
@pytest.mark.parametrize("ties", [False, True])
def test_list_of_kept_channels(F, share, ties):
    T, d = 33, 64
    k = max(1, round(F * share))
    g = torch.Generator(device="cuda").manual_seed(F + k)
    x = torch.randn(T, d, generator=g, device="cuda").bfloat16()
    wg, wu, wd = ((torch.randn(F, d, generator=g, device="cuda") * 0.1).bfloat16() for _ in range(3))
    if ties:
        wg[F // 3:] = wg[: F - F // 3].clone()   # pairs of equal gate values throughout
    ws = B.alloc_workspace(B.make_desc(T, d, F, k, x.dtype), B.MOC_OP_DECODE)
    ws.fill_(0xff)
    out = B.moc_ffn_decode(x, wg, wu, wd, k, workspace=ws)
    _, idx, _, _ = B.moc_ffn_forward(x, wg, wu, wd, k)
    torch.cuda.synchronize()
    assert B.moc_last_device_status() == B.MOC_OK
    gate = x.double() @ wg.double().T
    kept = torch.zeros_like(gate).scatter_(1, idx.long(), 1)
    ref = (torch.nn.functional.silu(gate) * (x.double() @ wu.double().T) * kept) @ wd.double()
    # both select from the same fp32 gate values; Z' and the sum are rounded to bf16: 2^-9 of each term and of the whole
    assert (out.double() - ref).norm() <= 2.0 ** -7 * ref.norm()
    assert ((out.double() - ref).norm(dim=1) <= 2.0 ** -6 * ref.norm(dim=1) + 1e-6 * ref.abs().max()).all()
