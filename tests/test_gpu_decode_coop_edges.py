"""The one-kernel decode form for one and two tokens (csrc/decode_coop.cuh): columns that the warps' shares do not divide, and gate
values where the parts of the threshold's bin decide, leave the choice open, or overflow."""
import numpy as np
import pytest
import torch

from oracle import moc_oracle as orc
from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu


# one vector of columns; parts of a warp's share; a share and a vector more; the widest row and one vector less; few rows to a CTA
@pytest.mark.parametrize("d,F", [(8, 300), (264, 333), (1032, 1200), (2056, 900), (4088, 640), (4096, 149), (4096, 5461)])
@pytest.mark.parametrize("T", [1, 2])
@pytest.mark.parametrize("block", [False, True])
def test_columns_that_the_shares_do_not_divide(d, F, T, block):
    g = torch.Generator(device="cuda").manual_seed(d + F + T)
    k = max(1, F // 8)
    x = torch.randn(T, d, generator=g, device="cuda").bfloat16()
    wg, wu, wd = ((torch.randn(F, d, generator=g, device="cuda") * 0.05).bfloat16() for _ in range(3))
    gamma = torch.ones(d, device="cuda", dtype=torch.bfloat16)
    if block:
        xin = (x.double() * torch.rsqrt(x.double().square().mean(1, keepdim=True) + 1e-5)).float().bfloat16()
        out = B.moc_ffn_decode_block(x, gamma, 1e-5, wg, wu, wd, k)
    else:
        xin = x
        out, kept = B.moc_ffn_decode_probe(x, wg, wu, wd, k)
        assert (kept.sum(1) == k).all()
    torch.cuda.synchronize()
    assert B.moc_last_device_status() == B.MOC_OK
    gate = xin.double() @ wg.double().T
    if block:
        kept = torch.zeros_like(gate).scatter_(1, gate.topk(k, dim=1).indices, 1)
    # a pick may differ only where sums in fp32 cannot tell the values apart: within 2^-24 sqrt(d) of the largest gate value or so
    least = (gate + (kept == 0) * 1e9).min(1).values
    assert (gate - (kept != 0) * 1e9).amax(1).le(least + 1e-5 * gate.abs().amax()).all()
    ref = (torch.nn.functional.silu(gate) * (xin.double() @ wu.double().T) * kept) @ wd.double() + (x.double() if block else 0)
    # half a unit of bf16's last place of the largest output; in the block form also of the layer's input, which the kernel rounds from
    # fp32 sums (a rare element one step off)
    assert (out.double() - ref).abs().max() <= (2.0 ** -8 if not block else 2.0 ** -6) * ref.abs().max()


def _probe(rows, k, d=16):
    """The kept masks of given gate rows: column i of W_gate under a one-hot x."""
    T, F = rows.shape
    wg = torch.zeros(F, d)
    x = torch.zeros(T, d)
    for t in range(T):
        wg[:, 3 + t] = torch.from_numpy(rows[t])
        x[t, 3 + t] = 1
    wg, x = wg.bfloat16().cuda(), x.bfloat16().cuda()
    zeros = torch.zeros_like(wg)
    kept = B.moc_ffn_decode_probe(x, wg, zeros, zeros, k)[1].cpu().numpy()
    assert B.moc_last_device_status() == B.MOC_OK
    return kept


@pytest.mark.parametrize("F", [2048, 11008])
@pytest.mark.parametrize("T", [1, 2])
def test_parts_of_the_threshold_bin(T, F):
    """bf16 values: 128 to an octave, so a narrow bin of [2^-5, 2^4) holds copies of one value.  Rows in which the K-th value is one
    of 1, 2, 15, 16, 17 or 300 equal ones, all or some of them kept, inside that range, at its ends and outside."""
    rng = np.random.default_rng(F + T)
    low = -np.abs(rng.standard_normal(F)).astype(np.float32) - 16
    for value in (2.0 ** -5, 2.0 ** -5 * (1 - 2.0 ** -8), 1.0, 1.5078125, 16.0 * (1 - 2.0 ** -8), 16.0, 40.0, 2.0 ** -20):
        for copies in (1, 2, 15, 16, 17, 300):
            for taken in {1, copies // 2, copies} - {0}:
                rows = np.stack([low] * T)
                for t in range(T):
                    at = rng.permutation(F)
                    rows[t, at[:copies]] = value
                    rows[t, at[copies:copies + 100]] = value * (1 + rng.integers(1, 100, 100) * 2.0 ** -7)
                rows = torch.from_numpy(rows).bfloat16().float().numpy()
                k = 100 + taken
                want = np.zeros((T, F), np.uint8)
                np.put_along_axis(want, orc.topk(rows, k).astype(np.int64), 1, axis=1)
                np.testing.assert_array_equal(_probe(rows, k), want, err_msg=f"{value} x {copies}, {taken} kept")
