"""The wide GEMM's epilogue at the edges of its chunks: 32 rows, 32 fp32 or 64 bf16 columns, one or two accumulators, tile after tile."""
import ctypes

import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("m", [31, 33, 257, 74 * 256 * 2 + 40])
@pytest.mark.parametrize("n", [32, 36, 100, 256, 260, 316, 508, 512, 520, 1100])
def test_fp32_columns(m, n):
    k = 136
    gen = torch.Generator(device="cuda").manual_seed(m + n)
    a = torch.randn(m, k, generator=gen, device="cuda").bfloat16()
    b = torch.randn(n, k, generator=gen, device="cuda").bfloat16()
    out = torch.full((m + 1, n), float("nan"), device="cuda")
    rc = B.load().moc_tc_gemm_bf16(m, n, k, _ptr(a), 0, k, _ptr(b), 0, k, _ptr(out), n,
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == B.MOC_OK
    want = a.double() @ b.double().t()
    # sums of k exact products, added in fp32
    assert (out[:m].double() - want).abs().max() <= k * 2.0 ** -24 * (a.double().abs() @ b.double().abs().t()).max()
    assert out[m:].isnan().all()
    assert B.moc_last_device_status() == B.MOC_OK


@pytest.mark.parametrize("tokens", [2049, 9500])
@pytest.mark.parametrize("d_model", [40, 264, 328, 520, 1000])
def test_bf16_columns(tokens, d_model):
    """With every channel kept the layer is the dense gated layer; d_model columns leave the down projection."""
    d_ff = 128
    gen = torch.Generator(device="cuda").manual_seed(tokens + d_model)
    x = torch.randn(tokens, d_model, generator=gen, device="cuda").bfloat16()
    wg, wu, wd = ((torch.randn(d_ff, d_model, generator=gen, device="cuda") * d_model ** -0.5).bfloat16() for _ in range(3))
    out = torch.full((tokens + 1, d_model), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.moc_ffn_forward(x, wg, wu, wd, d_ff, save=False, out=out[:tokens])
    g, u = x.double() @ wg.double().t(), x.double() @ wu.double().t()
    want = (g * torch.sigmoid(g) * u) @ wd.double()
    # u, z and the output are each rounded to bf16 (2^-9 of the value at most); the sums' errors are far smaller
    assert (out[:tokens].double() - want).norm() <= 3 * 2.0 ** -9 * want.norm()
    assert (out[:tokens].double() - want).abs().amax(0).max() <= 3 * 2.0 ** -7 * want.abs().max()
    assert out[tokens:].isnan().all()
    assert B.moc_last_device_status() == B.MOC_OK
