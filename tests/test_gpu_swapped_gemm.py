"""Forward on the tensor-core plan where its GEMMs may exchange their operands (a few hundred tokens), against fp32 products."""
import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu


# tokens at the edges of 64-column steps and of 256-row blocks; d_model and d_ff off every tile's size; contractions whose
# parts do not divide them
@pytest.mark.parametrize("tokens, d, F, pad, K", ((257, 1032, 5461, 43, 683), (320, 4096, 11008, 0, 1376), (321, 2048, 11000, 0, 1375),
                                                  (385, 768, 2048, 0, 256), (513, 2048, 5504, 0, 688), (577, 1000, 8200, 0, 100),
                                                  (1100, 1024, 2730, 6, 341), (1300, 4096, 11008, 0, 1376)))
def test_forward_against_fp32(tokens, d, F, pad, K):
    g = torch.Generator(device="cuda").manual_seed(tokens)
    x = torch.randn(tokens, d, generator=g, device="cuda").bfloat16()
    wg, wu, wd = ((torch.randn(F + pad, d, generator=g, device="cuda") / d ** 0.5).bfloat16() for _ in range(3))
    if pad:
        for w in (wg, wu, wd):
            w[F:] = 0
    out, idx, tg, tu = B.moc_ffn_forward(x, wg, wu, wd, K, d_ff=F)
    assert B.moc_last_device_status() == B.MOC_OK
    G, U = x.float() @ wg[:F].float().T, x.float() @ wu[:F].float().T
    at = idx.long()
    assert (at[:, 1:] > at[:, :-1]).all() and (at >= 0).all() and (at < F).all()
    tau = G.topk(K, dim=1).values[:, -1:]
    kept = torch.zeros_like(G, dtype=torch.bool).scatter_(1, at, True)
    assert (kept | (G < tau + 1e-3)).all() and (~kept | (G > tau - 1e-3)).all()
    for got, want in ((tg, G.gather(1, at)), (tu, U.gather(1, at))):
        assert (got.float() - want).abs().max() <= 2 ** -8 * want.abs().max() + 1e-3
    ref = (torch.nn.functional.silu(G) * U * kept).bfloat16().float() @ wd[:F].float()
    assert (out.float() - ref).norm() <= 1e-2 * ref.norm()
    assert (out.float() - ref).abs().max() <= 0.05 * ref.abs().max()


# one and two operand pairs per part; a part that ends inside a block; few and many tokens
@pytest.mark.parametrize("tokens, d, F, K", ((257, 1032, 5460, 683), (300, 4096, 2048, 256), (513, 2048, 5504, 688), (1111, 2048, 5461, 683),
                                             (1300, 520, 1000, 125), (2049, 768, 2048, 256)))
def test_backward_against_fp32(tokens, d, F, K):
    g = torch.Generator(device="cuda").manual_seed(tokens)
    x, dD = (torch.randn(tokens, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    wg, wu, wd = ((torch.randn(F, d, generator=g, device="cuda") / d ** 0.5).bfloat16() for _ in range(3))
    _, idx, tg, tu = B.moc_ffn_forward(x, wg, wu, wd, K)
    got = B.moc_ffn_backward(x, wg, wu, wd, idx, tg, tu, dD)
    assert B.moc_last_device_status() == B.MOC_OK
    at, gv, uv = idx.long(), tg.float(), tu.float()
    dz = (dD.float() @ wd.float().T).gather(1, at)
    s = torch.sigmoid(gv)
    dense = lambda v: torch.zeros(tokens, F, device="cuda").scatter_(1, at, v).bfloat16().float()  # noqa: E731
    z, du, dg = dense(s * gv * uv), dense(dz * s * gv), dense(dz * uv * s * (1 + gv * (1 - s)))
    want = {"grad_x": dg @ wg.float() + du @ wu.float(), "grad_w_down": z.T @ dD.float(), "grad_w_up": du.T @ x.float(),
            "grad_w_gate": dg.T @ x.float()}
    for name, w in want.items():
        v = got[name].float()
        assert (v - w).norm() <= 1e-2 * w.norm(), name
        assert (v - w).abs().max() <= 0.05 * w.abs().max(), name
