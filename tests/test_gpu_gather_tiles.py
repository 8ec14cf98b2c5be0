"""The gathered plan where its gate projection changes tiles and its row loops and channel lists have remainders."""
import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu


# tiles of 32, 64 and 128 with rows, columns and contraction off their sizes; K off the rows taken at once; one token, few
# and many token blocks of the channel lists, and the channels' pairs found without lists (up to 4096 tokens)
@pytest.mark.parametrize("tokens, d, F, K", ((1, 8, 9, 5), (33, 40, 31, 31), (256, 128, 512, 64), (257, 24, 1000, 127), (4096, 8, 64, 8),
                                             (4097, 8, 64, 8), (770, 24, 833, 7), (1665, 136, 1501, 33), (4100, 16, 600, 3)))
def test_f32_against_fp64(tokens, d, F, K):
    g = torch.Generator(device="cuda").manual_seed(tokens)
    x, dD = (torch.randn(tokens, d, generator=g, device="cuda") for _ in range(2))
    wg, wu, wd = (torch.randn(F, d, generator=g, device="cuda") / d ** 0.5 for _ in range(3))
    out, idx, tg, tu = B.moc_ffn_forward(x, wg, wu, wd, K)
    got = B.moc_ffn_backward(x, wg, wu, wd, idx, tg, tu, dD)
    assert B.moc_last_device_status() == B.MOC_OK
    X, D, Wg, Wu, Wd = (t.double() for t in (x, dD, wg, wu, wd))
    G, at = X @ Wg.T, idx.long()
    assert (at[:, 1:] > at[:, :-1]).all() and (at >= 0).all() and (at < F).all()
    kept = torch.zeros_like(G, dtype=torch.bool).scatter_(1, at, True)
    tau = G.topk(K, dim=1).values[:, -1:]
    assert (kept | (G < tau + 1e-5)).all() and (~kept | (G > tau - 1e-5)).all()
    gv, uv = G * kept, (X @ Wu.T) * kept
    s = torch.sigmoid(gv)
    dz = (D @ Wd.T) * kept
    z, du, dg = s * gv * uv, dz * s * gv, dz * uv * s * (1 + gv * (1 - s))
    pairs = {"out": (out, z @ Wd), "gate": (tg, G.gather(1, at)), "up": (tu, uv.gather(1, at)), "grad_x": (got["grad_x"], dg @ Wg + du @ Wu),
             "w_down": (got["grad_w_down"], z.T @ D), "w_up": (got["grad_w_up"], du.T @ X), "w_gate": (got["grad_w_gate"], dg.T @ X)}
    for name, (v, want) in pairs.items():
        assert (v.double() - want).abs().max() <= 2e-5 * max(1.0, want.abs().max().item()), name
