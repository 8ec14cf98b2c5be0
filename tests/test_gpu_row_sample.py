"""The backward element-wise step where its teams, its copies of the saved entries and its last form change."""
import numpy as np
import pytest
import torch

from oracle import parity
from paper_2511_09323_b200 import binding as B
from paper_2511_09323_b200 import synthetic as syn

pytestmark = pytest.mark.gpu


# widths on both sides of every team size, K that is and is not a multiple of 8 (bulk copies or plain loads of the saved
# rows), K = 1 and K = d_ff, and rows of which fewer than two fit an SM
@pytest.mark.parametrize("F,K", ((1024, 128), (1025, 7), (3072, 1), (3073, 384), (8192, 1023), (8193, 1024), (13000, 1624), (14000, 12),
                                 (200, 200)))
def test_backward_at_the_edges_of_the_element_wise_forms(F, K):
    w = syn.Workload(f"sample-{F}-{K}", "bf16", 301, 64, F, F, K, seed=F + K)
    wg, wu, wd = syn.make_weights(w)
    x, dD = syn.make_x(w), syn.make_grad_out(w)
    xd, wgd, wud, wdd, dDd = (t.cuda() for t in (x, wg, wu, wd, dD))
    _, idx, tg, tu = B.moc_ffn_forward(xd, wgd, wud, wdd, K)
    grads = B.moc_ffn_backward(xd, wgd, wud, wdd, idx, tg, tu, dDd)
    parity.check_backward({k: syn.to_f64(v) for k, v in grads.items()}, *map(syn.to_f64, (x, wg, wu, wd)), idx.cpu().numpy(),
                          syn.to_f64(tg), syn.to_f64(tu), syn.to_f64(dD), F, "bf16")
    # a saved index outside the row is left out and reported; the other tokens do not change
    bad = idx.clone()
    bad[300, 0] = -1
    got = B.moc_ffn_backward(xd, wgd, wud, wdd, bad, tg, tu, dDd, want=("x",))["grad_x"]
    assert B.moc_last_device_status() == B.MOC_ERR_BAD_INDEX
    np.testing.assert_array_equal(syn.to_f64(got[:300]), syn.to_f64(grads["grad_x"][:300]))
