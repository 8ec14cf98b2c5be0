"""The register form of the row selector at the edges of its warps, lanes and forms, bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import moc_oracle as orc
from paper_2511_09323_b200 import binding as B
from test_gpu_selector_plans import _adversarial_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", (2, 5, 127, 128, 129, 512, 513, 1024, 1025, 2048, 2049, 3073, 4096, 4097, 5632, 5633, 8193, 11264,
                               11265, 14336))
def test_register_form_bit_exact(n):
    rng = np.random.default_rng(n)
    rows = [_adversarial_rows(n), rng.standard_normal((40, n))]
    # the threshold inside a cluster: far more values in its bin, or right at the bin's edges, than are ranked at once
    tight = rng.standard_normal((12, n))
    tight[:, rng.permutation(n)[: max(1, n // 3)]] = 1.15 + 1e-4 * rng.standard_normal((12, max(1, n // 3)))
    # skewed and shifted rows, whose threshold lies far from where a normal row's would
    rows += [tight, rng.exponential(size=(8, n)) ** 3, -rng.exponential(size=(8, n)), rng.standard_normal((8, n)) * 1e-3 + 7.0]
    g = np.concatenate(rows).astype(np.float32)
    n_ld = (n + 7) // 8 * 8
    pad = np.full((g.shape[0], n_ld), 1e9, np.float32)
    pad[:, :n] = g
    for k in sorted({1, max(1, n // 16), max(1, n // 8), max(1, n // 2), n}):
        idx, variant = B.moc_topk_select_tc(torch.from_numpy(pad).cuda(), k, n=n)
        assert variant == ("team2" if n <= 3072 else "team4")
        np.testing.assert_array_equal(idx.cpu().numpy().astype(np.int32), orc.topk(g, k), err_msg=f"n={n} k={k}")
    assert B.moc_last_device_status() == B.MOC_OK
