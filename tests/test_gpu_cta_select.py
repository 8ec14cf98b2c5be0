"""The CTA-per-row selector at the edges of its sample window and of its ranked list, bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import moc_oracle as orc
from paper_2511_09323_b200 import binding as B
from test_gpu_selector_plans import _adversarial_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", (3, 127, 128, 1023, 1025, 4100, 11008, 12289))
def test_window_form_bit_exact(n):
    rng = np.random.default_rng(n)
    normal = rng.standard_normal((4, n))
    crowded = rng.standard_normal((4, n))  # clusters around the threshold: more keys in its bin than are ranked at once
    for r, width in enumerate((0.0, 1e-4, 2e-2, 1.0)):
        crowded[r, rng.permutation(n)[: max(1, n // 3)]] = 1.15 + width * rng.standard_normal(max(1, n // 3))
    rows = [_adversarial_rows(n), normal, normal * 1e-36, normal * 1e33, normal * 1e-3 + 7.0, crowded, rng.exponential(size=(4, n)) ** 3]
    g = np.concatenate(rows).astype(np.float32)
    for k in sorted({1, max(1, n // 16), max(1, n // 8), max(1, n // 2), n}):
        idx = B.moc_topk_select(torch.from_numpy(g).cuda(), k)
        np.testing.assert_array_equal(idx.cpu().numpy().astype(np.int32), orc.topk(g, k), err_msg=f"n={n} k={k}")
    assert B.moc_last_device_status() == B.MOC_OK
