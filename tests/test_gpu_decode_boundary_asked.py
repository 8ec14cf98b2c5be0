"""MOC_FFN_SB_MIN_TOKENS=n (read once per process) moves the boundary between the gathering plan and the small-batch plan to n tokens, for
every call below it."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu
ASKED = int(os.environ.get("MOC_FFN_SB_MIN_TOKENS", 0))


@pytest.mark.parametrize("tokens", [3, 4, 5, 6, 7])
def test_the_boundary_is_where_it_was_asked_for(tokens):
    if not ASKED:
        return   # (run by the test below)
    g = torch.Generator(device="cuda").manual_seed(tokens)
    x = torch.randn(tokens, 1440, generator=g, device="cuda").bfloat16()
    w = [(torch.randn(3840, 1440, generator=g, device="cuda") * 0.02).bfloat16() for _ in range(3)]
    B.moc_profile_enable(True)
    B.moc_ffn_decode(x, *w, 480)
    launched = {n for n, v in B.moc_profile_collect().items() if v[0]}
    B.moc_profile_enable(False)
    assert ("dec_down" in launched) == (tokens < ASKED), launched


def test_boundaries():
    if ASKED:
        return
    for asked in ("4", "7"):
        r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", __file__], env=dict(os.environ, MOC_FFN_SB_MIN_TOKENS=asked),
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0 and "6 passed" in r.stdout, r.stdout[-2000:]
