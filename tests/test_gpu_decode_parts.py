"""The one-kernel decode form's selection (csrc/decode_coop.cuh) on keys that differ inside the threshold's bin: parts that are kept whole, cut, first,
last, on both sides of a word of counters, overflowing; one token settled by its parts and the other by the exchange of the bin's keys."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import moc_oracle as orc
from paper_2511_09323_b200 import binding as B

pytestmark = pytest.mark.gpu
BINS, NARROW = 2048, 1152   # counters of the histogram, bins that have parts
D = 16


def _kept_and_exchanged(rows, k):
    """Masks and numbers of exchanged keys for given gate rows: a value is a sum of three bf16 weights, exact in fp32."""
    T, F = rows[0].shape[0], rows[0].shape[1]
    wg, x = torch.zeros(F, D), torch.zeros(T, D)
    for t in range(T):
        for i in range(3):
            wg[:, 3 * t + i] = torch.from_numpy(rows[i][t])
            x[t, 3 * t + i] = 1
    assert (wg.bfloat16().float() == wg).all()
    wg, x = wg.bfloat16().cuda(), x.bfloat16().cuda()
    zeros, out = torch.zeros_like(wg), torch.empty_like(x)
    desc, lib = B.make_desc(T, D, F, k, x.dtype), B.load()
    ws = torch.full((lib.moc_ffn_decode_probe_workspace_bytes(ctypes.byref(desc)),), 255, dtype=torch.uint8, device="cuda")
    kept = torch.full((T, F), 255, dtype=torch.uint8, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    rc = lib.moc_ffn_decode_probe(ctypes.byref(desc), p(x), p(wg), p(zeros), p(zeros), p(out), p(kept), p(ws), ws.numel(),
                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == B.MOC_OK and B.moc_last_device_status() == B.MOC_OK
    exchanged = ws[T * BINS * 4:][:4 * T].view(torch.int32).cpu().tolist()   # behind the histogram
    return kept.cpu().numpy(), exchanged


def _parts(T, F):
    """Parts of a narrow bin: what the workspace holds beside histogram, count, list and accumulator, half a byte each."""
    up = lambda n: (n + 255) // 256 * 256
    need = B.load().moc_ffn_decode_probe_workspace_bytes(ctypes.byref(B.make_desc(T, D, F, 8, torch.bfloat16)))
    return 2 * (need - up(T * BINS * 4) - up(T * 4) - up(T * F * 8) - up(T * D * 4)) // (T * NARROW)


def _patterns(P):
    """(keys of each part of the threshold's bin, how many of the bin are kept)"""
    h = P // 2
    spread = {P - 1: 3, h: 2, 0: 4}
    yield from ((spread, n) for n in (1, 3, 4, 5, 7, 9))             # cut and whole; the last part, one between, the first
    yield from (({h: 2, h - 1: 3, 1: 1}, n) for n in (2, 4, 5, 6))   # on both sides of a word of eight counters
    yield from (({h: 15, 2: 1}, n) for n in (15, 16))                # as many as a counter holds
    yield from (({h + 1: 16, h: 2, 1: 1}, n) for n in (16, 18, 19))  # one more: it carries into its neighbour
    yield from (({P - 1: 17, 1: 2}, n) for n in (17, 19))            # out of its word
    yield from (({h: 33, h + 1: 1}, n) for n in (1, 34))


@pytest.mark.parametrize("T,F,P", [(1, 700, 16), (1, 1000, 32), (1, 2048, 64), (1, 3000, 128), (1, 11008, 256), (2, 1000, 8), (2, 1300, 16),
                                   (2, 2048, 32), (2, 5504, 64), (2, 11008, 128), (2, 16384, 256)])
def test_values_that_differ_inside_the_bin(T, F, P):
    assert _parts(T, F) == P
    rng = np.random.default_rng(F + T)
    patterns = list(_patterns(P))
    for bottom in (2.0 ** -5, 1.5, 16.0 - 2.0 ** -4):                # the lowest narrow bin, one between, the highest
        step = float(np.spacing(np.float32(bottom)))
        for same in (False, True):                                   # keys of a part: all different, or equal
            for n, of_token_0 in enumerate(patterns):
                of_token_1 = patterns[(7 * n + 5) % len(patterns)]
                K, rows, settled, inside = None, [np.zeros((T, F), np.float32) for _ in range(3)], [], []
                # the same K for both tokens: as many more above the bin as one keeps fewer inside
                taken = [of_token_0[1], of_token_1[1]][:T]
                K = 100 + max(taken)
                for t, (counts, take) in enumerate([of_token_0, of_token_1][:T]):
                    at = rng.permutation(F)
                    rows[0][t] = -20
                    above = K - take
                    rows[0][t, at[:above]] = 32 * (1 + rng.integers(0, 128, above) * 2.0 ** -7)
                    at = at[above:]
                    for part, count in counts.items():
                        width = 65536 // P
                        inner = np.full(count, width - 1) if same else rng.choice(width, count, replace=False)
                        key = part * width + inner
                        rows[0][t, at[:count]] = bottom
                        rows[1][t, at[:count]] = (key >> 8) * 256 * step
                        rows[2][t, at[:count]] = (key & 255) * step
                        at = at[count:]
                    whole = np.cumsum([counts[p] for p in sorted(counts, reverse=True)])
                    settled.append(max(counts.values()) < 16 and take in whole)
                    inside.append(sum(counts.values()))
                values = rows[0] + rows[1] + rows[2]
                want = np.zeros((T, F), np.uint8)
                np.put_along_axis(want, orc.topk(values, K).astype(np.int64), 1, axis=1)
                kept, exchanged = _kept_and_exchanged(rows, K)
                what = f"{bottom}, {of_token_0}, {of_token_1 if T == 2 else ''}, same={same}"
                np.testing.assert_array_equal(kept, want, err_msg=what)
                assert exchanged == [0 if s else m for s, m in zip(settled, inside)], what
