"""The one-kernel decode form on gate values of every magnitude: the same channels, in the same time."""
import pytest
import torch

from paper_2511_09323_b200 import binding as B
from paper_2511_09323_b200 import synthetic as syn

pytestmark = pytest.mark.gpu


def _us(x, sets, k):
    """One call, in a graph of eight that rotate the weight sets; the fastest of twelve replays."""
    out = torch.empty_like(x)
    ws = B.alloc_workspace(B.make_desc(x.shape[0], x.shape[1], sets[0][0].shape[0], k, x.dtype), B.MOC_OP_DECODE)
    B.moc_ffn_decode(x, *sets[0], k, out=out, workspace=ws)
    torch.cuda.synchronize()
    graph, stream, times = torch.cuda.CUDAGraph(), torch.cuda.Stream(), []
    with torch.cuda.graph(graph, stream=stream):
        for i in range(8):
            B.moc_ffn_decode(x, *sets[i % 2], k, out=out, workspace=ws)
    for _ in range(12):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 1e3 / 8)
    return min(times)


@pytest.mark.parametrize("tokens", (1, 2))
def test_gate_magnitude_changes_neither_the_channels_nor_the_time(tokens):
    w = syn.C4
    sets = [[t.cuda() for t in syn.make_weights(w, seed_offset=s)] for s in range(2)]
    x = syn.make_x(w, tokens=tokens).cuda()
    _, kept = B.moc_ffn_decode_probe(x, *sets[0], w.k)
    base = _us(x, sets, w.k)
    for scale in (2.0 ** -20, 2.0 ** -7, 2.0 ** 10):   # powers of two: the same order, exactly
        scaled = [[s[0] * scale, *s[1:]] for s in sets]
        assert torch.equal(B.moc_ffn_decode_probe(x, *scaled[0], w.k)[1], kept), scale
        # (histogram bins of one width for some magnitudes and another for the rest: 20 % at two tokens)
        assert _us(x, scaled, w.k) < 1.1 * base, scale
    assert B.moc_last_device_status() == B.MOC_OK
