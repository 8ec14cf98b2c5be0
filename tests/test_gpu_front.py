"""The C++ host side of the PyTorch entry points (csrc/torch_front.cpp): argument errors and what it hands back."""
import pytest
import torch

from paper_2511_09323_b200 import binding as B
from paper_2511_09323_b200.autograd import moc_ffn


def _weights(device, d=64, F=96):
    return [torch.full((F, d), 0.01, dtype=torch.bfloat16, device=device) for _ in range(3)]


@pytest.mark.parametrize("call", ("forward", "decode", "decode_block", "ffn"))
def test_wrong_tensors_are_refused_before_the_library(call):
    x, w = torch.zeros(4, 64, dtype=torch.bfloat16), _weights("cpu")
    run = {"forward": lambda x: B.moc_ffn_forward(x, *w, 8), "decode": lambda x: B.moc_ffn_decode(x, *w, 8),
           "decode_block": lambda x: B.moc_ffn_decode_block(x, x[0], 1e-5, *w, 8), "ffn": lambda x: moc_ffn(x, *w, 8)}[call]
    with pytest.raises(ValueError, match="CUDA"):
        run(x)
    with pytest.raises(TypeError, match="Tensor"):
        run([[0.0]] * 4)


@pytest.mark.gpu
def test_library_errors_arrive_as_moc_error_from_both_threads():
    x, w = torch.zeros(40, 64, dtype=torch.bfloat16, device="cuda"), _weights("cuda")
    for run in (lambda: B.moc_ffn_forward(x, *w, 97), lambda: B.moc_ffn_decode(x, *w, 97), lambda: moc_ffn(x, *w, 97)):
        with pytest.raises(B.MocError) as e:
            run()
        assert e.value.status == B.MOC_ERR_INVALID_ARG
    with pytest.raises(ValueError, match="contiguous"):
        B.moc_ffn_forward(x.t().contiguous().t(), *w, 8)
    with pytest.raises(ValueError, match="multiple of 8"):
        B.moc_ffn_decode(x, *w, None, d_ff=90, grouped=True)
    # an error inside the backward call, on the autograd engine's thread: a gradient the library refuses (misaligned)
    leaf = x.clone().requires_grad_()
    y = moc_ffn(leaf, *w, 8)
    with pytest.raises(B.MocError) as e:
        torch.autograd.grad(y, leaf, torch.zeros(40 * 64 + 1, dtype=torch.bfloat16, device="cuda")[1:].view(40, 64))
    assert e.value.status == B.MOC_ERR_INVALID_ARG


@pytest.mark.gpu
def test_given_buffers_and_stream_are_used():
    x, w = torch.randn(40, 64, device="cuda").bfloat16(), _weights("cuda")
    out, saved = torch.empty_like(x), tuple(torch.empty((40, 8), dtype=t, device="cuda") for t in (torch.int16, x.dtype, x.dtype))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    got = B.moc_ffn_forward(x, *w, 8, out=out, saved=saved, stream=side)
    side.synchronize()
    assert got[0].data_ptr() == out.data_ptr() and [g.data_ptr() for g in got[1:]] == [s.data_ptr() for s in saved]
    assert B.moc_ffn_forward(x, *w, 8, save=False)[1:] == (None, None, None)
    x3 = x.view(5, 8, 64).transpose(0, 1).requires_grad_()   # three dimensions, not contiguous
    y = moc_ffn(x3, *w, 8)
    gx, = torch.autograd.grad(y, x3, torch.ones_like(y))
    assert y.shape == x3.shape == gx.shape
