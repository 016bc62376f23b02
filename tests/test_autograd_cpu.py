"""The bf16 forward of the autograd wrapper, which is plain torch and runs on the CPU: the bias is added to the rounded
product, so y has the bits (and under autocast the type) of ``x @ weight.t() + bias``."""
import pytest
import torch

from paper_2502_20586_b200.autograd import MxFp4LinearFunction

SHAPES = [(1, 64), (5, 64), (2, 3, 64), (64,)]


def _inputs(shape):
    gen = torch.Generator().manual_seed(len(shape) + shape[0])
    x, w, bias = (torch.randn(s, generator=gen).bfloat16() for s in (shape, (48, 64), (48,)))
    return x, w, bias


@pytest.mark.parametrize("shape", SHAPES)
def test_biased_forward_has_the_bits_of_product_plus_bias(shape):
    x, w, bias = _inputs(shape)
    y = MxFp4LinearFunction.apply(x, w, bias, 64, 0, 0)
    assert y.shape == (*shape[:-1], 48)
    assert torch.equal(y, x @ w.t() + bias)
    assert torch.equal(MxFp4LinearFunction.apply(x, w, bias[:1], 64, 0, 0), x @ w.t() + bias[:1])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
def test_biased_forward_under_autocast(dtype):
    x, w, bias = _inputs((2, 3, 64))
    with torch.autocast("cpu", dtype=dtype):
        want = x @ w.t() + bias                      # fp16 product + bf16 bias: promoted to fp32
        y = MxFp4LinearFunction.apply(x, w, bias, 64, 0, 0)
    assert y.dtype == want.dtype and torch.equal(y, want)
