"""The forward of the autograd wrapper with a plain product is torch and runs on the CPU: whatever the types, y has the type and
shape of ``x @ weight.t() + bias``, and outside the bf16 path with a whole bias its bits too."""
import pytest
import torch

from paper_2502_20586_b200.autograd import MxFp4LinearFunction


def _inputs(shape, dtypes):
    gen = torch.Generator().manual_seed(len(shape) + shape[0])
    return tuple(torch.randn(s, generator=gen).to(d) for s, d in zip((shape, (48, 64), (48,)), dtypes))


def _forward(x, w, bias):
    return MxFp4LinearFunction.apply(x, w, bias, 64, 0, 0)


@pytest.mark.parametrize("shape", [(1, 64), (5, 64), (2, 3, 64), (64,)])
def test_biased_bf16_forward(shape):
    x, w, bias = _inputs(shape, (torch.bfloat16,) * 3)
    y, product = _forward(x, w, bias), x.double() @ w.double().t()
    exact = product + bias.double()
    assert y.shape == exact.shape and y.dtype == torch.bfloat16
    u = 2.0 ** -8              # one rounding to bf16; room for one of the product, one of the sum, and 64 fp32 additions
    bound = u * product.abs() + u * (exact.abs() + u * product.abs()) + 64 * 2.0 ** -23 * (x.double().abs() @ w.double().abs().t())
    assert torch.all((y.double() - exact).abs() <= bound)
    assert torch.equal(_forward(x, w, bias[:1]), x @ w.t() + bias[:1])


@pytest.mark.parametrize("dtypes", [(torch.float32,) * 3, (torch.bfloat16, torch.bfloat16, torch.float32)])
def test_other_types(dtypes):
    x, w, bias = _inputs((5, 64), dtypes)
    y, want = _forward(x, w, bias), x @ w.t() + bias
    assert y.dtype == want.dtype and torch.equal(y, want)


@pytest.mark.parametrize("autocast", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_biased_forward_under_autocast(autocast, dtype):
    x, w, bias = _inputs((2, 3, 64), (dtype,) * 3)
    with torch.autocast("cpu", dtype=autocast):
        want = x @ w.t() + bias                      # the product in the autocast type, promoted by the bias
        y = _forward(x, w, bias)
    assert y.dtype == want.dtype and torch.equal(y, want)
