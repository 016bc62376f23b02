"""The tensors that the binding allocates are plain ones, whatever tensor class its inputs are.  The library is replaced by one
that accepts every call, so that no GPU is needed."""
import pytest
import torch

from paper_2502_20586_b200 import binding as mx


class Tagged(torch.Tensor):
    """A subclass, as frameworks use them to mark tensors; it passes for a GPU tensor here."""
    is_cuda = True


class _AcceptsEveryCall:
    def __getattr__(self, name):
        return lambda *args: 1 << 20 if name.endswith("_workspace") or name == "mxfp4_scale_bytes" else 0


@pytest.mark.parametrize("call", ["linear_backward", "linear_backward_ex", "linear_backward_static", "linear_backward_fused", "quantize_operands"])
def test_results_of_a_tensor_subclass_are_plain_tensors(call, monkeypatch):
    monkeypatch.setattr(mx, "_lib", _AcceptsEveryCall())
    monkeypatch.setattr(mx, "_stream", lambda: 0)
    args = [torch.zeros(shape, dtype=torch.bfloat16).as_subclass(Tagged) for shape in ((128, 128), (128, 8), (128, 8))]
    out = getattr(mx, "mxfp4_" + call)(*args, 64, 0, **({"with_bias": True} if call.endswith("_ex") else {}))
    flat = [t for o in out for t in (o if isinstance(o, tuple) else (o,))]
    assert flat and all(type(t) is torch.Tensor for t in flat)
