"""Per-tensor E4M3 quantisation at the edges of its spans, against the same arithmetic in torch (both are exact: bytes equal)."""
import pytest

pytestmark = pytest.mark.gpu


def _expected(x):
    import torch
    amax = x.abs().max().float()
    scale = 448.0 / amax if amax > 0 else torch.ones((), device="cuda")
    return (x.float() * scale).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8), scale, amax


# one vector, an odd number of vectors, exactly one step of a CTA and one vector more, several spans, rows with a gap
@pytest.mark.parametrize("rows,cols,ld", [(1, 8, 8), (3, 8, 8), (1, 16384, 16384), (1, 16392, 16392), (2049, 4104, 4104), (4096, 8192, 8192),
                                          (5, 24, 40), (1000, 1032, 1040)])
def test_codes_and_scale(rows, cols, ld):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows + cols)
    x = torch.randn((rows, ld), generator=gen, device="cuda").bfloat16()[:, :cols]
    for at in ((rows - 1, cols - 1), (0, 0)):                     # the largest value last, then first
        y = x.clone() if ld == cols else x.as_strided(x.shape, x.stride())
        y[at] = 100.0
        codes, scale = gpu.mxfp4_fp8_quantize(y)
        want, sf, amax = _expected(y)
        assert scale[0] == sf and scale[1] == amax
        assert torch.equal(codes, want)
        y[at] = 0.0
    assert gpu.mxfp4_device_status() == 0


# both operands of a forward product in the same launches: tensors of very different sizes, either way round
@pytest.mark.parametrize("b,n,m", [(1, 128, 8), (16, 4096, 4096), (8193, 256, 8), (1000, 1024, 4096)])
def test_two_tensors(b, n, m):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    gen = torch.Generator(device="cuda")
    gen.manual_seed(b + n + m)
    x, W = torch.randn((b, n), generator=gen, device="cuda").bfloat16(), (0.02 * torch.randn((m, n), generator=gen, device="cuda")).bfloat16()
    y = gpu.mxfp4_linear_forward_fp8(x, W, gpu.OUT_FP32)
    cx, sx = gpu.mxfp4_fp8_quantize(x)
    cw, sw = gpu.mxfp4_fp8_quantize(W)
    assert torch.equal(y, gpu.mxfp4_fp8_gemm(cx, sx, cw, sw, gpu.OUT_FP32))
    assert gpu.mxfp4_device_status() == 0
