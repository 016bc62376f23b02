"""The CTA-pair GEMM at the sizes where its tile walk and hand-overs change, against the fp64 product of the operands."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_20586_b200 import binding
    return binding


def _operand(gen, rows, K):
    """Random codes and scales of 2^-2 .. 2^2 (native tiling), and the fp64 values they stand for."""
    import torch
    codes = torch.randint(0, 256, (rows, K // 2), generator=gen, device="cuda", dtype=torch.uint8)
    nkc, rt = (K + 127) // 128, (rows + 127) // 128
    scales = torch.randint(125, 130, (rt, nkc, 32, 4, 4), generator=gen, device="cuda", dtype=torch.uint8)    # [row tile, k tile, row % 32, row / 32, block]
    grid = torch.tensor([0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0, -0.0, -0.5, -1.0, -1.5, -2.0, -3.0, -4.0, -6.0], dtype=torch.float64, device="cuda")
    values = torch.stack((grid[(codes & 15).long()], grid[(codes >> 4).long()]), 2).view(rows, K)
    per_block = scales.permute(0, 3, 2, 1, 4).reshape(rt * 128, nkc * 4)[:rows, :K // 32].double()
    return codes, scales.flatten(), values * torch.exp2(per_block - 127.0).repeat_interleave(32, 1)


# one K-step (or half of one) per tile over several tiles per pair: the two issuing threads alternate between tiles
@pytest.mark.parametrize("M,N,K", [(5120, 5000, 256), (4096, 8192, 128), (10240, 2560, 256)])
@pytest.mark.parametrize("fp32", [False, True])
def test_tile_walk(gpu, M, N, K, fp32):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M + N + K)
    ca, sa, a = _operand(gen, M, K)
    cb, sb, b = _operand(gen, N, K)
    want = a @ b.t()
    got = gpu.mxfp4_gemm(ca, sa, cb, sb, 1.0, gpu.OUT_FP32 if fp32 else gpu.OUT_BF16)
    assert gpu.mxfp4_device_status() == 0
    # fp32 sums of K exact products (16 head-room on the unit roundoff); bf16 output: half a unit in the last place
    tol = 16 * 2.0 ** -24 if fp32 else 2.0 ** -8
    assert torch.all((got.double() - want).abs() <= tol * (a.abs() @ b.abs().t() if fp32 else want.abs()) + 1e-30)
