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


# One tile to a pair, whose columns the two epilogue groups share in the 8-bit builds, against the same rows in a product of several tiles to
# a pair, whose groups take whole tiles: the same bits.  128-wide tiles, ragged rows and columns; 256-wide ones from 1000 rows on with
# 8-bit products of 4096 and 4128 columns (128 and 132 tiles of 128 columns take two rounds of the 74 pairs, 64 and 68 of 256 columns one)
@pytest.mark.parametrize("rows,more,N,K", [(200, 9000, 264, 256), (257, 19000, 136, 384), (512, 12000, 1000, 128), (1000, 9000, 1024, 384), (990, 9000, 1032, 256)])
@pytest.mark.parametrize("out", [0, 1])
def test_single_tile_of_a_pair(gpu, rows, more, N, K, out):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows + N + K)
    ca, sa, _ = _operand(gen, more, K)
    cb, sb, _ = _operand(gen, N * 4, K)
    few = sa[:(rows + 127) // 128 * ((K + 127) // 128) * 512]
    assert torch.equal(gpu.mxfp4_gemm(ca[:rows], few, cb[:N], sb, 1.5, out), gpu.mxfp4_gemm(ca, sa, cb[:N], sb, 1.5, out)[:rows])
    a, b = (torch.randint(0, 0x60, (n, K), generator=gen, device="cuda", dtype=torch.uint8) for n in (more, N * 4))      # E4M3, finite
    one = torch.ones(2, device="cuda")
    assert torch.equal(gpu.mxfp4_fp8_gemm(a[:rows], one, b, one, out), gpu.mxfp4_fp8_gemm(a, one, b, one, out)[:rows])
    for n in (N, N * 4):
        assert torch.equal(gpu.mxfp4_int4_gemm(a[:rows], few, b[:n], sb, 1.5, out), gpu.mxfp4_int4_gemm(a, sa, b[:n], sb, 1.5, out)[:rows])
    assert gpu.mxfp4_device_status() == 0


# The two products of a backward call go out as one launch: tile counts below and above the number of pairs (74), equal
# and unequal K, a first product that leaves some pairs with one tile more than the rest, both tile widths, ragged edges.
@pytest.mark.parametrize("b,n,m", [(256, 512, 512), (384, 8, 256), (8192, 1024, 1024), (8192, 1024, 3072), (4224, 1000, 1408), (1024, 4096, 4096),
                                   (2048, 2304, 2432), (6400, 520, 128 * 33), (256, 5000, 3840), (10240, 264, 384)])
def test_two_products_in_one_launch(gpu, b, n, m):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(b + n + m)
    dY, X, W = (torch.randn(shape, generator=gen, device="cuda").bfloat16() for shape in ((b, m), (b, n), (m, n)))
    dX = torch.full((b, n), float("nan"), dtype=torch.float32, device="cuda")
    dW = torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda")
    gpu.mxfp4_linear_backward(dY, X, W, 64, 5, gpu.ROUND_SR, gpu.OUT_FP32, dX=dX, dW=dW)
    q = gpu.mxfp4_quantize_operands(dY, X, W, 64, 5, gpu.ROUND_SR)
    assert torch.equal(dX, gpu.mxfp4_gemm(*q[0], *q[1], 16.0 / 9.0, gpu.OUT_FP32))
    assert torch.equal(dW, gpu.mxfp4_gemm(*q[2], *q[3], 16.0 / 9.0, gpu.OUT_FP32))
    assert gpu.mxfp4_device_status() == 0


# The 8-bit products: both tile widths, one and several tiles per pair (alternating accumulators), fewer rows than a CTA
# owns, ragged edges, one K-step, both output types.
@pytest.mark.parametrize("M,N,K", [(1, 8, 128), (16, 4096, 256), (129, 264, 128), (1000, 4096, 384), (5120, 4104, 128), (300, 20480, 256)])
@pytest.mark.parametrize("kind", ["fp8", "int4"])
@pytest.mark.parametrize("fp32", [False, True])
def test_eight_bit_products(gpu, M, N, K, kind, fp32):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M + N + K)
    out = gpu.OUT_FP32 if fp32 else gpu.OUT_BF16

    def codes(rows):
        if kind == "fp8":
            v = torch.randn((rows, K), generator=gen, device="cuda") * 8
        else:
            v = torch.randint(-7, 8, (rows, K), generator=gen, device="cuda").float()
        c = v.to(torch.float8_e4m3fn)
        return c.view(torch.uint8), c.double()

    (ca, a), (cb, b) = codes(M), codes(N)
    if kind == "fp8":
        sa, sb = (torch.tensor([s, 0.0], device="cuda") for s in (3.0, 0.25))
        got = gpu.mxfp4_fp8_gemm(ca, sa, cb, sb, out)
        a = a / 0.75
    else:
        _, sa, _ = _operand(gen, M, K)
        _, sb, _ = _operand(gen, N, K)
        got = gpu.mxfp4_int4_gemm(ca, sa, cb, sb, 1.0, out)

        def scale(s, rows):
            t = s.view((rows + 127) // 128, K // 128, 32, 4, 4).permute(0, 3, 2, 1, 4).reshape(-1, K // 32)[:rows].double()
            return torch.exp2(t - 127.0).repeat_interleave(32, 1)
        a, b = a * scale(sa, M), b * scale(sb, N)
    assert gpu.mxfp4_device_status() == 0
    want, size = a @ b.t(), a.abs() @ b.abs().t()
    # fp32 sums (and one rounding of the scale and of the product) of K terms; bf16 output: half a unit in the last place more
    bound = 16 * 2.0 ** -24 * size + (0.0 if fp32 else 2.0 ** -8) * want.abs()
    assert torch.all((got.double() - want).abs() <= bound + 1e-30)


# two pairs to a tile, each half of the K-steps: the fewest steps that split, an odd number of them, the most tiles, ragged edges
# (the bounds are those of whole tiles: one addition more)
@pytest.mark.parametrize("M,N,K", [(1, 8, 3072), (129, 136, 3200), (1000, 1016, 8192), (130, 4096, 3072)])
@pytest.mark.parametrize("kind", ["fp8", "int4"])
@pytest.mark.parametrize("fp32", [False, True])
def test_eight_bit_products_over_two_pairs(gpu, M, N, K, kind, fp32):
    test_eight_bit_products(gpu, M, N, K, kind, fp32)


# one output row: its pitch means nothing and may be larger than a tensor map can hold
@pytest.mark.parametrize("ldc", [264, 1 << 20, 1 << 40])
def test_pitch_of_a_single_row(gpu, ldc):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    a, b = ((torch.randn((rows, 256), generator=gen, device="cuda") * 8).to(torch.float8_e4m3fn).view(torch.uint8) for rows in (1, 264))
    one = torch.ones(2, device="cuda")
    want = gpu.mxfp4_fp8_gemm(a, one, b, one, gpu.OUT_FP32)
    got = torch.full((1, 264), float("nan"), device="cuda")
    assert gpu.lib().mxfp4_fp8_gemm(a.data_ptr(), one.data_ptr(), b.data_ptr(), one.data_ptr(), 1, 264, 256, got.data_ptr(), ldc, gpu.OUT_FP32,
                                    torch.cuda.current_stream().cuda_stream) == 0
    assert gpu.mxfp4_device_status() == 0 and torch.equal(got, want)


# at most 128 rows: one column tile more than pairs is where the one-CTA kernel takes over; the same bits as the pairs give for
# the halves of the columns
@pytest.mark.parametrize("M,N,K", [(1, 18952, 128), (128, 18952, 256), (17, 37896, 384), (100, 75784, 128)])
@pytest.mark.parametrize("kind", ["fp8", "int4"])
@pytest.mark.parametrize("fp32", [False, True])
def test_few_rows_and_many_columns(gpu, M, N, K, kind, fp32):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M + N + K)
    out = gpu.OUT_FP32 if fp32 else gpu.OUT_BF16
    a, b = ((torch.randn((rows, K), generator=gen, device="cuda") * 8).to(torch.float8_e4m3fn) for rows in (M, N))
    if kind == "int4":
        a, b = (t.float().clamp(-7, 7).round().to(torch.float8_e4m3fn) for t in (a, b))
    ca, cb = a.view(torch.uint8), b.view(torch.uint8)
    sa, sb = (_operand(gen, rows, K)[1] if kind == "int4" else torch.tensor([s, 0.0], device="cuda") for rows, s in ((M, 3.0), (N, 0.25)))
    whole = torch.full((M, N + 8), float("nan"), dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")[:, :N]

    def product(c0, c1, C):
        if kind == "fp8":
            return gpu.mxfp4_fp8_gemm(ca, sa, cb[c0:c1], sb, out, C_out=C)
        return gpu.mxfp4_int4_gemm(ca, sa, cb[c0:c1], sb[c0 // 128 * (K // 128) * 512:], 1.0, out, C_out=C)

    product(0, N, whole)
    assert gpu.mxfp4_device_status() == 0
    for c0 in range(0, N, 16384):
        c1 = min(N, c0 + 16384)
        assert torch.equal(whole[:, c0:c1], product(c0, c1, None))
    assert gpu.mxfp4_device_status() == 0
