"""The tensor-core quantiser's tile walk (bands, teams, several views, both views of one tensor), against the CUDA-core
quantiser or a walk of another shape: the transform is exact on small integers, so codes and scales are equal bytes."""
import pytest

from tests import helpers as hp

pytestmark = pytest.mark.gpu


def _small_integers(shape, seed):
    """Values whose transform is exact in any order of summation; scales differ from block to block."""
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.randint(-8, 9, shape, generator=gen, device="cuda").float()
    return x.bfloat16()


# numbers of 128-tiles across the walk that give bands of one, two and four tiles, fewer tiles than CTAs and many more
@pytest.mark.parametrize("rows,cols", [(128, 128), (128, 1032), (256, 4104), (384, 2056), (512, 8), (1152, 2048), (2048, 5128), (4608, 4096)])
@pytest.mark.parametrize("g", [64, 256])
@pytest.mark.parametrize("rounding", [0, 1, 2])
def test_transposing_view_equals_row_view_of_the_transpose(rows, cols, g, rounding):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    if rows % g:
        pytest.skip("reduce length not a multiple of g")
    x = _small_integers((rows, cols), rows + cols)
    codes, scales = gpu.mxfp4_rht_sr_quantize(x, 0, g, 3, 2, rounding)
    want, want_scales = gpu.mxfp4_rht_sr_quantize(x.t().contiguous(), 1, g, 3, 2, rounding)
    assert torch.equal(codes, want)
    linear = gpu.mxfp4_rht_sr_quantize(x, 0, g, 3, 2, rounding, gpu.SF_LINEAR)
    assert torch.equal(linear[0], want)
    per_tile = scales.view(-1, rows // 128, 32, 4, 4).permute(0, 3, 2, 1, 4).reshape(-1, rows // 32)[:cols]
    assert torch.equal(linear[1].view(cols, rows // 32), per_tile)
    assert torch.equal(linear[1], gpu.mxfp4_rht_sr_quantize(x.t().contiguous(), 1, g, 3, 2, rounding, gpu.SF_LINEAR)[1])
    assert want_scales.numel() == scales.numel() and gpu.mxfp4_device_status() == 0


# four views in one launch, and dY's two views from one read of it, against one launch per view
@pytest.mark.parametrize("b,n,m", [(128, 8, 128), (256, 1000, 384), (1152, 264, 2176), (4096, 512, 8192)])
@pytest.mark.parametrize("dual", ["0", "2"])
@pytest.mark.parametrize("rounding", [0, 1, 2])
def test_views_of_a_layer(b, n, m, dual, rounding, monkeypatch):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    monkeypatch.setenv("MXFP4_DUAL_DY", dual)
    dY, X, W = _small_integers((b, m), 1), _small_integers((b, n), 2), _small_integers((m, n), 3)
    q = gpu.mxfp4_quantize_operands(dY, X, W, 64, 9, rounding)
    for (codes, scales), (x, dim, tag) in zip(q, ((dY, 1, 1), (W, 0, 2), (dY, 0, 3), (X, 0, 4))):
        want = gpu.mxfp4_rht_sr_quantize(x, dim, 64, 9, tag, rounding)
        R = want[0].shape[0]
        assert torch.equal(codes, want[0])
        live = torch.arange(want[1].numel(), device="cuda").view(-1, want[0].shape[1] // 64, 32, 4, 4)       # rows beyond R are not written
        row = (torch.arange(live.shape[0], device="cuda").view(-1, 1, 1, 1, 1) * 128 + torch.arange(4, device="cuda").view(1, 1, 1, 4, 1) * 32
               + torch.arange(32, device="cuda").view(1, 1, 32, 1, 1)).expand_as(live) < R
        assert torch.equal(scales.view(live.shape)[row], want[1].view(live.shape)[row])
    assert gpu.mxfp4_device_status() == 0


# Nearest rounding reads dY once from 2^25 elements on: at the line and just below, the default against both forms asked for
@pytest.mark.parametrize("b", [8192, 8064])
def test_default_form_around_one_read(b, monkeypatch):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    n, m = 264, 4096
    assert (b * m >= gpu.one_read_elements(gpu.ROUND_RN)) == (b == 8192)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(b)
    dY, X, W = (torch.randn(s, generator=gen, device="cuda").bfloat16() for s in ((b, m), (b, n), (m, n)))
    out = {}
    for form in ("1", "0", "2"):
        monkeypatch.setenv("MXFP4_DUAL_DY", form)
        workspace = torch.zeros(gpu.mxfp4_linear_backward_workspace(b, m, n), dtype=torch.uint8, device="cuda")
        gpu.mxfp4_quantize_operands(dY, X, W, 64, 9, gpu.ROUND_RN, workspace=workspace)
        out[form] = (workspace, *gpu.mxfp4_linear_backward_ex(dY, X, W, 64, 9, gpu.ROUND_RN, gpu.OUT_FP32, with_bias=True))
        assert gpu.mxfp4_device_status() == 0
    for form in ("0", "2"):
        assert all(torch.equal(got, want) for got, want in zip(out["1"][:3], out[form][:3]))
    assert torch.equal(out["1"][3], out["2"][3])                         # band sums either way; form 0 sums in a pass of its own
    assert torch.all((out["1"][3].double() - dY.double().sum(0)).abs() <= b * 2.0 ** -24 * dY.double().abs().sum(0))


# Codes that start on a 16-byte and on no 32-byte boundary go out in 16-byte stores: the same bytes, and none beyond them
@pytest.mark.parametrize("rows,cols,reduce_dim", [(3, 256, 1), (130, 1280, 1), (512, 136, 0), (2048, 1000, 0)])
@pytest.mark.parametrize("g", [0, 32, 64, 128, 256])
@pytest.mark.parametrize("rounding", [0, 1, 2])
def test_codes_on_sixteen_bytes(rows, cols, reduce_dim, g, rounding):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows + g)
    x = torch.randn((rows, cols), generator=gen, device="cuda").bfloat16()
    want, want_scales = gpu.mxfp4_rht_sr_quantize(x, reduce_dim, g, 3, 2, rounding, gpu.SF_LINEAR)
    assert want.data_ptr() % 32 == 0
    for start in (16, 48):
        buffer = torch.full((want.numel() + 96,), 0xAA, dtype=torch.uint8, device="cuda")
        codes = buffer[start:start + want.numel()].view(want.shape)
        assert codes.data_ptr() % 32 == 16
        _, scales = gpu.mxfp4_rht_sr_quantize(x, reduce_dim, g, 3, 2, rounding, gpu.SF_LINEAR, codes=codes)
        assert torch.equal(codes, want) and torch.equal(scales, want_scales)
        assert torch.all(buffer[:start] == 0xAA) and torch.all(buffer[start + want.numel():] == 0xAA)
    assert gpu.mxfp4_device_status() == 0


# MXINT4 in one launch with the transform: rows that fill no tile (their scale bytes are zero), buffers on 16-byte and on
# 32-byte boundaries, against a pass over the transformed values in torch
@pytest.mark.parametrize("rows,cols,reduce_dim", [(1, 128, 1), (130, 1280, 1), (384, 136, 0), (1000, 2048, 1)])
@pytest.mark.parametrize("shift", [0, 16])
@pytest.mark.parametrize("rounding", [0, 1])
def test_mxint4_in_one_launch(rows, cols, reduce_dim, shift, rounding):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows + cols)
    x = torch.randn((rows, cols), generator=gen, device="cuda").bfloat16()
    R, K = (rows, cols) if reduce_dim == 1 else (cols, rows)
    codes = torch.full((R * K + 32,), 0xAA, dtype=torch.uint8, device="cuda")[shift:shift + R * K].view(R, K)
    y = torch.full((R * K + 8,), float("nan"), device="cuda")[shift // 4:shift // 4 + R * K].view(R, K)
    scales = torch.full((gpu.mxfp4_scale_bytes(R, K),), 0xAA, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    assert gpu.lib().mxfp4_int4_quantize(x.data_ptr(), rows, cols, cols, reduce_dim, 64, rounding, 5, 3, codes.data_ptr(), scales.data_ptr(),
                                         y.data_ptr(), stream) == 0
    assert gpu.mxfp4_device_status() == 0
    assert torch.equal(y, gpu.mxfp4_rht(x, reduce_dim, 64, 5))
    tiles = scales.view(-1, K // 128, 32, 4, 4).permute(0, 3, 2, 1, 4).reshape(-1, K // 32)
    assert torch.all(tiles[R:] == 0)
    exponent = torch.frexp(y.view(R, -1, 32).abs().amax(2))[1] - 3                     # floor(log2 amax) - 2
    assert torch.equal(tiles[:R].int(), (exponent + 127).clamp(min=0))
    q = codes.view(torch.float8_e4m3fn).double().view(R, -1, 32)
    w = y.double().view(R, -1, 32) / torch.exp2(tiles[:R].double() - 127.0).unsqueeze(2) * (1.0 if rounding else 0.75)
    if rounding:
        assert torch.equal(q, w.round().clamp(-7.0, 7.0))
    else:
        assert torch.all((q - w).abs() < 1.0) and torch.all(q == q.round()) and abs(float((q - w).mean())) < 0.05


# The CUDA-core row-wise quantiser with rows on 32-byte boundaries and off them (pitch, base) gives the same bytes
@pytest.mark.parametrize("rows,cols", [(1, 32), (7, 96), (300, 1056)])
@pytest.mark.parametrize("rounding", [0, 1, 2])
def test_row_alignment(rows, cols, rounding):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows)
    x = torch.randn((rows, cols), generator=gen, device="cuda").bfloat16()
    want = gpu.mxfp4_rht_sr_quantize(x, 1, 0, 3, 2, rounding)
    for pitch, start in ((cols + 8, 0), (cols + 16, 8), (cols + 16, 0)):
        y = torch.empty((rows * pitch + 16,), dtype=torch.bfloat16, device="cuda").as_strided((rows, cols), (pitch, 1), start)
        y.copy_(x)
        got = gpu.mxfp4_rht_sr_quantize(y, 1, 0, 3, 2, rounding, gpu.SF_LINEAR)
        assert torch.equal(got[0], want[0])
        assert torch.equal(got[1], gpu.mxfp4_rht_sr_quantize(x, 1, 0, 3, 2, rounding, gpu.SF_LINEAR)[1])


# The CUDA-core quantisers start while the product that writes their input still runs (few tiles, so SMs are free, and a long
# K): the bytes are those of a run that waits between the two
@pytest.mark.parametrize("reduce_dim", [0, 1])
@pytest.mark.parametrize("g", [0, 32])
@pytest.mark.parametrize("pad", [0, 8])
def test_product_quantised_by_the_next_launch(reduce_dim, g, pad):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    M, N, K = 288, 544, 16384                                            # no reduce length that the tensor-core quantiser takes
    gen = torch.Generator(device="cuda")
    gen.manual_seed(g + pad)
    a = [torch.randint(0, 256, (M, K // 2), generator=gen, device="cuda", dtype=torch.uint8) for _ in range(2)]
    b = torch.randint(0, 256, (N, K // 2), generator=gen, device="cuda", dtype=torch.uint8)
    ones = [torch.full((gpu.mxfp4_scale_bytes(rows, K),), 127, dtype=torch.uint8, device="cuda") for rows in (M, N)]
    C = torch.zeros((M, N + pad), dtype=torch.bfloat16, device="cuda")[:, :N]

    def product(i):
        gpu.mxfp4_gemm(a[i], ones[0], b, ones[1], 1.0, gpu.OUT_BF16, C_out=C)

    def quantise():
        return gpu.mxfp4_rht_sr_quantize(C, reduce_dim, g, 3, 2, gpu.ROUND_SR, gpu.SF_LINEAR)

    want = []
    for i in range(2):
        product(i)
        torch.cuda.synchronize()
        want.append(quantise())
        torch.cuda.synchronize()
    assert not torch.equal(want[0][0], want[1][0])
    got = []
    for i in range(40):
        product(i % 2)
        got.append(quantise())
    assert gpu.mxfp4_device_status() == 0
    for i, (codes, scales) in enumerate(got):
        assert torch.equal(codes, want[i % 2][0]) and torch.equal(scales, want[i % 2][1]), i


# A launch that is refused (here: more bands of rows than a grid holds) is the call's error and no other's
def test_refused_launch_leaves_no_error_behind():
    import torch
    from paper_2502_20586_b200 import binding as gpu
    x = torch.zeros((256 << 16, 8), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(gpu.MxFp4Error):
        gpu.mxfp4_rht_sr_quantize(x, 0, 0, 3, 2, gpu.ROUND_RN)
    codes, scales, _ = gpu.mxfp4_int4_quantize(x[:256], 0, 0, 3, 2, gpu.ROUND_RN)     # looks for a launch error after its last kernel
    assert gpu.mxfp4_device_status() == 0 and not torch.any(codes) and not torch.any(scales)


# As many tiles as the chip has SMs (half tiles to the epilogue groups) and one more (whole tiles): the rows that both have, row-wise and
# transposing, in either scale layout, a last tile of a few rows; with the sign vector's transform and with a caller's matrix
@pytest.mark.parametrize("K,g", [(128, 64), (256, 128), (512, 32)])
@pytest.mark.parametrize("rounding", [0, 2])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("given", [False, True])
def test_half_tiles(K, g, rounding, layout, given):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = sms // (K // 128) * 128
    x = _small_integers((rows + 128, K), K + g)
    T = _small_integers((g, g), g) / 8
    quantise = lambda y, dim: gpu.mxfp4_transform_quantize(y, dim, T, 7, 3, rounding, layout) if given else \
        gpu.mxfp4_rht_sr_quantize(y, dim, g, 7, 3, rounding, layout)
    linear = lambda s, n: s.view(n, K // 32) if layout == gpu.SF_LINEAR else \
        torch.from_numpy(hp.sf_native_to_linear(s.cpu().numpy(), n, K)).cuda()
    whole, scales = quantise(x, 1)
    scales = linear(scales, rows + 128)
    for n in (rows, rows - 100, 40):
        for y, dim in ((x[:n], 1), (x[:n].t()[:, :n // 8 * 8].contiguous(), 0)):
            codes, s = quantise(y, dim)
            n_rows = codes.shape[0]
            assert n_rows > n - 8 and torch.equal(codes, whole[:n_rows]) and torch.equal(linear(s, n_rows), scales[:n_rows])
    assert gpu.mxfp4_device_status() == 0


# The bias gradient's two passes inside the launches of a backward call: band sums in the one-list and in the one-read form,
# added up by the GEMM launch; against fp64, overwriting and accumulating
@pytest.mark.parametrize("b,n,m", [(128, 264, 128), (640, 8, 1152), (2048, 1000, 5120)])
@pytest.mark.parametrize("dual", ["0", "1", "2"])
def test_bias_gradient_inside_the_launches(b, n, m, dual, monkeypatch):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    monkeypatch.setenv("MXFP4_DUAL_DY", dual)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(b + m)
    dY, X, W = (torch.randn(s, generator=gen, device="cuda").bfloat16() for s in ((b, m), (b, n), (m, n)))
    _, dW, db = gpu.mxfp4_linear_backward_ex(dY, X, W, 64, 5, gpu.ROUND_SR, gpu.OUT_FP32, with_bias=True)
    want, bound = dY.double().sum(0), b * 2.0 ** -24 * dY.double().abs().sum(0)      # fp32 sums in any order
    assert torch.all((db.double() - want).abs() <= bound)
    gpu.mxfp4_linear_backward_ex(dY, X, W, 64, 6, gpu.ROUND_SR, gpu.OUT_FP32, dW=dW, db=db, accumulate=True)
    assert torch.all((db.double() - 2.0 * want).abs() <= 4.0 * bound)
    assert gpu.mxfp4_device_status() == 0


# Band sums of values whose fp32 sums are exact in any order (the largest and smallest bf16 exponents of small integers, subnormal
# ones among them), and of infinities and NaN
@pytest.mark.parametrize("scale", [2.0 ** -133, 2.0 ** -126, 1.0, 2.0 ** 100])
@pytest.mark.parametrize("b,m,dual", [(128, 128, "0"), (384, 1152, "0"), (384, 1152, "2")])
def test_band_sums_are_exact(scale, b, m, dual, monkeypatch):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    monkeypatch.setenv("MXFP4_DUAL_DY", "1" if dual == "0" else dual)              # (0 sums in a pass of its own)
    dY = (_small_integers((b, m), 5).double() * scale).to(torch.bfloat16)
    assert torch.equal(dY.double(), _small_integers((b, m), 5).double() * scale)
    dY[5, 3], dY[b - 1, m - 1], dY[7, 64], dY[9, 64] = float("inf"), float("nan"), float("inf"), -float("inf")
    X, W = (torch.zeros(s, dtype=torch.bfloat16, device="cuda") for s in ((b, 8), (m, 8)))
    db = gpu.mxfp4_linear_backward_ex(dY, X, W, 64, 5, gpu.ROUND_SR, gpu.OUT_FP32, with_bias=True)[2]
    assert torch.equal(db.double().nan_to_num(7.0, 8.0, 9.0), dY.double().sum(0).nan_to_num(7.0, 8.0, 9.0))


# An operand of eight rows with more than 2^23 scale tiles (its scales fill more than 4 GB), against the same quantiser on the
# operand's first and last columns: nearest rounding, so the bytes do not depend on where a block lies
@pytest.mark.parametrize("kind,reduce_dim,g", [("mxfp4", 1, 64), ("mxfp4", 0, 32), ("mxfp4", 1, 256), ("mxint4", 1, 128)])
def test_more_than_four_gigabytes_of_scales(kind, reduce_dim, g):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    if torch.cuda.mem_get_info()[0] < (90 << 30):
        pytest.skip("needs 90 GB of device memory")
    K = (1 << 30) + 256

    def quantise(x):
        if kind == "mxint4":
            return gpu.mxfp4_int4_quantize(x, reduce_dim, g, 3, 2, gpu.ROUND_RN)[:2]
        return gpu.mxfp4_rht_sr_quantize(x, reduce_dim, g, 3, 2, gpu.ROUND_RN)

    x = torch.zeros((8, K) if reduce_dim == 1 else (K, 8), dtype=torch.bfloat16, device="cuda")
    ends = [x.narrow(reduce_dim, 0, 1024), x.narrow(reduce_dim, 1 << 30, 256)]
    for i, end in enumerate(ends):
        end.copy_(_small_integers(tuple(end.shape), i + 1) * (1 << 4 * i))
    codes, scales = quantise(x)
    assert gpu.mxfp4_device_status() == 0
    tiles = scales.view(-1, 32, 4, 4)[:, :8, 0, :]                       # the eight rows' bytes of every tile
    per_tile = codes.shape[1] // (K // 128)
    for end, t0 in ((ends[0], 0), (ends[1], 1 << 23)):
        want, want_scales = quantise(end.contiguous())
        n = want_scales.numel() // 512
        assert torch.equal(tiles[t0:t0 + n], want_scales.view(-1, 32, 4, 4)[:, :8, 0, :])
        assert torch.equal(codes[:, t0 * per_tile:(t0 + n) * per_tile], want)
    assert not torch.any(tiles[8:1 << 23])
    del x, ends, codes, scales, tiles, end
    torch.cuda.empty_cache()
