"""The native host call of a layer's backward (csrc/host_calls.cpp) against the Python one, which serves tensors of a subclass: the same
bits, buffers, streams and refusals."""
import pytest

pytestmark = pytest.mark.gpu


def _layer(b=256, n=264, m=384):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(b + n + m)
    return [torch.randn(s, generator=gen, device="cuda").bfloat16() for s in ((b, m), (b, n), (m, n))]


def _tagged(t):
    import torch

    class Tagged(torch.Tensor):
        pass
    return t.as_subclass(Tagged)


@pytest.mark.parametrize("seed", [0, -1, 2 ** 64 - 1, 2 ** 64 + 5])
@pytest.mark.parametrize("out_dtype", [0, 1])
@pytest.mark.parametrize("with_bias", [False, True])
def test_both_host_paths_give_the_same(seed, out_dtype, with_bias):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    dY, X, W = _layer()
    want = gpu.mxfp4_linear_backward_ex(_tagged(dY), X, W, 64, seed, 0, out_dtype, with_bias=with_bias)
    got = gpu.mxfp4_linear_backward_ex(dY.requires_grad_(True), X, torch.nn.Parameter(W), 64, seed, 0, out_dtype, with_bias=with_bias)
    plain = gpu.mxfp4_linear_backward(dY, X, W, 64, seed, 0, out_dtype)
    for a, b in zip(want, got):
        assert (a is None and b is None) or (type(b) is torch.Tensor and a.dtype == b.dtype and torch.equal(a, b) and not b.requires_grad)
    assert torch.equal(plain[0], want[0]) and torch.equal(plain[1], want[1])
    with torch.cuda.stream(torch.cuda.Stream()):
        side = gpu.mxfp4_linear_backward(dY, X, W, 64, seed, 0, out_dtype, dX=torch.empty_like(want[0]), dW=torch.empty_like(want[1]))
        torch.cuda.current_stream().synchronize()
    assert torch.equal(side[0], want[0]) and torch.equal(side[1], want[1]) and gpu.mxfp4_device_status() == 0


def test_buffers_of_the_caller_come_back():
    import torch
    from paper_2502_20586_b200 import binding as gpu
    dY, X, W = _layer()
    dX, dW, db = (torch.zeros(s, device="cuda") for s in ((256, 264), (384, 264), (384,)))
    ws = torch.empty(gpu.mxfp4_linear_backward_ex_workspace(256, 384, 264, True), dtype=torch.uint8, device="cuda")
    out = gpu.mxfp4_linear_backward_ex(dY, X, W, 64, 3, 0, 1, dX=dX, dW=dW, db=db, accumulate=True, workspace=ws)
    assert out[0] is dX and out[1] is dW and out[2] is db
    ref = gpu.mxfp4_linear_backward_ex(dY, X, W, 64, 3, 0, 1, with_bias=True)
    assert torch.equal(ref[0], dX) and torch.equal(ref[1], dW) and torch.equal(ref[2], db)      # accumulated onto zeros


def test_refusals():
    import torch
    from paper_2502_20586_b200 import binding as gpu
    dY, X, W = _layer()
    for bad in ((dY.float(), X, W), (dY, X.cpu(), W), (dY, X, W.t()), (dY[:, ::2], X, W)):
        with pytest.raises(AssertionError):
            gpu.mxfp4_linear_backward(*bad, 64, 0)
    with pytest.raises(ValueError):
        gpu.mxfp4_linear_backward(dY.view(2, 128, 384), X, W, 64, 0)
    with pytest.raises(AssertionError):
        gpu.mxfp4_linear_backward_ex(dY, X, W, 64, 0, 0, 1, accumulate=True)
    with pytest.raises(gpu.MxFp4Error) as e:
        gpu.mxfp4_linear_backward(dY, X, W, 48, 0)
    assert e.value.code == 4
    with pytest.raises(gpu.MxFp4Error) as e:
        gpu.mxfp4_linear_backward(dY, X, W, 64, 0, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    assert e.value.code == 6
    with pytest.raises(TypeError):
        gpu.mxfp4_linear_backward(dY, X, W, 64.0, 0)
    with pytest.raises(RuntimeError):                        # a batched tensor has no memory of its own
        torch.vmap(lambda d: gpu.mxfp4_linear_backward(d, X, W, 64, 0)[0])(dY[None])
    del dY, X, W
    free = torch.cuda.mem_get_info()[0]
    wide = torch.empty(1, dtype=torch.bfloat16, device="cuda").expand(1 << 20, 1 << 20)         # expanded: not contiguous
    with pytest.raises(AssertionError):
        gpu.mxfp4_linear_backward(wide, wide, wide, 64, 0)
    assert torch.cuda.mem_get_info()[0] >= free - (64 << 20) and gpu.mxfp4_device_status() == 0


def test_out_of_memory_is_an_exception():
    """A result that does not fit what this process may take of the device: torch's own exception, and the library keeps working."""
    import torch
    from paper_2502_20586_b200 import binding as gpu
    dY, X, W = _layer(4096, 8192, 128)
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (16 << 20)) / torch.cuda.mem_get_info()[1])
    try:
        with pytest.raises(torch.OutOfMemoryError):          # 128 MB, sixteen of which there are
            gpu.mxfp4_linear_backward(dY, X, W, 64, 0, gpu.ROUND_SR, gpu.OUT_FP32)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    dY, X, W = _layer()
    gpu.mxfp4_linear_backward(dY, X, W, 64, 0)
    assert gpu.mxfp4_device_status() == 0


# Tensors and buffers that are smaller than the sizes say, or laid out or typed otherwise: refused by either host path before the library
# is called, whose kernels would read and write past them
@pytest.mark.parametrize("subclass", [False, True])
def test_tensors_that_do_not_fit_are_refused(subclass):
    import torch
    from paper_2502_20586_b200 import binding as gpu
    dY, X, W = _layer()                                                          # b 256, n 264, m 384
    make = lambda *size, dtype=torch.float32: torch.zeros(size, dtype=dtype, device="cuda")
    bf16 = dict(dtype=torch.bfloat16)
    tag = _tagged if subclass else (lambda t: t)
    for x, w in ((X[:128], W), (X[:255], W), (make(384, 264, **bf16), W), (X, W[:256]), (X, make(264, 384, **bf16)), (X, make(384, 256, **bf16)), (X, W.view(-1)[8:])):
        for call in (gpu.mxfp4_linear_backward, gpu.mxfp4_linear_backward_ex, gpu.mxfp4_linear_backward_static, gpu.mxfp4_linear_backward_fused,
                     gpu.mxfp4_quantize_operands):
            with pytest.raises(AssertionError):
                call(tag(dY), x, w, 64, 0)
    need = gpu.mxfp4_linear_backward_ex_workspace(256, 384, 264, True)
    good = dict(dX=make(256, 264), dW=make(384, 264), db=make(384), workspace=make(need, dtype=torch.uint8))
    bad = dict(dX=(make(255, 264), make(256, 264, **bf16), make(256, 272), make(264, 256).t(), make(256, 528)[:, ::2], make(256, 264).cpu(),
                   make(1).expand(256, 264)),
               dW=(make(383, 264), make(384, 264, **bf16), make(264, 384), make(264, 384).t(), make(384, 264).cpu()),
               db=(make(383), make(384, **bf16), make(768)[::2], make(384).cpu()),
               workspace=(make(2 * need, dtype=torch.uint8)[::2], make(1, dtype=torch.uint8).expand(need), torch.zeros(need, dtype=torch.uint8)))
    for name, buffers in bad.items():
        for t in buffers:
            with pytest.raises(AssertionError):
                gpu.mxfp4_linear_backward_ex(tag(dY), X, W, 64, 0, 0, gpu.OUT_FP32, accumulate=True, **{**good, name: t})
            if name == "db":
                continue
            with pytest.raises(AssertionError):
                gpu.mxfp4_linear_backward(tag(dY), X, W, 64, 0, 0, gpu.OUT_FP32, **{name: t})
            for call in (gpu.mxfp4_linear_backward_static, gpu.mxfp4_linear_backward_fused):
                if name != "workspace" or call is gpu.mxfp4_linear_backward_fused:
                    with pytest.raises(AssertionError):
                        call(tag(dY), X, W, 64, 0, 0, gpu.OUT_FP32, **{name: t})
            if name == "workspace":
                with pytest.raises(AssertionError):
                    gpu.mxfp4_quantize_operands(tag(dY), X, W, 64, 0, workspace=t)
    assert not any(torch.any(t) for t in good.values())                          # nothing ran
    # larger buffers, and W or buffers of one dimension, serve as before: the results stand at the buffers' start
    want = gpu.mxfp4_linear_backward_ex(dY, X, W, 64, 0, 0, gpu.OUT_FP32, with_bias=True)
    flat = dict(dX=make(256 * 264 + 24), dW=make(400, 264), db=make(1, 400), workspace=make(need, dtype=torch.int32))
    got = gpu.mxfp4_linear_backward_ex(tag(dY), X, W.view(-1), 64, 0, 0, gpu.OUT_FP32, **flat)
    for a, t in zip(want, got):
        assert torch.equal(t.view(-1)[:a.numel()], a.view(-1)) and not torch.any(t.view(-1)[a.numel():])
    assert gpu.mxfp4_device_status() == 0


def test_other_threads_run_while_a_call_allocates():
    """A result for which the caching allocator first has to free blocks, which waits for the GPU (a torch kernel of about half a
    second): another Python thread keeps running all the while."""
    import threading
    import time

    import torch
    from paper_2502_20586_b200 import binding as gpu
    torch.cuda.empty_cache()                                                    # no room left over from another test's segments
    dY, X, W = (torch.zeros(s, dtype=torch.bfloat16, device="cuda") for s in ((4096, 128), (4096, 4096), (128, 4096)))
    dW = torch.empty((128, 4096), device="cuda")
    workspace = torch.empty(gpu.mxfp4_linear_backward_workspace(4096, 128, 4096), dtype=torch.uint8, device="cuda")
    call = lambda: gpu.mxfp4_linear_backward(dY, X, W, 64, 0, gpu.ROUND_SR, gpu.OUT_FP32, dW=dW, workspace=workspace)[0]
    call()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    blocks = [torch.empty(48 << 20, dtype=torch.uint8, device="cuda") for _ in range(2)]      # dX takes 64 MB: neither will do
    del blocks
    ticks, stop = [], threading.Event()

    def tick():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.001)
    other = threading.Thread(target=tick)
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (16 << 20)) / torch.cuda.mem_get_info()[1])
    try:
        other.start()
        torch.cuda._sleep(10 ** 9)
        start = time.perf_counter()
        dX = call()
        end = time.perf_counter()
    finally:
        stop.set()
        other.join()
        torch.cuda.set_per_process_memory_fraction(1.0)
    seen = [start, *(t for t in ticks if start < t < end), end]
    assert end - start > 0.2                                                    # the call did wait
    assert max(b - a for a, b in zip(seen, seen[1:])) < 0.5 * (end - start)
    assert not torch.any(dX) and gpu.mxfp4_device_status() == 0


class _Parameter:
    """An argument as ctypes lets a class of the caller's pass for one."""
    def __init__(self, value):
        self._as_parameter_ = value


# Integers in every form that ctypes takes for one, and forms that it does not: by either host path
@pytest.mark.parametrize("subclass", [False, True])
def test_integers_of_every_kind(subclass):
    import ctypes

    import numpy as np
    import torch
    from paper_2502_20586_b200 import binding as gpu
    dY, X, W = _layer()
    want = gpu.mxfp4_linear_backward(dY, X, W, 64, 5, gpu.ROUND_SR, gpu.OUT_FP32)
    if subclass:
        dY = _tagged(dY)
    i, u = ctypes.c_int, ctypes.c_uint64
    for ints in ((i(64), u(5), i(0), i(1)), (64, u(5), 0, i(1)), (np.int64(64), np.uint64(5), False, True), (_Parameter(64), 5, 0, _Parameter(i(1)))):
        got = gpu.mxfp4_linear_backward_ex(dY, X, W, *ints, with_bias=True)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        assert torch.equal(gpu.mxfp4_linear_backward(dY, X, W, *ints)[1], want[1])
    for ints in ((64.0, 5, 0, 1), (64, "5", 0, 1), (64, 5, None, 1), (64, 5, 0, ctypes.c_float(1)), (ctypes.c_long(64), 5, 0, 1)):
        for error in (TypeError, ctypes.ArgumentError):
            with pytest.raises(error):
                gpu.mxfp4_linear_backward(dY, X, W, *ints)
            with pytest.raises(error):
                gpu.mxfp4_linear_backward_ex(dY, X, W, *ints)
    assert gpu.mxfp4_device_status() == 0


# out_dtype in every form that stands for 1 to the library: results of four bytes an element from every call that makes them itself
def test_every_form_of_fp32_makes_fp32_results():
    import ctypes

    import torch
    from paper_2502_20586_b200 import binding as gpu
    dY, X, W = _layer(m=512)
    q = gpu.mxfp4_quantize_operands(dY, X, W, 64, 5)
    a, b = gpu.mxfp4_int4_quantize(X[:, :256], 1, 64, 5)[:2], gpu.mxfp4_int4_quantize(W[:, :256], 1, 64, 5)[:2]
    one = torch.ones(2, device="cuda")
    calls = [lambda o: gpu.mxfp4_linear_backward(dY, X, W, 64, 5, 0, o), lambda o: gpu.mxfp4_linear_backward(_tagged(dY), X, W, 64, 5, 0, o),
             lambda o: gpu.mxfp4_linear_backward_static(dY, X, W, 64, 5, 0, o), lambda o: gpu.mxfp4_linear_backward_fused(dY, X, W, 64, 5, 0, o),
             lambda o: gpu.mxfp4_gemm(*q[0], *q[1], out_dtype=o), lambda o: gpu.mxfp4_gemm_fused(dY, 1, 64, 5, 0, 0, *q[1], out_dtype=o),
             lambda o: gpu.mxfp4_linear_forward_fp8(X[:, :256].contiguous(), W[:, :256].contiguous(), o),
             lambda o: gpu.mxfp4_fp8_gemm(a[0], one, b[0], one, o), lambda o: gpu.mxfp4_int4_gemm(*a, *b, out_dtype=o)]
    flat = lambda r: [r] if isinstance(r, torch.Tensor) else list(r)
    for call in calls:
        want = flat(call(gpu.OUT_FP32))
        for o in (True, ctypes.c_int(1), _Parameter(1), _Parameter(ctypes.c_int(1)), (1 << 32) + 1):
            got = flat(call(o))
            assert all(t.dtype == torch.float32 and torch.equal(t, w) for t, w in zip(got, want))
        assert all(t.dtype == torch.bfloat16 for t in flat(call(ctypes.c_int(0))))
    assert gpu.mxfp4_device_status() == 0


def test_forward_tensors_that_do_not_fit_are_refused():
    import torch
    from paper_2502_20586_b200 import binding as gpu
    x, W = (torch.ones(s, dtype=torch.bfloat16, device="cuda") for s in ((200, 256), (136, 256)))
    make = lambda *size, dtype=torch.float32: torch.zeros(size, dtype=dtype, device="cuda")
    for w in (W[:, :128].contiguous(), make(136, 264, dtype=torch.bfloat16), make(136, dtype=torch.bfloat16)):
        with pytest.raises(AssertionError):
            gpu.mxfp4_linear_forward_fp8(x, w)
    for y in (make(199, 136), make(200, 136, dtype=torch.bfloat16), make(136, 200).t(), make(200, 144), make(200, 136).cpu()):
        with pytest.raises(AssertionError):
            gpu.mxfp4_linear_forward_fp8(x, W, gpu.OUT_FP32, y=y)
    for workspace in (make(1 << 20)[::2], torch.zeros(1 << 20, dtype=torch.uint8)):
        with pytest.raises(AssertionError):
            gpu.mxfp4_linear_forward_fp8(x, W, workspace=workspace)
    y = make(200 * 136 + 8)
    gpu.mxfp4_linear_forward_fp8(x, W.view(136, 16, 16), gpu.OUT_FP32, y=y, workspace=make(1 << 20, dtype=torch.uint8))
    assert torch.all(y[:-8] == 256.0) and not torch.any(y[-8:]) and gpu.mxfp4_device_status() == 0
