"""The work a training program gives this library, as timed cases.

Every case goes through the public Python entry points.  Shapes are those of ``workloads.CONFIGS`` (one 256 x 512 layer,
the GPT 345M / 1.3B / 6.7B linears), of the ablation sweep, and generic ragged ones; values follow the same
descriptions (activations with a few large feature columns, heavy-tailed sparse gradients, N(0, 0.02^2) weights).

Names as in ``workloads.Linear``: tokens b, in-features n, out-features m; dY [b, m], X [b, n], W [m, n].
"""
import torch

from paper_2502_20586_b200 import binding as mx
from paper_2502_20586_b200.ablation import mxfp4_product
from paper_2502_20586_b200.autograd import MxFp4LinearFunction

ROUNDING = {"sr": mx.ROUND_SR, "rn": mx.ROUND_RN, "sr16": mx.ROUND_SR16}

# A backward call of the largest layer (6.7B FC1 / FC2): b * m * n of it bounds what draw() may ask for.
LARGEST = 16384 * 4096 * 16384


def listed():
    return [
        # One small layer (unit-test and fine-tuning scale): nothing but latency, launches and host work.
        dict(name="backward_256x512", kind="backward", b=256, n=512, m=512, g=64, rounding="sr", keep=False),
        # The smallest and the widest linear of the 345M model, the call a training framework makes per layer.
        dict(name="backward_345m_attn_out", kind="backward", b=8192, n=1024, m=1024, g=64, rounding="sr", keep=False),
        dict(name="backward_345m_fc1", kind="backward", b=8192, n=1024, m=4096, g=64, rounding="sr", keep=True),
        # A 1.3B linear with the buffers kept by the caller.
        dict(name="backward_1p3b_fc2", kind="backward", b=16384, n=8192, m=2048, g=128, rounding="sr", keep=True),
        # The largest call: FC1 of the 6.7B model, the benchmark's widest layer.
        dict(name="backward_6p7b_fc1", kind="backward", b=16384, n=4096, m=16384, g=128, rounding="sr", keep=True),
        # Sizes that fill no tile: 33 and 11 tiles of 128, 1000 in-features, the smallest transform block.
        dict(name="backward_ragged", kind="backward", b=4224, n=1000, m=1408, g=32, rounding="sr16", keep=False),
        # Gradient accumulation in fp32 with a bias: two micro-batches of the 1.3B QKV layer.
        dict(name="accumulate_1p3b_qkv", kind="accumulate", b=4096, n=2048, m=6144, g=128, rounding="sr", keep=True),
        # One layer's training step through autograd: bf16 forward (345M QKV, with bias), then the MXFP4 backward.
        dict(name="train_345m_qkv", kind="train", b=8192, n=1024, m=3072, g=64, rounding="sr", forward="bf16", bias=True),
        # The same with the E4M3 forward pass and hardware rounding, at the 6.7B attention output.
        dict(name="train_6p7b_attn_out_fp8", kind="train", b=16384, n=4096, m=4096, g=128, rounding="sr16", forward="fp8", bias=False),
        # E4M3 forward pass alone on a ragged evaluation batch (345M FC1).
        dict(name="forward_fp8_ragged", kind="forward_fp8", b=1000, n=1024, m=4096),
        # The ablation's product on the 1.3B FC1 shape: quantise both operands, one GEMM, fp32 result; without a transform.
        dict(name="product_rn_1p3b_fc1", kind="product", M=16384, N=8192, K=2048, g=0, rounding="rn"),
        # The other element format: MXINT4 operands and product, weight gradient of the 345M attention output.
        dict(name="product_int4_345m", kind="int4", M=1024, N=1024, K=8192, g=64, rounding="sr"),
    ]


def _size(rng, lo, hi, step):
    """Log-uniform in [lo, hi], a multiple of `step`."""
    v = lo * (hi / lo) ** rng.random()
    return max(lo, int(v) // step * step)


def _short_and_many(M, N, K):
    """An MXFP4 product of one 256-element K-step over more than two 256 x 256 tiles per CTA pair."""
    return K <= 256 and -(-M // 256) * -(-N // 256) > 148


def draw(rng):
    while True:
        kind = rng.choice(["backward", "backward", "backward", "accumulate", "train", "forward_fp8", "product", "product", "int4"])
        if kind in ("backward", "accumulate", "train"):
            g = rng.choice([32, 64, 128, 256] if kind == "backward" else [64, 128])
            c = dict(kind=kind, b=_size(rng, 256, 16384, max(g, 128)), n=_size(rng, 256, 16384, 8), m=_size(rng, 256, 16384, max(g, 128)),
                     g=g, rounding=rng.choice(["sr", "sr", "sr16", "rn"]))
            volume = c["b"] * c["m"] * c["n"]
            if kind == "train":
                c["forward"] = rng.choice(["bf16", "fp8"])
                c["bias"] = rng.random() < 0.5
                if c["forward"] == "fp8":
                    c["n"] = _size(rng, 256, 8192, 128)
                volume = 4 * c["b"] * c["m"] * c["n"]         # the bf16 forward product takes as long as the backward
            else:
                c["keep"] = rng.random() < 0.5
                if kind == "accumulate":
                    volume *= 3                               # two micro-batches, fp32 gradients
        elif kind == "forward_fp8":
            c = dict(kind=kind, b=_size(rng, 16, 16384, 1), n=_size(rng, 256, 16384, 128), m=_size(rng, 256, 16384, 8))
            volume = 2 * c["b"] * c["m"] * c["n"]
        else:
            g = rng.choice([0, 32, 64, 128, 256] if kind == "product" else [0, 64, 128])
            c = dict(kind=kind, M=_size(rng, 128, 16384, 1), N=_size(rng, 256, 8192, 8), K=_size(rng, 256, 8192, max(g, 128)),
                     g=g, rounding=rng.choice(["sr", "rn", "sr16"] if kind == "product" else ["sr", "rn"]))
            volume = 4 * c["M"] * c["N"] * c["K"]
        if kind == "product":
            products = [(c["M"], c["N"], c["K"])]
        elif kind in ("backward", "accumulate", "train"):
            products = [(c["b"], c["n"], c["m"]), (c["m"], c["n"], c["b"])]
        else:
            products = []
        # Such products are left out: the GEMM ran into its wait limit on them when these cases were chosen.
        if volume <= LARGEST and not any(_short_and_many(*p) for p in products):
            return c


# ---------------------------------------------------------------- inputs
def _normal(gen, shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)


def _activation(gen, rows, cols):
    """N(0, 1) with eight feature columns twenty times as large."""
    a = _normal(gen, (rows, cols))
    a[:, torch.randperm(cols, generator=gen, device="cuda")[:8]] *= 20.0
    return a.to(torch.bfloat16)


def _gradient(gen, rows, cols):
    """Student-t with three degrees of freedom, standard deviation 1e-4."""
    chi2 = _normal(gen, (rows, cols)).square_()
    chi2 += _normal(gen, (rows, cols)).square_()
    chi2 += _normal(gen, (rows, cols)).square_()
    return _normal(gen, (rows, cols)).div_(chi2.div_(3.0).sqrt_()).mul_(1e-4 / 3.0 ** 0.5).to(torch.bfloat16)


def _weight(gen, rows, cols):
    return _normal(gen, (rows, cols)).mul_(0.02).to(torch.bfloat16)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = dict(case, seed=seed & 0xFFFFFFFF)
    s["mode"] = ROUNDING.get(case.get("rounding"))
    kind = case["kind"]
    if kind in ("product", "int4"):
        s["A"], s["B"] = _gradient(gen, case["M"], case["K"]), _weight(gen, case["N"], case["K"])
        return s
    b, n, m = case["b"], case["n"], case["m"]
    s["W"] = _weight(gen, m, n)
    if kind == "forward_fp8":
        s["X"] = _activation(gen, b, n)
        return s
    if kind == "train":
        rows = b // 8                                         # a batch of eight sequences
        s["X"] = _activation(gen, b, n).view(8, rows, n).requires_grad_(True)
        s["dY"] = _gradient(gen, b, m).view(8, rows, m)
        s["W"].requires_grad_(True)
        s["bias_param"] = _weight(gen, 1, m).view(m).requires_grad_(True) if case["bias"] else None
        return s
    if kind == "accumulate":
        s["batches"] = [(_gradient(gen, b, m), _activation(gen, b, n)) for _ in range(2)]
        s["dW"] = torch.empty((m, n), dtype=torch.float32, device="cuda")
        s["db"] = torch.empty((m,), dtype=torch.float32, device="cuda")
        s["workspace"] = torch.empty(mx.mxfp4_linear_backward_ex_workspace(b, m, n, True), dtype=torch.uint8, device="cuda") if case["keep"] else None
        return s
    s["dY"], s["X"] = _gradient(gen, b, m), _activation(gen, b, n)
    s["buffers"] = {}
    if case["keep"]:                                          # a program that owns its gradient buffers and one workspace
        s["buffers"] = dict(dX=torch.empty((b, n), dtype=torch.bfloat16, device="cuda"), dW=torch.empty((m, n), dtype=torch.bfloat16, device="cuda"),
                            workspace=torch.empty(mx.mxfp4_linear_backward_workspace(b, m, n), dtype=torch.uint8, device="cuda"))
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "backward":
        return mx.mxfp4_linear_backward(s["dY"], s["X"], s["W"], s["g"], s["seed"], s["mode"], **s["buffers"])
    if kind == "accumulate":                                  # the first micro-batch overwrites the gradients, the second adds to them
        dXs = []
        for i, (dY, X) in enumerate(s["batches"]):
            dX, dW, db = mx.mxfp4_linear_backward_ex(dY, X, s["W"], s["g"], s["seed"] + i, s["mode"], mx.OUT_FP32, dW=s["dW"], db=s["db"],
                                                     accumulate=i > 0, workspace=s["workspace"])
            dXs.append(dX)
        return dXs, dW, db
    if kind == "train":
        y = MxFp4LinearFunction.apply(s["X"], s["W"], s["bias_param"], s["g"], s["seed"], s["mode"], s["forward"] == "fp8")
        leaves = [t for t in (s["X"], s["W"], s["bias_param"]) if t is not None]
        return y, torch.autograd.grad(y, leaves, s["dY"])
    if kind == "forward_fp8":
        return mx.mxfp4_linear_forward_fp8(s["X"], s["W"])
    if kind == "product":
        return mxfp4_product(s["A"], s["B"], s["g"], s["mode"], s["seed"])
    qa = mx.mxfp4_int4_quantize(s["A"], 1, s["g"], s["seed"], 1, s["mode"])
    qb = mx.mxfp4_int4_quantize(s["B"], 1, s["g"], s["seed"], 2, s["mode"])
    return qa, qb, mx.mxfp4_int4_gemm(*qa[:2], *qb[:2], 16.0 / 9.0 if s["mode"] != mx.ROUND_RN else 1.0)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind in ("product", "int4"):
        M, N, K = case["M"], case["N"], case["K"]
        read = 2 * (M + N) * K
        if kind == "product":
            return dict(bytes=read + 4 * M * N, flops=2 * M * N * K)
        # codes (one byte) and the fp32 transformed values are results of the quantiser
        return dict(bytes=read + (M + N) * K * (1 + 1 / 32 + 4) + 2 * M * N, flops=2 * M * N * K)
    b, n, m = case["b"], case["n"], case["m"]
    X, dY, W = 2 * b * n, 2 * b * m, 2 * m * n
    if kind == "forward_fp8":
        return dict(bytes=X + W + 2 * b * m, flops=2 * b * m * n)
    if kind == "backward":
        return dict(bytes=dY + X + W + 2 * b * n + 2 * m * n, flops=4 * b * m * n)
    if kind == "accumulate":
        return dict(bytes=2 * (dY + X + 4 * b * n) + W + 4 * m * n, flops=8 * b * m * n)
    return dict(bytes=2 * X + 2 * dY + 2 * W + 2 * b * n, flops=6 * b * m * n)


def tolerance(case):
    """The quantised operands are whole numbers and stay the same bytes; products of them differ only by the order of their
    fp32 sums and, for a bf16 result, by its last bit.  About four times what the results differ by from the fp64 product
    of the same operands (for the bias gradient: from the fp64 column sums)."""
    if case["kind"] in ("product", "accumulate"):             # fp32 results: 2.7e-8, largest 6.6e-8; bias gradient 1.2e-7, largest 5.9e-7
        return {"rel": 1e-6, "max": 5e-6}
    return {"rel": 7e-3, "max": 1.6e-2}                       # bf16 results: 1.7e-3, largest 3.9e-3 (half a unit in the last place)


# ---------------------------------------------------------------- the same results in 64 bits, plain torch
_M32 = 0xFFFFFFFF


def _philox(index, tag, domain, seed):
    """Philox4x32-10 of the counters (index, 0, tag, domain), indices below 2^32: four int64 tensors of 32-bit words."""
    c = [index, torch.zeros_like(index), torch.full_like(index, tag), torch.full_like(index, domain)]
    k0, k1 = seed & _M32, seed >> 32
    for _ in range(10):
        hi, lo = [], []
        for mult, x in ((0xD2511F53, c[0]), (0xCD9E8D57, c[2])):
            low, high = mult * (x & 0xFFFF), mult * (x >> 16)
            hi.append((high + (low >> 16)) >> 16)
            lo.append(((high << 16) + low) & _M32)
        c = [hi[1] ^ c[1] ^ k0, lo[1], hi[0] ^ c[3] ^ k1, lo[0]]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c


def _reverse16(v):
    for s, m in ((1, 0x5555), (2, 0x3333), (4, 0x0F0F), (8, 0x00FF)):
        v = ((v >> s) & m) | ((v & m) << s)
    return v


def _transform(x, g, seed):
    """x diag(S) H_g / sqrt(g) on every g-chunk of the rows of x (fp64)."""
    if g == 0:
        return x
    j = torch.arange(g, device=x.device)
    words = torch.stack(_philox(j // 128, 0, 0, seed))                     # [4, g]
    sign = 1.0 - 2.0 * ((words[(j % 128) // 32, j] >> (j % 32)) & 1).double()
    H = torch.ones((1, 1), dtype=torch.float64, device=x.device)
    while H.shape[0] < g:
        H = torch.cat((torch.cat((H, H), 1), torch.cat((H, -H), 1)), 0)
    return ((x.reshape(-1, g) * sign) @ H).view(x.shape) / g ** 0.5


def _quantised(x, g, mode, seed, tag, int4=False):
    """What the quantiser keeps of the rows of x (fp64): values, not codes."""
    R, K = x.shape
    out = torch.empty((R, K), dtype=torch.float64, device=x.device)
    rows = max(1, (1 << 24) // K)
    for r0 in range(0, R, rows):
        y = _transform(x[r0:r0 + rows].double(), g, seed).reshape(-1, 32)
        X = torch.ldexp(torch.ones_like(y[:, :1]), (torch.frexp(y.abs().amax(1, keepdim=True))[1] - 3).clamp(min=-127))
        w = y.abs() / X * (1.0 if mode == mx.ROUND_RN else 0.75)
        step = torch.ones_like(w) if int4 else torch.where(w < 2, 0.5, torch.where(w < 4, 1.0, 2.0)).double()
        if mode == mx.ROUND_RN:
            q = ((w / step).round() * step).clamp(max=7.0 if int4 else 6.0)
        else:
            call = torch.arange(r0 * K // 16, r0 * K // 16 + y.numel() // 16, device=x.device)
            b = torch.stack(_philox(call, tag, 1, seed), 1)                # [calls, 4 words of 4 draws]
            b = torch.stack([(b >> s) & 0xFF for s in (0, 8, 16, 24)], 2)
            low = (w / step).floor()
            frac = w / step - low
            if mode == mx.ROUND_SR16:
                even, odd = 256 * b[..., 2] + b[..., 0], 256 * b[..., 3] + b[..., 1]
                dither = torch.stack((even, _reverse16(even), odd, _reverse16(odd)), 2).view(y.shape)
                up = (65536 * frac).floor() + dither >= 65536
            else:
                up = 256 * frac >= b.view(y.shape) + 0.5
            q = (low + up) * step
        out[r0:r0 + rows] = (q * X * y.sign()).view(-1, K)
    return out


def _backward64(dY, X, W, g, mode, seed):
    alpha = 1.0 if mode == mx.ROUND_RN else 16.0 / 9.0
    dX = alpha * _quantised(dY, g, mode, seed, 1) @ _quantised(W.t(), g, mode, seed, 2).t()
    return dX, alpha * _quantised(dY.t(), g, mode, seed, 3) @ _quantised(X.t(), g, mode, seed, 4).t()


def _fp8_64(x, W):
    def e4m3(t):
        scale = 448.0 / t.abs().max().float()
        return (t.float() * scale).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).double(), scale.double()
    (a, sa), (b, sb) = e4m3(x), e4m3(W)
    return a @ b.t() / (sa * sb)


def exact(case, seed):
    s = prepare(dict(case, keep=False), seed)
    kind, g, mode, seed = case["kind"], case.get("g"), s["mode"], s["seed"]
    if kind in ("product", "int4"):
        alpha = 1.0 if mode == mx.ROUND_RN else 16.0 / 9.0
        C = alpha * _quantised(s["A"], g, mode, seed, 1, kind == "int4") @ _quantised(s["B"], g, mode, seed, 2, kind == "int4").t()
        if kind == "product":
            return C
        return (None, None, _transform(s["A"].double(), g, seed)), (None, None, _transform(s["B"].double(), g, seed)), C
    if kind == "forward_fp8":
        return _fp8_64(s["X"], s["W"])
    if kind == "backward":
        return _backward64(s["dY"], s["X"], s["W"], g, mode, seed)
    if kind == "accumulate":
        grads = [_backward64(dY, X, s["W"], g, mode, seed + i) for i, (dY, X) in enumerate(s["batches"])]
        return [dX for dX, _ in grads], grads[0][1] + grads[1][1], sum(dY.double().sum(0) for dY, _ in s["batches"])
    X, dY, W = s["X"].detach().flatten(0, 1), s["dY"].flatten(0, 1), s["W"].detach()
    y = _fp8_64(X, W) if case["forward"] == "fp8" else X.double() @ W.double().t()
    dX, dW = _backward64(dY, X, W, g, mode, seed)
    grads = [dX.view(s["X"].shape), dW]
    if case["bias"]:
        y = y + s["bias_param"].detach().double()
        grads.append(dY.double().sum(0))
    return y.view(s["dY"].shape), grads
