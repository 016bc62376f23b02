// Element-wise kernels of the two extensions of the recipe (the GEMMs are in gemm_pair.cu and gemm_f8.cu):
//   - per-tensor E4M3 quantisation for the FP8 forward pass (Section 4.1; supplementary FP8 results);
//   - MXINT4 elements (Section 3, opening remark): Algorithm 1 / 2 with 4-bit integers in place of E2M1.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.h"
#include "ptx.cuh"
#include "quant_math.cuh"

namespace mx {
namespace {

// ---------------------------------------------------------------- FP8 forward: one scale per tensor
// Both passes are bound by memory; both operands of a product go through each in one launch.  The tensors are cut into
// spans, one per CTA (two CTAs of 1024 threads per SM, each working on one tensor); a thread takes 16 elements (two 16-byte
// loads, one 16-byte store) per step and two steps at a time.  The second pass walks its span from the end, where the
// first pass has left it in L2.
// Before -> now, amax and convert: x 16384 x 4096 and W 4096 x 4096 106 -> 70 us (x alone 91 -> 53: 335 MB at 6.3 TB/s), x
// 1000 x 1024 and W 4096 x 1024 38 -> 9.  Before: a launch per tensor and pass, a memset each, a 64-bit division per load.
struct Fp8Span {
    const __nv_bfloat16* x;
    uint8_t* codes;
    float* scale;                          // [0] 448 / amax, [1] amax
    int64_t cols, ld, pairs;               // pairs of 8-element vectors, the last one possibly half
    int64_t vecs;
    int64_t per_cta;                       // pairs in a CTA's span
    int cta_begin, ctas;
};
struct Fp8Tensors {
    Fp8Span t[2];
    int n;
    uint16_t* partial;                     // one bf16 magnitude per CTA, or null: atomicMax on scale[1]
};
constexpr int kFp8Threads = 1024, kFp8Ctas = 2 * 148;

// Vector v (8 elements) of a tensor; DENSE: rows follow each other without a gap.
template <bool DENSE>
__device__ __forceinline__ uint4 fp8_load(const Fp8Span& t, int64_t v) {
    if (DENSE) return reinterpret_cast<const uint4*>(t.x)[v];
    const int64_t per_row = t.cols >> 3, r = v / per_row;
    return *reinterpret_cast<const uint4*>(t.x + r * t.ld + ((v - r * per_row) << 3));
}
__device__ __forceinline__ uint32_t magnitude_max(uint32_t m, const uint4& v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) m = max(m, max(w[j] & 0x7FFFu, (w[j] >> 16) & 0x7FFFu));
    return m;
}
__device__ __forceinline__ uint32_t block_max(uint32_t m) {
    __shared__ uint32_t warp_max[kFp8Threads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
    __syncthreads();
    m = warp_max[threadIdx.x & 31];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    return m;
}

// Pass 1: amax of |x| as a bf16 bit pattern (magnitudes order like their 15-bit patterns); the maximum is
// order-independent, so the result is reproducible.
template <bool DENSE>
__global__ void __launch_bounds__(kFp8Threads, 2) fp8_amax_kernel(const __grid_constant__ Fp8Tensors p) {
    pdl_launch_dependents();
    pdl_wait();
    const Fp8Span& t = p.t[p.n == 2 && (int)blockIdx.x >= p.t[1].cta_begin ? 1 : 0];
    const int64_t begin = (int64_t)((int)blockIdx.x - t.cta_begin) * t.per_cta, end = min(t.pairs, begin + t.per_cta);
    uint32_t m = 0;
    int64_t i = begin + threadIdx.x;
    for (; i + kFp8Threads < end; i += 2 * kFp8Threads) {
        const int64_t k = i + kFp8Threads;                 // (of the first pair both vectors exist: a later pair follows it)
        const uint4 a = fp8_load<DENSE>(t, 2 * i), b = fp8_load<DENSE>(t, 2 * i + 1), c = fp8_load<DENSE>(t, 2 * k);
        const uint4 d = 2 * k + 1 < t.vecs ? fp8_load<DENSE>(t, 2 * k + 1) : c;
        m = magnitude_max(magnitude_max(magnitude_max(magnitude_max(m, a), b), c), d);
    }
    if (i < end) {
        m = magnitude_max(m, fp8_load<DENSE>(t, 2 * i));
        if (2 * i + 1 < t.vecs) m = magnitude_max(m, fp8_load<DENSE>(t, 2 * i + 1));
    }
    m = block_max(m);
    if (threadIdx.x == 0) {
        if (p.partial != nullptr) p.partial[blockIdx.x] = (uint16_t)m;
        else if (m != 0) atomicMax(reinterpret_cast<uint32_t*>(t.scale + 1), m << 16);
    }
}

// cvt.rn.satfinite.e4m3x2.f32: two floats -> two E4M3 bytes (`lo` in the low byte); nearest-even, saturating at 448.
__device__ __forceinline__ uint32_t cvt_e4m3x2_rn(float lo, float hi) {
    uint16_t d;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(d) : "f"(hi), "f"(lo));
    return d;
}

// Pass 2: scale = 448 / amax in fp32 (1 for an all-zero tensor); code = E4M3(fp32(x * scale)).
__device__ __forceinline__ uint2 fp8_convert(const uint4& v, float sf) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t out[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float a0 = __fmul_rn(__uint_as_float(w[2 * j] << 16), sf), a1 = __fmul_rn(__uint_as_float(w[2 * j] & 0xFFFF0000u), sf);
        const float a2 = __fmul_rn(__uint_as_float(w[2 * j + 1] << 16), sf), a3 = __fmul_rn(__uint_as_float(w[2 * j + 1] & 0xFFFF0000u), sf);
        out[j] = cvt_e4m3x2_rn(a0, a1) | (cvt_e4m3x2_rn(a2, a3) << 16);
    }
    return make_uint2(out[0], out[1]);
}
template <bool DENSE>
__global__ void __launch_bounds__(kFp8Threads, 2) fp8_quantize_kernel(const __grid_constant__ Fp8Tensors p) {
    pdl_launch_dependents();
    pdl_wait();
    const Fp8Span& t = p.t[p.n == 2 && (int)blockIdx.x >= p.t[1].cta_begin ? 1 : 0];
    float amax;
    if (p.partial != nullptr) {                            // at most kFp8Ctas < kFp8Threads spans
        amax = __uint_as_float(block_max((int)threadIdx.x < t.ctas ? p.partial[t.cta_begin + threadIdx.x] : 0u) << 16);
        if ((int)blockIdx.x == t.cta_begin && threadIdx.x == 0) t.scale[1] = amax;
    } else {
        amax = t.scale[1];
    }
    const float sf = amax > 0.0f ? 448.0f / amax : 1.0f;
    if ((int)blockIdx.x == t.cta_begin && threadIdx.x == 0) t.scale[0] = sf;
    const int64_t begin = (int64_t)((int)blockIdx.x - t.cta_begin) * t.per_cta, end = min(t.pairs, begin + t.per_cta);
    auto pair = [&](int64_t i) {
        const uint4 a = fp8_load<DENSE>(t, 2 * i);
        if (2 * i + 1 < t.vecs) {
            const uint2 lo = fp8_convert(a, sf), hi = fp8_convert(fp8_load<DENSE>(t, 2 * i + 1), sf);
            reinterpret_cast<uint4*>(t.codes)[i] = make_uint4(lo.x, lo.y, hi.x, hi.y);
        } else {
            reinterpret_cast<uint2*>(t.codes)[2 * i] = fp8_convert(a, sf);
        }
    };
    int64_t i = end - 1 - threadIdx.x;
    for (; i - kFp8Threads >= begin; i -= 2 * kFp8Threads) {
        const int64_t k = i - kFp8Threads;                 // (both of its vectors exist: a later pair follows it)
        const uint4 a = fp8_load<DENSE>(t, 2 * k), b = fp8_load<DENSE>(t, 2 * k + 1);
        pair(i);
        const uint2 lo = fp8_convert(a, sf), hi = fp8_convert(b, sf);
        reinterpret_cast<uint4*>(t.codes)[k] = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
    if (i >= begin) pair(i);
}

// ---------------------------------------------------------------- MXINT4: integers -7..7 with one E8M0 scale per 32
// The separate pass over transformed values (no transform, g = 256, reduce lengths the tensor-core transform does not take;
// otherwise quantize_tc.cu rounds them where it has them): one thread per MX block.
__global__ void mxint4_quantize_kernel(const float* __restrict__ y, int64_t R, int64_t K, int rounding, uint64_t seed, uint32_t stream_tag,
                                       uint8_t* __restrict__ codes, uint8_t* __restrict__ scales) {
    const int64_t nkb = K >> 5, blk = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (blk >= R * nkb) return;
    const int64_t r = blk / nkb, kb = blk - r * nkb;
    float v[32];
    const float4* src = reinterpret_cast<const float4*>(y + r * K + kb * 32);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float4 f = src[i];
        v[4 * i] = f.x; v[4 * i + 1] = f.y; v[4 * i + 2] = f.z; v[4 * i + 3] = f.w;
    }
    uint32_t out[8], byte, rw[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (rounding == 0) {
        sr_draws32(seed, stream_tag, (uint64_t)(r * K + kb * 32), rw);
        quantize_block32_int4<true>(v, rw, out, byte);
    } else {
        quantize_block32_int4<false>(v, rw, out, byte);
    }
    scales[sf_native_offset(r, kb, (nkb + 3) >> 2)] = (uint8_t)byte;
    uint4* dst = reinterpret_cast<uint4*>(codes + r * K + kb * 32);
    dst[0] = make_uint4(out[0], out[1], out[2], out[3]);
    dst[1] = make_uint4(out[4], out[5], out[6], out[7]);
}

}  // namespace

cudaError_t launch_fp8_quantize(const Fp8QuantArgs* a, int n, uint16_t* partial, cudaStream_t stream) {
    if (n < 1 || n > 2) return cudaErrorInvalidValue;
    Fp8Tensors p = {};
    p.n = n;
    p.partial = partial;
    int64_t pairs = 0;
    bool dense = true;
    for (int i = 0; i < n; ++i) {
        Fp8Span& t = p.t[i];
        t.x = static_cast<const __nv_bfloat16*>(a[i].x);
        t.codes = a[i].codes; t.scale = a[i].scale;
        t.cols = a[i].cols; t.ld = a[i].ld;
        t.vecs = a[i].rows * (a[i].cols >> 3);
        t.pairs = (t.vecs + 1) / 2;
        pairs += t.pairs;
        dense = dense && a[i].ld == a[i].cols;
    }
    // spans of whole steps of a CTA, so that at most kFp8Ctas of them cover both tensors
    int64_t span = (pairs + kFp8Ctas - 3) / (kFp8Ctas - 2);
    span = (span + kFp8Threads - 1) / kFp8Threads * kFp8Threads;
    int ctas = 0;
    for (int i = 0; i < n; ++i) {
        p.t[i].per_cta = span;
        p.t[i].cta_begin = ctas;
        p.t[i].ctas = (int)((p.t[i].pairs + span - 1) / span);
        ctas += p.t[i].ctas;
    }
    if (partial == nullptr)
        for (int i = 0; i < n; ++i) {
            const cudaError_t e = cudaMemsetAsync(a[i].scale + 1, 0, sizeof(float), stream);
            if (e != cudaSuccess) return e;
        }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas); cfg.blockDim = dim3(kFp8Threads); cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    const cudaError_t e = launch_result(cudaLaunchKernelEx(&cfg, dense ? fp8_amax_kernel<true> : fp8_amax_kernel<false>, p));
    return e != cudaSuccess ? e : launch_result(cudaLaunchKernelEx(&cfg, dense ? fp8_quantize_kernel<true> : fp8_quantize_kernel<false>, p));
}

cudaError_t launch_mxint4_quantize(const float* y, int64_t R, int64_t K, int rounding, uint64_t seed, uint32_t stream_tag,
                                   uint8_t* codes, uint8_t* scales, cudaStream_t stream) {
    // rows and K-blocks that only fill the last scale tiles are zero
    if (R % 128 != 0 || K % 128 != 0) {
        const cudaError_t e = cudaMemsetAsync(scales, 0, (size_t)((R + 127) / 128 * ((K + 127) / 128) * 512), stream);
        if (e != cudaSuccess) return e;
    }
    const int64_t blocks = R * (K >> 5);
    mxint4_quantize_kernel<<<(unsigned)((blocks + 127) / 128), 128, 0, stream>>>(y, R, K, rounding, seed, stream_tag, codes, scales);
    return cudaGetLastError();
}

}  // namespace mx
