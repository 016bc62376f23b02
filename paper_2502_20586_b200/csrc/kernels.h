// Internal launch interfaces between the C-ABI layer (api.cu) and the kernel files.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace mx {

// What a launch returned, taken out of the runtime's record if it is an error: checks after later launches are not to find it again.
inline cudaError_t launch_result(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

struct QuantArgs {
    const void* x;        // bf16 [rows, cols], leading dimension ld
    int64_t rows, cols, ld;
    int reduce_dim;       // 1: reduce along cols; 0: reduce along rows (transposed output)
    int g;                // 0, 32, 64, 128, 256
    int rounding;         // 0 SR, 1 RN, 2 SR with the 16-bit dither
    uint64_t seed;
    uint32_t stream_tag;
    uint8_t* codes;
    uint8_t* scales;
    int sf_native;
    float* y_out;         // only for the transform dump
    CUtensorMap tmap_x;   // x as [rows, cols] bf16, box 64 cols x 128 rows, 128-byte swizzle (tensor-core path)
    bool has_tmap;
    const void* custom_t = nullptr;   // bf16 [g, g] row-major: transform matrix given by the caller instead of diag(S) H_g / sqrt(g) (tensor-core path, g <= 128)
    bool layer = false;     // one of the four operand views of a layer's backward call: the call's products read its codes next
    bool mxint4 = false;    // MXINT4 codes (one byte per element) and y_out in one pass (tensor-core path, g <= 128, rounding 0 or 1, native scales)
};

// Whether a launch of the tensor-core quantiser marks x's lines as the first to leave L2, so that codes are still there when a
// GEMM reads them.  Counted are 2 bytes read and 17/32 written an element of every view.
// The views of a backward call: where that is more than L2 holds (126 MB).  Whole calls of 8192 tokens, 1024 in, not marked / marked, SR, RN, SR16
// in us: 3072 out (157 MB) 53.9, 49.4, 51.0 / 52.3, 47.5, 49.3; 4096 out (202 MB) 65.6, 59.8, 63.5 / 64.0, 58.5, 62.9; larger layers the same
// within their repeats.  Below the line: 1024 out (66 MB) 28.6, 25.0, 27.4 / 29.0, 25.4, 27.5; 8192 x 512 x 2304 (105 MB) RN 32.4 / 33.2.  Two
// views from one read count twice: every line is read once in any case.  2^25 elements (103 MB moved, 170 counted) RN 8192 x 1024 x 4096 60.5 / 57.6.
// One view, quantised by a call of its own: only up to 180 MB, since x may be read again next and a marked stream of several times L2's
// size is slower.  RN in us, the view alone, both views in turn, a product with 2048 rows: 8192 x 6144 (127 MB) 23.4, 46.0, 73.0 / 20.2, 43.4, 68.5;
// 8192 x 8192 (170) 29.3, 58.4, 90.0 / 25.5, 60.4, 87.8; 10240 x 8192 (212) 35.3, 70.8, 107.4 / 30.6, 76.4, 105.7; 16384 x 8192 (340) 54.7, 109, 151 / 59.0, 121,
// 156; 16384 x 16384 104, 207, 305 / 117, 235, 310.  Not where the transformed values are written (dump of 8192 x 6144: 57.5 / 60.0).
inline bool quant_input_leaves_l2(const QuantArgs* a, int n) {
    double bytes = 0.0;
    for (int v = 0; v < n; ++v) bytes += (double)a[v].rows * (double)a[v].cols * 2.53125;
    if (a[0].layer) return bytes > 126e6;
    return n == 1 && a[0].y_out == nullptr && bytes > 126e6 && bytes <= 180e6;
}

// Tensor-core transform path (quantize_tc.cu): g in {32, 64, 128} and reduce length a multiple of 128.
bool quant_tc_eligible(const QuantArgs& a);
cudaError_t quant_tc_init();
cudaError_t launch_quantize_tc(const QuantArgs& a, bool dump_y, cudaStream_t stream);
// Up to kQuantMaxViews eligible views sharing g, seed, rounding and scale layout, in ONE launch.
constexpr int kQuantMaxViews = 4;
// lite: the small-footprint build (g <= 128) that can share an SM with the small build of the pair GEMM.
// dual: n = 2, a[0] / a[1] = the row-wise and the transposed view of ONE tensor (both extents multiples of 128): every tile of it is read once.
// col_sums (full-size build, g <= 128, may be null): fp32 [rows / 128, cols] receives the column sums of every 128-row band of a[0]'s
// tensor (reduce_dim 1, rows a multiple of 128).
cudaError_t launch_quantize_tc_group(const QuantArgs* a, int n, bool dump_y, cudaStream_t stream, bool lite = false, bool dual = false,
                                     float* col_sums = nullptr);
// Second pass of the bias gradient: db [m] = (accumulate ? db : 0) + the rows of partial [bands, m] added in order.
struct BandSums {
    const float* partial = nullptr;
    float* db = nullptr;
    int64_t m = 0;
    int bands = 0, accumulate = 0;
};

cudaError_t launch_quantize(const QuantArgs& a, cudaStream_t stream);
cudaError_t launch_rht_dump(const QuantArgs& a, cudaStream_t stream);

struct GemmArgs {
    CUtensorMap tmap_a;   // codes [M, K/2] bytes, box 128 B x 128 rows, 128-byte swizzle
    CUtensorMap tmap_b;   // codes [N, K/2] bytes, box 128 B x BN rows (pair kernel: x tile_n / 2 rows, each CTA loads half a B tile)
    CUtensorMap tmap_sfa; // scale tiles of A as [row tiles * K tiles, 512 bytes]: box = two consecutive tiles (pair kernel)
    CUtensorMap tmap_sfb; // ... of B
    CUtensorMap tmap_c;   // output [M, N] (leading dimension ldc): box 64 bytes x 32 rows, 64-byte swizzle (pair kernel's stores)
    bool use_pair;        // run the CTA-pair kernel (gemm_pair.cu)
    bool lite = false;    // pair kernel only: the small-footprint build that leaves room on the SM for a co-resident quantiser
    const uint8_t* sfa;   // native scale layout
    const uint8_t* sfb;
    int64_t M, N, K;
    float alpha;
    void* C;
    int64_t ldc;
    int out_fp32;
    int accumulate;       // C += alpha A B^T instead of C = (fp32 output only)
};

constexpr int kGemmBM = 128;
constexpr int kGemmBN = 256;
constexpr int kGemmBKBytes = 128;   // 256 E2M1 elements per pipeline stage

// Bias gradient: db [m] (fp32) = (accumulate ? db : 0) + column sums of bf16 dY [b, m]; `partial` is scratch of
// bias_grad_workspace(b, m) bytes.
size_t bias_grad_workspace(int64_t b, int64_t m);
cudaError_t launch_bias_grad(const void* dY, int64_t b, int64_t m, int64_t ld, int accumulate, float* db, float* partial, cudaStream_t stream);
// Each kernel file keeps its own device status word (set when a bounded wait expires); these read and clear them.
cudaError_t fetch_gemm_status(unsigned int* word);
cudaError_t fetch_gemm_pair_status(unsigned int* word);
cudaError_t fetch_quant_tc_status(unsigned int* word);
cudaError_t fetch_fp4_ceiling_status(unsigned int* word);

// GEMM with the RHT + quantiser of its A operand fused into the kernel (gemm_fused.cu): A = x or x^T in bf16.
struct FusedGemmArgs {
    CUtensorMap tmap_x;   // x as [rows, cols] bf16, box 64 cols x 128 rows, 128-byte swizzle
    bool has_tmap_x;
    CUtensorMap tmap_b;   // codes [N, K/2] bytes, box 128 B x 128 rows
    const uint8_t* sfb;   // native scale layout
    int64_t M, N, K;
    float alpha;
    void* C;
    int64_t ldc;
    int out_fp32;
    int g;                // 32, 64, 128
    int reduce_dim;       // 1: A = x; 0: A = x^T
    int rounding;
    uint64_t seed;
    uint32_t stream_tag;
};
bool gemm_fused_eligible(const FusedGemmArgs& a);
cudaError_t launch_gemm_fused(const FusedGemmArgs& a, cudaStream_t stream);
cudaError_t gemm_fused_init();
cudaError_t fetch_gemm_fused_status(unsigned int* word);

// GEMM on 8-bit element containers (gemm_pair.cu, and gemm_f8.cu for few rows and many columns): E4M3 operands with per-tensor scales (FP8 forward pass), or E4M3
// containers of MXINT4 integers with one UE8M0 scale per 32 elements (native scale layout, K % 128 == 0).
struct Gemm8Args {
    CUtensorMap tmap_a;   // bytes [M, K], box 128 B x 128 rows, 128-byte swizzle
    CUtensorMap tmap_b;   // bytes [N, K], box 128 B x tile_n / 2 rows (one-CTA kernel: 256 rows)
    CUtensorMap tmap_c;   // output, as in GemmArgs (pair kernel)
    bool block_scaled;
    CUtensorMap tmap_sfa; // block_scaled: scale tiles (native layout) as [row tiles * K tiles, 512 bytes], box = one tile
    CUtensorMap tmap_sfb;
    const uint8_t* sfa;   // block_scaled: the same scales for the one-CTA kernel
    const uint8_t* sfb;
    const float* scale_a; // plain: device pointers to the per-tensor scales; C = A B^T / (scale_a scale_b)
    const float* scale_b;
    int64_t M, N, K;
    float alpha;          // block_scaled only
    void* C;
    int64_t ldc;
    int out_fp32;
};
int gemm_f8_tile_n(const Gemm8Args& a);            // from M, N, K
cudaError_t launch_gemm_f8(const Gemm8Args& a, int tile_n, cudaStream_t stream);
bool gemm_f8_one_cta(const Gemm8Args& a);          // from M, N: the one-CTA kernel is the better one
cudaError_t launch_gemm_f8_one_cta(const Gemm8Args& a, cudaStream_t stream);
cudaError_t gemm_f8_init();
cudaError_t fetch_gemm_f8_status(unsigned int* word);

// Element-wise kernels of the extensions (variants.cu).
// Per-tensor E4M3 quantisation of one or two tensors: scale[0] = 448 / amax(x) (1 for an all-zero tensor), scale[1] = amax,
// codes = E4M3(x * scale).  `partial` (kFp8PartialBytes of scratch, may be null) saves the memset of the amax words.
struct Fp8QuantArgs {
    const void* x;        // bf16 [rows, cols], leading dimension ld
    int64_t rows, cols, ld;
    uint8_t* codes;       // [rows, cols]
    float* scale;         // [2]
};
constexpr size_t kFp8PartialBytes = 2 * 2 * 148;
cudaError_t launch_fp8_quantize(const Fp8QuantArgs* a, int n, uint16_t* partial, cudaStream_t stream);
// MXINT4 from fp32 pre-quantisation values y [R, K]: per 32-block E8M0 scale (Algorithm 1 / 2 rule), elements rounded
// to integers in [-7, 7] (rounding 0: 3/4 pre-scale + stochastic rounding with the path's Philox draws; 1: nearest),
// stored as E4M3 bytes; scales in the native layout.
cudaError_t launch_mxint4_quantize(const float* y, int64_t R, int64_t K, int rounding, uint64_t seed, uint32_t stream_tag,
                                   uint8_t* codes, uint8_t* scales, cudaStream_t stream);

cudaError_t launch_gemm(const GemmArgs& a, cudaStream_t stream);
cudaError_t gemm_init();            // one-time: opt in to large dynamic shared memory
// One product, or two independent ones in one launch; tile_n = what gemm_pair_tile_n says for them (the B maps' boxes depend on it).
int gemm_pair_tile_n(const GemmArgs* a, int n);
// `bias` (may be null): warps that are idle otherwise add up the band sums.
cudaError_t launch_gemm_pair(const GemmArgs* a, int n, int tile_n, cudaStream_t stream, const BandSums* bias = nullptr);
cudaError_t gemm_pair_init();

}  // namespace mx
