// Blockwise RHT + MXFP4 quantiser with the transform on the tensor cores (g in {32, 64, 128, 256}).
//
// Section 3.2 builds the blockwise RHT as a dense matrix product with a small g x g matrix, which keeps it
// memory-bound in the operand.  Here that product is a tcgen05.mma kind::f16: per tile of 128 output rows x 128
// reduce-dim elements,
//     D[128 x 128] = A[128 x 128] * T,   T = blockdiag over 128/g chunks of diag(S) H_g (x 1/sqrt(g) when exact),
// with bf16 inputs (T is +-1, +-1/8 or 0: exact) and fp32 accumulation in TMEM.  The accumulator comes back with
// one output row per TMEM lane and its 128 transformed values in consecutive columns, so each epilogue thread
// owns whole MX blocks: amax, scale, stochastic rounding and packing need no shuffles.  The same kernel serves
// both access patterns: for a contiguous reduce dimension the x tile is the K-major A operand; for the transposing
// views (W, dY^T, X^T of Algorithm 3) the very same TMA tile is handed to the MMA as an MN-major operand, so the
// transposition costs nothing.
//
// g = 256 spans two 128-wide k-tiles: H_256 = [[H_128, H_128], [H_128, -H_128]], so the two k-tiles of a 256-chunk
// go through their own half-transform T_h = diag(S_{128h..128h+127}) H_128 / 16 into two accumulators u and v, and
// the epilogue forms u + v and u - v in fp32 (one add per element more than g <= 128).
//
// One launch can quantise up to four operand views that share g, seed and rounding (the four views of one
// backward call, Algorithm 3 lines 3-6): their tiles form one list that the persistent CTAs walk, which removes
// three launch / prologue / drain gaps per layer.
//
//   warp 0        TMA producer (two 64-column x 128-row boxes per tile, 128-byte swizzle, 4-stage ring)
//   warp 1        MMA issuer (8 K=16 MMAs per tile, N = g, into one of four 128-column TMEM accumulators)
//   warps 2, 3    column sums of dY when a bias gradient is wanted, else idle; they complete warp group 0, which hands
//                 registers (setmaxnreg) to the epilogue groups
//   warps 4..15   epilogue, three groups of four warps on alternate tiles: warp = TMEM lane quadrant, a thread owns one
//                 output row of the tile: tcgen05.ld 32 columns at a time, scale / SR / pack / store per MX block
//                 (g = 256: four groups, warps 4..19)
//
// What bounds it: SR by the epilogue's logic pipe and, in calls that last, by the board's power (950 - 1000 W at 1.4 - 1.7 GHz: time is
// energy, an instruction per element about a hundredth of a call); RN and SR16 by the memory.  What brought it there:
//   - issue.  MMAs issued from a lane-0 branch have their descriptors moved to uniform registers every time, and every epilogue
//     warp waited for an accumulator; a converged warp with one elected lane, and three epilogue groups with a spare accumulator instead of
//     four without one;
//   - whole sectors of codes in one store (store_codes), SR through the convert (quantize_block32_rw), tiles described once
//     (TileInfo), MMAs without T's zero blocks, T eight entries at a time (hadamard_row8).
// 16384 x 16384 views, before the last five -> now, in bursts: SR row-wise 124 -> 112 us, transposing 140 -> 113, g = 64 118 / 138 -> 107, g = 256
// 132 -> 125, SR16 111 / 130 -> 103 - 105, RN 108 / 119 -> 105 (6.5 TB/s); the operands of a backward call, 16384 x 4096 x 4096 105 -> 95 - 102 (g = 128),
// 8192 x 1024 x 4096 38.5 -> 35 (g = 64).
// Slower were: the block loop rolled up (SR 127), four groups with accumulators handed back by halves (128), TMEM loads a block
// ahead (134), part of the Philox rounds folded into constants of the view (more moves than it saved: 96 instructions a block for 85), a fifth
// stage (RN 110).
// Every mbarrier wait is bounded; on expiry the CTA records a status word and unwinds.
#include <cuda_bf16.h>

#include "kernels.h"
#include "ptx.cuh"
#include "quant_math.cuh"

namespace mx {
namespace {

constexpr int kTile = 128;                          // output rows per tile and reduce-dim elements per tile
constexpr uint32_t kBoxBytes = 64 * 2 * 128;        // one TMA box: 64 bf16 columns x 128 rows = 16 KB
constexpr uint32_t kTileBytes = 2 * kBoxBytes;      // 32 KB
constexpr uint32_t kTBytes = 2 * kBoxBytes;         // transform matrix, 128 x 128 bf16

// What the epilogue has to know of a tile.  The producer thread, which works out where the tile lies in any case, leaves it in
// shared memory: each epilogue thread did the same arithmetic for every tile of its own.
struct __align__(16) TileInfo {
    uint8_t* codes;            // codes of the tile's first row
    uint8_t* scales;           // native layout: the tile's 512 bytes; linear: scales of its first row
    uint32_t blk;              // index in the view of the first row's first MX block
    uint32_t k_blocks;         // MX blocks from one row to the next
    uint32_t rows;             // rows of the tile that exist
    uint32_t view;
};
// The producer is at most kStages tiles ahead of the MMA issuer and that one kAccBufs ahead of an epilogue group which has not
// read its accumulator out: sixteen entries are never overwritten before they are read.
constexpr uint32_t kInfoSlots = 16;

// Two builds of the kernel.  FULL owns its SM: a 4-stage ring, four TMEM accumulators, three epilogue warp groups on
// alternate tiles (g = 256: two teams of two groups, each with its pair of accumulators).  LITE is sized to run beside the small build of the pair GEMM (gemm_pair.cu) on the same SM, so that
// the operands of one product are quantised while the other product's GEMM keeps the FP4 pipe busy: one 32 KB stage,
// one accumulator (128 TMEM columns), two epilogue warp groups that share every tile (two MX blocks of each row per
// group), 64 registers per thread at launch.  g <= 128 only.  Codes and scales are the same bytes in both builds.
template <bool LITE, int KW>
struct QCfg {
    static constexpr int kStages = LITE ? 1 : 4;
    static constexpr int kAccBufs = LITE ? 1 : 4;                        // x 128 TMEM columns
    static constexpr int kTmemCols = LITE ? 128 : 512;
    static constexpr int kEpiGroups = LITE ? 2 : KW == 2 ? 4 : 3;       // epilogue warp groups (one warp per TMEM lane quadrant)
    static constexpr int kEpiWarps = 4 * kEpiGroups;
    static constexpr int kTransforms = KW;                               // g = 256: two half-transforms
    static constexpr uint32_t kSmem = kStages * kTileBytes + kTransforms * kTBytes + kInfoSlots * (uint32_t)sizeof(TileInfo) + 1024 + 512;
    static_assert((2 * kStages + 2 * kAccBufs + (int)kInfoSlots) * 8 + 8 <= 512, "barriers");
    // Register hand-over (setmaxnreg): warp group 0 shrinks to kRegsLight, the epilogue groups grow to kRegsEpi.  The
    // increase can only draw on what the CTA itself holds, i.e. threads x registers-per-thread at launch: the init
    // routine checks that budget against the compiled kernel, because an increase that cannot be met waits forever.
    static constexpr int kRegsLight = LITE ? 32 : 40, kRegsEpi = LITE ? 80 : kEpiGroups == 3 ? 152 : 104;
    static constexpr int kThreads = (4 + kEpiWarps) * 32;                // warp group 0: producer, MMA issuer, two idle warps; then the epilogue warp groups
    static constexpr int kLaunchRegs = LITE ? 64 : kEpiGroups == 3 ? 128 : 96;
    static_assert(kThreads * kLaunchRegs >= 128 * kRegsLight + (kThreads - 128) * kRegsEpi, "warp groups ask for more registers than the CTA holds");
};

struct QView {                 // one operand view: output operand [R, K] read from x [rows, cols]
    uint32_t R, k_blocks;      // output rows; MX blocks of 32 along K (R * k_blocks < 2^31)
    uint32_t r_tiles, k_tiles;
    uint32_t tile_begin;       // first index of this view in the launch's tile list
    uint32_t n_tiles;          // r_tiles * k_tiles
    uint32_t minor_count;      // tiles along the fast direction of the view's tile order (see locate_tile)
    uint32_t lg_band;          // log2 of the tiles across the fast direction that are walked side by side (TilePos)
    int reduce_dim;            // 1: K runs along x columns (x tile is the K-major operand); 0: along x rows (MN-major)
    uint32_t stream_tag;
    uint8_t* codes;
    uint8_t* scales;
    float* y_out;              // transform dump only
};

struct QParams {
    QView view[kQuantMaxViews];
    int n_views;
    uint32_t n_tiles;          // over all views
    int g, sf_native;
    bool x_passes;             // x's lines are the first to leave L2 (quant_input_leaves_l2)
    bool wide_stores;          // y_out and the codes of every view start on 32-byte boundaries
    const uint16_t* custom_t;  // bf16 [g, g] row-major transform matrix given by the caller, or null (then diag(S) H_g / sqrt(g))
    uint64_t seed;
    float* col_sums;           // partial column sums [x rows / 128][x cols] of view 0's x in fp32 (bias gradient), or null
    PipeConsts pipe;           // see quant_math.cuh: constants kept opaque to the compiler
    PhiloxKeys keys;           // the ten Philox round keys of `seed` (key schedule only; the rounds run on the device)
};

struct QMaps {
    CUtensorMap x[kQuantMaxViews];
};

// Position of a tile in the launch's list: its view and where it lies there.  Tiles of a view with a contiguous reduce
// dimension run along k first, the transposing ones along the output rows first, so that CTAs working side by side read
// neighbouring 256-byte row segments of x; across that direction four tiles (two, one where the count is not a multiple)
// go side by side, so that a transposing view's 64-byte code segments of a row are written as whole lines at nearly the
// same time (16384 x 16384 transposing: 142 -> 139 us).  major counts bands, minor walks a band.
// DUAL launches: view 0 (reduce along x columns) and view 1 (reduce along x rows) are the two views of ONE tensor x
// (dY of Algorithm 3, lines 3 and 5).  A unit is one 128 x 128 tile of x, loaded once, in the same order for both views;
// it yields two logical tiles, 2 u (view 0) and 2 u + 1 (view 1).
struct TilePos {
    int v;
    uint32_t major, minor;
    uint32_t local;            // index inside the view (DUAL: the unit)
};
template <bool DUAL>
__device__ __forceinline__ TilePos locate_tile(const QParams& p, uint32_t t) {
    TilePos pos;
    if (DUAL) {
        pos.v = (int)(t & 1u);
        pos.local = t >> 1;
    } else {
        pos.v = 0;
#pragma unroll
        for (int i = 1; i < kQuantMaxViews; ++i)
            if (i < p.n_views && t >= p.view[i].tile_begin) pos.v = i;
        pos.local = t - p.view[pos.v].tile_begin;
    }
    pos.major = pos.local / p.view[pos.v].minor_count;
    pos.minor = pos.local - pos.major * p.view[pos.v].minor_count;
    return pos;
}
__device__ __forceinline__ uint32_t along_minor(const QView& vw, const TilePos& pos) { return pos.minor >> vw.lg_band; }
__device__ __forceinline__ uint32_t across_minor(const QView& vw, const TilePos& pos) { return (pos.major << vw.lg_band) | (pos.minor & ((1u << vw.lg_band) - 1u)); }
__device__ __forceinline__ uint32_t row_tile(const QView& vw, const TilePos& pos) { return vw.reduce_dim == 1 ? across_minor(vw, pos) : along_minor(vw, pos); }
__device__ __forceinline__ uint32_t k_tile(const QView& vw, const TilePos& pos) { return vw.reduce_dim == 1 ? along_minor(vw, pos) : across_minor(vw, pos); }
template <int KW, bool INT4>
__device__ __forceinline__ void describe_tile(const QParams& p, const TilePos& pos, TileInfo& out) {
    const QView& vw = p.view[pos.v];
    const uint32_t rt = row_tile(vw, pos), kt = k_tile(vw, pos) * KW;
    const uint32_t blk = rt * (uint32_t)kTile * vw.k_blocks + kt * 4u;
    out.codes = vw.codes + (uint64_t)blk * (INT4 ? 32u : 16u);
    out.scales = vw.scales + (p.sf_native ? sf_row_offset(rt * ((vw.k_blocks + 3) >> 2) + kt, 0, 0) : (uint64_t)blk);
    out.blk = blk;
    out.k_blocks = vw.k_blocks;
    out.rows = vw.R - rt * (uint32_t)kTile;
    out.view = (uint32_t)pos.v;
}

// kModeInt4*: MXINT4 elements, one byte each, together with the transformed values that were rounded (g <= 128): what a pass
// of its own over the fp32 values did before.  Bound by writing them; 32-byte stores, since a thread owns a row: 1024 x 8192
// 37 -> 15.7 us, 16384 x 4096 252 -> 89 (the dump alone 175 -> 72: 402 MB at 5.6 TB/s).
enum { kModeSR = 0, kModeRN = 1, kModeDump = 2, kModeSR16 = 3, kModeInt4SR = 4, kModeInt4RN = 5 };
constexpr bool mode_draws(int mode) { return mode == kModeSR || mode == kModeSR16 || mode == kModeInt4SR; }
constexpr bool mode_int4(int mode) { return mode == kModeInt4SR || mode == kModeInt4RN; }
constexpr bool mode_keeps_y(int mode) { return mode == kModeDump || mode_int4(mode); }
// template argument of quantize_block32_rw
constexpr int mode_rounding(int mode) { return mode == kModeSR16 ? 2 : mode; }

// Codes of block j of a thread's row: two blocks go out together, 32 bytes, a whole L2 sector where the operand starts on one.
// A block at a time wrote every sector in two halves: 16384 x 16384 SR transposing 140 -> 124 us, row-wise 126 -> 124, RN 118.5 -> 105
// (the memory's rate) and 109 -> 105; the operands of 16384 x 4096 x 16384 324 -> 308.
__device__ __forceinline__ void store_codes(uint8_t* dst, int j, const uint32_t (&packed)[4], uint32_t (&kept)[4], bool wide) {
    if ((j & 1) == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) kept[i] = packed[i];
    } else {
        const uint32_t both[8] = {kept[0], kept[1], kept[2], kept[3], packed[0], packed[1], packed[2], packed[3]};
        st_global_32B(dst + 16 * (j - 1), both, wide);
    }
}
// sum += the eight bf16 values of v, each widened exactly and added in fp32 (one instruction an element).
__device__ __forceinline__ void add_bf16x8(float (&sum)[8], const uint4& v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
        asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.f32.bf16 %0, lo, %0;\n\tadd.f32.bf16 %1, hi, %1;\n\t}"
            : "+f"(sum[2 * i]), "+f"(sum[2 * i + 1]) : "r"(w[i]));
}
// Tiles (units) that a round-robin deal of n gives this CTA.
__device__ __forceinline__ uint32_t tiles_of_cta(uint32_t n) { return blockIdx.x < n ? (n - blockIdx.x + gridDim.x - 1u) / gridDim.x : 0u; }

// KW = 128-wide k-tiles per entry of the tile list: 1, or 2 for g = 256 (a tile then spans one 256-chunk).
template <int MODE, int KW, bool LITE, bool DUAL, bool HALVES = false>
__device__ __forceinline__ void quantize_tc_body(const QMaps& maps, const QParams& p) {
    using Cfg = QCfg<LITE, KW>;
    static_assert(!DUAL || (KW == 1 && !LITE), "one load for two views: g <= 128, full-size build");
    constexpr int kStagesQ = Cfg::kStages, kAccBufs = Cfg::kAccBufs, kEpiGroups = Cfg::kEpiGroups, kThreadsQ = Cfg::kThreads;
    static_assert(!(LITE && KW == 2), "the small build serves g <= 128");
    static_assert(!HALVES || (KW == 1 && !LITE && !DUAL), "half tiles: g <= 128, one view's tile at a time");
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* smem_t = smem + kStagesQ * kTileBytes;
    TileInfo* info = reinterpret_cast<TileInfo*>(smem_t + Cfg::kTransforms * kTBytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(info + kInfoSlots);
    uint64_t* full_bar = bars;                          // [kStagesQ]  TMA -> MMA
    uint64_t* empty_bar = bars + kStagesQ;              // [kStagesQ]  MMA -> TMA
    uint64_t* acc_full = bars + 2 * kStagesQ;           // [kAccBufs]  MMA -> epilogue
    uint64_t* acc_empty = bars + 2 * kStagesQ + kAccBufs;   // [kAccBufs]  epilogue -> MMA
    uint64_t* info_full = acc_empty + kAccBufs;         // [kInfoSlots] producer -> epilogue
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(info_full + kInfoSlots);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (warp-uniform, and known to be)
    const uint32_t num_tiles = p.n_tiles;

    if (threadIdx.x == 0) {
        // a stage is free when its transforms have read it (one commit) and, with column sums on, the two summing warps too
        const uint32_t n_readers = (KW == 1 && !LITE && p.col_sums != nullptr) ? 3u : 1u;
        for (int s = 0; s < kStagesQ; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], n_readers); }
        for (int b = 0; b < kAccBufs; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], (KW == 2 || LITE || HALVES) ? 8 : 4); }
        for (uint32_t i = 0; i < kInfoSlots; ++i) mbar_init(&info_full[i], 1);
        *abort_flag = 0;
        mbar_fence_init();
        for (int v = 0; v < p.n_views; ++v) prefetch_tensormap(&maps.x[v]);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, Cfg::kTmemCols);
        tmem_relinquish();
    }
    {
        if (KW == 1 && p.custom_t != nullptr) pdl_wait();                // the matrix may come from the kernel before this one
        // Transform operand, written in the 128-byte-swizzled K-major layout the MMA descriptor expects:
        // entry (n, k) at box (k / 64), row n (128 B pitch), 16-byte chunk ((k % 64) / 8) ^ (n % 8).  Only the g x g block at the
        // origin is read (g = 256: the two 128 x 128 half-transforms).
        const int lg_c = p.g == 32 ? 2 : p.g == 64 ? 3 : 4;                  // chunks of eight k to a row: 2^lg_c
#pragma unroll
        for (int h = 0; h < KW; ++h) {                                   // KW = 2: sign bits 128 h .. 128 h + 127 come from Philox call h
            const uint4 sign = philox4x32_10((uint32_t)h, 0u, 0u, 0u, (uint32_t)p.seed, (uint32_t)(p.seed >> 32));
            const uint32_t mag = KW == 2 ? 0x3D803D80u : p.g == 64 ? 0x3E003E00u : 0x3F803F80u;    // 1/16, 1/8: exact 1/sqrt(g); else 1
            for (int task = threadIdx.x; task < 8 << (2 * lg_c); task += kThreadsQ) {
                const int n = task >> lg_c, c = task & ((1 << lg_c) - 1);
                uint32_t w[4];
                if (KW == 1 && p.custom_t != nullptr) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {                        // entry (n, k) of the operand = T[k][n] (Section 3.2: any orthogonal matrix)
                        const int k = c * 8 + 2 * j;
                        w[j] = p.custom_t[k * p.g + n] | ((uint32_t)p.custom_t[(k + 1) * p.g + n] << 16);
                    }
                } else {
                    hadamard_row8(n, c, sign, mag, w);
                }
                const uint32_t off = (uint32_t)(c >> 3) * kBoxBytes + (uint32_t)n * 128u + (uint32_t)(((c & 7) ^ (n & 7)) << 4);
                *reinterpret_cast<uint4*>(smem_t + h * kTBytes + off) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        fence_proxy_async_smem();                                        // generic-proxy writes -> tensor-core reads
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    pdl_launch_dependents();                            // the next kernel of the stream may set itself up behind this one
    pdl_wait();                                         // the set-up above overlapped the previous kernel's tail; its data is needed now

    if (warp < 4) {
    // ============================ warp group 0: producer, MMA issuer, two idle warps; it gives registers to the others
    reg_dealloc<Cfg::kRegsLight>();
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t it = 0, n_info = 0;
            bool ok = true;
            const uint64_t evict_first = l2_policy_evict_first();
            // DUAL: one load per unit (two logical tiles), in the coordinates of its row-wise view
            for (uint32_t t = DUAL ? 2u * blockIdx.x : blockIdx.x; t < num_tiles && ok; t += (DUAL ? 2u : 1u) * gridDim.x) {
                TilePos pos = locate_tile<DUAL>(p, t);
                // x coordinates: (column, row).  reduce_dim 1: output rows = x rows, k = x columns; else swapped.
                const bool rowwise = p.view[pos.v].reduce_dim == 1;
#pragma unroll
                for (int h = 0; h < KW; ++h, ++it) {
                    const int s = it % kStagesQ;
                    if (!(ok = mbar_wait(&empty_bar[s], ((it / kStagesQ) & 1) ^ 1, abort_flag))) break;
                    const uint32_t rt = row_tile(p.view[pos.v], pos), kt = k_tile(p.view[pos.v], pos) * KW + h;   // 128-wide k-tile
                    const int32_t cx = (int32_t)((rowwise ? kt : rt) * kTile), cy = (int32_t)((rowwise ? rt : kt) * kTile);
                    uint8_t* st = smem + s * kTileBytes;
                    mbar_expect_tx(&full_bar[s], kTileBytes);
                    if (p.x_passes) {
                        tma_load_2d_hint(st, &maps.x[pos.v], &full_bar[s], cx, cy, evict_first);
                        tma_load_2d_hint(st + kBoxBytes, &maps.x[pos.v], &full_bar[s], cx + 64, cy, evict_first);
                    } else {
                        tma_load_2d(st, &maps.x[pos.v], &full_bar[s], cx, cy);
                        tma_load_2d(st + kBoxBytes, &maps.x[pos.v], &full_bar[s], cx + 64, cy);
                    }
                }
                if (!ok) break;
#pragma unroll
                for (int h = 0; h < (DUAL ? 2 : 1); ++h, ++n_info) {
                    if (DUAL) pos.v = h;
                    describe_tile<KW, mode_int4(MODE)>(p, pos, info[n_info % kInfoSlots]);
                    mbar_arrive(&info_full[n_info % kInfoSlots]);
                }
            }
            if (!ok) *abort_flag = 1;
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        // The whole warp walks the loop and one elected lane issues: with warp-uniform control flow the descriptors live in
        // uniform registers.
        // kind::f16 instruction descriptor: D = fp32 (bits 4-5 = 1), A = B = bf16 (bits 7-9, 10-12 = 1),
        // A major at bit 15 (0 = K-major, 1 = MN-major), B K-major, N >> 3 at bit 17, M >> 4 at bit 24.
        const uint32_t gt = p.g < kTile ? (uint32_t)p.g : (uint32_t)kTile, lg_steps = gt == 32 ? 1u : gt == 64 ? 2u : 3u;   // K-steps of a chunk
        const uint32_t idesc_k = (1u << 4) | (1u << 7) | (1u << 10) | ((gt >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
        const uint32_t t_addr = smem_u32(smem_t), s_addr = smem_u32(smem);
        uint32_t it = 0;
        bool ok = true;
        auto wait = [&](uint64_t* bar, uint32_t parity) { return ok = __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)); };
        auto transform = [&](uint32_t a_addr, bool rowwise, int h, int b) {      // 8 MMAs (K = 16 each): stage -> accumulator b
            const uint32_t idesc = idesc_k | ((rowwise ? 0u : 1u) << 15), d = tmem_base + b * kTile;
            const uint64_t bdesc = make_smem_desc(t_addr + h * kTBytes, 16, 1024, 2);
            // K-major: box ks/4, 32 bytes of K per step inside the 128-byte swizzle atom; MN-major: 16 k-rows of 128 B per
            // step, the second 64 output rows sit one box further
            const uint64_t adesc = rowwise ? make_smem_desc(a_addr, 16, 1024, 2) : make_smem_desc(a_addr, kBoxBytes, 1024, 2);
            const uint32_t a_half = rowwise ? kBoxBytes >> 4 : 4 * 2048 >> 4, a_step = rowwise ? 32 >> 4 : 2048 >> 4;
            // T is block-diagonal with equal blocks: chunk c of the tile's 128 / g takes its own columns of A against the first block.
            // (With the zero blocks multiplied as well the tensor cores did two or four times the work, at the board's power limit.  g = 64,
            // when that changed and other parts still took longer: operands of 8192 x 1024 x 4096 41.0 -> 39.8 us (now 35), nearest rounding
            // 32.6 -> 31.6 (now 30 - 31); 16384 x 16384 SR 110 -> 108.)
#pragma unroll
            for (uint32_t ks = 0; ks < 8; ++ks) {
                const uint32_t c = ks >> lg_steps, kc = ks & ((1u << lg_steps) - 1u);
                tc_mma_f16(d + c * gt, adesc + (ks >> 2) * a_half + (ks & 3) * a_step, bdesc + (kc >> 2) * (kBoxBytes >> 4) + (kc & 3) * (32 >> 4), idesc, kc != 0 ? 1u : 0u);
            }
        };
        if (DUAL) {
            // per unit: the stage is the K-major operand of view 0's transform and the MN-major operand of view 1's
            uint32_t is = 0;                                             // stage counter (units)
            for (uint32_t u = blockIdx.x; 2u * u < num_tiles && ok; u += gridDim.x, ++is) {
                const int s = is % kStagesQ;
                if (!wait(&full_bar[s], (is / kStagesQ) & 1)) break;
                const uint32_t a_addr = s_addr + s * kTileBytes;
#pragma unroll
                for (int h = 0; h < 2; ++h, ++it) {
                    const int b = it % kAccBufs;
                    if (!wait(&acc_empty[b], ((it / kAccBufs) & 1) ^ 1)) break;
                    tc_fence_after_sync();
                    if (elect_one()) {
                        transform(a_addr, h == 0, 0, b);
                        tc_commit(&acc_full[b]);
                        if (h == 1) tc_commit(&empty_bar[s]);            // both transforms have read the stage
                    }
                    __syncwarp();
                }
            }
        } else {
            const bool sums = KW == 1 && !LITE && p.col_sums != nullptr;
            for (uint32_t t = blockIdx.x; t < num_tiles && ok; t += gridDim.x) {
                int v = 0;
#pragma unroll
                for (int i = 1; i < kQuantMaxViews; ++i)
                    if (i < p.n_views && t >= p.view[i].tile_begin) v = i;
                const bool rowwise = p.view[v].reduce_dim == 1;
#pragma unroll
                for (int h = 0; h < KW; ++h, ++it) {                       // KW = 2: k-tile h goes through T_h into its own accumulator
                    const int s = it % kStagesQ, b = it % kAccBufs;
                    if (!wait(&acc_empty[b], ((it / kAccBufs) & 1) ^ 1)) break;
                    if (!wait(&full_bar[s], (it / kStagesQ) & 1)) break;
                    tc_fence_after_sync();
                    if (elect_one()) {
                        transform(s_addr + s * kTileBytes, rowwise, h, b);
                        tc_commit(&empty_bar[s]);
                        tc_commit(&acc_full[b]);
                        if (sums && v != 0) mbar_arrive(&empty_bar[s], 2);   // in place of the two summing warps, which only read view 0
                    }
                    __syncwarp();
                }
            }
        }
        if (!ok && lane == 0) *abort_flag = 1;
    } else if (KW == 1 && !LITE && p.col_sums != nullptr) {
        // ------------------------------------------------------------------ warps 2, 3: column sums of the x tile (dL/db = 1 dL/dy)
        // The tile is in shared memory anyway: warp w sums columns 64 w .. 64 w + 63 (one TMA box).  A lane takes eight adjacent columns
        // (one 16-byte chunk, moved by the 128-byte swizzle; eight lanes read a whole row, so no bank conflicts) of every fourth row, rows
        // in order; the four row groups are added pairwise: a fixed summation order.  One partial sum per (128-row band of x, column);
        // the GEMM launch adds the bands in order.  (A launch of several views: only the tiles of view 0, the row-wise view of dY, are
        // summed; for the others, which follow, the MMA issuer counts these warps' arrivals.)
        // These two warps set the pace of view 0's tiles when they take long over one (each shares its scheduler with three epilogue warps):
        // two columns a lane, 128 rows in a chain of additions and widening by shift and mask took 9 us of a call of 4096 x 2048 x 6144, and
        // the other views' tiles passed through their hands as well.  Calls with db (without), before -> now, SR, fp32 results: 4096 x 2048 x
        // 6144 86.0 -> 79.8 us (77.3), 8192 x 1024 x 4096 78.1 -> 70.3 (67.4), 8192 x 1024 x 1024 36.6 -> 33.9 (32.6), 4224 x 1000 x 1408 27.5 -> 25.3 (24.8).
        const int w = warp - 2;
        const uint32_t chunk = (uint32_t)lane & 7u, rg = (uint32_t)lane >> 3;
        const uint32_t off0 = rg * 128u + ((chunk ^ rg) << 4), off1 = (rg + 4u) * 128u + ((chunk ^ (rg + 4u)) << 4);   // rows rg and rg + 4
        uint32_t is = 0;
        bool ok = true;
        for (uint32_t u = blockIdx.x; u < (DUAL ? num_tiles >> 1 : p.view[0].n_tiles); u += gridDim.x, ++is) {
            const int s = is % kStagesQ;
            ok = mbar_wait(&full_bar[s], (is / kStagesQ) & 1, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const uint8_t* box = smem + s * kTileBytes + w * kBoxBytes;
            float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
            for (int r = 0; r < kTile; r += 8) {
                const uint4 a = *reinterpret_cast<const uint4*>(box + r * 128 + off0), b = *reinterpret_cast<const uint4*>(box + r * 128 + off1);
                add_bf16x8(sum, a);
                add_bf16x8(sum, b);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty_bar[s]);                   // this warp is done with the stage
            // rows: groups 0 and 1, 2 and 3, then the two pairs; a lane ends up with two of its chunk's eight columns
            const bool odd = (rg & 1u) != 0, high = (rg & 2u) != 0;
            float half[4], quarter[2];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float got = __shfl_xor_sync(0xffffffffu, odd ? sum[i] : sum[4 + i], 8);
                half[i] = (odd ? sum[4 + i] : sum[i]) + got;
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float got = __shfl_xor_sync(0xffffffffu, high ? half[i] : half[2 + i], 16);
                quarter[i] = (high ? half[2 + i] : half[i]) + got;
            }
            const TilePos pos = locate_tile<DUAL>(p, DUAL ? 2u * u : u);
            const uint32_t xr = row_tile(p.view[0], pos), xc = k_tile(p.view[0], pos);
            float* dst = p.col_sums + (int64_t)xr * (32 * (int64_t)p.view[0].k_blocks) + (int64_t)xc * kTile + w * 64 + 8 * chunk + (odd ? 4 : 0) + (high ? 2 : 0);
            *reinterpret_cast<float2*>(dst) = make_float2(quarter[0], quarter[1]);
        }
        if (!ok && lane == 0) *abort_flag = 1;
    }
    } else {
        // ------------------------------------------------------------------ epilogue (the warp groups after the first)
        reg_alloc<Cfg::kRegsEpi>();
        // Groups of four warps (FULL: three, four for g = 256; LITE: two) take alternate tiles or share them, see below; inside
        // a group a warp owns one TMEM lane quadrant, i.e. a thread owns one output row of the tile: four MX blocks, 64 bytes of
        // codes, 4 scale bytes.  The SR draws of a block depend on element indices only and are computed while the accumulator is
        // on its way to the registers.
        const int e = warp - 4;
        const int q = warp & 3;                      // TMEM lane quadrant this warp may read
        const int grp = e >> 2;
        const float cg = p.custom_t != nullptr ? 1.0f : p.g == 32 ? 0.17677669529663687f : p.g == 128 ? 0.08838834764831845f : 1.0f;
        // A team takes every kTeams-th tile of the CTA.  FULL: a group is a team (g = 256: two groups are, one for each half of
        // the 256-chunk), a thread handles all four blocks of its row.
        // LITE: the two groups share every tile, group 0 the row's MX blocks 0 and 1, group 1 blocks 2 and 3.
        constexpr int kTeams = KW == 2 ? 2 : LITE ? 1 : kEpiGroups;
        // HALVES: a group takes half a tile, two blocks of every row, at a time (quantise_by_halves).
        constexpr int kBlocksPerThread = LITE || HALVES ? 2 : 4;
        constexpr uint32_t kUnits = HALVES ? 2u : 1u;                                   // units of work a tile gives the groups
        const uint32_t lane_row = (uint32_t)(q * 32 + lane);
        const uint32_t scale_off = (uint32_t)sf_row_offset(KW == 2 ? grp & 1 : 0, q, lane);   // native layout, from the tile's first byte
        bool ok = true;
        auto wait = [&](uint64_t* bar, uint32_t parity) { return ok = __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)); };

        // i-th accumulator of the CTA.  Tiles are dealt out round-robin; in a DUAL launch whole units are (two consecutive tiles,
        // one per view), so that both transforms of a unit read the same stage.
        const uint32_t n_mine = DUAL ? 2u * tiles_of_cta(num_tiles >> 1) : tiles_of_cta(num_tiles);
        for (uint32_t un = KW == 2 ? (uint32_t)(grp >> 1) : LITE ? 0u : (uint32_t)grp; un < kUnits * n_mine; un += kTeams) {
            const uint32_t it = un / kUnits;
            const uint32_t part = KW == 2 ? 4u * (grp & 1) : LITE ? 2u * grp : 2u * (un % kUnits);    // first MX block of the row this thread handles
            if (!wait(&info_full[it % kInfoSlots], (it / kInfoSlots) & 1)) break;
            const TileInfo ti = info[it % kInfoSlots];
            const QView& vw = p.view[ti.view];
            const bool live = lane_row < ti.rows;
            const uint32_t row_blk = lane_row * ti.k_blocks + part, blk = ti.blk + row_blk;   // this thread's first MX block
            uint8_t* code_dst = ti.codes + (uint64_t)row_blk * (mode_int4(MODE) ? 32u : 16u);
            uint8_t* scale_dst = ti.scales + (p.sf_native ? scale_off + (KW == 2 ? 0u : part) : row_blk);
            float* y_dst = mode_keeps_y(MODE) ? vw.y_out + (uint64_t)blk * 32u : nullptr;
            uint32_t sb_all = 0, kept[4];
            if constexpr (KW == 2) {
                // g = 256: a tile is one 256-chunk of 128 rows; its two k-tiles went through T_0 and T_1 into the accumulator
                // pair (b0, b0 + 1): u = A_lo T_0, v = A_hi T_1.  The transformed values are y[0..127] = u + v and
                // y[128..255] = u - v (H_256 = [[H, H], [H, -H]]).  Tiles alternate between the two accumulator pairs; pair
                // pr is drained by groups 2 pr (the u + v half) and 2 pr + 1 (the u - v half), so every barrier is used by
                // the same warps each time and its phases alternate for them.
                const int b0 = 2 * (grp >> 1), hh = grp & 1;
                const uint32_t ph = (it >> 1) & 1;                               // this pair's (it / 2)-th use
                uint32_t rw[8];
                if (mode_draws(MODE)) sr_draws32_block(p.keys, vw.stream_tag, blk, rw);
                if (!wait(&acc_full[b0], ph) || !wait(&acc_full[b0 + 1], ph)) break;
                tc_fence_after_sync();
                const uint32_t ta = tmem_base + ((uint32_t)(q * 32) << 16) + b0 * kTile;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t nx[8], packed[4], sb = 0;
                    float y[32];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {                           // sixteen columns of u and of v at a time
                        uint32_t u[16], v[16];
                        tmem_ld_32x32b_x16(ta + 32 * j + 16 * c, u);
                        tmem_ld_32x32b_x16(ta + kTile + 32 * j + 16 * c, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            y[16 * c + i] = hh == 0 ? __uint_as_float(u[i]) + __uint_as_float(v[i]) : __uint_as_float(u[i]) - __uint_as_float(v[i]);
                    }
                    if (j == 3) {                                           // this group is done with both accumulators
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) { mbar_arrive(&acc_empty[b0]); mbar_arrive(&acc_empty[b0 + 1]); }
                    }
                    if (mode_draws(MODE) && j < 3) sr_draws32_block(p.keys, vw.stream_tag, blk + (j + 1), nx);   // beside the rounding of this block
                    if (MODE == kModeDump) {
                        if (live) {
                            float4* dst = reinterpret_cast<float4*>(y_dst + 32 * j);
#pragma unroll
                            for (int i = 0; i < 8; ++i) dst[i] = make_float4(y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
                        }
                    } else {
                        quantize_block32_rw<mode_rounding(MODE)>(y, rw, packed, sb, p.pipe);
                        if (live) store_codes(code_dst, j, packed, kept, p.wide_stores);
                        sb_all |= sb << (8 * j);
                    }
                    if (mode_draws(MODE) && j < 3) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) rw[i] = nx[i];
                    }
                }
                if (MODE != kModeDump && live) *reinterpret_cast<uint32_t*>(scale_dst) = sb_all;
            } else {
                const int b = it % kAccBufs;
                if (!wait(&acc_full[b], (it / kAccBufs) & 1)) break;
                tc_fence_after_sync();
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + b * kTile + 32 * part;
#pragma unroll
                for (int j = 0; j < kBlocksPerThread; ++j) {
                    uint32_t raw[32], rw[8], packed[4], sb = 0;
                    float y[32];
                    tmem_ld_32x32b_x32(taddr + 32 * j, raw);
                    if (mode_draws(MODE)) {                         // while the load is under way
                        sr_draws32_block(p.keys, vw.stream_tag, blk + j, rw);
                        tmem_ld_wait_after(rw);
                    } else {
                        tmem_ld_wait();
                    }
                    if (j == kBlocksPerThread - 1) {                // the accumulator is free once it has been read
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&acc_empty[b]);
                    }
#pragma unroll
                    for (int i = 0; i < 32; ++i) y[i] = __uint_as_float(raw[i]);
                    if (cg != 1.0f) {                               // g = 32, 128: 1/sqrt(g) is not a power of two (for g = 64 it is folded into T)
#pragma unroll
                        for (int i = 0; i < 32; i += 2) mul2_rn(y[i], y[i + 1], cg, y[i], y[i + 1]);
                    }
                    if (mode_keeps_y(MODE) && live) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) st_global_32B(y_dst + 32 * j + 8 * i, reinterpret_cast<const uint32_t*>(y) + 8 * i, p.wide_stores);
                    }
                    if constexpr (mode_int4(MODE)) {
                        uint32_t bytes[8];
                        quantize_block32_int4<MODE == kModeInt4SR>(y, rw, bytes, sb);
                        if (live) st_global_32B(code_dst + 32 * j, bytes, p.wide_stores);
                        sb_all |= sb << (8 * j);
                    } else if constexpr (MODE != kModeDump) {
                        quantize_block32_rw<mode_rounding(MODE)>(y, rw, packed, sb, p.pipe);
                        if (live) store_codes(code_dst, j, packed, kept, p.wide_stores);
                        sb_all |= sb << (8 * j);
                    }
                }
                if (MODE != kModeDump && (live || mode_int4(MODE))) {   // (MXINT4: rows that only fill the last tile are zero)
                    if (mode_int4(MODE) && !live) sb_all = 0;
                    // this thread's two or four consecutive bytes, in either scale layout
                    if (LITE || HALVES) *reinterpret_cast<uint16_t*>(scale_dst) = (uint16_t)sb_all;
                    else *reinterpret_cast<uint32_t*>(scale_dst) = sb_all;
                }
            }
        }
        if (!ok && lane == 0) *abort_flag = 1;
    }

    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, Cfg::kTmemCols);
    }
}

template <int MODE, int KW>
__global__ void __launch_bounds__(QCfg<false, KW>::kThreads, 1)
quantize_tc_kernel(const __grid_constant__ QMaps maps, const __grid_constant__ QParams p) {
    quantize_tc_body<MODE, KW, false, false>(maps, p);
}

// Half tiles to the epilogue groups (see quantise_by_halves), g <= 128.
template <int MODE>
__global__ void __launch_bounds__(QCfg<false, 1>::kThreads, 1)
quantize_tc_halves_kernel(const __grid_constant__ QMaps maps, const __grid_constant__ QParams p) {
    quantize_tc_body<MODE, 1, false, false, true>(maps, p);
}

// Both views of one tensor from one read of it (Algorithm 3 lines 3 and 5 use the same dL/dy), g <= 128.
template <int MODE>
__global__ void __launch_bounds__(QCfg<false, 1>::kThreads, 1)
quantize_tc_dual_kernel(const __grid_constant__ QMaps maps, const __grid_constant__ QParams p) {
    quantize_tc_body<MODE, 1, false, true>(maps, p);
}

// The small-footprint build (see QCfg), g <= 128.
using LiteQCfg = QCfg<true, 1>;
template <int MODE>
__global__ void __maxnreg__(LiteQCfg::kLaunchRegs)
quantize_tc_lite_kernel(const __grid_constant__ QMaps maps, const __grid_constant__ QParams p) {
    quantize_tc_body<MODE, 1, true, false>(maps, p);
}

}  // namespace

bool quant_tc_eligible(const QuantArgs& a) {
    const int64_t K = a.reduce_dim == 1 ? a.cols : a.rows;
    const int64_t R = a.reduce_dim == 1 ? a.rows : a.cols;
    const int64_t tiles = ((R + kTile - 1) / kTile) * (K / kTile);          // tile indices are 32-bit in the kernel
    // below 2^36 elements the index of a block's two Philox calls fits the low counter word
    return (a.g == 32 || a.g == 64 || a.g == 128 || a.g == 256) && K % kTile == 0 && tiles < (int64_t(1) << 28) && a.has_tmap &&
           R * K < (int64_t(1) << 36);
}

cudaError_t fetch_quant_tc_status(unsigned int* word) { return device_status_fetch(word); }

template <bool LITE, int KW>
static cudaError_t quant_kernel_init(const void* k) {
    using Cfg = QCfg<LITE, KW>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem);
    if (e != cudaSuccess) return e;
    // all of the SM's configurable memory as shared memory (see gemm_pair.cu: kernels share an SM only under one carve-out)
    e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, k);
    if (e != cudaSuccess) return e;
    // registers the CTA holds at launch must cover the limits the warp groups set for themselves
    if (fa.numRegs * Cfg::kThreads < 128 * Cfg::kRegsLight + (Cfg::kThreads - 128) * Cfg::kRegsEpi) return cudaErrorLaunchOutOfResources;
    return cudaSuccess;
}

cudaError_t quant_tc_init() {
    const void* kernels[10] = {(const void*)quantize_tc_kernel<kModeSR, 1>, (const void*)quantize_tc_kernel<kModeRN, 1>,
                               (const void*)quantize_tc_kernel<kModeDump, 1>, (const void*)quantize_tc_kernel<kModeSR16, 1>,
                               (const void*)quantize_tc_kernel<kModeInt4SR, 1>, (const void*)quantize_tc_kernel<kModeInt4RN, 1>,
                               (const void*)quantize_tc_kernel<kModeSR, 2>, (const void*)quantize_tc_kernel<kModeRN, 2>,
                               (const void*)quantize_tc_kernel<kModeDump, 2>, (const void*)quantize_tc_kernel<kModeSR16, 2>};
    for (int i = 0; i < 10; ++i) {
        const cudaError_t e = i < 6 ? quant_kernel_init<false, 1>(kernels[i]) : quant_kernel_init<false, 2>(kernels[i]);
        if (e != cudaSuccess) return e;
    }
    const void* halves[2] = {(const void*)quantize_tc_halves_kernel<kModeSR>, (const void*)quantize_tc_halves_kernel<kModeSR16>};
    for (const void* k : halves) {
        const cudaError_t e = quant_kernel_init<false, 1>(k);
        if (e != cudaSuccess) return e;
    }
    const void* dual[3] = {(const void*)quantize_tc_dual_kernel<kModeSR>, (const void*)quantize_tc_dual_kernel<kModeRN>,
                           (const void*)quantize_tc_dual_kernel<kModeSR16>};
    for (const void* k : dual) {
        const cudaError_t e = quant_kernel_init<false, 1>(k);
        if (e != cudaSuccess) return e;
    }
    const void* lite[3] = {(const void*)quantize_tc_lite_kernel<kModeSR>, (const void*)quantize_tc_lite_kernel<kModeRN>,
                           (const void*)quantize_tc_lite_kernel<kModeSR16>};
    for (const void* k : lite) {
        const cudaError_t e = quant_kernel_init<true, 1>(k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Launches that give no CTA more than one tile: the groups take half of it each, where a tile otherwise waits for one group's four
// blocks in a row.  256 x 512 x 512, operands 4.57 -> 4.23 us (SR), 4.35 -> 4.08 (SR16), 3.73 -> 3.80 (nearest rounding, whose blocks are short: not
// there); whole calls with SR 10.1 -> 9.75.  Single views of K = 128, whole tiles / halves in us a launch: SR 16 tiles 4.13 / 3.70, 100 tiles 4.59 / 3.89,
// 148 tiles 4.95 / 4.23; SR16 3.87 / 3.44, 4.15 / 3.68, 4.53 / 4.00.  The line is the mechanism's, short of where the two cross: with two or three tiles to a CTA the
// halves still gain (296 tiles SR 5.45 / 5.31, SR16 5.28 / 4.95; 440 tiles 6.03 / 5.80, 5.64 / 5.35), with eleven a group's own tile hides the others' and
// they cost: 8192 x 1024 x 1024 14.7 / 15.5 (SR), 16384 x 4096 x 4096 96.4 / 101.3.
static bool quantise_by_halves(uint32_t tiles, int sms, int g, int rounding) { return tiles <= (uint32_t)sms && g != 256 && rounding != 1; }

// Quantise n (1..kQuantMaxViews) eligible operand views that share g, seed, rounding and scale layout in one launch.
cudaError_t launch_quantize_tc_group(const QuantArgs* a, int n, bool dump_y, cudaStream_t stream, bool lite, bool dual, float* col_sums) {
    if (n < 1 || n > kQuantMaxViews) return cudaErrorInvalidValue;
    // dual: a[0] and a[1] are the row-wise and the transposed view of one tensor, whose tiles are then loaded once for both
    if (dual && (n != 2 || lite || dump_y || a[0].g == 256 || a[0].custom_t != nullptr || a[0].x != a[1].x || a[0].rows != a[1].rows ||
                 a[0].cols != a[1].cols || a[0].ld != a[1].ld || a[0].reduce_dim != 1 || a[1].reduce_dim != 0 || a[0].rows % kTile != 0))
        return cudaErrorInvalidValue;
    if (a[0].mxint4 && (n != 1 || dual || lite || dump_y || a[0].g == 256 || a[0].custom_t != nullptr || a[0].y_out == nullptr)) return cudaErrorInvalidValue;
    if (lite && (dump_y || a[0].g == 256 || a[0].custom_t != nullptr)) return cudaErrorInvalidValue;   // the small build: RHT with g <= 128, quantising
    QParams p;
    QMaps maps;
    uint32_t tiles = 0;
    for (int v = 0; v < n; ++v) {
        QView& w = p.view[v];
        w.R = (uint32_t)(a[v].reduce_dim == 1 ? a[v].rows : a[v].cols);
        w.k_blocks = (uint32_t)((a[v].reduce_dim == 1 ? a[v].cols : a[v].rows) / 32);
        w.r_tiles = (w.R + kTile - 1) / kTile;
        w.k_tiles = w.k_blocks / (a[v].g == 256 ? 8u : 4u);                    // g = 256: a tile spans one 256-chunk
        w.tile_begin = tiles;
        w.n_tiles = w.r_tiles * w.k_tiles;
        tiles += w.n_tiles;
        w.reduce_dim = a[v].reduce_dim;
        w.stream_tag = a[v].stream_tag;
        w.codes = a[v].codes; w.scales = a[v].scales; w.y_out = a[v].y_out;
        maps.x[v] = a[v].tmap_x;
    }
    for (int v = n; v < kQuantMaxViews; ++v) { p.view[v] = p.view[0]; p.view[v].tile_begin = 0xFFFFFFFFu; maps.x[v] = maps.x[0]; }
    p.n_views = n;
    p.n_tiles = tiles;
    p.x_passes = quant_input_leaves_l2(a, n);
    p.g = a[0].g; p.sf_native = a[0].sf_native; p.seed = a[0].seed;
    uintptr_t stores = reinterpret_cast<uintptr_t>(a[0].y_out);
    for (int v = 0; v < n; ++v) stores |= reinterpret_cast<uintptr_t>(a[v].codes);
    p.wide_stores = (stores & 31u) == 0;
    p.custom_t = static_cast<const uint16_t*>(a[0].custom_t);
    if (p.custom_t != nullptr && p.g == 256) return cudaErrorInvalidValue;
    // column sums: of view 0's tensor, read row-wise in whole 128-row bands
    if (col_sums != nullptr && (lite || dump_y || a[0].g == 256 || a[0].mxint4 || a[0].reduce_dim != 1 || a[0].rows % kTile != 0)) return cudaErrorInvalidValue;
    p.col_sums = col_sums;
    p.pipe = make_pipe_consts();
    {   // Philox key schedule: key_i = key_0 + i * (0x9E3779B9, 0xBB67AE85)
        uint32_t k0 = (uint32_t)p.seed, k1 = (uint32_t)(p.seed >> 32);
        for (int i = 0; i < 10; ++i) {
            p.keys.k0[i] = k0; p.keys.k1[i] = k1;
            k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
        }
    }
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const uint32_t units = dual ? tiles / 2 : tiles;       // loads: in a dual launch the two views' tiles pair up
    const unsigned grid = units < (uint32_t)sms ? units : (unsigned)sms;
    for (int v = 0; v < kQuantMaxViews; ++v) {
        QView& w = p.view[v];
        w.lg_band = 0;         // bands of four tiles along the reduce dimension where it runs across the walk
        const uint32_t across = w.reduce_dim == 1 ? w.r_tiles : w.k_tiles;
        if (dual || w.reduce_dim == 0) while (w.lg_band < 2 && (across >> w.lg_band) % 2 == 0) ++w.lg_band;
        w.minor_count = (w.reduce_dim == 1 ? w.k_tiles : w.r_tiles) << w.lg_band;
        if (dual) w.n_tiles = units;
    }
    const bool wide = p.g == 256, mxint4 = a[0].mxint4;
    void (*kernel)(QMaps, QParams);
    if (dual) kernel = a[0].rounding == 0 ? quantize_tc_dual_kernel<kModeSR> : a[0].rounding == 2 ? quantize_tc_dual_kernel<kModeSR16> : quantize_tc_dual_kernel<kModeRN>;
    else if (lite) kernel = a[0].rounding == 0 ? quantize_tc_lite_kernel<kModeSR> : a[0].rounding == 2 ? quantize_tc_lite_kernel<kModeSR16> : quantize_tc_lite_kernel<kModeRN>;
    else if (mxint4) kernel = a[0].rounding == 0 ? quantize_tc_kernel<kModeInt4SR, 1> : quantize_tc_kernel<kModeInt4RN, 1>;
    else if (dump_y) kernel = wide ? quantize_tc_kernel<kModeDump, 2> : quantize_tc_kernel<kModeDump, 1>;
    else if (quantise_by_halves(tiles, sms, p.g, a[0].rounding)) kernel = a[0].rounding == 0 ? quantize_tc_halves_kernel<kModeSR> : quantize_tc_halves_kernel<kModeSR16>;
    else if (a[0].rounding == 0) kernel = wide ? quantize_tc_kernel<kModeSR, 2> : quantize_tc_kernel<kModeSR, 1>;
    else if (a[0].rounding == 2) kernel = wide ? quantize_tc_kernel<kModeSR16, 2> : quantize_tc_kernel<kModeSR16, 1>;
    else kernel = wide ? quantize_tc_kernel<kModeRN, 2> : quantize_tc_kernel<kModeRN, 1>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.stream = stream;
    cfg.blockDim = dim3(lite ? LiteQCfg::kThreads : wide ? QCfg<false, 2>::kThreads : QCfg<false, 1>::kThreads);
    cfg.dynamicSmemBytes = lite ? LiteQCfg::kSmem : wide ? QCfg<false, 2>::kSmem : QCfg<false, 1>::kSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return launch_result(cudaLaunchKernelEx(&cfg, kernel, maps, p));
}

cudaError_t launch_quantize_tc(const QuantArgs& a, bool dump_y, cudaStream_t stream) {
    return launch_quantize_tc_group(&a, 1, dump_y, stream, false, false, nullptr);
}

}  // namespace mx
