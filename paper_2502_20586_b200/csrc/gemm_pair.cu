// Block-scaled FP4 GEMM (and 8-bit ones), CTA-pair variant (tcgen05 cta_group::2): two CTAs of a 2-CTA cluster share one
// 256 x 256 output tile.  Each CTA loads 128 rows of A and only HALF of the B tile (128 of its 256 rows); the pair MMA reads
// both halves, so per MMA a tensor core pulls 4 KB + 4 KB from its own shared memory instead of 4 KB + 8 KB.  The
// 1-CTA kernel (gemm.cu) is bound by exactly that operand traffic.  Each CTA keeps the accumulator of its own 128
// rows (all 256 columns) in its TMEM.
//
// Shared memory (all 227 KB): six operand stages of 32 KB, a six-slot scale ring of 3 KB, 16 KB of epilogue staging.
// TMEM: 256 accumulator columns + six scale slots of 24 columns.
//
// Roles per CTA (12 warps in three warp groups), all waits bounded as in gemm.cu:
//   warp 0       TMA producer: own A rows, own half of B (completion counted on the LEADER's barrier);
//   warp 3       scale loader: own A-row scale tiles and the scale tiles of all 256 B rows, tiled copies into ring slot
//                s of stage s, counted on the same leader barrier as the operands, so the issuer waits once per step;
//   warps 1, 2   MMA issuers, leader CTA only, taking the K-steps in turn under a baton, one elected lane each.  Per
//                step: six tcgen05.cp carry the step's scale tiles from the ring into TMEM slot s of BOTH CTAs (the copy
//                itself replicates them to the four lane quadrants and reads shared memory once; they are issued while
//                the other warp still issues its MMAs), then four K = 64 pair-MMAs; ONE multicast tcgen05.commit per
//                step frees operand stage, ring slot and TMEM scale slot in both CTAs;
//   warps 4..11  epilogue of the CTA's own 128 x 256 half tile, a warp 32 rows x 128 columns: accumulator -> registers
//                (all 128 columns in flight) -> hand the accumulator back -> scale, convert -> swizzled staging -> TMA
//                stores (or reduce-adds when accumulating).
// A-row scales are per CTA; every CTA needs the scales of all 256 B rows.
//
// What bounds it, in cycles of the SM: the tensor pipe in the steady state (a K-step of a pair tile 515 - 550; the same MMAs on operands that
// stay in shared memory 512.8, fp4_ceiling.cu: 8.1 PFLOP/s in a burst, 7.1 sustained), and per tile a hand-over in which the pipe stands still,
// since TMEM has no room for a second 256-column accumulator beside the scale slots: 1500 - 2300 with bf16 output (1.0 - 1.5 us at 1.55 GHz), 3300
// with fp32 (2.1 us at 1.6), 660 where the tile is not stored: the stores and the next tile's loads share the way out of the SM.  The clock is what the
// board's power leaves: 1.44 - 1.6 GHz in the first launches of a run, 1.18 - 1.33 in a long one.  Two things got it there:
//   - issue.  From a lane-0 branch the descriptors of every MMA, scale copy and commit go to uniform registers one by one, and
//     two issuing threads did not keep up with the pipe.  With warp-uniform control flow and an elected lane the issuers wait
//     for operands instead.  Back to back, before -> now: 16384 x 4096 x 16384 382 -> 349 us (alone 372 -> 333: 6.6 PFLOP/s),
//     16384 x 4096 x 4096 105 -> 97, 1024 x 1024 x 8192 16.2 -> 12.5.  One issuing warp without the baton: 376, 103, 16.5;
//   - the hand-over.  Eight warps take the accumulator out unconverted, in place of four that had to convert the first
//     half before reading the second, and for fp32 stored every 32 columns before reading the next: 16384 x 8192 x 2048
//     bf16 125 -> 115 us, fp32 197 -> 143 (537 MB written, but memory is not the bound: a fill of that buffer takes 74 us, the
//     same product with K = 128 84, with K = 2048 135 beside them.  Per pair tile the fp32 stores take about 3.0 us and the MMAs
//     2.7, and they overlap in part only; a second staging buffer, stores without the evict-first hint, and 32-byte stores
//     straight from the registers gained nothing).
// A 256 x 384 pair tile (two N = 192 MMAs from one A) was slower everywhere: 391 -> 414 us at K = 16384, 106 -> 115 at 4096
// (before the issue change).
//
// The 8-bit products (FP8 forward pass, MXINT4; enum Kind) run on the same roles: a one-CTA kernel of 128 x 256 tiles with
// one accumulator and stores from registers served them before.  E4M3 16384 x 4096 x 4096: 221 -> 168 us (3.3 PFLOP/s,
// twice the measured bf16 rate), 8192 x 3072 x 1024 50 -> 23, 16 x 4096 x 4096 16.5 -> 11.4; MXINT4
// 16384 x 4096 x 4096 245 -> 178, 1024 x 1024 x 8192 34 -> 20.  Since then the issue above and the split products: 168 - 172, 20.3, 10.0 and 167, 13.2.
// The one-CTA kernel still serves few rows and many columns (gemm_f8.cu).
#include <cuda_bf16.h>

#include <cstdlib>

#include "kernels.h"
#include "ptx.cuh"

namespace mx {
namespace {

constexpr int PM = 256;                                     // rows of a pair tile
constexpr uint32_t kAB = 128 * kGemmBKBytes;                // 16 KB: 128 A rows x 128 B
constexpr uint32_t kSfTile = 512;                           // scales of 128 rows x 128 elements
constexpr uint32_t kEpiBuf = 2048;                          // epilogue staging: 32 rows x 64 B, one buffer per epilogue warp (8 warps)
constexpr uint32_t kEpiB = 8 * kEpiBuf;
constexpr uint32_t kBarB = 256;
constexpr int kThreadsP = 12 * 32;

// Four builds of the kernel.  PN = 256 (256 x 256 pair tile): six operand stages (all 227 KB of shared memory), one
// 512-column TMEM allocation, every register of the SM.  PN = 128 (256 x 128): eight stages, and TMEM room for two
// accumulators, so that a tile's MMAs run while the tile before is taken out; see gemm_pair_tile_n() for when it is the better
// one, and for its SPLIT form, of 8-bit products only, split_pays().  LITE (PN = 256) leaves room for a second, independent kernel on the same SM (the tensor-core quantiser's small
// build, quantize_tc.cu, which quantises the OTHER product's operands meanwhile): four stages, TMEM taken as 256 + 128
// columns, 104 registers per thread at launch.
// Operand kinds: E2M1 with one UE8M0 scale per 32 elements (the method's GEMM); E4M3 with one scale per tensor (FP8 forward
// pass, Section 4.1); E4M3 containers of the integers -7..7 with one UE8M0 scale per 32 elements (MXINT4, Section 3).  A
// K-step is 128 bytes of every row and four MMAs in all of them.  Without scale slots in TMEM the plain E4M3 build has two
// 256-column accumulators.
enum Kind { kMxf4, kF8, kMxf8 };

template <Kind KIND, bool LITE, int PN>
struct PairCfg {
    static constexpr int kSfTiles = KIND == kMxf4 ? 2 : KIND == kMxf8 ? 1 : 0;   // scale tiles of 128 rows in a K-step
    static constexpr int kAccBufs = PN == 128 || KIND == kF8 ? 2 : 1;
    static constexpr int kWarpCols = kAccBufs == 2 ? PN : PN / 2;                // accumulator columns an epilogue warp takes
    static constexpr int kStages = LITE ? 4 : PN == 128 ? 8 : 6;
    static constexpr uint32_t kBB = PN / 2 * kGemmBKBytes;  // half of the B tile
    static constexpr uint32_t kStageB = kAB + kBB;
    static constexpr uint32_t kSfaB = kSfTiles * kSfTile;   // own 128 A rows
    static constexpr uint32_t kSfSlotB = kSfaB + PN / 128 * kSfaB;               // and all PN B rows
    static constexpr uint32_t kSfCols = kSfSlotB / 128;     // TMEM columns of a slot: 4 per 512-byte tile
    // scale ring: shared-memory slot i feeds TMEM slot i; same ring index as the operand stages so ONE commit frees both
    // The dynamic shared-memory window is at least 256-byte aligned, so rounding its base up to 1024 costs at most 768 bytes.
    static constexpr uint32_t kSmem = kStages * (kStageB + kSfSlotB) + kEpiB + kBarB + 768;
    // Register hand-over (setmaxnreg) between warp group 0 and the two epilogue groups; an increase can only
    // draw on what the CTA holds at launch (threads x registers per thread), which gemm_pair_init checks: an increase
    // that cannot be met waits forever.
    static constexpr int kRegsLight = LITE ? 56 : 72, kRegsEpi = LITE ? 128 : 216;
    static constexpr int kBatch = LITE ? 2 : 4;             // 32-column accumulator loads an epilogue warp keeps in flight
    static constexpr int kLaunchRegs = LITE ? 104 : 168;    // registers per thread the CTA is given at launch
    static_assert(!LITE || (KIND == kMxf4 && PN == 256), "the small build has one 256-column accumulator");
    static_assert(kSmem <= 232448, "over the 227 KB shared-memory limit");
    static_assert((2 * kStages + 2 + 2 * kAccBufs) * 8 + 16 <= kBarB, "barriers");
    static_assert(kStages * kSfCols <= (LITE ? 128 : 512 - kAccBufs * PN), "scale slots do not fit their TMEM allocation");
    static_assert(kThreadsP * kLaunchRegs >= 128 * (kRegsLight + 2 * kRegsEpi), "warp groups ask for more registers than the CTA holds");
};

struct ProblemP {                                           // one product of a launch
    int64_t M, N;
    int nkc, num_kt;                                        // 128-element scale tiles along K; pipeline steps
    int m_tiles, n_tiles;                                   // in pair tiles
    int group_m;                                            // rasterisation: this many pair-tile rows share the B tiles in L2 (fill_problem)
    float alpha;
    const float *scale_a, *scale_b;                         // kF8: alpha is 1 / (*scale_a * *scale_b)
    int out_fp32;
    int accumulate;                                         // fp32 output only: C += instead of C =
};

// A launch runs one product, or two that do not depend on each other (the two GEMMs of a backward call) with the one of
// the longer K first.  Every pair knows its own tiles without asking: the first product's n0 tiles go round-robin; the
// n0 mod P = `rest` pairs that got one more of them sit out while the others take `early` tiles of the second product
// each; what is left of that goes round-robin over all, the others first.
struct ParamsP {
    ProblemP prob[2];
    int n0, n1;                                             // tiles of the two products
    int rest, early;
    BandSums bias;                                          // partial == nullptr: none
};
struct MapsP {
    CUtensorMap a[2], b[2], sfa[2], sfb[2], c[2];
};

__device__ __forceinline__ void tile_coords_p(int t, int m_tiles, int n_tiles, int kGroupMP, int& mt, int& nt) {
    const int per_group = kGroupMP * n_tiles;
    const int grp = t / per_group;
    const int first_m = grp * kGroupMP;
    const int gm = min(kGroupMP, m_tiles - first_m);
    const int r = t - grp * per_group;
    mt = first_m + r % gm;
    nt = r / gm;
}

// The tiles of one pair (see ParamsP).
struct TileWalk {
    int pair, pairs, n_first, n_early, order;               // order: this pair's place among the takers of the second product's late tiles
    uint32_t count;
    __device__ __forceinline__ TileWalk(const ParamsP& p, int pair_, int pairs_) : pair(pair_), pairs(pairs_) {
        const int others = pairs - p.rest;
        const bool extra = pair < p.rest;
        n_first = p.n0 / pairs + (extra ? 1 : 0);
        n_early = extra ? 0 : p.early;
        order = extra ? pair + others : pair - p.rest;
        const int late = p.n1 - p.early * others;
        count = (uint32_t)(n_first + n_early + (late > order ? (late - order + pairs - 1) / pairs : 0));
    }
    // tile tl (< count) of this pair: the product it belongs to and its coordinates there
    __device__ __forceinline__ int locate(const ParamsP& p, uint32_t tl, int& mt, int& nt) const {
        const int x = (int)tl - n_first, others = pairs - p.rest;
        const int which = x < 0 ? 0 : 1;
        const int t = x < 0 ? (int)tl * pairs + pair : x < n_early ? x * others + order : p.early * others + (x - n_early) * pairs + order;
        const ProblemP& q = p.prob[which];
        tile_coords_p(t, q.m_tiles, q.n_tiles, q.group_m, mt, nt);
        return which;
    }
};

// Pair MMAs on 8-bit operands, K = 32: E4M3 (formats in the instruction descriptor), and the same with one UE8M0 scale per
// row and the MMA's 32 elements.
__device__ __forceinline__ void tc_mma_f8_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_mma_mxf8_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                 uint32_t sfa_tmem, uint32_t sfb_tmem, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)
        : "memory");
}

// SPLIT: two pairs of a 4-CTA cluster share ONE output tile, each with half of its K-steps (see split_pays and the epilogue).
template <Kind KIND, bool LITE, int PN, bool SPLIT = false>
__device__ __forceinline__ void gemm_pair_body(const MapsP& maps, const ParamsP& p) {
    using Cfg = PairCfg<KIND, LITE, PN>;
    static_assert(!SPLIT || (PN == 128 && KIND != kMxf4), "split products: 8-bit kinds, 128-wide tiles");
    constexpr int kStagesP = Cfg::kStages, kAccBufs = Cfg::kAccBufs;
    constexpr uint32_t kStageB = Cfg::kStageB, kSfSlotB = Cfg::kSfSlotB;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sf_ring = smem + kStagesP * kStageB;
    uint8_t* epi_ring = sf_ring + kStagesP * kSfSlotB;
    uint64_t* bars = reinterpret_cast<uint64_t*>(epi_ring + kEpiB);
    uint64_t* full_bar = bars;                              // [kStagesP] leader: operands and scale tiles of both CTAs landed
    uint64_t* empty_bar = full_bar + kStagesP;              // [kStagesP] per CTA: stage and scale slot free (pair commit)
    uint64_t* turn = empty_bar + kStagesP;                  // [2] leader: baton between the two MMA issuers
    uint64_t* tmem_full = turn + 2;                         // [kAccBufs] per CTA: accumulator complete (pair commit)
    uint64_t* tmem_empty = tmem_full + kAccBufs;            // [kAccBufs] leader: both CTAs drained the accumulator
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tmem_empty + kAccBufs);   // [2] base columns of the TMEM allocation(s)
    volatile uint32_t* abort_flag = tmem_slot + 2;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // (warp-uniform, and known to be)
    const uint32_t rank = SPLIT ? cluster_ctarank() & 1u : cluster_ctarank();    // in the pair: 0 = leader
    const uint32_t half_k = SPLIT ? cluster_ctarank() >> 1 : 0u;                 // this pair's half of the K-steps
    constexpr int kLgCtas = SPLIT ? 2 : 1;
    const TileWalk walk(p, (int)(blockIdx.x >> kLgCtas), (int)(gridDim.x >> kLgCtas));
    // K-steps of a tile that are this pair's: all of them, or the first or second half
    auto first_step = [&](int num_kt) { return SPLIT && half_k != 0 ? (num_kt + 1) >> 1 : 0; };
    auto end_step = [&](int num_kt) { return SPLIT && half_k == 0 ? (num_kt + 1) >> 1 : num_kt; };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStagesP; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&turn[0], 1); mbar_init(&turn[1], 1);
        for (int b = 0; b < kAccBufs; ++b) { mbar_init(&tmem_full[b], 1); mbar_init(&tmem_empty[b], 16 / kAccBufs); }
        *abort_flag = 0;
        mbar_fence_init();
        for (int i = 0; i < (p.n1 > 0 ? 2 : 1); ++i) {
            prefetch_tensormap(&maps.a[i]);
            prefetch_tensormap(&maps.b[i]);
            if (KIND != kF8) {
                prefetch_tensormap(&maps.sfa[i]);
                prefetch_tensormap(&maps.sfb[i]);
            }
            prefetch_tensormap(&maps.c[i]);
        }
    }
    if (warp == 1) {
        if (LITE) {                                         // accumulator and scale slots as two allocations: 128 columns stay free
            tmem_alloc_pair(&tmem_slot[0], 256);
            tmem_alloc_pair(&tmem_slot[1], 128);
        } else {
            tmem_alloc_pair(&tmem_slot[0], 512);
        }
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();                                     // both CTAs' barriers exist before anyone signals across
    tc_fence_after_sync();
    const uint32_t tmem_acc = tmem_slot[0];                 // accumulator columns
    const uint32_t tmem_sf = LITE ? tmem_slot[1] : tmem_slot[0] + kAccBufs * PN;   // scale slots of kSfCols columns
    // Warp group 0 (producer, issuers, scale loader) needs few registers; the epilogue groups take them to hold 128 columns
    // of the accumulator each.
    // Each warp group (four warps) sets its register limit once, at the head of its own branch: all four warps must
    // execute the same setmaxnreg, and the limit must dominate the code that relies on it.
    pdl_launch_dependents();                                // the next kernel of the stream may set itself up behind this one
    pdl_wait();                                             // everything above overlapped the previous kernel's tail; its data is needed now

    if (warp < 4) {
    // ============================ warp group 0: producer, two MMA issuers, scale loader (few registers each)
    reg_dealloc<Cfg::kRegsLight>();
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        // The whole warp walks the loop and one elected lane issues, here and in the scale loader, as the MMA issuers do: from a lane-0 branch,
        // with divisions by the ring's size, a step's loads took 425 cycles of this thread, more than a 128-wide tile's MMAs (256), and the ring
        // filled as slowly at every start; now 240.  Before -> now: 1024 x 1024 x 8192 11.7 -> 11.2 us, 256 x 512 x 512 5.2 -> 5.0,
        // 16384 x 4096 x 4096 98 -> 96.5, 16384 x 8192 x 2048 111 -> 108.5 (bf16 output; with fp32 it did not move); backward 8192 x 1024 x 1024 29.1 -> 27.9.
        uint32_t s = 0, ph = 1;
        bool ok = true;
        for (uint32_t tl = 0; tl < walk.count && ok; ++tl) {
            int mt, nt;
            const int w = walk.locate(p, tl, mt, nt);
            const int end_kt = end_step(p.prob[w].num_kt);
            const CUtensorMap *map_a = &maps.a[w], *map_b = &maps.b[w];
            const int32_t a_row = (2 * mt + (int)rank) * 128, b_row = nt * PN + (int)rank * (PN / 2);   // this CTA's rows of A, half of B's
            for (int kt = first_step(p.prob[w].num_kt); kt < end_kt; ++kt) {
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(&empty_bar[s], ph, abort_flag)))) break;
                if (elect_one()) {
                    uint8_t* st = smem + s * kStageB;
                    if (rank == 0) mbar_expect_tx(&full_bar[s], 2 * (kStageB + kSfSlotB));   // operands and scales of both CTAs
                    tma_load_2d_pair(st, map_a, &full_bar[s], kt * kGemmBKBytes, a_row);
                    tma_load_2d_pair(st + kAB, map_b, &full_bar[s], kt * kGemmBKBytes, b_row);
                }
                __syncwarp();
                if (++s == (uint32_t)kStagesP) { s = 0; ph ^= 1; }
            }
        }
        if (!ok && lane == 0) *abort_flag = 1;
    } else if (warp == 1 || warp == 2) {
        // ------------------------------------------------------------------ MMA issuers (leader CTA only)
        // Two warps take the steps in turn (even steps warp 1, odd steps warp 2): while one issues its MMAs, the other has
        // already waited for its operands and copied its scales.  A baton (mbarrier turn[]) keeps the MMAs in step order,
        // so accumulation order is fixed.  The whole warp walks the loop (every wait ends for all lanes or none) and one
        // elected lane issues.
        if (rank == 0) {
            // instruction descriptor: K-major, N >> 3 at bit 17, M >> 4 at bit 24; A, B = E2M1 (1) or E4M3 (0) at bits 7 and 10;
            // scaled kinds: scale = UE8M0 (bit 23), scale byte ids at bits 4 (B) and 29 (A); plain: D = fp32 (bit 4)
            const uint32_t idesc0 = ((uint32_t)(PN >> 3) << 17) | ((uint32_t)(PM >> 4) << 24) |
                                    (KIND == kMxf4 ? (1u << 7) | (1u << 10) | (1u << 23) : KIND == kMxf8 ? 1u << 23 : 1u << 4);
            const uint32_t idesc1 = idesc0 | (2u << 29) | (2u << 4);          // scale bytes 2, 3 of the 32-bit column
            const uint64_t desc0 = make_smem_desc(smem_u32(smem), 16, 1024, 2);
            const uint32_t desc_hi = (uint32_t)(desc0 >> 32);
            const uint32_t a_lo0 = (uint32_t)desc0;
            const uint32_t me = warp == 1 ? 0u : 1u;
            uint32_t s = me % kStagesP, ph = 0, tile_i = 0, n = 0;
            auto steps_of = [&](uint32_t tile) {
                const int all = p.prob[(int)tile < walk.n_first ? 0 : 1].num_kt;
                return end_step(all) - first_step(all);
            };
            int kt = (int)me, num_kt = steps_of(0);
            while (tile_i < walk.count && kt >= num_kt) { kt -= num_kt; num_kt = steps_of(++tile_i); }
            bool ok = true;
            for (; tile_i < walk.count; ++n) {
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(&full_bar[s], ph, abort_flag)))) break;
                tc_fence_after_sync();
                const uint32_t a_lo = a_lo0 + s * (kStageB >> 4), b_lo = a_lo + (kAB >> 4);
                const uint32_t sfa_t = tmem_sf + s * Cfg::kSfCols, sfb_t = sfa_t + 4 * Cfg::kSfTiles;
                constexpr uint32_t kSfbChunk = PN / 32;      // TMEM columns of one 128-element chunk's B scales
                if (Cfg::kSfTiles != 0 && elect_one()) {
                    // the step's scales: shared memory -> TMEM of both CTAs, replicated to the four lane quadrants by the copy;
                    // issued while the other warp still issues its MMAs (a different TMEM slot), ordered before this
                    // lane's MMAs by program order
                    const uint32_t sf_s = smem_u32(sf_ring + s * kSfSlotB);
#pragma unroll
                    for (int c = 0; c < Cfg::kSfTiles; ++c) {
                        tc_cp_32x128b_warpx4_pair(sfa_t + 4 * c, make_smem_desc(sf_s + c * kSfTile, 0, 128, 0));
#pragma unroll
                        for (int j = 0; j < PN / 128; ++j)
                            tc_cp_32x128b_warpx4_pair(sfb_t + kSfbChunk * c + 4 * j,
                                                      make_smem_desc(sf_s + Cfg::kSfaB + (Cfg::kSfTiles * j + c) * kSfTile, 0, 128, 0));
                    }
                }
                if (!(ok = __all_sync(0xffffffffu, mbar_wait_spin(&turn[me], (n & 1) ^ me ^ 1, abort_flag)))) break;   // the step before mine is issued
                // The copies above did not need the accumulator.  Waited for under the baton: with one K-step per tile the
                // two threads alternate between tiles, and a thread that waited before its turn could see an earlier tile's
                // hand-back as its own (a phase parity only tells neighbouring phases apart).
                const uint32_t buf = tile_i % kAccBufs, acc = tmem_acc + buf * PN;
                if (kt == 0) {
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait_spin(&tmem_empty[buf], ((tile_i / kAccBufs) & 1) ^ 1, abort_flag)))) break;
                }
                tc_fence_after_sync();                       // the other warp's MMAs on this accumulator come before mine, in every step
                const uint32_t hi2 = 2u << 30;
                const bool last = kt == num_kt - 1;
                auto D = [&](uint32_t lo) { return ((uint64_t)desc_hi << 32) | lo; };
                // an odd number of 128-element chunks: the last step holds one only
                const bool two_chunks = KIND != kMxf4 || !(last && (p.prob[(int)tile_i < walk.n_first ? 0 : 1].nkc & 1) != 0);
                if (elect_one()) {
                    if constexpr (KIND == kMxf4) {
                        tc_mma_mxf4_pair(acc, D(a_lo), D(b_lo), idesc0, sfa_t, sfb_t, kt != 0 ? 1u : 0u);
                        tc_mma_mxf4_pair(acc, D(a_lo + 2), D(b_lo + 2), idesc1, sfa_t | hi2, sfb_t | hi2, 1u);
                        if (two_chunks) {
                            tc_mma_mxf4_pair(acc, D(a_lo + 4), D(b_lo + 4), idesc0, sfa_t + 4, sfb_t + kSfbChunk, 1u);
                            tc_mma_mxf4_pair(acc, D(a_lo + 6), D(b_lo + 6), idesc1, (sfa_t + 4) | hi2, (sfb_t + kSfbChunk) | hi2, 1u);
                        }
                    } else {
    #pragma unroll
                        for (uint32_t kb = 0; kb < 4; ++kb) {        // scale byte kb of the 32-bit column: K-block kb of the step
                            if (KIND == kF8) tc_mma_f8_pair(acc, D(a_lo + 2 * kb), D(b_lo + 2 * kb), idesc0, (uint32_t)kt | kb ? 1u : 0u);
                            else tc_mma_mxf8_pair(acc, D(a_lo + 2 * kb), D(b_lo + 2 * kb), idesc0 | (kb << 29) | (kb << 4), sfa_t | (kb << 30), sfb_t | (kb << 30),
                                                  (uint32_t)kt | kb ? 1u : 0u);
                        }
                    }
                    tc_fence_before_sync();
                    mbar_arrive(&turn[me ^ 1]);                                    // pass the baton
                    tc_commit_pair(&empty_bar[s], 2u * half_k);                    // frees the operand stage and the scale slot
                    if (last) tc_commit_pair(&tmem_full[buf], 2u * half_k);
                }
                __syncwarp();
                s += 2;
                if (s >= (uint32_t)kStagesP) { s -= kStagesP; ph ^= 1; }
                kt += 2;
                while (tile_i < walk.count && kt >= num_kt) { kt -= num_kt; num_kt = steps_of(++tile_i); }
            }
            if (!ok && lane == 0) *abort_flag = 1;
        } else if (KIND == kMxf4 && !LITE && p.bias.partial != nullptr) {
            // The second CTA of a pair issues nothing: its two warps add up the bands of dY's column sums (the quantiser launch
            // before this one made them), a thread per column, bands in order.  Bound by the latency of its loads, hidden by
            // the GEMM; as a kernel of its own behind it this took 4 to 5 us and a launch gap.
            const float* partial = p.bias.partial;
            const uint32_t m = (uint32_t)p.bias.m, end = m * (uint32_t)p.bias.bands;       // below 2^29: operands are below 2^36 elements
#pragma unroll 1
            for (uint32_t c = (blockIdx.x >> 1) * 64u + (uint32_t)(warp - 1) * 32u + (uint32_t)lane; c < m; c += (gridDim.x >> 1) * 64u) {
                float sum = p.bias.accumulate ? p.bias.db[c] : 0.f;
                uint32_t k = c;
#pragma unroll 1
                for (; k + 3u * m < end; k += 4u * m) {
                    const float v0 = partial[k], v1 = partial[k + m], v2 = partial[k + 2u * m], v3 = partial[k + 3u * m];
                    sum += v0; sum += v1; sum += v2; sum += v3;
                }
#pragma unroll 1
                for (; k < end; k += m) sum += partial[k];
                p.bias.db[c] = sum;
            }
        }
    } else {
        // ------------------------------------------------------------------ scale loader (both CTAs)
        // One box = the one or two 512-byte scale tiles of a 128-row tile for this K-step (box rows past the operand read zeros; a
        // box that runs over the end of an odd K reads the next row tile's first, which no MMA uses).
        if (KIND != kF8) {
            uint32_t s = 0, ph = 1;
            bool ok = true;
            for (uint32_t tl = 0; tl < walk.count && ok; ++tl) {
                int mt, nt;
                const int w = walk.locate(p, tl, mt, nt);
                const int end_kt = end_step(p.prob[w].num_kt), nkc = p.prob[w].nkc;
                const CUtensorMap *map_a = &maps.sfa[w], *map_b = &maps.sfb[w];
                const int32_t a_row = (2 * mt + (int)rank) * nkc, b_row = nt * (PN / 128) * nkc;
                for (int kt = first_step(p.prob[w].num_kt); kt < end_kt; ++kt) {
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(&empty_bar[s], ph, abort_flag)))) break;
                    if (elect_one()) {
                        uint8_t* dst = sf_ring + s * kSfSlotB;
                        tma_load_2d_pair(dst, map_a, &full_bar[s], 0, a_row + Cfg::kSfTiles * kt);
#pragma unroll
                        for (int j = 0; j < PN / 128; ++j)
                            tma_load_2d_pair(dst + Cfg::kSfaB * (1 + j), map_b, &full_bar[s], 0, b_row + j * nkc + Cfg::kSfTiles * kt);
                    }
                    __syncwarp();
                    if (++s == (uint32_t)kStagesP) { s = 0; ph ^= 1; }
                }
            }
            if (!ok && lane == 0) *abort_flag = 1;
        }
    }
    if (SPLIT) {                                            // the two barriers of the exchange below
        __syncwarp();
        cluster_sync_all();
        cluster_sync_all();
    }
    } else {
        // ------------------------------------------------------------------ epilogue (both CTAs, own 128 rows)
        reg_alloc<Cfg::kRegsEpi>();                                  // the epilogue groups take the registers the others gave up
        // A warp owns one TMEM lane quadrant.  One accumulator: the second group takes columns 128 .. 255 of every tile; two:
        // the groups take alternate tiles, each its own accumulator.
        const int q = warp & 3, half = (warp - 4) >> 2;
        uint8_t* stage = epi_ring + (warp - 4) * kEpiBuf;
        const uint64_t pol_c = l2_policy_evict_first();         // the output is not read again here: let the operands keep L2
        bool ok = true;
        // One staged block: 16 registers = 64 bytes of this lane's row, columns [col, col + 64 B), into this warp's buffer
        // (64-byte swizzle: the row-per-lane writes are conflict-free) and out by TMA.
        auto put = [&](const uint32_t (&w)[16], const CUtensorMap* map, bool add, int32_t col, int32_t row0, bool in_range) {
            if (lane == 0) bulk_wait_group_read<0>();           // the store before this one must have left the buffer
            __syncwarp();
            uint4* dst = reinterpret_cast<uint4*>(stage + lane * 64);
            const int sw = (lane >> 1) & 3;
#pragma unroll
            for (int j = 0; j < 4; ++j) dst[j ^ sw] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                if (in_range) {
                    if (add) tma_reduce_add_2d(map, stage, col, row0);
                    else tma_store_2d_hint(map, stage, col, row0, pol_c);
                }
                bulk_commit_group();
            }
        };
        if constexpr (SPLIT) {
            // One tile a cluster.  CTA r of either pair holds the same 128 rows x 128 columns, summed over half of K.  Pair 0
            // finishes the first 64 columns, pair 1 the others: each sends what the other finishes into that CTA's operand ring, which
            // is idle by then (first barrier: every MMA of all four CTAs is done), and adds what it gets (second barrier: it is
            // there).  One fp32 addition, the same whichever side makes it.  A warp takes 32 columns of its lane quadrant.
            int mt, nt;
            walk.locate(p, 0, mt, nt);
            const ProblemP& pr = p.prob[0];
            const CUtensorMap* map = &maps.c[0];
            ok = __all_sync(0xffffffffu, mbar_wait_spin(&tmem_full[0], 0, abort_flag));
            tc_fence_after_sync();
            cluster_sync_all();
            uint32_t mine[32];
            const uint32_t taddr = tmem_acc + ((uint32_t)(q * 32) << 16) + 32 * half;
            // 16 bytes of a row at a time, a warp's 32 rows side by side
            const uint32_t slot = smem_u32(smem) + (uint32_t)(half * 8 * 128 + q * 32 + lane) * 16u;
            if (ok) {
                uint32_t other[32];
                tmem_ld_32x32b_x32(taddr + 64 * (1 - half_k), other);
                tmem_ld_32x32b_x32(taddr + 64 * half_k, mine);
                tmem_ld_wait();
                const uint32_t dst = peer_smem(slot, (1 - half_k) * 2 + rank);
#pragma unroll
                for (int i = 0; i < 8; ++i) st_peer_16B(dst + i * 2048, other[4 * i], other[4 * i + 1], other[4 * i + 2], other[4 * i + 3]);
            }
            cluster_sync_all();
            if (ok) {
                const float alpha = KIND == kF8 ? 1.0f / (*pr.scale_a * *pr.scale_b) : pr.alpha;
                const int64_t row0 = (int64_t)mt * PM + (int64_t)rank * 128 + q * 32, col = (int64_t)nt * PN + 64 * half_k + 32 * half;
                float v[32];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 o = *reinterpret_cast<const float4*>(smem + (slot - smem_u32(smem)) + i * 2048);
                    v[4 * i] = (__uint_as_float(mine[4 * i]) + o.x) * alpha;
                    v[4 * i + 1] = (__uint_as_float(mine[4 * i + 1]) + o.y) * alpha;
                    v[4 * i + 2] = (__uint_as_float(mine[4 * i + 2]) + o.z) * alpha;
                    v[4 * i + 3] = (__uint_as_float(mine[4 * i + 3]) + o.w) * alpha;
                }
                const bool in_range = row0 < pr.M && col < pr.N;
                uint32_t o[16];
                if (pr.out_fp32) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(v[16 * h + j]);
                        put(o, map, pr.accumulate != 0, (int32_t)col + 16 * h, (int32_t)row0, in_range && col + 16 * h < pr.N);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
                        o[j] = *reinterpret_cast<const uint32_t*>(&h);
                    }
                    put(o, map, false, (int32_t)col, (int32_t)row0, in_range);
                }
            }
        } else if (KIND != kMxf4 && kAccBufs == 2 && walk.count == 1) {
            // One tile to this pair (8-bit builds): the groups share it, half of its columns each, instead of one taking it and the other nothing.
            // Whole E4M3 forward passes, tokens x out x in: 1000 x 4096 x 1024 17.4 -> 16.8 us, 2000 x 2048 x 1024 15.2 -> 14.7, 4096 x 1024 x 2048
            // 22.1 -> 21.6.  Code of its own: woven into the loop below it cost the other builds (backward 8192 x 1024 x 1024 27.9 -> 28.3).  Not the
            // MXFP4 builds: a backward call of 256 x 512 x 512 gained (9.75 -> 9.4), 8192 x 1024 x 1024 (28.65 -> 28.9) and 1024 x 1024 x 8192
            // (29.0 -> 30.2), where some pairs have one tile and others several, lost.
            int mt, nt;
            walk.locate(p, 0, mt, nt);
            const ProblemP& pr = p.prob[0];
            const CUtensorMap* map = &maps.c[0];
            ok = __all_sync(0xffffffffu, mbar_wait_spin(&tmem_full[0], 0, abort_flag));
            if (ok) {
                tc_fence_after_sync();
                constexpr int kChunks = PN / 64;                     // of 32 columns
                const int64_t row0 = (int64_t)mt * PM + (int64_t)rank * 128 + q * 32, col0 = (int64_t)nt * PN + half * (PN / 2);
                const float alpha = KIND == kF8 ? 1.0f / (*pr.scale_a * *pr.scale_b) : pr.alpha;
                uint32_t r[kChunks][32];
#pragma unroll
                for (int c = 0; c < kChunks; ++c) tmem_ld_32x32b_x32(tmem_acc + ((uint32_t)(q * 32) << 16) + half * (PN / 2) + c * 32, r[c]);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < kChunks; ++c) {
                    const int64_t col = col0 + c * 32;
                    const bool in_range = row0 < pr.M && col < pr.N;
                    uint32_t o[16];
                    if (pr.out_fp32) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(r[c][16 * h + j]) * alpha);
                            put(o, map, false, (int32_t)col + 16 * h, (int32_t)row0, in_range && col + 16 * h < pr.N);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[c][2 * j]) * alpha,
                                                                           __uint_as_float(r[c][2 * j + 1]) * alpha);
                            o[j] = *reinterpret_cast<const uint32_t*>(&h);
                        }
                        put(o, map, false, (int32_t)col, (int32_t)row0, in_range);
                    }
                }
            }
        } else
        for (uint32_t tl = kAccBufs == 2 ? half : 0; tl < walk.count; tl += kAccBufs) {
            int mt, nt;
            const int w = walk.locate(p, tl, mt, nt);
            const ProblemP& pr = p.prob[w];
            const CUtensorMap* map = &maps.c[w];
            const uint32_t buf = kAccBufs == 2 ? half : 0;
            ok = __all_sync(0xffffffffu, mbar_wait_spin(&tmem_full[buf], (tl / kAccBufs) & 1, abort_flag));
            if (!ok) break;
            tc_fence_after_sync();
            const int64_t row0 = (int64_t)mt * PM + (int64_t)rank * 128 + q * 32;
            const uint32_t taddr = tmem_acc + ((uint32_t)(q * 32) << 16) + half * Cfg::kWarpCols;   // (two accumulators: its own, kWarpCols = PN)
            constexpr int kBatches = Cfg::kWarpCols / 32 / Cfg::kBatch;
            const float alpha = KIND == kF8 ? 1.0f / (*pr.scale_a * *pr.scale_b) : pr.alpha;
#pragma unroll 1
            for (int hb = 0; hb < kBatches; ++hb) {
                uint32_t r[Cfg::kBatch][32];
#pragma unroll
                for (int c = 0; c < Cfg::kBatch; ++c) tmem_ld_32x32b_x32(taddr + (hb * Cfg::kBatch + c) * 32, r[c]);
                tmem_ld_wait();
                if (hb == kBatches - 1) {                // the accumulator is in registers: the next tile's MMAs may start
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(&tmem_empty[buf], 0);
                }
                const int64_t colb = (int64_t)nt * PN + (kAccBufs == 1 ? half * Cfg::kWarpCols : 0) + hb * Cfg::kBatch * 32;
#pragma unroll
                for (int c = 0; c < Cfg::kBatch; ++c) {
                    const int64_t col = colb + c * 32;
                    const bool in_range = row0 < pr.M && col < pr.N;
                    uint32_t o[16];
                    if (pr.out_fp32) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(r[c][16 * h + j]) * alpha);
                            put(o, map, pr.accumulate != 0, (int32_t)col + 16 * h, (int32_t)row0, in_range && col + 16 * h < pr.N);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[c][2 * j]) * alpha,
                                                                           __uint_as_float(r[c][2 * j + 1]) * alpha);
                            o[j] = *reinterpret_cast<const uint32_t*>(&h);
                        }
                        put(o, map, false, (int32_t)col, (int32_t)row0, in_range);
                    }
                }
            }
        }
        if (lane == 0) bulk_wait_group<0>();                         // every store has left shared memory and is visible
        if (!ok && lane == 0) *abort_flag = 1;
    }

    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);      // let copies in flight land
        __syncthreads();
    }
    cluster_sync_all();                                     // neither CTA leaves while the other may still signal it
    if (warp == 1) {
        tc_fence_after_sync();
        if (LITE) {
            tmem_dealloc_pair(tmem_slot[1], 128);
            tmem_dealloc_pair(tmem_slot[0], 256);
        } else {
            tmem_dealloc_pair(tmem_slot[0], 512);
        }
    }
}

template <int PN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreadsP, 1)
gemm_mxf4_pair_kernel(const __grid_constant__ MapsP maps, const __grid_constant__ ParamsP p) {
    gemm_pair_body<kMxf4, false, PN>(maps, p);
}
template <Kind KIND, int PN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreadsP, 1)
gemm_8bit_pair_kernel(const __grid_constant__ MapsP maps, const __grid_constant__ ParamsP p) {
    gemm_pair_body<KIND, false, PN>(maps, p);
}

template <Kind KIND>
__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(kThreadsP, 1)
gemm_split_kernel(const __grid_constant__ MapsP maps, const __grid_constant__ ParamsP p) {
    gemm_pair_body<KIND, false, 128, true>(maps, p);
}

// The small-footprint build (see PairCfg): same roles, same arithmetic, same accumulation order.
using LiteCfg = PairCfg<kMxf4, true, 256>;
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(LiteCfg::kLaunchRegs)
gemm_mxf4_pair_lite_kernel(const __grid_constant__ MapsP maps, const __grid_constant__ ParamsP p) {
    gemm_pair_body<kMxf4, true, 256>(maps, p);
}

}  // namespace

cudaError_t fetch_gemm_pair_status(unsigned int* word) { return device_status_fetch(word); }

template <typename Cfg, typename K>
static cudaError_t pair_kernel_init(K kernel) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem);
    if (e != cudaSuccess) return e;
    // All of the SM's configurable memory as shared memory: two kernels can only share an SM under one carve-out, and
    // the small builds of GEMM and quantiser together need nearly all of it.
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    if (fa.numRegs * kThreadsP < 128 * (Cfg::kRegsLight + 2 * Cfg::kRegsEpi)) return cudaErrorLaunchOutOfResources;
    return cudaSuccess;
}

cudaError_t gemm_pair_init() {
    cudaError_t e = pair_kernel_init<PairCfg<kMxf4, false, 256>>(gemm_mxf4_pair_kernel<256>);
    if (e == cudaSuccess) e = pair_kernel_init<PairCfg<kMxf4, false, 128>>(gemm_mxf4_pair_kernel<128>);
    if (e == cudaSuccess) e = pair_kernel_init<PairCfg<kF8, false, 256>>(gemm_8bit_pair_kernel<kF8, 256>);
    if (e == cudaSuccess) e = pair_kernel_init<PairCfg<kF8, false, 128>>(gemm_8bit_pair_kernel<kF8, 128>);
    if (e == cudaSuccess) e = pair_kernel_init<PairCfg<kMxf8, false, 256>>(gemm_8bit_pair_kernel<kMxf8, 256>);
    if (e == cudaSuccess) e = pair_kernel_init<PairCfg<kMxf8, false, 128>>(gemm_8bit_pair_kernel<kMxf8, 128>);
    if (e == cudaSuccess) e = pair_kernel_init<PairCfg<kF8, false, 128>>(gemm_split_kernel<kF8>);
    if (e == cudaSuccess) e = pair_kernel_init<PairCfg<kMxf8, false, 128>>(gemm_split_kernel<kMxf8>);
    return e != cudaSuccess ? e : pair_kernel_init<LiteCfg>(gemm_mxf4_pair_lite_kernel);
}

namespace {
int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// How the tiles of one or two products spread over the pairs (see ParamsP), and how long the last pair takes: a tile
// costs cost[i].  `early` is the best of the numbers around cost[0] / cost[1].
struct Spread {
    int rest, early;
    double time;
};
Spread spread_tiles(int n0, int n1, const double (&cost)[2], int pairs) {
    Spread best{n0 % pairs, 0, 0.0};
    const int rest = best.rest, others = pairs - rest;
    const int most = rest != 0 ? n1 / others : 0, around = (int)(cost[0] / cost[1]) < most ? (int)(cost[0] / cost[1]) : most;
    for (int e = around > 0 ? around - 1 : 0; e <= around + 1 && e <= most; ++e) {
        const int late = n1 - e * others, rounds = late / pairs, left = late % pairs;
        const double t_others = (n0 / pairs) * cost[0] + (e + rounds + (left > 0 ? 1 : 0)) * cost[1];
        const double t_rest = rest == 0 ? 0.0 : (n0 / pairs + 1) * cost[0] + (rounds + (left > others ? 1 : 0)) * cost[1];
        const double t = t_others > t_rest ? t_others : t_rest;
        if (best.time == 0.0 || t < best.time) { best.early = e; best.time = t; }
    }
    return best;
}

// Microseconds a pair spends on one tile of a launch that does not reach the board's power limit, for comparing plans: per K-step, and
// per tile what the hand-over of the accumulator (256) or the stores (128, two accumulators) add.  Fitted to the times of whole launches with bf16
// output, which overlap a part of the hand-over (head of this file); fp32 output and addition, whose hand-over is about twice as long, are planned
// with the same figures.
double tile_cost(int pn, int64_t K) {
    const double steps = (double)ceil_div(K, 256);
    return pn == 256 ? 0.34 * steps + 0.65 : 0.245 * steps + 0.3;
}

// Whether an 8-bit product goes out with two pairs to a tile (SPLIT): its 128-wide tiles leave half of the pairs idle (32 clusters
// of four SMs fit the chip's GPCs at once), and half of its K-steps take longer than the exchange, about 2 us.  Whole tiles / split
// in us, 1024 x 1024 (512 x 2048 and 130 x 4096 the same within 0.3): MXINT4 K = 3072 8.9 / 8.8, 4096 10.5 / 9.8, 8192 17.1 / 13.2; E4M3 8.9 / 8.7, 10.6 / 9.5,
// 17.1 / 12.8.  Below the line split lost: MXINT4 K = 1024 6.6 / 7.4, 2048 8.3 / 8.3 (as separate calls, a microsecond more each).
// What it costs: the sum over K is then one of two halves, so the last bits of a row of an 8-bit product depend on how many rows and
// columns are computed with it, as they do in no product of whole tiles (mxfp4.h says so).  MXFP4 products keep whole tiles: a backward
// call's bits are those of its products one by one, and with twice the elements to a K-step they would gain from K = 8192 on only (11.7 / 10.4).
constexpr int kSplitClusters = 32, kSplitSteps = 24;
bool split_pays(int64_t M, int64_t N, int64_t steps) {
    return (int64_t)ceil_div(M, PM) * ceil_div(N, 128) <= kSplitClusters && steps >= kSplitSteps;
}

void fill_problem(ProblemP& p, const GemmArgs& a, int pn) {
    p.M = a.M; p.N = a.N;
    p.nkc = (int)(a.K >> 7);
    p.num_kt = (p.nkc + 1) >> 1;
    p.alpha = a.alpha; p.scale_a = p.scale_b = nullptr;
    p.out_fp32 = a.out_fp32; p.accumulate = a.accumulate;
    p.m_tiles = ceil_div(a.M, PM);
    p.n_tiles = ceil_div(a.N, pn);
    // Tile order: groups of group_m pair-tile rows x all n-tiles.  Inside a group the A rows stay in L2 and B streams
    // through once; B is fetched from DRAM once for the whole launch only if it survives in L2 from one group to the
    // next, i.e. if a group's A rows + all of B + the group's output fit the part of L2 that behaves as one cache
    // (about half of the 126 MB: 48 MB is used here).  Eight rows where that holds, else four: on 16384 x 4096 x 16384
    // eight rows read 348 MB from DRAM, four 243 MB (operands: 168 MB) at the same speed inside a backward step;
    // groups of two or one row read a little less still but cost 0.3 % / 2.5 % of the step (fewer pairs share a B tile
    // at any moment).
    const double b_bytes = (double)a.N * (double)a.K * 0.53125, out_b = a.out_fp32 ? 4.0 : 2.0;
    p.group_m = 8.0 * 256.0 * (double)a.K * 0.53125 + b_bytes + 8.0 * 256.0 * (double)a.N * out_b > 48.0 * 1024 * 1024 ? 4 : 8;
    const char* e = getenv("MXFP4_GEMM_GROUP_M");                  // tuning switch: fixed group size (1..64) instead of the rule above
    if (e != nullptr && atoi(e) >= 1 && atoi(e) <= 64) p.group_m = atoi(e);
}

cudaError_t pair_count(int* pairs) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    *pairs = sms / 2;
    return e;
}
cudaError_t launch_pairs(void (*kernel)(MapsP, ParamsP), int pairs, uint32_t smem, const MapsP& maps, const ParamsP& p, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs); cfg.blockDim = dim3(kThreadsP); cfg.stream = stream;
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return launch_result(cudaLaunchKernelEx(&cfg, kernel, maps, p));
}
}  // namespace

// Columns of a pair tile for a launch of these products (n = 1 or 2): the width with which the last pair is done first.
// 128 wins where 256-wide tiles leave pairs idle: backward 8192 x 1024 x 1024 (dW has 16 tiles of 32 steps) 31.7 -> 28.3 us,
// 1024 x 1024 x 8192 alone 15.2 -> 12.3; it loses wherever the chip is full (16384 x 4096 x 4096: 98 -> 124).
int gemm_pair_tile_n(const GemmArgs* a, int n) {
    int pairs = 0;
    if (a[0].lite || pair_count(&pairs) != cudaSuccess) return 256;
    double time[2];
    for (int i = 0; i < 2; ++i) {
        const int pn = i == 0 ? 256 : 128;
        const int lo = n == 2 && a[1].K > a[0].K ? 1 : 0;
        const int n0 = ceil_div(a[lo].M, PM) * ceil_div(a[lo].N, pn), n1 = n == 2 ? ceil_div(a[1 - lo].M, PM) * ceil_div(a[1 - lo].N, pn) : 0;
        const double cost[2] = {tile_cost(pn, a[lo].K), tile_cost(pn, a[n == 2 ? 1 - lo : lo].K)};
        time[i] = spread_tiles(n0, n1, cost, n0 + n1 < pairs ? n0 + n1 : pairs).time;
    }
    return time[1] < time[0] ? 128 : 256;
}

cudaError_t launch_gemm_pair(const GemmArgs* a, int n, int pn, cudaStream_t stream, const BandSums* bias) {
    if (n < 1 || n > 2 || (pn != 128 && pn != 256) || (a[0].lite && (n != 1 || pn != 256))) return cudaErrorInvalidValue;
    int pairs = 0;
    const cudaError_t e = pair_count(&pairs);
    if (e != cudaSuccess) return e;
    ParamsP p;
    MapsP maps;
    const int first = n == 2 && a[1].K > a[0].K ? 1 : 0;
    int tiles[2] = {0, 0};
    double cost[2];
    for (int i = 0; i < 2; ++i) {
        const GemmArgs& g = a[n == 2 ? (i == 0 ? first : 1 - first) : 0];
        fill_problem(p.prob[i], g, pn);
        maps.a[i] = g.tmap_a; maps.b[i] = g.tmap_b; maps.sfa[i] = g.tmap_sfa; maps.sfb[i] = g.tmap_sfb; maps.c[i] = g.tmap_c;
        cost[i] = tile_cost(pn, g.K);
        if (i < n) tiles[i] = p.prob[i].m_tiles * p.prob[i].n_tiles;
    }
    if (tiles[0] + tiles[1] < pairs) pairs = tiles[0] + tiles[1];
    const Spread s = spread_tiles(tiles[0], tiles[1], cost, pairs);
    p.n0 = tiles[0]; p.n1 = tiles[1]; p.rest = s.rest; p.early = s.early;
    if (bias != nullptr && a[0].lite) return cudaErrorInvalidValue;
    p.bias = bias != nullptr ? *bias : BandSums{};
    const uint32_t smem = a[0].lite ? LiteCfg::kSmem : pn == 128 ? PairCfg<kMxf4, false, 128>::kSmem : PairCfg<kMxf4, false, 256>::kSmem;
    void (*kernel)(MapsP, ParamsP) = a[0].lite ? gemm_mxf4_pair_lite_kernel : pn == 128 ? gemm_mxf4_pair_kernel<128> : gemm_mxf4_pair_kernel<256>;
    return launch_pairs(kernel, pairs, smem, maps, p, stream);
}

// Columns of a pair tile for an 8-bit product: the width with which the last pair is done first.  Measured per tile: 0.36 us
// a K-step + 0.1 (256 wide), 0.245 + 0.1 (128 wide).  E4M3, 256 / 128 wide: 128 wins where 256-wide tiles leave pairs idle (16 x 4096 x
// 4096 13.8 / 10.2 us, 1024 x 1024 x 2048 9.8 / 7.3), 256 elsewhere (8192 x 3072 x 1024 20.3 / 26.9, 16384 x 4096 x 4096 170 / 236).
int gemm_f8_tile_n(const Gemm8Args& a) {
    int pairs = 0;
    if (pair_count(&pairs) != cudaSuccess) return 256;
    if (split_pays(a.M, a.N, a.K >> 7)) return 128;
    const double steps = (double)(a.K >> 7), cost[2] = {0.36 * steps + 0.1, 0.245 * steps + 0.1};
    double time[2];
    for (int i = 0; i < 2; ++i) time[i] = ceil_div((int64_t)ceil_div(a.M, PM) * ceil_div(a.N, i == 0 ? 256 : 128), pairs) * cost[i];
    return time[1] < time[0] ? 128 : 256;
}

cudaError_t launch_gemm_f8(const Gemm8Args& a, int pn, cudaStream_t stream) {
    if (pn != 128 && pn != 256) return cudaErrorInvalidValue;
    int pairs = 0;
    const cudaError_t e = pair_count(&pairs);
    if (e != cudaSuccess) return e;
    ParamsP p = {};
    MapsP maps = {};
    ProblemP& q = p.prob[0];
    q.M = a.M; q.N = a.N;
    q.nkc = q.num_kt = (int)(a.K >> 7);
    q.alpha = a.alpha; q.scale_a = a.scale_a; q.scale_b = a.scale_b;
    q.out_fp32 = a.out_fp32;
    q.m_tiles = ceil_div(a.M, PM);
    q.n_tiles = ceil_div(a.N, pn);
    q.group_m = 8;
    p.n0 = q.m_tiles * q.n_tiles;
    if (p.n0 < pairs) pairs = p.n0;
    p.rest = p.n0 % pairs;
    maps.a[0] = a.tmap_a; maps.b[0] = a.tmap_b; maps.c[0] = a.tmap_c;
    if (a.block_scaled) { maps.sfa[0] = a.tmap_sfa; maps.sfb[0] = a.tmap_sfb; }
    if (pn == 128 && split_pays(a.M, a.N, q.num_kt)) {
        p.rest = 0;
        return launch_pairs(a.block_scaled ? gemm_split_kernel<kMxf8> : gemm_split_kernel<kF8>, 2 * p.n0,
                            a.block_scaled ? PairCfg<kMxf8, false, 128>::kSmem : PairCfg<kF8, false, 128>::kSmem, maps, p, stream);
    }
    if (a.block_scaled)
        return pn == 128 ? launch_pairs(gemm_8bit_pair_kernel<kMxf8, 128>, pairs, PairCfg<kMxf8, false, 128>::kSmem, maps, p, stream)
                         : launch_pairs(gemm_8bit_pair_kernel<kMxf8, 256>, pairs, PairCfg<kMxf8, false, 256>::kSmem, maps, p, stream);
    return pn == 128 ? launch_pairs(gemm_8bit_pair_kernel<kF8, 128>, pairs, PairCfg<kF8, false, 128>::kSmem, maps, p, stream)
                     : launch_pairs(gemm_8bit_pair_kernel<kF8, 256>, pairs, PairCfg<kF8, false, 256>::kSmem, maps, p, stream);
}

}  // namespace mx
