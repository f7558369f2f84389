// BCSR SpMM kernel for sm_100a (Sec. 3.1 - 3.3 of the paper, re-designed for Blackwell).
//
// Work unit ("tile"): one block-row I of A times BN_T = 128 * GROUPS columns of B
// ("tokens").  For every stored block p of the block-row the tile accumulates
//     D[n, r] += sum_c  B[J_p*b + c, n0 + n] * A_p[r, c]
// i.e. the tokens sit on the 128 TMEM lanes (MMA M side, operand read MN-major straight
// from row-major B) and the b rows of the block are the MMA N side (operand = the stored
// block, K-major).  One shape therefore serves b = 16, 32, 64 and 128, and an epilogue thread
// holds one token: a warp's registers are a [C row][32 tokens] tile, row-major like C.
//
// Roles (192 to 288 threads, one CTA per SM, persistent):
//   warps 0, 6 ..   TMA producers (one to four, BcsrProducers), taking the stages in turn: per pipeline
//               stage (1, 2 or 4 stored blocks) one request for the A blocks and one 3-D request per
//               block for its B tile (2*GROUPS boxes of b x 64 tokens), issued by different lanes of
//               one warp-instruction, into a STAGES-deep shared-memory ring; full/empty mbarriers
//               with phase bits.
//   warp 1      MMA issuer: one thread issues tcgen05.mma into one of two TMEM accumulator
//               buffers; tcgen05.commit frees the ring slot / publishes the accumulator.
//   warps 2-5   epilogue: tcgen05.ld -> registers -> one of the warp's staging tiles in shared
//               memory (16 fp32 or 32 16-bit C rows x 32 tokens = 2 KB; a ring of as many tiles
//               per warp as fit beside the stage ring, so that the warp fills the next tile
//               while earlier TMA stores are still reading theirs) -> one TMA store per tile,
//               which also clips at the edges of C (zeros for empty block-rows); overlaps the
//               next tile's MMAs thanks to the second TMEM buffer.  (Column-major 16-bit results:
//               straight from the registers, see BcsrCfg::kDirect.)
// Value types (FMT): fp16, bf16 (K = 16 per MMA), TF32 (fp32 storage, K = 8; the token tile then
// uses the 128-byte swizzle with 32-byte atoms, and blocks wider than 32 columns pass through the
// ring in 32-column slices), E4M3 (K = 32): a K step is 32 bytes of an operand row in all of them.
// A tile of one part of a K-split block-row (record x < 0) stores an fp32 partial tile through
// map P instead of C; bcsr_merge_kernel adds the parts in order.
// Optional variants, all template parameters:
//   CT = 1   C is written in the input's 16-bit type instead of fp32.
//   CM = 1   "column-major" operands (the layout of the paper's BCSR kernel, Sec. 3.2, and of a
//            linear layer Y = X W^T, Sec. 4.4): B is given as X[N][k] (one row per token, k
//            contiguous) and C as Y[N][m].  The token tile is then a K-major MMA operand
//            (rows of min(b, 64) elements, swizzle = row bytes; b = 128 as two K halves), and
//            the staging tile is [32 tokens][16 columns of Y] (fp32).
//   DYN = 1  dynamic tile scheduling with Cluster Launch Control (the direction Sec. 5 points
//            to after the paper's atomic-counter scheduler lost to the hardware block
//            scheduler, Sec. 3.6): the grid has one CTA per tile, in the schedule's global order
//            (slab by slab, longest block-row first); a CTA runs tile blockIdx.x and then
//            keeps cancelling the launch of not-yet-started CTAs and running their tiles.  A
//            seventh warp fetches the tile indices ahead of time into a four-deep ring that
//            the six working warps read.
// The host deals tiles to CTAs ahead of time: slab by slab (a slab = token tiles whose B rows
// fit in L2), longest block-row first, each tile to the least loaded CTA; CTA c walks its list.
#include <mutex>
#include <type_traits>

#include "kernels.h"
#include "ptx.cuh"

namespace spmm {

namespace {

// ES = bytes per input element: 2 (fp16 / bf16), 4 (fp32 storage, TF32 arithmetic), or 1 (E4M3,
// column-major operands only).
// H = rows of one stored block = the MMA's N extent: B for the format's own b x b blocks, 128 for
// the stacked blocks of a row group (128 / b block-rows on top of one another, see format.h).
// CS = bytes per element of C, CM = column-major operands: they fix the epilogue's staging tile.
// A pipeline stage holds one "unit": kBps whole blocks (small b), or one of the kKS column
// slices a block is cut into where its rows are longer than 128 bytes of 4-byte elements
// (b = 64 / 128 with TF32: units of 32 columns, so that a stage stays a fraction of shared memory).
// SPLIT = 1: a tile of 128 tokens is computed by two CTAs: 64 tokens in either (MMA M = 64), or, with stacked blocks, 64 of
// their 128 rows (MMA N = 64).
template <int B, int H, int GROUPS, int STAGES, int ES, int CS, int CM, int SPLIT>
struct BcsrCfg {
    static constexpr int kKS = (H == B) ? bcsr_k_split(B, ES) : 1;     // stage units per block
    static constexpr int kKB = B / kKS;                      // columns of A (= rows of B) per unit
    static constexpr int kBB = kKB * ES;                     // bytes of one unit row (its K extent)
    static constexpr int kKSteps = kBB / 32;                 // MMAs per unit and token group (32 bytes of K each)
    static constexpr int kBnT = 128 * GROUPS;
    static constexpr bool kHalfTok = SPLIT && H == B, kHalfRows = SPLIT && H != B;
    static constexpr int kTok = kHalfTok ? 64 : kBnT;        // tokens and block rows that this CTA stages
    static constexpr int kRows = kHalfRows ? H / 2 : H;
    static constexpr int kWarpTok = kHalfTok ? 16 : 32;      // tokens of an epilogue warp (M = 64: a quarter of them in 16 of its lanes)
    static constexpr int kTokBox = 128 / ES;                 // tokens per 128-byte box row (row-major B)
    static constexpr int kNBox = kTok / kTokBox;             // boxes per unit (row-major B)
    static constexpr int kBoxBytes = kKB * 128;              // kKB k-rows x 128 B (row-major B)
    static constexpr int kDenseBytes = kTok * kBB;           // B tile of one unit
    static constexpr int kABytes = kRows * kBB;
    // Small blocks carry too little work for the fixed cost of a pipeline stage (barrier
    // round trip, request issue, MMA hand-off): a stage holds several consecutive stored
    // blocks of the block-row, their B tiles first, then their A blocks (one request).  So do
    // blocks of 32 and 64 in tiles of 128 tokens, where the issuer's part of a stage (about 170
    // cycles) is as long as a block's four MMAs of 48: twice as many blocks per stage, half as many
    // stages, so that the staging tiles keep their room.  Down-projection 3584 x 18944, density
    // 0.1, N = 128, bf16 9.5 -> 7.9 us; N = 2048, E4M3 34.4 -> 31.6; b = 32, 2048 x 8192 both ways,
    // N = 700, bf16 25.2 -> 23.9.  Not for b = 16, whose stages already hold four blocks: with eight,
    // 50 blocks a row 11.1 -> 10.7, but two blocks a row 6.8 -> 7.2 (half as many tiles in flight).
    // Halves of stacked rows, whose MMAs are half as long, have twice the blocks as well: 3000 x
    // 16000, b = 16, 10 % full rows, bf16, N = 256 75.3 -> 67.8, 600 x 6000 TF32, N = 200 44.0 ->
    // 41.1 (whole stacked blocks, three stages of 64 KB for six of 32: 49.0 -> 50.5 on 6000 x 5000).
    // A stage that is at most half full asks for half of the A blocks (map A0): kFew.
    static constexpr int kBps = H == B ? bcsr_blocks_per_stage(B, ES, GROUPS) : bcsr_stacked_per_stage(B, ES) * (SPLIT ? 2 : 1);
    static constexpr int kFew = H == B ? bcsr_blocks_per_stage(B, ES, 2) : kBps;
    static constexpr int kStageBytes = ((kBps * (kDenseBytes + kABytes) + 1023) / 1024) * 1024;
    static constexpr int kAOff = kBps * kDenseBytes;         // A blocks inside the stage
    static constexpr int kARowBytes = kBB < 128 ? kBB : 128;
    static constexpr uint32_t kASwizzle = kARowBytes == 128 ? SWZ_128B : (kARowBytes == 64 ? SWZ_64B : SWZ_32B);
    // column-major operands: a token group's tile is 128 rows x kXRowBytes, K-major
    static constexpr int kXRowBytes = kARowBytes;
    static constexpr int kXGroupBytes = (kHalfTok ? 64 : 128) * kXRowBytes;    // one K half of one token group
    static constexpr int kAccCols = GROUPS * kRows;
    static constexpr int kTmemCols = (2 * kAccCols <= 32) ? 32 : (2 * kAccCols <= 64 ? 64 : (2 * kAccCols <= 128 ? 128 : (2 * kAccCols <= 256 ? 256 : 512)));
    static constexpr int kBarrierBytes = 512;                // mbarriers, TMEM slot, flags, tile-index ring
    // Epilogue staging: a tile is kEpiCols accumulator columns (rows of C) x 32 tokens.  Every
    // epilogue warp owns a ring of kEpiBufs tiles: as many as fit beside the stage ring (the
    // operand stream comes first: a deeper stage ring gains more than more staging), at most
    // eight.  With more than one tile a warp fills the next tile while earlier TMA stores are
    // still reading theirs.
    // Column-major 16-bit results leave straight from the registers instead: a lane holds consecutive elements of its
    // token's row of Y, whole 128-byte lines of it at b >= 64, and does not wait for a staging tile (the 512-token
    // shapes have room for one per warp).  Up-projection 18944 x 3584, density 0.1, bf16, N = 9001: 195.6 -> 176.6 us
    // (3584 x 18944, eight times the blocks per tile, 151 either way).  fp32 results keep the staging tiles: E4M3,
    // N = 2048, 44.0 us with them, 45.5 without.
    static constexpr bool kDirect = CM != 0 && CS == 2;
    static constexpr int kEpiCols = bcsr_epi_cols(B, CS == 2, CM != 0);
    static constexpr int kEpiTileBytes = kEpiCols * kWarpTok * CS;
    static constexpr int kEpiRoom = (227 * 1024 - 1024 /*align*/ - kBarrierBytes - STAGES * kStageBytes) / (4 * kEpiTileBytes);
    static constexpr int kEpiBufs = kEpiRoom < 8 ? kEpiRoom : 8;
    static constexpr int kStagingBytes = kDirect ? 0 : 4 * kEpiBufs * kEpiTileBytes;
    static constexpr int kSmemBytes = STAGES * kStageBytes + kStagingBytes + 1024 /*align*/ + kBarrierBytes;
    static_assert(kEpiBufs >= 1 && kEpiBufs <= 8, "no room for the epilogue's staging tiles");
    static_assert(kEpiCols <= B && H % kEpiCols == 0, "a staging tile never straddles two block-rows");
    static_assert(2 * kAccCols <= 512, "accumulators exceed TMEM");
    static_assert(kSmemBytes <= 227 * 1024, "stage ring exceeds shared memory");
    static_assert((2 * STAGES + 7 + 8) * 8 + 64 + 32 <= kBarrierBytes, "barrier area");
    static_assert(!SPLIT || (GROUPS == 1 && (CM || kNBox >= 1)), "half of a 128-token tile");
    static_assert(kBps == 1 || (B <= 64 && kKS == 1), "multi-block stages are for the small block sizes");
    static_assert(kKS == 1 || kBB <= 128, "a column slice is at most one 128-byte row piece");
    static_assert(kBB % 32 == 0, "a block row must hold whole K steps");
    static_assert(H == B || (H == 128 && B < 128), "stacked blocks are 128 rows high");
};

// Ring depth for a shape: CAP stages, fewer where they would leave no room for one staging tile
// per epilogue warp.
template <int B, int H, int GROUPS, int CAP, int ES, int CS, int CM, int SPLIT>
constexpr int bcsr_fit_stages() {
    using C1 = BcsrCfg<B, H, GROUPS, 1, ES, CS, CM, SPLIT>;
    const int s = (227 * 1024 - 1024 - C1::kBarrierBytes - 4 * C1::kEpiTileBytes) / C1::kStageBytes;
    return s > CAP ? CAP : (s < 2 ? 2 : s);
}

constexpr int kSchedDepth = 4;      // tile indices fetched ahead by the dynamic scheduler

// TMA producer warps.  One warp takes ~470 cycles per stage to see it free and to issue its two to five requests,
// whatever their size (one CTA alone, 64 x 64 blocks at 128 tokens, 24 KB a stage: 471 cycles a block without the
// MMAs, 311 with the MMAs and without the loads, 517 with both), so up to four warps take the stages in turn.
// Measured with one -> four warps (us): down-projection 3584 x 18944, N = 128, bf16 21.1 -> 14.3; N = 2048, E4M3
// 68.1 -> 36.9; TF32, 64 x 64, N = 3000 115.5 -> 91.1; b = 32, N = 1000 229 -> 161; the prefill shapes within 1 %.
// 512-token stages of 64-row blocks (or of 1-byte values) stay with one: a request is 32 KB there and the loads
// are not short of issue; with four, E4M3 with fp32 C was slower, the loads crowding out the stores (N = 9001
// 185 -> 234).
// At most one warp per stage: a warp's parity wait on a stage's empty barrier is exact only while that barrier is
// at most one phase behind the use the warp is about to fill, that is, while unit it - 2 STAGES has been consumed;
// the warp's own previous unit it - NP tells it that unit it - NP - STAGES has.
template <int B, int GROUPS, int STAGES, int ES, int DYN>
struct BcsrProducers {
    static constexpr int kMost = STAGES < 4 ? STAGES : 4;
    static constexpr int n = (DYN || (GROUPS == 4 && (B >= 64 || ES == 1))) ? 1 : kMost;
    static constexpr int kThreads = DYN ? 224 : 160 + 32 * n;
};

// What the tensor core takes of a 4-byte operand.
__device__ __forceinline__ float tf32_operand(float x) { return x != x ? x : __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// C[row][n] of a TF32 matrix from the blocks its block-row stores.  A stacked block multiplies the absent sub-blocks
// of its other block-rows as zeros, and a zero times Inf or NaN is NaN: where a row group's accumulator is NaN, this
// says whether the row's own blocks make it one.  Never reached with finite operands and sums.
template <int B, int CM>
__device__ __noinline__ float plain_product(const int32_t* block_row_ptr, const int32_t* block_col_idx, const float* vals,
                                            const float* dense, int64_t k, int64_t N, int64_t row, int64_t n) {
    const int64_t I = row / B;
    const int q1 = block_row_ptr[I + 1];
    float s = 0.f;
    for (int q = block_row_ptr[I]; q < q1; ++q) {
        const int64_t k0 = static_cast<int64_t>(block_col_idx[q]) * B;
        const float* a = vals + (static_cast<int64_t>(q) * B + (row - I * B)) * B;
        const int width = static_cast<int>(min_i64(B, k - k0));
        for (int j = 0; j < width; ++j)
            s = fmaf(tf32_operand(a[j]), tf32_operand(CM ? dense[n * k + k0 + j] : dense[(k0 + j) * N + n]), s);
    }
    return s;
}

// The maps that a kernel reads: a launch's parameters are copied for every call (three to five maps in
// place of six, host time of a call, 512 x 512, N = 256: row-major 3.76 -> 3.70 us, column-major 3.73 -> 3.63, 16-bit result 3.58).
struct BcsrOperandMaps { CUtensorMap A, B, B3; };
template <bool HAS> struct BcsrMapA0 {};
template <> struct BcsrMapA0<true> { CUtensorMap A0; };
template <bool HAS> struct BcsrMapC {};
template <> struct BcsrMapC<true> { CUtensorMap C; };
template <bool HAS> struct BcsrMapP {};
template <> struct BcsrMapP<true> { CUtensorMap P; };
template <int BS, int H, int GROUPS, int FMT, int CT, int CM, int DYN, int SPLIT, int ES = FMT == 3 ? 1 : (FMT == 2 ? 4 : 2)>
struct BcsrKernelMaps : BcsrOperandMaps,
                        BcsrMapA0<H == BS && (bcsr_blocks_per_stage(BS, ES, 2) < bcsr_blocks_per_stage(BS, ES, GROUPS))>,
                        BcsrMapC<!(CM && CT)>,
                        BcsrMapP<H == BS && !CT && !CM && !DYN && !SPLIT> {
    static constexpr bool kParts = H == BS && !CT && !CM && !DYN && !SPLIT;     // K-split: static schedule, fp32, row-major
    explicit BcsrKernelMaps(const BcsrMaps& m) : BcsrOperandMaps{m.A, m.B, m.B3} {
        if constexpr (std::is_base_of_v<BcsrMapA0<true>, BcsrKernelMaps>) this->A0 = m.A0;
        if constexpr (std::is_base_of_v<BcsrMapC<true>, BcsrKernelMaps>) this->C = m.C;
        if constexpr (kParts) this->P = m.P;
    }
};

template <int B, int H, int GROUPS, int STAGES, int FMT, int CT, int CM, int DYN, int SPLIT>
__global__ void __launch_bounds__((BcsrProducers<B, GROUPS, STAGES, FMT == 3 ? 1 : (FMT == 2 ? 4 : 2), DYN>::kThreads), 1)
bcsr_spmm_kernel(const __grid_constant__ BcsrKernelMaps<B, H, GROUPS, FMT, CT, CM, DYN, SPLIT> tm, const BcsrParams p) {
    constexpr int ES = FMT == 3 ? 1 : (FMT == 2 ? 4 : 2);
    static_assert(FMT != 2 || (!CT && !DYN && (H == B || B <= 32)), "TF32: fp32 C, static schedule, row groups of rows up to 128 bytes");
    static_assert(H == B || !DYN, "stacked blocks: static schedule only");
    using CElem = typename CType<FMT, CT>::type;
    using Cfg = BcsrCfg<B, H, GROUPS, STAGES, ES, static_cast<int>(sizeof(CElem)), CM, SPLIT>;
    using Maps = BcsrKernelMaps<B, H, GROUPS, FMT, CT, CM, DYN, SPLIT>;
    static_assert(!SPLIT || !DYN, "half tiles: static schedule only");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_al = smem_raw + (smem_base - smem_u32(smem_raw));
    // stage ring | staging tiles of the epilogue warps | barriers
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_al + STAGES * Cfg::kStageBytes + Cfg::kStagingBytes);
    // barrier slots: full[STAGES], empty[STAGES], acc_full[2], acc_empty[2]
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
    auto accf_bar = [&](int a) { return bar0 + 8u * (2 * STAGES + a); };
    auto acce_bar = [&](int a) { return bar0 + 8u * (2 * STAGES + 2 + a); };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars + 2 * STAGES + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 2 * STAGES + 5);
    const uint32_t drain_bar = bar0 + 8u * (2 * STAGES + 6);   // abort path: MMAs still in flight
    // dynamic scheduling: ring of fetched tile indices (16-byte answers) with full / empty barriers
    auto schf_bar = [&](int s) { return bar0 + 8u * (2 * STAGES + 7 + s); };
    auto sche_bar = [&](int s) { return bar0 + 8u * (2 * STAGES + 7 + kSchedDepth + s); };
    const uint32_t sched_resp = (bar0 + 8u * (2 * STAGES + 7 + 2 * kSchedDepth) + 15u) & ~15u;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = SPLIT ? blockIdx.x & 1 : 0;          // which half of the tile's tokens or of the blocks' rows
    WaitCtl ctl{abort_flag, p.status, p.wait_limit_ns};

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(accf_bar(a), 1); mbar_init(acce_bar(a), 4); }
        mbar_init(drain_bar, 1);
        if constexpr (DYN) {
            for (int s = 0; s < kSchedDepth; ++s) { mbar_init(schf_bar(s), 1); mbar_init(sche_bar(s), 6); }
        }
        *abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tm.A);
        if constexpr (Cfg::kFew < Cfg::kBps) prefetch_tmap(&tm.A0);
        prefetch_tmap(&tm.B);
        prefetch_tmap(&tm.B3);
        if constexpr (!Cfg::kDirect) prefetch_tmap(&tm.C);
        if constexpr (Maps::kParts) prefetch_tmap(&tm.P);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), Cfg::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    const int64_t N = p.N;
    // Static schedule: this CTA's range of the tile list.  Dynamic: tile blockIdx.x, then the
    // indices the scheduler warp obtains; every working warp walks the same sequence.
    int tile_begin = 0, tile_end = 0;
    int4 rec0 = make_int4(0, 0, 0, 0);               // record of this CTA's first tile
    if constexpr (!DYN) {
        const int list = SPLIT ? blockIdx.x / 2 : blockIdx.x;
        tile_begin = __ldg(p.cta_ptr + list);
        tile_end = __ldg(p.cta_ptr + list + 1);
        if (tile_begin < tile_end) rec0 = __ldg(p.tiles + tile_begin);
    }
    // The row groups' launch (overlap = 1): the launch of the remaining block-rows runs beside this one (the two
    // write disjoint rows of C), so it is let go only when the operands are ready.
    if (p.overlap != 1) grid_trigger();
    // What a role does before this is with the handle's own data only (complete on every stream once the handle
    // exists): the producers request their first stored blocks, see below.
    auto operands_ready = [&]() {
        if (p.overlap != 2) grid_wait();
        if (p.overlap == 1) grid_trigger();
    };
    // Next tile of this warp's walk; nth = number of tiles it has taken so far.  A tile's record
    // {block-row, token tile, first stored block, end block} is all a role needs to know about
    // it; with the static schedule the following tile's record is requested one tile ahead
    // (*rec_next), so that its latency is not paid between tiles.
    auto next_tile = [&](uint32_t nth, int4* rec, int4* rec_next, bool* ok) -> bool {
        if constexpr (!DYN) {
            const int ti = tile_begin + static_cast<int>(nth);
            if (ti >= tile_end) return false;
            *rec = nth == 0 ? rec0 : *rec_next;
            if (ti + 1 < tile_end) *rec_next = __ldg(p.tiles + ti + 1);
            return true;
        } else {
            int ti_dyn;
            int* ti = &ti_dyn;
            if (nth == 0) { *rec = __ldg(p.tiles + blockIdx.x); return true; }
            // fetched tile nth is entry nth - 1 of the ring
            const int slot = (nth - 1u) % kSchedDepth;
            const uint32_t use = (nth - 1u) / kSchedDepth;
            if (!__all_sync(0xffffffffu, mbar_wait(schf_bar(slot), use & 1u, ctl, 5))) { *ok = false; return false; }
            uint32_t x;
            const bool valid = clc_query(sched_resp + 16u * slot, &x);
            fence_proxy_async_smem();           // the slot is rewritten by the asynchronous proxy later
            __syncwarp();
            if (lane == 0) mbar_arrive(sche_bar(slot));
            if (valid && x >= gridDim.x) {
                // cannot happen with a well-formed answer; recorded instead of trusted
                if (lane == 0 && atomicCAS(p.status, 0, 2) == 0) { p.status[1] = 8; p.status[2] = static_cast<int>(x); }
                *ok = false;
                return false;
            }
            *ti = static_cast<int>(x);
            if (valid) *rec = __ldg(p.tiles + *ti);
            return valid;
        }
    };

    constexpr int NP = BcsrProducers<B, GROUPS, STAGES, ES, DYN>::n;
    static_assert(NP <= STAGES && NP <= 4, "parity waits; slots of `issued`");
    // units issued by every producer warp (its own among those below this count): for the abort path
    volatile uint32_t* issued = reinterpret_cast<volatile uint32_t*>(reinterpret_cast<uint8_t*>(bars) + Cfg::kBarrierBytes - 16);
    if (warp == 0 || (!DYN && warp >= 6)) {
        // ------------------------------------------------------------------ TMA producers
        // A warp serialises the TMA requests of its lanes (~60 cycles each) but needs far
        // longer for requests issued one after the other by a single thread, so the loads of
        // a stage are spread over the lanes: lane x < nbox fetches B box x, lanes 8 / 9 the
        // A block (two halves when b = 128).  Lane 0 posts the stage's byte count first.
        {
            const uint32_t pw = warp == 0 ? 0 : warp - 5;   // this warp takes the stage units pw, pw + NP, ...
            uint32_t it = 0;
            bool ok = true;
            // A blocks and the B slab are re-read by other CTAs while the slab lasts: ask L2 to
            // keep them in preference to the C lines streaming through
            const uint64_t keep = l2_policy_evict_last();
            int4 tcd, tcd_next;
            int Jl_next = 0;                 // block columns of the next tile's first 32 blocks, fetched a tile ahead
            bool have_next = false;
            // tokens of this CTA's part of the tile that exist
            auto valid_tokens = [&](int n0) -> int {
                if constexpr (Cfg::kHalfTok) return static_cast<int>(min_i64(Cfg::kTok, N > n0 + half * Cfg::kTok ? N - n0 - half * Cfg::kTok : 0));
                return static_cast<int>(min_i64(Cfg::kBnT, N - n0));
            };
            // the A request always brings kBps or kFew blocks (the boxes of the tensor maps)
            auto few_blocks = [&](int nb) { return Cfg::kFew < Cfg::kBps && nb <= Cfg::kFew; };
            // the stage of unit it, nb stored blocks: its byte count, before any of its requests
            auto expect_stage = [&](uint32_t it, int nb, int nvalid) {
                const int nbox = (nvalid + Cfg::kTokBox - 1) / Cfg::kTokBox;
                const uint32_t dense_tx = CM ? (Cfg::kHalfTok ? (nvalid > 0 ? Cfg::kDenseBytes : 0)
                                                              : ((p.use_3d && nvalid == Cfg::kBnT) ? Cfg::kDenseBytes : ((nvalid + 127) >> 7) * (128 * Cfg::kBB)))
                                             : nbox * Cfg::kBoxBytes;
                // (stacked blocks: one request per block, a box holds at most 256 rows)
                if (lane == 0)
                    mbar_arrive_expect_tx(full_bar(it % STAGES), (H == B ? (few_blocks(nb) ? Cfg::kFew : Cfg::kBps) : nb) * Cfg::kABytes + nb * dense_tx);
                __syncwarp();
            };
            // and its stored blocks q .. q + nb - 1 (columns kx .. of them)
            auto request_blocks = [&](uint32_t it, int q, int kx, int nb) {
                const int s = it % STAGES;
                const uint32_t sb = smem_base + s * Cfg::kStageBytes;
                if constexpr (H == B) {
                    if (lane == 8) {
                        const CUtensorMap* blocks = &tm.A;
                        if constexpr (Cfg::kFew < Cfg::kBps) blocks = few_blocks(nb) ? &tm.A0 : &tm.A;
                        tma_load_2d_hint(sb + Cfg::kAOff, blocks, full_bar(s), kx, q * B, keep);
                    } else if (Cfg::kBB > 128 && lane == 9) {
                        tma_load_2d_hint(sb + Cfg::kAOff + B * 128, &tm.A, full_bar(s), 128 / ES, q * B, keep);
                    }
                } else {
                    if (lane >= 8 && lane < 8 + nb)
                        tma_load_2d_hint(sb + Cfg::kAOff + (lane - 8) * Cfg::kABytes, &tm.A, full_bar(s), 0, (q + lane - 8) * H + half * (H - Cfg::kRows), keep);
                }
            };
            // The first tile's first units: their block columns and stored blocks belong to the handle and are
            // fetched while the launch before this one may still be running (a short launch is a chain of index,
            // request, MMA and store latencies, and the weights of a decode step come from HBM); the units' B tiles
            // follow in the loop below.  Back to back, us:
            // both projections 18944 x 3584, bf16, N = 128 19.4 -> 17.7; 512 x 512, N = 256 4.12 -> 3.79 (4.21 -> 4.03
            // on another box).
            uint32_t early = 0;
            if (!DYN && tile_begin < tile_end && rec0.w > rec0.z) {
                Jl_next = (rec0.z + lane < rec0.w) ? __ldg(p.block_col_idx + rec0.z + lane) : 0;
                have_next = true;
                const int nq = min(32, rec0.w - rec0.z);
                early = min(STAGES, (nq + Cfg::kBps - 1) / Cfg::kBps * Cfg::kKS);
                const int nvalid = valid_tokens(rec0.y * Cfg::kBnT);
                for (uint32_t u = pw; u < early; u += NP) {
                    const int jq = static_cast<int>(u) / Cfg::kKS * Cfg::kBps;
                    expect_stage(u, min(Cfg::kBps, nq - jq), nvalid);
                    request_blocks(u, rec0.z + jq, static_cast<int>(u) % Cfg::kKS * Cfg::kKB, min(Cfg::kBps, nq - jq));
                }
            }
            operands_ready();
            // The order of a stage's requests, see bcsr_tiles_first in api.cu, is chosen outside the loop, and only in the
            // shapes that gain from it: a test of it per stage cost small launches up to 5 % (15,584 x 2008, b = 64, TF32,
            // N = 680, us: 37.4 so, 39.3 with the test), and so did a second loop beside the one in use where a stage is
            // short (TF32, b = 64, column-major, 512 x 11264, N = 128: 21.1 with it, 19.6 without).
            auto walk = [&](auto order) {
            constexpr bool kTilesFirst = decltype(order)::value;
            for (uint32_t nth = 0; ok && next_tile(nth, &tcd, &tcd_next, &ok); ++nth) {
                const int nvalid = valid_tokens(tcd.y * Cfg::kBnT);
                const int n0 = tcd.y * Cfg::kBnT + (Cfg::kHalfTok ? half * Cfg::kTok : 0);         // this CTA's first token
                [[maybe_unused]] const int nbox = (nvalid + Cfg::kTokBox - 1) / Cfg::kTokBox;
                const bool whole_tile = !Cfg::kHalfTok && p.use_3d && nvalid == Cfg::kBnT;
                const int pb = tcd.z, pe = tcd.w;
                const int Jl_first = have_next ? Jl_next : ((pb + lane < pe) ? __ldg(p.block_col_idx + pb + lane) : 0);
                if constexpr (!DYN) {
                    // the record of the following tile was requested when this one was taken
                    have_next = tile_begin + static_cast<int>(nth) + 1 < tile_end;
                    if (have_next) Jl_next = (tcd_next.z + lane < tcd_next.w) ? __ldg(p.block_col_idx + tcd_next.z + lane) : 0;
                }
                for (int q0 = pb; q0 < pe && ok; q0 += 32) {
                    // block columns of up to 32 stored blocks with one coalesced load
                    const int Jl = q0 == pb ? Jl_first : ((q0 + lane < pe) ? __ldg(p.block_col_idx + q0 + lane) : 0);
                    const int nq = min(32, pe - q0);
                    for (int jq = 0; jq < nq && ok; jq += Cfg::kBps)
#pragma unroll 1
                    for (int kp = 0; kp < Cfg::kKS; ++kp, ++it) {       // column slices of the block (1 unless TF32, b >= 64)
                        if (NP > 1 && it % NP != pw) continue;
                        const int q = q0 + jq;
                        const int kx = kp * Cfg::kKB;                    // first column of A / first row of B of this unit
                        const int nb = min(Cfg::kBps, nq - jq);          // stored blocks in this stage
                        const int s = it % STAGES;
                        const uint32_t ph = (it / STAGES) & 1u;
                        // (an early unit's stage is fresh; it may even have been used already, where it has no tokens)
                        if (it >= early) {
                            if (!__all_sync(0xffffffffu, mbar_wait(empty_bar(s), ph ^ 1u, ctl, 1))) { ok = false; break; }
                            expect_stage(it, nb, nvalid);
                            if (!kTilesFirst) request_blocks(it, q, kx, nb);
                        }
                        const uint32_t sb = smem_base + s * Cfg::kStageBytes;
                        if constexpr (CM) {
                            // X as [N / 128][128][k]: box = GROUPS x 128 tokens x min(b, 64) elements
                            // of block column J (b = 128: lanes nb.. fetch the second K half)
                            constexpr int kHalves = Cfg::kBB > 128 ? 2 : 1;
                            const int blk = lane % Cfg::kBps, hf = lane / Cfg::kBps;
                            const int J = __shfl_sync(0xffffffffu, Jl, jq + (blk < nb ? blk : 0));
                            if (whole_tile) {
                                if (blk < nb && hf < kHalves)
                                    tma_load_3d_hint(sb + blk * Cfg::kDenseBytes + hf * (GROUPS * Cfg::kXGroupBytes), &tm.B3,
                                                     full_bar(s), J * B + kx + hf * (128 / ES), 0, n0 >> 7, keep);
                            } else {
                                // ragged tile, or half of one: one request per token group, rows >= N are zero filled
                                const int ngrp = (nvalid + 127) >> 7;
                                for (int g = 0; g < ngrp; ++g)
                                    if (blk < nb && hf < kHalves)
                                        tma_load_2d_hint(sb + blk * Cfg::kDenseBytes + hf * (GROUPS * Cfg::kXGroupBytes) + g * Cfg::kXGroupBytes,
                                                         &tm.B, full_bar(s), J * B + kx + hf * (128 / ES), n0 + g * 128, keep);
                            }
                        } else
                        if (whole_tile) {
                            // all boxes of a unit with one request: B seen as [token box][k][128 bytes of
                            // tokens], box = kNBox x kKB x 128 bytes; lane i takes block i
                            const int J = __shfl_sync(0xffffffffu, Jl, jq + (lane < nb ? lane : 0));
                            if (lane < nb) tma_load_3d_hint(sb + lane * Cfg::kDenseBytes, &tm.B3, full_bar(s), 0, J * B + kx, n0 / Cfg::kTokBox, keep);
                        } else {
                            for (int i = 0; i < nb; ++i) {
                                const int J = __shfl_sync(0xffffffffu, Jl, jq + i);
                                if (lane < nbox)
                                    tma_load_2d_hint(sb + i * Cfg::kDenseBytes + lane * Cfg::kBoxBytes, &tm.B, full_bar(s),
                                                     n0 + lane * Cfg::kTokBox, J * B + kx, keep);
                            }
                        }
                        if (kTilesFirst && it >= early) request_blocks(it, q, kx, nb);
                    }
                }
            }
            };
            constexpr bool kEither = H == B && !CM && !SPLIT && !DYN && (B == 128 || (B == 64 && GROUPS > 1));
            if (kEither && p.tiles_first) walk(std::bool_constant<kEither>());
            else walk(std::false_type());
            if (lane == 0) issued[pw] = it;
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        // Warp-uniform control flow (all lanes wait and compute the uniform descriptors); one
        // elected lane issues the tcgen05 instructions.
        {
            // 8-bit floats: format code 0 = E4M3 in both operand fields
            constexpr uint32_t idesc = make_idesc(FMT == 3 ? 0 : FMT, Cfg::kHalfTok ? 64 : 128, Cfg::kRows, CM ? 0 : 1, 0);
            // row-major B: the token tile is MN-major; 4-byte elements need the 128-byte swizzle with
            // 32-byte atoms (a pattern of 4 k-rows), 2-byte elements the plain one (8 k-rows)
            const uint64_t adesc0 = CM ? make_smem_desc(0, 16, 8 * Cfg::kXRowBytes, Cfg::kASwizzle)
                                       : make_smem_desc(0, Cfg::kBoxBytes, ES == 4 ? 512 : 1024, ES == 4 ? SWZ_128B_BASE32B : SWZ_128B);
            constexpr int kStepBytes = (32 / ES) * 128;     // k-rows of one MMA x 128 bytes (row-major token tile)
            const uint64_t bdesc0 = make_smem_desc(0, 16, 8 * Cfg::kARowBytes, Cfg::kASwizzle);
            const bool leader = elect_one();
            // Whether the next stage's full barrier was already seen complete: with one token group and b < 128 the
            // next stage is tested before this stage's MMAs are issued, so that its answer is there when they have
            // been (a stage cost the issuer 172 cycles beside its four MMAs of 48, during which the tensor pipe ran
            // dry; down-projection 3584 x 18944, N = 128: 11.3 -> 10.6 us, b = 32, N = 1000: 87.7 -> 80.3).  Wider
            // tiles have MMAs enough to cover it and measured up to 3 % slower with the extra test; so have blocks of 128
            // (8192 x 8192, b = 128, density 0.2: 156.1 us with it, 154.2 without).
            uint32_t it = 0, tile_i = 0;
            bool ready = false;
            bool ok = true;
            operands_ready();               // (the time its waits may take is not to include the launch before this one)
            int4 tcd, tcd_next;
            for (; ok && next_tile(tile_i, &tcd, &tcd_next, &ok); ++tile_i) {
                const int n0 = tcd.y * Cfg::kBnT;
                const int nvalid = static_cast<int>(min_i64(Cfg::kBnT, N - n0));
                const int ngrp = (nvalid + 127) >> 7;
                const int acc = tile_i & 1;
                const uint32_t aph = (tile_i >> 1) & 1u;
                if (!__all_sync(0xffffffffu, mbar_wait(acce_bar(acc), aph ^ 1u, ctl, 2))) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t d0 = tmem_base + acc * Cfg::kAccCols;
                const int pb = tcd.z, pe = tcd.w;
                for (int q = pb; q < pe && ok; q += Cfg::kBps)
#pragma unroll 1
                for (int kp = 0; kp < Cfg::kKS; ++kp, ++it) {
                    // stages never straddle the producer's 32-block windows (kBps divides 32)
                    const int nb = min(Cfg::kBps, min(pe - q, 32 - ((q - pb) & 31)));
                    const int s = it % STAGES;
                    const uint32_t ph = (it / STAGES) & 1u;
                    if (!ready && !__all_sync(0xffffffffu, mbar_wait(full_bar(s), ph, ctl, 3))) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint32_t sb = smem_base + s * Cfg::kStageBytes;
                    if constexpr (GROUPS == 1 && B < 128)
                        ready = __all_sync(0xffffffffu, mbar_test_wait(full_bar((it + 1) % STAGES), ((it + 1) / STAGES) & 1u));
#pragma unroll
                    for (int i = 0; i < Cfg::kBps; ++i) {
                        if (i < nb) {
                            // descriptors differ only in their start-address field (bytes >> 4)
                            const uint64_t a0 = adesc0 + ((sb + i * Cfg::kDenseBytes) >> 4);
                            const uint64_t b0 = bdesc0 + ((sb + Cfg::kAOff + i * Cfg::kABytes) >> 4);
                            const uint32_t accum0 = (q > pb || i > 0 || kp > 0) ? 1u : 0u;
#pragma unroll
                            for (int ks = 0; ks < Cfg::kKSteps; ++ks) {
                                const uint32_t boff = Cfg::kBB <= 128 ? ks * 32 : (ks >> 2) * (B * 128) + (ks & 3) * 32;
#pragma unroll
                                for (int g = 0; g < GROUPS; ++g)
                                    if (leader && g < ngrp)
                                        umma_kind<FMT == 3 ? 2 : (FMT == 2 ? 1 : 0)>(d0 + g * Cfg::kRows,
                                                       a0 + ((CM ? (Cfg::kBB <= 128 ? g * Cfg::kXGroupBytes + ks * 32
                                                                            : (ks >> 2) * (GROUPS * Cfg::kXGroupBytes) + g * Cfg::kXGroupBytes + (ks & 3) * 32)
                                                                 : g * (Cfg::kNBox / GROUPS) * Cfg::kBoxBytes + ks * kStepBytes) >> 4),
                                                       b0 + (boff >> 4), idesc, ks > 0 ? 1u : accum0);
                            }
                        }
                    }
                    if (leader) tc_commit(empty_bar(s));
                }
                if (!ok) break;
                if (leader) {
                    if (pe > pb) tc_commit(accf_bar(acc));
                    else mbar_arrive(accf_bar(acc));
                }
            }
        }
    } else if (warp < 6) {
        // ------------------------------------------------------------------ epilogue warps
        const int qd = warp & 3;                    // TMEM lane quarter this warp may read
        const bool mine = lane < Cfg::kWarpTok;     // this lane holds a token
        uint32_t tile_i = 0;
        uint32_t chunk = 0;                         // staging tiles this warp has filled so far
        const uint32_t stg0 = smem_base + STAGES * Cfg::kStageBytes + (warp - 2) * (Cfg::kEpiBufs * Cfg::kEpiTileBytes);
        bool ok = true;
        [[maybe_unused]] const bool wide = ((reinterpret_cast<uintptr_t>(p.C) | static_cast<uintptr_t>(p.m * sizeof(CElem))) & 31) == 0;
        operands_ready();
        int4 tcd, tcd_next;
        for (; ok && next_tile(tile_i, &tcd, &tcd_next, &ok); ++tile_i) {
            const int tI = tcd.x;
            const int n0 = tcd.y * Cfg::kBnT;
            const int nvalid = static_cast<int>(min_i64(Cfg::kBnT, N - n0));
            const int ngrp = (nvalid + 127) >> 7;
            const int acc = tile_i & 1;
            const uint32_t aph = (tile_i >> 1) & 1u;
            const bool has_blocks = tcd.w > tcd.z;
            // stacked blocks: the block-rows the group's 128 accumulator columns belong to
            int member = 0;
            if constexpr (H != B) member = lane < H / B ? __ldg(p.stack_rows + tI * (H / B) + lane) : 0;
            if (!__all_sync(0xffffffffu, mbar_wait(accf_bar(acc), aph, ctl, 4))) { ok = false; break; }
            tc_fence_after_sync();
            // K-split: a tile of one part of a long block-row (record x = -1 - slot) writes its fp32
            // partial tile, rows slot * b .. of the partial array, instead of C (fp32 row-major C only)
            const bool part = Maps::kParts && tI < 0;
            const int64_t row0 = static_cast<int64_t>(part ? -1 - tI : tI) * B;
            constexpr int W = Cfg::kDirect ? (B < 64 ? B : 64) : Cfg::kEpiCols;     // accumulator columns at a time
            for (int g = 0; g < ngrp; ++g) {
                const int nw = n0 + g * 128 + (Cfg::kHalfTok ? half * 64 : 0) + qd * Cfg::kWarpTok;          // first token of this warp
                if (nw >= N) break;                             // the whole warp is beyond the last token
#pragma unroll 1
                for (int c0 = 0; c0 < Cfg::kRows; c0 += W) {
                    uint32_t v[W];
                    if (has_blocks) {
                        const uint32_t ta = tmem_base + (static_cast<uint32_t>(qd * 32) << 16) +
                                            acc * Cfg::kAccCols + g * Cfg::kRows + c0;
                        tmem_ld_cols<W>(ta, v);
                        tmem_ld_wait();
                    } else {
#pragma unroll
                        for (int j = 0; j < W; ++j) v[j] = 0u;
                    }
                    int32_t crow = static_cast<int32_t>(row0) + c0;
                    if constexpr (H != B) crow = __shfl_sync(0xffffffffu, member, (half * (H - Cfg::kRows) + c0) / B) * B + (c0 % B);
                    if constexpr (H != B && FMT == 2) {
                        float most = 0.f;                     // NaN if any value is
#pragma unroll
                        for (int j = 0; j < W; j += 2)
                            asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(most) : "f"(__uint_as_float(v[j])), "f"(__uint_as_float(v[j + 1])));
                        if (__any_sync(0xffffffffu, mine && most != most)) {
#pragma unroll
                            for (int j = 0; j < W; ++j)
                                if (__uint_as_float(v[j]) != __uint_as_float(v[j]) && mine && crow + j < p.m && nw + lane < N)
                                    v[j] = __float_as_uint(plain_product<B, CM>(p.block_row_ptr, p.plain_col_idx, p.plain_vals, p.B, p.k, N,
                                                                               crow + j, nw + lane));
                            __syncwarp();
                        }
                    }
                    if constexpr (Cfg::kDirect) {
                        // this lane's token: W consecutive columns of its row of Y, straight from the registers in
                        // pieces of 32 bytes (16 where a row or the end of Y does not allow it)
                        constexpr int kPer = 32 / static_cast<int>(sizeof(CElem));
                        if (mine && nw + lane < N) {
                            CElem* dst = static_cast<CElem*>(p.C) + (nw + lane) * p.m + crow;
#pragma unroll
                            for (int c = 0; c < W; c += kPer) {
                                uint32_t w8[8];
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    const CElem lo = from_f32<CElem>(__uint_as_float(v[c + 2 * i]));
                                    const CElem hi = from_f32<CElem>(__uint_as_float(v[c + 2 * i + 1]));
                                    w8[i] = static_cast<uint32_t>(*reinterpret_cast<const unsigned short*>(&lo)) |
                                            (static_cast<uint32_t>(*reinterpret_cast<const unsigned short*>(&hi)) << 16);
                                }
                                if (wide && crow + c + kPer <= p.m) {
                                    st_global_vec<32>(dst + c, w8);
                                } else {
                                    if (crow + c + kPer / 2 <= p.m) st_global_vec<16>(dst + c, w8);
                                    if (crow + c + kPer <= p.m) st_global_vec<16>(dst + c + kPer / 2, w8 + 4);
                                }
                            }
                        }
                    } else {
                    // registers -> the next tile of this warp's staging ring -> one TMA store.  The
                    // store that used this tile kEpiBufs chunks ago must have read it first.
                    const uint32_t stg = stg0 + (chunk % Cfg::kEpiBufs) * Cfg::kEpiTileBytes;
                    ++chunk;
                    if (lane == 0) bulk_wait_read<Cfg::kEpiBufs - 1>();
                    __syncwarp();
                    if constexpr (!CM) {
                        // tile [W rows][32 tokens], no swizzle: 128-byte rows of fp32 (64-byte rows
                        // of 2-byte elements); a warp's store covers one row, so no bank is hit twice
#pragma unroll
                        for (int j = 0; j < W; ++j) {
                            if constexpr (sizeof(CElem) == 4) {
                                if (mine) st_shared_u32(stg + (j * Cfg::kWarpTok + lane) * 4, v[j]);
                            } else {
                                const CElem h = from_f32<CElem>(__uint_as_float(v[j]));
                                if (mine) st_shared_u16(stg + (j * Cfg::kWarpTok + lane) * 2, *reinterpret_cast<const unsigned short*>(&h));
                            }
                        }
                    } else {
                        // tile [32 tokens][16 fp32]: this lane's row, in 16-byte chunks; its 64 bytes are stored with
                        // the tensor map's 64-byte swizzle (chunk index XOR (row / 2) % 4), which also keeps the
                        // warp's stores off each other's banks
                        static_assert(W == 16 && sizeof(CElem) == 4, "64-byte rows");
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (mine) st_shared_v4(stg + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4), v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        const CUtensorMap* tm_out = &tm.C;
                        if constexpr (Maps::kParts) tm_out = part ? &tm.P : &tm.C;
                        // row-major: box = 32 tokens x W rows at (token, row); column-major: box =
                        // W columns x 32 tokens at (column, token).  Out-of-range parts are clipped.
                        if constexpr (!CM) tma_store_2d(tm_out, stg, nw, crow);
                        else tma_store_2d(tm_out, stg, crow, nw);
                        bulk_commit_group();
                    }
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce_bar(acc));
        }
        if (lane == 0) bulk_wait_all<false>();          // this warp's last stores have landed
    }

    if constexpr (DYN) {
        if (warp == 6 && lane == 0) {
            // -------------------------------------------------------------- tile scheduler
            // One request at a time (a request after a failed one is not allowed), up to
            // kSchedDepth tiles ahead of the slowest working warp.
            for (uint32_t r = 0;; ++r) {             // ring entry r = the CTA's tile r + 1
                const int slot = r % kSchedDepth;
                const uint32_t use = r / kSchedDepth;
                if (use > 0 && !mbar_wait(sche_bar(slot), (use - 1u) & 1u, ctl, 6)) break;
                mbar_arrive_expect_tx(schf_bar(slot), 16);
                clc_try_cancel(sched_resp + 16u * slot, schf_bar(slot));
                if (!mbar_wait(schf_bar(slot), use & 1u, ctl, 7)) {
                    // leaving early: the answer of the request just issued must still land in
                    // this CTA's shared memory before the CTA may exit (bounded)
                    mbar_drain_wait(schf_bar(slot), use & 1u, ctl, 22);
                    break;
                }
                uint32_t x;
                if (!clc_query(sched_resp + 16u * slot, &x)) break;      // no CTA left to cancel: the walk ends
            }
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) {
        // leave no bulk copy in flight: wait (bounded) for the last fill issued into every stage
        uint32_t most = 0;
        for (int w = 0; w < NP; ++w) most = issued[w] > most ? issued[w] : most;
        bool ok = true;
        for (uint32_t s = 0; s < STAGES && ok; ++s) {
            for (uint32_t j = most; j-- > 0;) {              // a stage's last fill is among the last few units
                if (j % STAGES != s || j >= issued[j % NP]) continue;
                ok = mbar_drain_wait(full_bar(s), (j / STAGES) & 1u, ctl, 21);
                break;
            }
        }
    }
    // launched while the previous grid of the stream was still running: do not finish before it
    if (p.overlap == 2) grid_wait();
    if (warp == 1) {
        if (*abort_flag) {
            // abort path: let the MMAs this warp's elected lane already issued finish before
            // TMEM is freed (kept out of the role loop above on purpose: placed there it
            // slowed the normal path measurably)
            if (elect_one()) {
                tc_commit(drain_bar);
                mbar_drain_wait(drain_bar, 0, ctl, 23);
            }
            __syncwarp();
        }
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, Cfg::kTmemCols);
    }
}

// CAP = the deepest ring the shape is given; the ring actually used also leaves room for the
// epilogue's staging tiles (bcsr_fit_stages).
template <int B, int H, int GROUPS, int CAP, int FMT, int CT, int CM, int DYN, int SPLIT = 0>
cudaError_t launch_one(const BcsrMaps& tm, const BcsrParams& p,
                       int grid, cudaStream_t stream) {
    constexpr int ES = FMT == 3 ? 1 : (FMT == 2 ? 4 : 2);
    constexpr int CS = static_cast<int>(sizeof(typename CType<FMT, CT>::type));
    constexpr int STAGES = bcsr_fit_stages<B, H, GROUPS, CAP, ES, CS, CM, SPLIT>();
    using Cfg = BcsrCfg<B, H, GROUPS, STAGES, ES, CS, CM, SPLIT>;
    constexpr int kThreads = BcsrProducers<B, GROUPS, STAGES, ES, DYN>::kThreads;
    auto kfn = bcsr_spmm_kernel<B, H, GROUPS, STAGES, FMT, CT, CM, DYN, SPLIT>;
    // the attribute belongs to the (function, device) pair: set it once per device
    static std::mutex mu;
    static bool attr_done[kMaxDevices] = {};
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(mu);
        if (!attr_done[dev]) {
            e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kSmemBytes);
            if (e != cudaSuccess) return e;
            attr_done[dev] = true;
        }
    }
    const BcsrKernelMaps<B, H, GROUPS, FMT, CT, CM, DYN, SPLIT> maps(tm);
    if constexpr (DYN) {        // (its grid is a queue of CTAs that running ones cancel: launched when the stream gets there)
        kfn<<<grid, kThreads, Cfg::kSmemBytes, stream>>>(maps, p);
        return cudaGetLastError();
    } else {
        return launch_dependent(kfn, dim3(static_cast<unsigned>(SPLIT ? 2 * grid : grid)), kThreads, Cfg::kSmemBytes, stream, maps, p);
    }
}

template <int FMT, int CT, int CM, int DYN>
cudaError_t launch_shape(int b, int groups, const BcsrMaps& tm, const BcsrParams& p, int grid, cudaStream_t stream) {
    switch (b * 10 + groups) {
        case 161: return launch_one<16, 16, 1, 10, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 162: return launch_one<16, 16, 2, 5, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 164: return launch_one<16, 16, 4, 3, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 321: return launch_one<32, 32, 1, 5, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 322: return launch_one<32, 32, 2, 5, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 324: return launch_one<32, 32, 4, 3, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 641: return launch_one<64, 64, 1, 4, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 642: return launch_one<64, 64, 2, 5, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 644: return launch_one<64, 64, 4, 3, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 1281: return launch_one<128, 128, 1, 3, FMT, CT, CM, DYN>(tm, p, grid, stream);
        case 1282: return launch_one<128, 128, 2, 2, FMT, CT, CM, DYN>(tm, p, grid, stream);
        default: break;
    }
    if constexpr (!DYN) {
        switch (b * 10 + groups) {
            case 160: return launch_one<16, 16, 1, 16, FMT, CT, CM, 0, 1>(tm, p, grid, stream);
            case 320: return launch_one<32, 32, 1, 8, FMT, CT, CM, 0, 1>(tm, p, grid, stream);
            case 640: return launch_one<64, 64, 1, 5, FMT, CT, CM, 0, 1>(tm, p, grid, stream);
            case 1280: return launch_one<128, 128, 1, 4, FMT, CT, CM, 0, 1>(tm, p, grid, stream);
            default: break;
        }
    }
    return cudaErrorInvalidValue;
}

// Stacked blocks (row groups): 128 rows x b; token tile 256 and four stages of 48 KB, or 128 and six of 32 KB.
template <int FMT, int CT, int CM>
cudaError_t launch_stack_shape(int b, int groups, const BcsrMaps& tm, const BcsrParams& p, int grid, cudaStream_t stream) {
    switch (b * 10 + groups) {
        case 161: return launch_one<16, 128, 1, 6, FMT, CT, CM, 0>(tm, p, grid, stream);
        case 162: return launch_one<16, 128, 2, 4, FMT, CT, CM, 0>(tm, p, grid, stream);
        case 321: return launch_one<32, 128, 1, 6, FMT, CT, CM, 0>(tm, p, grid, stream);
        case 322: return launch_one<32, 128, 2, 4, FMT, CT, CM, 0>(tm, p, grid, stream);
        case 160: return launch_one<16, 128, 1, 4, FMT, CT, CM, 0, 1>(tm, p, grid, stream);
        case 320: return launch_one<32, 128, 1, 4, FMT, CT, CM, 0, 1>(tm, p, grid, stream);
        default: break;
    }
    if constexpr (FMT != 2) {
        if (b == 64 && groups == 1) return launch_one<64, 128, 1, 6, FMT, CT, CM, 0>(tm, p, grid, stream);
        if (b == 64 && groups == 2) return launch_one<64, 128, 2, 4, FMT, CT, CM, 0>(tm, p, grid, stream);
    }
    return cudaErrorInvalidValue;
}

template <int FMT>
cudaError_t launch_stack_fmt(int b, int groups, int c16, int cm, const BcsrMaps& tm, const BcsrParams& p, int grid, cudaStream_t stream) {
    if constexpr (FMT != 2) {
        if (c16) return cm ? launch_stack_shape<FMT, 1, 1>(b, groups, tm, p, grid, stream)
                           : launch_stack_shape<FMT, 1, 0>(b, groups, tm, p, grid, stream);
    }
    if (c16) return cudaErrorInvalidValue;
    return cm ? launch_stack_shape<FMT, 0, 1>(b, groups, tm, p, grid, stream)
              : launch_stack_shape<FMT, 0, 0>(b, groups, tm, p, grid, stream);
}

// E4M3 inputs: fp32 C, static schedule; b = 32, 64 or 128 (a block row must hold at least one
// 32-element K step).  Stages are half the bytes of the 16-bit ones.
template <int CM>
cudaError_t launch_fp8(int b, int groups, const BcsrMaps& tm, const BcsrParams& p, int grid, cudaStream_t stream) {
    switch (b * 10 + groups) {
        case 321: return launch_one<32, 32, 1, 8, 3, 0, CM, 0>(tm, p, grid, stream);
        case 322: return launch_one<32, 32, 2, 10, 3, 0, CM, 0>(tm, p, grid, stream);
        case 324: return launch_one<32, 32, 4, 6, 3, 0, CM, 0>(tm, p, grid, stream);
        case 641: return launch_one<64, 64, 1, 7, 3, 0, CM, 0>(tm, p, grid, stream);
        case 642: return launch_one<64, 64, 2, 10, 3, 0, CM, 0>(tm, p, grid, stream);
        case 644: return launch_one<64, 64, 4, 5, 3, 0, CM, 0>(tm, p, grid, stream);
        case 1281: return launch_one<128, 128, 1, 6, 3, 0, CM, 0>(tm, p, grid, stream);
        case 1282: return launch_one<128, 128, 2, 4, 3, 0, CM, 0>(tm, p, grid, stream);
        default: break;
    }
    if constexpr (CM) {
        switch (b * 10 + groups) {
            case 320: return launch_one<32, 32, 1, 8, 3, 0, 1, 0, 1>(tm, p, grid, stream);
            case 640: return launch_one<64, 64, 1, 8, 3, 0, 1, 0, 1>(tm, p, grid, stream);
            case 1280: return launch_one<128, 128, 1, 8, 3, 0, 1, 0, 1>(tm, p, grid, stream);
            default: break;
        }
    }
    return cudaErrorInvalidValue;
}

// TF32 (fp32 storage): fp32 C, static schedule; the deepest rings the stage sizes allow.
template <int CM>
cudaError_t launch_tf32(int b, int groups, const BcsrMaps& tm, const BcsrParams& p, int grid, cudaStream_t stream) {
    switch (b * 10 + groups) {
        case 161: return launch_one<16, 16, 1, 5, 2, 0, CM, 0>(tm, p, grid, stream);
        case 162: return launch_one<16, 16, 2, 3, 2, 0, CM, 0>(tm, p, grid, stream);
        case 321: return launch_one<32, 32, 1, 5, 2, 0, CM, 0>(tm, p, grid, stream);
        case 322: return launch_one<32, 32, 2, 3, 2, 0, CM, 0>(tm, p, grid, stream);
        case 641: return launch_one<64, 64, 1, 8, 2, 0, CM, 0>(tm, p, grid, stream);
        case 642: return launch_one<64, 64, 2, 5, 2, 0, CM, 0>(tm, p, grid, stream);
        case 644: return launch_one<64, 64, 4, 3, 2, 0, CM, 0>(tm, p, grid, stream);
        case 1281: return launch_one<128, 128, 1, 6, 2, 0, CM, 0>(tm, p, grid, stream);
        case 1282: return launch_one<128, 128, 2, 4, 2, 0, CM, 0>(tm, p, grid, stream);
        case 320: return launch_one<32, 32, 1, 8, 2, 0, CM, 0, 1>(tm, p, grid, stream);
        case 640: return launch_one<64, 64, 1, 10, 2, 0, CM, 0, 1>(tm, p, grid, stream);
        case 1280: return launch_one<128, 128, 1, 8, 2, 0, CM, 0, 1>(tm, p, grid, stream);
        case 160: return launch_one<16, 16, 1, 10, 2, 0, CM, 0, 1>(tm, p, grid, stream);
        default: return cudaErrorInvalidValue;
    }
}

template <int FMT>
cudaError_t launch_fmt(int b, int groups, int c16, int cm, int dyn, const BcsrMaps& tm, const BcsrParams& p, int grid, cudaStream_t stream) {
    // dynamic scheduling is built for the default output (fp32, row-major) only
    if (dyn) return (c16 || cm) ? cudaErrorInvalidValue : launch_shape<FMT, 0, 0, 1>(b, groups, tm, p, grid, stream);
    if (cm) return c16 ? launch_shape<FMT, 1, 1, 0>(b, groups, tm, p, grid, stream)
                       : launch_shape<FMT, 0, 1, 0>(b, groups, tm, p, grid, stream);
    return c16 ? launch_shape<FMT, 1, 0, 0>(b, groups, tm, p, grid, stream)
               : launch_shape<FMT, 0, 0, 0>(b, groups, tm, p, grid, stream);
}

}  // namespace

// Widest token tile per block size, in 128-token groups.  b = 64 with row-major fp32 C writes
// the most bytes of C per staged operand byte: there a 256-token tile with five 40 KB stages and
// three staging tiles per epilogue warp measured 3 % faster than 512 tokens with three 72 KB
// stages and one staging tile; every other combination measured equal or slower with 256.
// TF32: elements are twice as wide, so b = 16 / 32 stop at 256 tokens (a 512-token stage of
// several blocks would not fit twice).
int bcsr_token_groups_max(int dtype, int b, int c16, int col_major) {
    if (b == 128) return 2;
    if (dtype == 2 && b <= 32) return 2;
    return (b == 64 && !c16 && !col_major) ? 2 : 4;
}

cudaError_t launch_bcsr(int dtype, int b, int groups, int c16, int col_major, int dynamic, const BcsrMaps& tm, const BcsrParams& p,
                        int grid, cudaStream_t stream) {
    if (dtype == 1) return launch_fmt<0>(b, groups, c16, col_major, dynamic, tm, p, grid, stream);   // fp16
    if (dtype == 0) return launch_fmt<1>(b, groups, c16, col_major, dynamic, tm, p, grid, stream);   // bf16
    if (dtype == 3) {
        if (c16 || dynamic) return cudaErrorInvalidValue;
        return col_major ? launch_fp8<1>(b, groups, tm, p, grid, stream)
                         : launch_fp8<0>(b, groups, tm, p, grid, stream);
    }
    if (dtype == 2) {
        if (c16 || dynamic) return cudaErrorInvalidValue;
        return col_major ? launch_tf32<1>(b, groups, tm, p, grid, stream)
                         : launch_tf32<0>(b, groups, tm, p, grid, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_bcsr_stacked(int dtype, int b, int groups, int c16, int col_major, const BcsrMaps& tm, const BcsrParams& p, int grid,
                                cudaStream_t stream) {
    if (dtype == 1) return launch_stack_fmt<0>(b, groups, c16, col_major, tm, p, grid, stream);   // fp16
    if (dtype == 0) return launch_stack_fmt<1>(b, groups, c16, col_major, tm, p, grid, stream);   // bf16
    if (dtype == 2) return launch_stack_fmt<2>(b, groups, c16, col_major, tm, p, grid, stream);   // TF32: b = 16, 32
    if (dtype == 3 && !c16 && col_major) {
        // E4M3: half the bytes per stage, deeper rings
        switch (b * 10 + groups) {
            case 321: return launch_one<32, 128, 1, 10, 3, 0, 1, 0>(tm, p, grid, stream);
            case 322: return launch_one<32, 128, 2, 8, 3, 0, 1, 0>(tm, p, grid, stream);
            case 641: return launch_one<64, 128, 1, 10, 3, 0, 1, 0>(tm, p, grid, stream);
            case 642: return launch_one<64, 128, 2, 8, 3, 0, 1, 0>(tm, p, grid, stream);
            case 320: return launch_one<32, 128, 1, 6, 3, 0, 1, 0, 1>(tm, p, grid, stream);
            default: break;
        }
    }
    return cudaErrorInvalidValue;
}

namespace {

// One CTA per (split block-row, run of 1024 four-column pieces of its b x N output); a thread sums
// four pieces over the parts, in part order (run-to-run identical results), all loads of a
// piece in flight together.
constexpr int kMergePieces = 4;
__global__ void __launch_bounds__(256) bcsr_merge_kernel(const BcsrMergeParams p) {
    const int i = blockIdx.x;
    const int I = p.row[i], first = p.first[i], nparts = p.nparts[i];
    // the partial tiles belong to the SpMM kernel launched just before on the same stream
    grid_trigger();
    grid_wait();
    const int64_t N = p.N, n4 = N >> 2;                 // N is a multiple of 4 (16-byte rows)
    const int64_t row0 = static_cast<int64_t>(I) * p.b;
    const int64_t rows = min_i64(p.b, p.m - row0);
    const int64_t total = rows * n4;
    const float4* part = reinterpret_cast<const float4*>(p.partial) + static_cast<int64_t>(first) * p.b * n4;
    float4* out = reinterpret_cast<float4*>(p.C + row0 * N);
    const int64_t slot_stride = static_cast<int64_t>(p.b) * n4;
    const int64_t e0 = static_cast<int64_t>(blockIdx.y) * (256 * kMergePieces) + threadIdx.x;
    float4 acc[kMergePieces];
#pragma unroll
    for (int k = 0; k < kMergePieces; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 0; s < nparts; ++s) {
#pragma unroll
        for (int k = 0; k < kMergePieces; ++k) {
            const int64_t e = e0 + k * 256;
            if (e < total) {
                const float4 v = __ldg(part + s * slot_stride + e);
                acc[k].x += v.x; acc[k].y += v.y; acc[k].z += v.z; acc[k].w += v.w;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < kMergePieces; ++k) {
        const int64_t e = e0 + k * 256;
        if (e < total) out[e] = acc[k];
    }
}

}  // namespace

cudaError_t launch_bcsr_merge(const BcsrMergeParams& p, cudaStream_t stream) {
    if (p.n <= 0) return cudaSuccess;
    const int64_t pieces = static_cast<int64_t>(p.b) * (p.N >> 2);
    const dim3 grid(static_cast<unsigned>(p.n), static_cast<unsigned>((pieces + 256 * kMergePieces - 1) / (256 * kMergePieces)));
    return launch_dependent(bcsr_merge_kernel, grid, 256, 0, stream, p);
}

}  // namespace spmm
