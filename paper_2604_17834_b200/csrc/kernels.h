// Launch interfaces between the C-ABI layer (api.cu) and the kernels.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace spmm {

// Launch with programmatic stream serialisation (see grid_wait in ptx.cuh).  Measured back to back: BCSR
// 512 x 512, N = 256 6.15 -> 4.25 us, 3584 x 18944 N = 128
// 14.3 -> 11.4; WCSR 4000 rows, N = 36 8.2 -> 6.5, 100,000 rows, N = 128 38.0 -> 35.1; long launches unchanged.
template <class... P, class... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// per-device caches (kernel attributes, the built-in scratch address) are arrays of this length
constexpr int kMaxDevices = 64;

struct BcsrParams {
    const int32_t* block_row_ptr;
    const int32_t* block_col_idx;
    const int4* tiles;        // {block-row, token tile, first stored block, end block}, CTA-major
    const int32_t* cta_ptr;   // [grid+1] ranges of tiles
    void* C;            // fp32 or the input's 16-bit type; [m][N], or [N][m] with column-major operands
    int64_t m, N;
    int* status;
    uint64_t wait_limit_ns;
    int32_t use_3d;     // tmB3 is valid: whole token tiles are fetched with one 3-D request
    int32_t tiles_first;        // a stage's B tiles are requested before its stored blocks (row-major whole tiles of plain blocks of 128, or of 64 with groups > 1)
    // stacked launch only: [groups][128 / b] block-rows of every row group (see BcsrStack); the
    // tile records then name {group, token tile, first stacked block, end stacked block} and
    // block_col_idx is the stacked blocks' column index
    const int32_t* stack_rows;
    // TF32 row groups: the format's own blocks and the dense operand (see plain_product in bcsr_kernel.cu)
    const int32_t* plain_col_idx;
    const float* plain_vals;
    const float* B;
    int64_t k;
    // 0: waits for the launch before it in the stream before it touches an operand (grid_wait).
    // 1: the same, and the next launch may run beside it: it is let go (grid_trigger) after that wait.
    // 2: such a next launch: it may start at once, and waits for the one before it before its CTAs exit
    int32_t overlap;
};

// dtype: 0 bf16, 1 fp16, 2 tf32 (fp32 storage; fp32 C, static schedule), 3 E4M3 (column-major
// operands, fp32 C).  groups: token tile = 128 * groups columns of B (1, 2 or 4).
// c16: C in the input's 16-bit type.  With es = bytes per element, t = 128 / es tokens per
// 128-byte box row and kb = b / bcsr_k_split(b, es) rows of B per stage unit --
// row-major operands: map B = B as [k][N], box kb x t; B3 = B as [N / t][k][t], box
// (es * groups) x kb x t; 128-byte swizzle (with 32-byte atoms for es = 4).  Column-major operands
// (col_major): B = X as [N][k], box 128 tokens x min(kb * es, 128) bytes; B3 = X as
// [N / 128][128][k], box groups x 128 x the same; both with the swizzle of that row length.
// A: the stored blocks as [blocks * b][b], box (b * bcsr_blocks_per_stage) rows x min(kb * es, 128) bytes.
// A0: A as wider tiles have it, fewer blocks to a box (read by 128-token tiles whose stages hold more).
// C: C as [m][N], box 32 x bcsr_epi_cols, no swizzle; or fp32 Y as [N][m], box 16 x 32, 64-byte swizzle (16-bit Y: not
// read, it is stored without a map).
// P: K-split, the partial tiles as [slots * b][N] fp32, box as C's (the tile record of a part holds -1 - slot in place of the
// block-row); C where the plan has no parts.
// dynamic: the grid is one CTA per tile (grid = number of tiles, p.tiles in the schedule's global
// order, p.cta_ptr unused) and CTAs steal tiles through Cluster Launch Control; fp32 row-major only.
struct BcsrMaps { CUtensorMap A, A0, B, B3, C, P; };
cudaError_t launch_bcsr(int dtype, int b, int groups, int c16, int col_major, int dynamic, const BcsrMaps& tm, const BcsrParams& p,
                        int grid, cudaStream_t stream);
// Row groups: the same kernel with 128 x b stacked blocks (MMA N = 128) and a 256-token tile (groups = 2), or a
// 128-token one (groups = 1; see ensure_schedule).
// A: the stacked values as [blocks * 128][b], box 128 x b; B3 built for `groups`; b = 16, 32, 64 (tf32: 16, 32).
// `groups` of a launch by half tiles (both kinds of launch): the lists of a 128-token schedule, two CTAs to each, with 64 of
// its tiles' tokens in either (C: boxes of 16 tokens instead of 32; column-major B: box of 64 tokens; E4M3: column-major
// operands only) or, for stacked blocks of b = 16 and 32, 64 of their rows (A: box of 64 rows).
constexpr int kSplitGroups = 0;
constexpr int kStackRows = 128;
constexpr int kStackGroups = 2;
cudaError_t launch_bcsr_stacked(int dtype, int b, int groups, int c16, int col_major, const BcsrMaps& tm, const BcsrParams& p,
                                int grid, cudaStream_t stream);
// K-split, the merge: C rows of every split block-row = sum of its parts' partial tiles in part order.
struct BcsrMergeParams {
    const int32_t* row;      // [n] split block-rows
    const int32_t* first;    // first slot
    const int32_t* nparts;
    const float* partial;    // [slots][b][N]
    float* C;                // [m][N]
    int64_t m, N;
    int32_t n, b;
};
cudaError_t launch_bcsr_merge(const BcsrMergeParams& p, cudaStream_t stream);
int bcsr_token_groups_max(int dtype, int b, int c16, int col_major);
// Accumulator columns (= rows of A's block) an epilogue warp handles at a time: it stages them
// in a 2 KB (1 KB for b = 16 with 16-bit C) shared-memory tile and stores the tile with one TMA
// request whose box is 32 tokens x this many rows (row-major C) or this many columns x 32 tokens
// (column-major fp32 Y).  Larger tiles (up to 64 rows) were measured slower: the stage ring needs the room.
constexpr int bcsr_epi_cols(int b, bool c16, bool col_major) { return (b < 32 || !c16) ? 16 : 32; }
// stored blocks that share one pipeline stage (and one A request): 4 / 2 / 1 for b = 16 / 32 / 64 and more; twice as many
// for b = 32 and 64 with tiles of 128 tokens (groups <= 1) and up to 2-byte values, see BcsrCfg::kBps
constexpr int bcsr_blocks_per_stage(int b, int es, int groups) {
    return (b == 16 ? 4 : (b == 32 ? 2 : 1)) * (groups <= 1 && es <= 2 && (b == 32 || b == 64) ? 2 : 1);
}
// stacked blocks (row groups) per stage: 4 / 2 / 1 blocks; 4-byte values are twice as wide
constexpr int bcsr_stacked_per_stage(int b, int es) { return bcsr_blocks_per_stage(b, es, 2) / (es == 4 ? 2 : 1); }
// Column slices a stored block is cut into, one pipeline stage each: blocks of 4-byte elements
// with rows longer than 128 bytes (TF32, b = 64 / 128) go through the ring 32 columns at a time;
// every other block is one unit.
constexpr int bcsr_k_split(int b, int es) { return (es == 4 && b > 32) ? b / 32 : 1; }

// WCSR pipeline shape, shared by the host schedule (fills are cut to the stage size) and the
// kernel.  A stage holds 128 / es columns (64 of a 2-byte type, 32 of TF32) of one 128-token
// tile: 16 KB of gathered B rows + the A tile (2 KB at window height 16, 8 KB at 64).  Per value
// size and window height: ring depth, producer warps (each owns STAGES / PW stages) and resident
// CTAs per SM, which is also the number of bins per SM of the static schedule (every resident
// CTA walks one bin).  Measured on B200 at height 16: 2-byte types run fastest as three small
// CTAs per SM (4 stages, 4 producer warps), TF32 as two deeper ones (6 stages, 6 producer warps);
// both fill the SM's shared memory.  Height 64: two CTAs per SM, 4 stages of 24 KB, 4 producer
// warps (the accumulators of two CTAs fill the 512 TMEM columns).
#ifndef WCSR_STAGE_ROW_BYTES
#define WCSR_STAGE_ROW_BYTES 128
#endif
constexpr int wcsr_stage_cols(int es) { return WCSR_STAGE_ROW_BYTES / es; }
// Narrow dense operands (2-byte types, window height 16, N <= 64): a gathered row is one 128-byte
// segment instead of two, so a stage of the same size class holds 96 columns (12 KB of rows +
// 3 KB of A): a third fewer stage hand-shakes per column, which is what bounds the narrow case.
constexpr int kWcsrNarrowCols = 96;
constexpr int kWcsrNarrowMaxN = 64;
constexpr int wcsr_stages(int es, int wh) { return wh == 64 ? 4 : (es == 4 ? 6 : 4); }
constexpr int wcsr_producer_warps(int es, int wh) { return wh == 64 ? 4 : (es == 4 ? 6 : 4); }
constexpr int wcsr_bins_per_sm(int es, int wh) { return wh == 64 ? 2 : (es == 4 ? 2 : 3); }

// Device task descriptor of the WCSR kernel (one per sub-task of the split plan).
struct WcsrDevTask {
    int32_t col_begin;   // absolute position of the task's first padded column
    int32_t count;       // columns (multiple of b_col)
    int32_t window;
    int32_t slot;        // partial tile index, or -1: write C directly
};

struct WcsrParams {
    const int32_t* bin_ptr;      // [n_bins+1] ranges of items
    const int4* items;           // {window, partial slot or -1, columns, 0} of every task, bin-major
    const int2* fills;           // {first padded column, count | first<<16 | last<<17}, bin-major (cut to the launch's stage size)
    const int32_t* bin_fill;     // [n_bins+1] fill ranges
    const int32_t* col_idx;      // window_col_idx [P]
    const uint8_t* grp_class;    // reuse class of every four padded columns [P / 4], or null: no gather hints
    int32_t hot_min;             // groups of this class and above are gathered with the evict-last priority
    int32_t hint_flags;          // 1: the packed A tiles are fetched evict-first
    const uint8_t* packed;       // packed A values
    const void* B;               // k x N row-major
    void* C;                     // [m][N] fp32, or the input's 16-bit type
    float* partial;              // [n_slots][window height][N]
    int64_t m, N;
    int32_t n_bins;
    int32_t n_tt;                // token tiles = ceil(N / (128 * groups))
    int* status;
    uint64_t wait_limit_ns;
};

// dtype: 0 bf16, 1 fp16, 2 tf32, 3 E4M3 (fp32 C).  tmB: 2-D map of B (k rows x N), box = 128
// bytes x 1 row, 128-byte swizzle (32-byte atoms for tf32), used in row-gather mode.
// narrow: the N <= 64 variant for 2-byte types at window height 16 (p.fills / p.bin_fill cut to kWcsrNarrowCols).
// lsu_gather: the comparison variant whose producers gather B rows with 16-byte cp.async copies through the
// load/store units instead of TMA (window height 16, fp32 C, not narrow); tmB is then unused.
cudaError_t launch_wcsr(int dtype, int wh, int c16, int narrow, int lsu_gather, const CUtensorMap& tmB, const WcsrParams& p,
                        int sms, cudaStream_t stream);

struct MergeParams {
    const int32_t* window;   // [n] windows the merge writes
    const int32_t* first;    // first slot or -1
    const int32_t* nparts;   // slots to add (0 = zero fill)
    const float* partial;
    void* C;
    int64_t m, N;
    int32_t n;
};
cudaError_t launch_wcsr_merge(const MergeParams& p, int wh, int ctype, cudaStream_t stream);   // ctype: 0 fp32, 1 fp16, 2 bf16

// WCSR product from the row stream (wcsr_rows_kernel.cu; the stream: WcsrRowStream in format.h).
struct WcsrRowsParams {
    const int4* tasks;           // [n_tasks] {first entry, entries, position in order of the first row, 0}
    const int4* parts;           // [n_parts] {first entry, entries, long row, part}: one CTA per column tile, first in the grid
    const int4* longs;           // [long rows] {row, first partial slot, parts, 0}
    const int32_t* order;        // rows in task order
    const int32_t* col;          // entries: column, sign bit = last of its row, 0x7fffffff = no gather
    const uint8_t* val;
    unsigned* counters;          // [long rows][kRowsMaxTiles], zero between launches
    float* partial;              // [slots][tiles of the launch][tile columns]
    const uint8_t* zeros;        // 32 zero bytes
    const void* B;
    void* C;
    int64_t N;
    int32_t n_tasks, n_parts;
    int32_t lanes, groups, tile0;    // set by launch_wcsr_rows
};
constexpr int kRowsThreads = 128;
constexpr int kRowsMaxTiles = 8;     // column tiles one launch covers at most
// How a dense width is cut: a column tile is lanes vectors of vec bytes (a group of lanes).
struct RowsShape { int vec, lanes, tiles, tile_cols; };
// aligned32: every row of B and of C starts on a 32-byte boundary.
RowsShape wcsr_rows_shape(int64_t N, int es, bool aligned32);
// bf16, fp16, tf32; threads: kRowsThreads or 256; plain: tf32 in 16-byte vectors only, see wcsr_rows_kernel.  Column tiles [tile0, tile0 + tiles), at most kRowsMaxTiles of them.
cudaError_t launch_wcsr_rows(int dtype, int c16, const RowsShape& s, WcsrRowsParams p, int tile0, int tiles, int threads, bool plain, cudaStream_t stream);

// In the row kernel's place where the wait limit is zero, which makes the kernels that wait give up at their first wait:
// the row kernel waits for nothing, and this reports to `status` what they would.
cudaError_t launch_wcsr_rows_give_up(int* status, cudaStream_t stream);

// Device address and size in bytes of the library's built-in partial-tile scratch on the
// current device (resolved on the first call per device).
cudaError_t wcsr_static_scratch(float** ptr, size_t* bytes);

}  // namespace spmm
