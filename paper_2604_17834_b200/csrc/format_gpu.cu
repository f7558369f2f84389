// GPU-side construction of the BCSR format (Sec. 2.3) from a CSR matrix that already lives in
// device memory: block mask and index (which (I, J) blocks hold a stored entry, block columns
// ascending inside a block-row) and value packing into zero-filled b x b tiles.  Same arrays,
// bit for bit, as the host builder in format.cpp.
//
// One CTA per block-row.  The entries of a block-row are one contiguous range of the CSR
// arrays (rows I*b .. I*b + b - 1), and its block columns are collected in a shared-memory
// bitmap of ceil(k / b) bits:
//   count pass   bitmap -> number of stored blocks of the block-row
//   scan         exclusive prefix sum over block-rows -> block_row_ptr
//   fill pass    bitmap again, prefix popcounts over its words -> block_col_idx (ascending by
//                construction) and the slot of every entry's block; values scattered into
//                blocks[slot][row in block][column in block]
// A bitmap needs 2 * ceil(k / b) / 8 bytes of shared memory (bits + word prefix), at most 200 KB:
// k / b <= 819,200.
//
// WCSR (window condensation of Sec. 2.3): a window's entries are one contiguous range of the CSR arrays, wh ascending
// runs.  A short window is sorted by one warp in registers, a longer one goes through a bitmap of its columns or, where
// the matrix is too wide for that, is merged run by run in shared memory; one too long for that is cut into pieces by
// column, which go either way, a CTA each.  An entry gets its place among the window's distinct columns.  A prefix sum of the lengths padded to b_col is window_row_ptr; a last pass, entry by entry, writes the
// columns over a -1 fill and the values straight into the packed tile layout.
#include <cstring>
#include <numeric>
#include <type_traits>
#include <algorithm>
#include <new>

#include "device_memory.h"
#include "format.h"
#include "kernels.h"
#include "ptx.cuh"
#include "spmm_b200.h"

namespace spmm {

namespace {

constexpr int kThreads = 256;

// Which of its kernels condenses a window of n entries (below: sort_window, bitmap_window, merge_window).  The bitmap of a
// window costs about a word per 32 columns of the matrix, so short windows of a wide matrix are merged instead, up to
// what fits shared memory.
constexpr int kWarpWindow = 256, kMergeWindow = 2048, kLargeWindow = 18432;
constexpr int kColumnsPerEntry = 256;        // a bitmap from one entry per that many columns on
enum { kListBitmap, kListMerge, kListLarge, kLists };
constexpr int kMostBitmap = 216 * 1024;      // bits and their prefixes, 8 bytes per 32 columns
constexpr int64_t kBitmapColumns = kMostBitmap / 8 * 32;
static_assert(kLargeWindow * 12 <= kMostBitmap, "the merging kernels' shared memory");
// Windows of more than kLargeWindow entries are cut into pieces of about kPiece, at columns chosen so that no piece holds more
// than kPieceCap (wcsr_cut_windows_kernel), unless a bitmap reads no more than kBitmapReads entries for them: the four launches
// for the pieces cost a small handle about as much as that (R-MAT 2^15, 24 a row, all windows above 18,432 entries cut:
// 254 -> 267 us).
constexpr int kBitmapReads = 48 * 1024;
constexpr int kPiece = 4032, kPieceSlack = 512, kPieceCap = kPiece + kPieceSlack + 64;
__host__ __device__ constexpr int64_t pieces_of(int64_t n) { return (n + kPiece - 1) / kPiece; }
constexpr int64_t kMostLong = (int64_t{1} << 31) / kLargeWindow + 1;      // windows there can be, with less than 2^31 entries
constexpr int kLongShift = 40;               // a count of windows above this bit, of their pieces below it
struct WindowLists {
    int wh;                                  // 0: no lists are wanted
    int64_t k;
    int32_t* list[kLists];                   // kListBitmap: its first place; the others are filled from their last place down
    int* count;                              // [kLists], zero before
    int32_t *long_window, *long_first;       // [max_long] the windows that are cut, and their first pieces
    unsigned long long* long_count;          // both counts in one, zero before: the first pieces ascend with the windows' places
    int64_t max_long;
    int64_t long_from;                       // they have that many entries and more
    __device__ __forceinline__ int which(int64_t n) const {                  // kLists: it is cut
        if (n >= long_from) return kLists;
        if (n * kColumnsPerEntry >= k) return kListBitmap;
        return n <= kMergeWindow ? kListMerge : kListLarge;
    }
};

// Validation in two passes, so that the second one never reads past the arrays: once row_ptr is
// known to start at 0 and to be monotone, every position below row_ptr[m] lies inside col_idx.
// (nnz: receives row_ptr[m] where the caller reads it together with *err; may be null.  longer, where not null: lists
// of the windows of wh rows that one warp does not condense, see WindowLists.)
__global__ void csr_check_rows_kernel(int64_t m, const int64_t* row_ptr, int* err, int64_t* nnz, const WindowLists longer) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (row_ptr[0] != 0) atomicMin(err, SPMM_ERR_INVALID_ARG);
        if (nnz) *nnz = row_ptr[m];
    }
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < m;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        if (row_ptr[i + 1] < row_ptr[i]) atomicMin(err, SPMM_ERR_INVALID_ARG);
        if (longer.wh && i % longer.wh == 0) {
            const int64_t n = row_ptr[min(i + longer.wh, m)] - row_ptr[i];
            if (n <= kWarpWindow) continue;
            const int which = longer.which(n);
            if (which < kLists) {
                // (chosen, not indexed: an index puts the parameters on the stack.  400,000 power-law rows: 8.9 -> 5.5 us)
                int32_t* const list = which == kListBitmap ? longer.list[kListBitmap] : which == kListMerge ? longer.list[kListMerge] : longer.list[kListLarge];
                const int at = atomicAdd(longer.count + which, 1);
                list[which == kListBitmap ? at : -at] = static_cast<int32_t>(i / longer.wh);
            } else if (n < (int64_t{1} << 31)) {
                const unsigned long long one = 1ull << kLongShift, before = atomicAdd(longer.long_count, one + static_cast<unsigned long long>(pieces_of(n)));
                const int64_t at = static_cast<int64_t>(before >> kLongShift);
                if (at < longer.max_long) {              // (not so with a row_ptr that is refused)
                    longer.long_window[at] = static_cast<int32_t>(i / longer.wh);
                    longer.long_first[at] = static_cast<int32_t>(before & (one - 1));
                }
            }
        }
    }
}

__global__ void csr_check_cols_kernel(int64_t m, int64_t k, const int64_t* row_ptr, const int32_t* col_idx, int* err) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < m;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int64_t prev = -1;
        for (int64_t p = row_ptr[i]; p < row_ptr[i + 1]; ++p) {
            const int64_t c = col_idx[p];
            if (c < 0 || c >= k) { atomicMin(err, SPMM_ERR_OUT_OF_RANGE); break; }
            if (c <= prev) { atomicMin(err, SPMM_ERR_UNSORTED); break; }
            prev = c;
        }
    }
}

// The same rules entry by entry, whatever the row lengths (a row of 5000 entries kept one thread of the kernel
// above busy for 140 us): *bad is set when any entry breaks one; the row-wise kernel then finds the error code.
// A column that does not ascend must be the first of its row: its position is looked up in row_ptr.
__global__ void csr_check_entries_kernel(int64_t m, int64_t k, const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx, int* bad) {
    const int64_t nnz = row_ptr[m];
    for (int64_t p = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; p < nnz;
         p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t c = col_idx[p];
        bool ok = c >= 0 && c < k;
        if (ok && p > 0 && c <= col_idx[p - 1]) {
            int64_t lo = 0, hi = m;                      // first row that starts at or behind p
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (row_ptr[mid] < p) lo = mid + 1; else hi = mid;
            }
            ok = row_ptr[lo] == p;
        }
        if (!ok) *bad = 1;
    }
}

// Checks the columns of a CSR matrix whose row pointers are known to be sound; synchronises `st`.
int check_csr_cols(int64_t m, int64_t k, int64_t nnz, const int64_t* d_row_ptr, const int32_t* d_col_idx, int* d_bad, int* d_err, cudaStream_t st) {
    const unsigned entry_grid = static_cast<unsigned>(std::min<int64_t>((nnz + 255) / 256, 8192));
    csr_check_entries_kernel<<<entry_grid, 256, 0, st>>>(m, k, d_row_ptr, d_col_idx, d_bad);
    int bad = 0, err = 0;
    if (cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return SPMM_ERR_CUDA;
    if (!bad) return SPMM_OK;
    csr_check_cols_kernel<<<static_cast<unsigned>(std::min<int64_t>((m + 255) / 256, 2048)), 256, 0, st>>>(m, k, d_row_ptr, d_col_idx, d_err);
    if (cudaMemcpyAsync(&err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return SPMM_ERR_CUDA;
    return err;
}

// Shared-memory bitmap of the block columns of block-row I.
__device__ __forceinline__ void mark_block_columns(uint32_t* bits, int words, int64_t I, int64_t m, int b,
                                                   const int64_t* row_ptr, const int32_t* col_idx) {
    for (int w = threadIdx.x; w < words; w += blockDim.x) bits[w] = 0u;
    __syncthreads();
    const int64_t r1 = (I + 1) * b < m ? (I + 1) * b : m;
    const int64_t p0 = row_ptr[I * b], p1 = row_ptr[r1];
    for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        const int J = col_idx[p] / b;
        atomicOr(&bits[J >> 5], 1u << (J & 31));
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kThreads)
bcsr_count_kernel(int64_t m, int b, int words, const int64_t* row_ptr, const int32_t* col_idx, int32_t* counts) {
    extern __shared__ uint32_t smem[];
    __shared__ int total;
    if (threadIdx.x == 0) total = 0;
    mark_block_columns(smem, words, blockIdx.x, m, b, row_ptr, col_idx);
    int n = 0;
    for (int w = threadIdx.x; w < words; w += blockDim.x) n += __popc(smem[w]);
    for (int o = 16; o > 0; o >>= 1) n += __shfl_down_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(&total, n);
    __syncthreads();
    if (threadIdx.x == 0) counts[blockIdx.x] = total;
}

// Exclusive sums over a CTA of THREADS threads, one value each; *total gets the sum of all.  scratch: 32 values.
template <int THREADS = 1024>
__device__ __forceinline__ long long block_exclusive_sum(long long v, long long* scratch, long long* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();                         // (the scratch may still be read from the call before)
    if (lane == 31) scratch[warp] = x;
    __syncthreads();
    if (warp == 0) {
        long long t = lane < THREADS / 32 ? scratch[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        scratch[lane] = t;
    }
    __syncthreads();
    *total = scratch[31];
    return (warp ? scratch[warp - 1] : 0) + x - v;
}

// out[0] = 0, out[i + 1] = c[0] + ... + c[i] with every count rounded up to a multiple of `unit`; *overflow set if the
// total passes int32.  One CTA of 1024 threads, eight counts a thread and step.
__device__ __forceinline__ void scan_counts(const int32_t* counts, int64_t n, int unit, int32_t* out, int* overflow) {
    __shared__ long long scratch[32];
    constexpr int kPer = 8;
    long long carry = 0;
    if (threadIdx.x == 0) out[0] = 0;
    for (int64_t base = 0; base < n; base += 1024 * kPer) {
        const int64_t i0 = base + static_cast<int64_t>(threadIdx.x) * kPer;
        int c[kPer];
        long long sum = 0, total;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            c[j] = i0 + j < n ? (counts[i0 + j] + unit - 1) / unit * unit : 0;
            sum += c[j];
        }
        long long at = carry + block_exclusive_sum(sum, scratch, &total);
        carry += total;
        if (at + sum >= (1ll << 31)) *overflow = 1;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            at += c[j];
            if (i0 + j < n) out[i0 + j + 1] = static_cast<int32_t>(at);
        }
    }
}

__global__ void __launch_bounds__(1024) exclusive_scan_kernel(const int32_t* counts, int64_t n, int32_t* out, int* overflow) {
    scan_counts(counts, n, 1, out, overflow);
}

template <int ES>
__global__ void __launch_bounds__(kThreads)
bcsr_fill_kernel(int64_t m, int b, int words, const int64_t* row_ptr, const int32_t* col_idx, const uint8_t* vals,
                 const int32_t* block_row_ptr, int32_t* block_col_idx, uint8_t* blocks) {
    extern __shared__ uint32_t smem[];
    uint32_t* bits = smem;
    uint32_t* prefix = smem + words;         // set bits in the words before this one
    __shared__ int warp_sum[kThreads / 32];
    __shared__ int carry;
    const int64_t I = blockIdx.x;
    mark_block_columns(bits, words, I, m, b, row_ptr, col_idx);
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int base = 0; base < words; base += blockDim.x) {
        const int w = base + threadIdx.x;
        const int v = w < words ? __popc(bits[w]) : 0;
        int x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        if (warp == 0 && lane < kThreads / 32) {
            int s = warp_sum[lane];
            for (int o = 1; o < kThreads / 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffu, s, o);
                if (lane >= o) s += y;
            }
            warp_sum[lane] = s;
        }
        __syncthreads();
        const int incl = carry + (warp ? warp_sum[warp - 1] : 0) + x;
        if (w < words) prefix[w] = static_cast<uint32_t>(incl - v);
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = incl;
        __syncthreads();
    }
    const int32_t slot0 = block_row_ptr[I];
    // block columns, ascending: word by word, bit by bit
    for (int w = threadIdx.x; w < words; w += blockDim.x) {
        uint32_t x = bits[w];
        int32_t pos = slot0 + static_cast<int32_t>(prefix[w]);
        while (x) {
            const int bit = __ffs(x) - 1;
            block_col_idx[pos++] = w * 32 + bit;
            x &= x - 1;
        }
    }
    // values: one warp per row of the block-row
    const int64_t r1 = (I + 1) * b < m ? (I + 1) * b : m;
    const size_t tile_bytes = static_cast<size_t>(b) * b * ES;
    for (int64_t i = I * b + warp; i < r1; i += kThreads / 32) {
        const int64_t p0 = row_ptr[i], p1 = row_ptr[i + 1];
        for (int64_t p = p0 + lane; p < p1; p += 32) {
            const int c = col_idx[p];
            const int J = c / b;
            const uint32_t below = bits[J >> 5] & ((1u << (J & 31)) - 1u);
            const size_t slot = static_cast<size_t>(slot0) + prefix[J >> 5] + __popc(below);
            uint8_t* dst = blocks + slot * tile_bytes + (static_cast<size_t>(i - I * b) * b + (c - J * b)) * ES;
            const uint8_t* src = vals + static_cast<size_t>(p) * ES;
            if constexpr (ES == 1) *dst = *src;
            else if constexpr (ES == 2) *reinterpret_cast<uint16_t*>(dst) = *reinterpret_cast<const uint16_t*>(src);
            else *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(src);
        }
    }
}

}  // namespace

void finish_bcsr_host(BcsrHost* out) {
    const int64_t nbr = out->nbr;
    std::vector<uint8_t> col_used(static_cast<size_t>(out->nbc), 0);
    for (int32_t J : out->block_col_idx) col_used[J] = 1;
    out->distinct_bcols = std::count(col_used.begin(), col_used.end(), uint8_t{1});
    out->row_order.resize(static_cast<size_t>(nbr));
    std::iota(out->row_order.begin(), out->row_order.end(), 0);
    std::stable_sort(out->row_order.begin(), out->row_order.end(), [&](int32_t x, int32_t y) {
        const int32_t lx = out->block_row_ptr[x + 1] - out->block_row_ptr[x];
        const int32_t ly = out->block_row_ptr[y + 1] - out->block_row_ptr[y];
        return lx > ly;
    });
    out->n_empty = 0;
    for (int64_t I = 0; I < nbr; ++I)
        if (out->block_row_ptr[I + 1] == out->block_row_ptr[I]) out->n_empty++;
}

// One thread per 16-byte piece of the stacked values: sub-block r of stacked block s is stored
// block src[s][r] (b x b, row-major) or zeros.
__global__ void bcsr_stack_kernel(const uint4* __restrict__ blocks, const int32_t* __restrict__ src, uint4* __restrict__ out,
                                  int R, int pieces_per_block, int64_t n_pieces) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n_pieces) return;
    const int64_t sub = i / pieces_per_block;          // = s * R + r
    const int piece = static_cast<int>(i % pieces_per_block);
    const int32_t p = __ldg(src + sub);
    out[i] = p >= 0 ? __ldg(blocks + static_cast<int64_t>(p) * pieces_per_block + piece) : make_uint4(0u, 0u, 0u, 0u);
    (void)R;
}

int stack_bcsr_device(const uint8_t* d_blocks, const BcsrStack& st, int b, int es, uint8_t** d_stacked) {
    *d_stacked = nullptr;
    if (st.ns == 0) return SPMM_OK;
    const int pieces = b * b * es / 16;
    const int64_t n_pieces = st.ns * st.R * pieces;
    int32_t* d_src = nullptr;
    if (!dev_alloc_ok(&d_src, st.src.size() * 4, nullptr)) return SPMM_ERR_ALLOC;
    if (!dev_alloc_ok(d_stacked, static_cast<size_t>(n_pieces) * 16, nullptr)) {
        dev_free(d_src, nullptr);
        return SPMM_ERR_ALLOC;
    }
    int rc = SPMM_OK;
    if (cudaMemcpy(d_src, st.src.data(), st.src.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess) rc = SPMM_ERR_CUDA;
    if (!rc) {
        const int threads = 256;
        const int64_t grid = (n_pieces + threads - 1) / threads;
        bcsr_stack_kernel<<<static_cast<unsigned>(grid), threads>>>(reinterpret_cast<const uint4*>(d_blocks), d_src,
                                                                   reinterpret_cast<uint4*>(*d_stacked), st.R, pieces, n_pieces);
        if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) rc = SPMM_ERR_CUDA;
    }
    if (rc) cudaGetLastError();
    dev_free(d_src, nullptr);
    if (rc) { dev_free(*d_stacked, nullptr); *d_stacked = nullptr; }
    return rc;
}

int build_bcsr_device(int64_t m, int64_t k, const int64_t* d_row_ptr, const int32_t* d_col_idx, const uint8_t* d_vals,
                      int es, int b, cudaStream_t st, BcsrHost* out, int64_t* nnz_out, int32_t** d_block_row_ptr,
                      int32_t** d_block_col_idx, uint8_t** d_blocks) {
    if (b != 16 && b != 32 && b != 64 && b != 128) return SPMM_ERR_UNSUPPORTED;
    if (es != 1 && es != 2 && es != 4) return SPMM_ERR_UNSUPPORTED;
    if (m < 0 || k < 0 || !d_row_ptr) return SPMM_ERR_INVALID_ARG;
    const int64_t nbr = (m + b - 1) / b, nbc = (k + b - 1) / b;
    const int words = static_cast<int>((nbc + 31) / 32);
    const size_t smem = static_cast<size_t>(2) * (words > 0 ? words : 1) * 4;
    constexpr int kMostSmem = 200 * 1024;
    if (smem > kMostSmem) return SPMM_ERR_TOO_LARGE;
    *d_block_row_ptr = nullptr;
    *d_block_col_idx = nullptr;
    *d_blocks = nullptr;
    out->b = b;
    out->nbr = nbr;
    out->nbc = nbc;
    out->block_row_ptr.assign(static_cast<size_t>(nbr) + 1, 0);        // (may throw: before anything is held on the device)

    int* d_flags = nullptr;                     // [0] CSR error code (min), [1] scan overflow, [2] a bad entry
    int32_t* d_counts = nullptr;
    auto fail = [&](int code) {
        cudaGetLastError();                  // (of a call that failed: not for a later check to find)
        dev_free(d_flags, st);
        dev_free(d_counts, st);
        dev_free(*d_block_row_ptr, st);
        dev_free(*d_block_col_idx, st);
        dev_free(*d_blocks, st);
        *d_block_row_ptr = nullptr;
        *d_block_col_idx = nullptr;
        *d_blocks = nullptr;
        return code;
    };
    if (!dev_alloc_ok(&d_flags, 4 * sizeof(int), st)) return fail(SPMM_ERR_ALLOC);
    if (cudaMemsetAsync(d_flags, 0, 4 * sizeof(int), st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    if (!dev_alloc_ok(&d_counts, static_cast<size_t>(nbr + 1) * 4, st)) return fail(SPMM_ERR_ALLOC);
    if (!dev_alloc_ok(d_block_row_ptr, static_cast<size_t>(nbr + 1) * 4, st)) return fail(SPMM_ERR_ALLOC);

    // 1. the CSR must be canonical (the count and fill passes rely on in-range columns)
    int64_t nnz = 0;
    int flags[2] = {0, 0};
    const unsigned check_grid = static_cast<unsigned>(std::min<int64_t>((m + 255) / 256, 2048));
    if (m > 0) {
        csr_check_rows_kernel<<<check_grid, 256, 0, st>>>(m, d_row_ptr, d_flags, nullptr, WindowLists{});
        if (cudaMemcpyAsync(&nnz, d_row_ptr + m, sizeof(int64_t), cudaMemcpyDeviceToHost, st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    }
    if (cudaMemcpyAsync(flags, d_flags, sizeof(flags), cudaMemcpyDeviceToHost, st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    if (cudaStreamSynchronize(st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    if (flags[0] != 0) return fail(flags[0]);
    if (nnz < 0 || (nnz > 0 && (!d_col_idx || !d_vals))) return fail(SPMM_ERR_INVALID_ARG);
    if (nnz > 0) {
        if (int rc = check_csr_cols(m, k, nnz, d_row_ptr, d_col_idx, d_flags + 2, d_flags, st)) return fail(rc);
    }
    *nnz_out = nnz;

    // 2. stored blocks per block-row, 3. block_row_ptr
    if (smem > 48 * 1024) {                  // (the most there may be: threads that build for other widths set it too)
        cudaFuncSetAttribute(bcsr_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem);
        cudaFuncSetAttribute(bcsr_fill_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem);
        cudaFuncSetAttribute(bcsr_fill_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem);
        cudaFuncSetAttribute(bcsr_fill_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem);
    }
    if (nbr > 0) bcsr_count_kernel<<<static_cast<unsigned>(nbr), kThreads, smem, st>>>(m, b, words, d_row_ptr, d_col_idx, d_counts);
    exclusive_scan_kernel<<<1, 1024, 0, st>>>(d_counts, nbr, *d_block_row_ptr, d_flags + 1);
    if (cudaMemcpyAsync(out->block_row_ptr.data(), *d_block_row_ptr, static_cast<size_t>(nbr + 1) * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return fail(SPMM_ERR_CUDA);
    if (cudaMemcpyAsync(flags, d_flags, sizeof(flags), cudaMemcpyDeviceToHost, st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    if (cudaStreamSynchronize(st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    if (flags[1]) return fail(SPMM_ERR_TOO_LARGE);
    const int64_t nnzb = out->block_row_ptr[static_cast<size_t>(nbr)];
    out->nnzb = nnzb;

    // 4. block columns and values
    const size_t tile_bytes = static_cast<size_t>(b) * b * es;
    const size_t idx_bytes = static_cast<size_t>(nnzb) * 4, val_bytes = static_cast<size_t>(nnzb) * tile_bytes;
    if (!dev_alloc_ok(d_block_col_idx, idx_bytes ? idx_bytes : 16, st)) return fail(SPMM_ERR_ALLOC);
    if (!dev_alloc_ok(d_blocks, val_bytes ? val_bytes : 16, st)) return fail(SPMM_ERR_ALLOC);
    if (val_bytes && cudaMemsetAsync(*d_blocks, 0, val_bytes, st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    if (nbr > 0 && nnzb > 0) {
        if (es == 1)
            bcsr_fill_kernel<1><<<static_cast<unsigned>(nbr), kThreads, smem, st>>>(m, b, words, d_row_ptr, d_col_idx, d_vals, *d_block_row_ptr, *d_block_col_idx, *d_blocks);
        else if (es == 4)
            bcsr_fill_kernel<4><<<static_cast<unsigned>(nbr), kThreads, smem, st>>>(m, b, words, d_row_ptr, d_col_idx, d_vals, *d_block_row_ptr, *d_block_col_idx, *d_blocks);
        else
            bcsr_fill_kernel<2><<<static_cast<unsigned>(nbr), kThreads, smem, st>>>(m, b, words, d_row_ptr, d_col_idx, d_vals, *d_block_row_ptr, *d_block_col_idx, *d_blocks);
    }
    try {
        out->block_col_idx.assign(static_cast<size_t>(nnzb), 0);
    } catch (const std::bad_alloc&) {
        return fail(SPMM_ERR_ALLOC);
    }
    if (nnzb && cudaMemcpyAsync(out->block_col_idx.data(), *d_block_col_idx, idx_bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return fail(SPMM_ERR_CUDA);
    if (cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess) return fail(SPMM_ERR_CUDA);
    dev_free(d_flags, st);
    dev_free(d_counts, st);
    finish_bcsr_host(out);       // row order, empty block-rows, distinct block columns: host, from the index arrays
    return SPMM_OK;
}

namespace {

// ---- window condensation
// Per entry: its row, and its place among the window's condensed columns; per window: how many it has; per column: how
// many windows hold it.  An entry out of range or not ascending in its row sets *bad and counts as column 0; nothing
// below leaves its arrays then, and the results are not used.
struct CondenseParams {
    int64_t m, k, nwin;
    const int64_t* row_ptr;
    const int32_t* col_idx;
    int32_t* row_of;                         // [nnz]
    int32_t* pos_of;                         // [nnz]
    int32_t* ucount;                         // [nwin]
    int32_t* refs;                           // [k], zero before
    int* bad;
    const int32_t* list;                     // the windows of this launch, where it does not go over all
};

__device__ __forceinline__ int32_t checked_column(const CondenseParams& p, int64_t at, int64_t row_start) {
    const int32_t c = p.col_idx[at];
    if (c < 0 || c >= p.k || (at > row_start && p.col_idx[at - 1] >= c)) {
        *p.bad = 1;
        return 0;
    }
    return c;
}

// off[0 .. rows]: where the rows of the window start, relative to its first entry.
template <int WH>
__device__ __forceinline__ int row_in_window(const int* off, int j) {
    int r = 0;                               // the last row that starts at or before entry j
#pragma unroll
    for (int step = WH / 2; step > 0; step >>= 1)
        if (off[r + step] <= j) r += step;
    return r;
}

// Where the entries of a window, or of a piece of one, lie: entry j, of its row r.
struct WholeWindow {
    int64_t p0;
    const int* off;
    __device__ __forceinline__ int64_t at(int, int j) const { return p0 + j; }
    __device__ __forceinline__ int64_t row_start(int r) const { return p0 + off[r]; }
};
struct WindowPiece {
    const int64_t *base, *start;             // per row: the place of its first entry here minus that entry's number; its start
    __device__ __forceinline__ int64_t at(int r, int j) const { return base[r] + j; }
    __device__ __forceinline__ int64_t row_start(int r) const { return start[r]; }
};

// One warp: at most 32 * ITEMS entries, sorted in registers by a bitonic network over positions lane * ITEMS + i; the
// distinct ones then lie ascending in cols (padded to 32 * ITEMS with the largest int), where every entry looks its own up.
// For 60,000 power-law rows the network takes about four warp instructions per entry, merging in shared memory 44.
template <int WH, int ITEMS>
__device__ __forceinline__ void sort_window(const CondenseParams& p, int64_t w, int64_t p0, int n, const int* off, int32_t* own, int32_t* cols) {
    constexpr int kPad = 0x7fffffff;
    constexpr int N = 32 * ITEMS;
    const int lane = threadIdx.x & 31;
    int32_t key[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int j = i * 32 + lane;
        key[i] = kPad;
        if (j < n) {
            const int r = row_in_window<WH>(off, j);
            key[i] = checked_column(p, p0 + j, p0 + off[r]);
            p.row_of[p0 + j] = static_cast<int32_t>(w * WH + r);
        }
        own[j] = key[i];
        cols[j] = kPad;
    }
#pragma unroll
    for (int size = 2; size <= N; size *= 2)
#pragma unroll
        for (int stride = size / 2; stride > 0; stride /= 2) {
            if (stride >= ITEMS) {
                // partner in another lane; ascending where the position's `size` bit is clear
                const bool up = size >= N || ((lane * ITEMS) & size) == 0;
                const bool low = (lane & (stride / ITEMS)) == 0;
#pragma unroll
                for (int i = 0; i < ITEMS; ++i) {
                    const int32_t other = __shfl_xor_sync(0xffffffffu, key[i], stride / ITEMS);
                    key[i] = up == low ? min(key[i], other) : max(key[i], other);
                }
            } else {
#pragma unroll
                for (int i = 0; i < ITEMS; ++i) {
                    if (i & stride) continue;
                    const bool up = size >= N || ((lane * ITEMS + i) & size) == 0;
                    const int32_t a = min(key[i], key[i | stride]), b = max(key[i], key[i | stride]);
                    key[i] = up ? a : b;
                    key[i | stride] = up ? b : a;
                }
            }
        }
    const int32_t before = __shfl_up_sync(0xffffffffu, key[ITEMS - 1], 1);
    unsigned first = 0;                      // bit i: the first of its column
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const bool f = key[i] != kPad && ((lane == 0 && i == 0) || key[i] != (i ? key[i - 1] : before));
        first |= static_cast<unsigned>(f) << i;
    }
    int at = __popc(first);
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += y;
    }
    if (lane == 31) p.ucount[w] = at;
    at -= __popc(first);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if (first >> i & 1u) {
            cols[at++] = key[i];
            atomicAdd(p.refs + key[i], 1);
        }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int j = i * 32 + lane;
        const int32_t c = own[j];
        int pos = 0;
#pragma unroll
        for (int step = N / 2; step > 0; step /= 2)
            if (cols[pos + step - 1] < c) pos += step;
        if (j < n) p.pos_of[p0 + j] = pos;
    }
}

// n entries: keys[2][cap], rank[cap] in shared memory; off has WH + 1 entries.  Returns the number of distinct columns.
template <int WH, int THREADS, class Entries>
__device__ __forceinline__ int merge_window(const CondenseParams& p, int64_t w, const Entries& e, int n, const int* off, int32_t* keys, int cap, uint32_t* rank) {
    __shared__ int warp_sum[THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int j = threadIdx.x; j < n; j += THREADS) {
        const int r = row_in_window<WH>(off, j);
        const int64_t at = e.at(r, j);
        keys[j] = checked_column(p, at, e.row_start(r));
        rank[j] = static_cast<uint32_t>(j) | static_cast<uint32_t>(r) << 16;     // the row stays beside the rank
        p.row_of[at] = static_cast<int32_t>(w * WH + r);
    }
    __syncthreads();
    int32_t *src = keys, *dst = keys + cap;
    // runs of 2^level rows: an entry's rank in the merged pair of runs = its place in its own + the entries of the other
    // that go before it (equal ones: the earlier run first)
    for (int span = 1; span < WH; span *= 2) {
        for (int j = threadIdx.x; j < n; j += THREADS) {
            const uint32_t row = rank[j] >> 16;
            const int g = static_cast<int>(row) & ~(span - 1);                   // first row of this entry's run
            const bool right = (g & span) != 0;
            const int sib = right ? g - span : g + span;
            const int at = static_cast<int>(rank[j] & 0xffffu);
            const int32_t c = src[at];
            const int s0 = off[sib];
            int lo = s0, hi = off[sib + span];
            const int32_t bound = right ? c : c - 1;                             // entries of the other run up to here go before
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (src[mid] <= bound) lo = mid + 1; else hi = mid;
            }
            const int to = at + (right ? lo - off[g] : lo - s0);
            dst[to] = c;
            rank[j] = static_cast<uint32_t>(to) | row << 16;
        }
        __syncthreads();
        int32_t* t = src;
        src = dst;
        dst = t;
    }
    // dst[r] = condensed columns up to and with rank r
    int carry = 0;
    for (int base = 0; base < n; base += THREADS) {
        const int r = base + threadIdx.x;
        const bool first = r < n && (r == 0 || src[r] != src[r - 1]);
        if (first && static_cast<uint32_t>(src[r]) < static_cast<uint32_t>(p.k)) atomicAdd(p.refs + src[r], 1);     // (any value, after a bad entry)
        const unsigned ball = __ballot_sync(0xffffffffu, first);
        if (lane == 0) warp_sum[warp] = __popc(ball);
        __syncthreads();
        int before = carry, all = carry;
        for (int i = 0; i < THREADS / 32; ++i) {
            const int x = warp_sum[i];
            if (i < warp) before += x;
            all += x;
        }
        if (r < n) dst[r] = before + __popc(ball & ((2u << lane) - 1u));
        carry = all;
        __syncthreads();
    }
    for (int j = threadIdx.x; j < n; j += THREADS) p.pos_of[e.at(static_cast<int>(rank[j] >> 16), j)] = dst[rank[j] & 0xffffu] - 1;
    return carry;
}

// One warp per window; the last of the launches that run side by side, it ends after the others.
constexpr int kSortWarps = 4;
template <int WH>
__global__ void __launch_bounds__(32 * kSortWarps) wcsr_sort_windows_kernel(const CondenseParams p) {
    __shared__ int32_t own[kSortWarps][kWarpWindow], cols[kSortWarps][kWarpWindow];
    __shared__ int offs[kSortWarps][WH + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w = blockIdx.x * int64_t{kSortWarps} + warp;
    if (w < p.nwin) {
        const int64_t r0 = w * WH, p0 = p.row_ptr[r0];
        int* off = offs[warp];
        for (int i = lane; i <= WH; i += 32) off[i] = static_cast<int>(p.row_ptr[min(r0 + i, p.m)] - p0);
        __syncwarp();
        const int n = off[WH];
        if (n <= 64) sort_window<WH, 2>(p, w, p0, n, off, own[warp], cols[warp]);
        else if (n <= 128) sort_window<WH, 4>(p, w, p0, n, off, own[warp], cols[warp]);
        else if (n <= kWarpWindow) sort_window<WH, 8>(p, w, p0, n, off, own[warp], cols[warp]);
    }
    grid_wait();
}

template <int WH, int THREADS>
__device__ __forceinline__ void load_offsets(const CondenseParams& p, int64_t w, int* off) {
    const int64_t r0 = w * WH;
    const int64_t p0 = p.row_ptr[r0];
    for (int i = threadIdx.x; i <= WH; i += THREADS) off[i] = static_cast<int>(p.row_ptr[min(r0 + i, p.m)] - p0);
    __syncthreads();
}

// One CTA per listed window.  shared memory: two key arrays and the ranks.
template <int WH, int THREADS>
__global__ void __launch_bounds__(THREADS) wcsr_merge_windows_kernel(const CondenseParams p) {
    constexpr int kCap = THREADS == 1024 ? kLargeWindow : kMergeWindow;
    extern __shared__ int32_t dyn[];
    __shared__ int off[WH + 1];
    grid_trigger();
    const int64_t w = p.list[blockIdx.x];
    load_offsets<WH, THREADS>(p, w, off);
    const int found = merge_window<WH, THREADS>(p, w, WholeWindow{p.row_ptr[w * WH], off}, off[WH], off, dyn, kCap, reinterpret_cast<uint32_t*>(dyn + 2 * kCap));
    if (threadIdx.x == 0) p.ucount[w] = found;
    grid_wait();
}

// Bits of the columns [c0, c0 + 32 words) and the set bits before each word, as many at a time as there is room for, of the
// columns [begin, end) that the entries lie in.  Returns the number of distinct columns.
constexpr int kBitmapThreads = 512;
template <int WH, class Entries>
__device__ __forceinline__ int bitmap_window(const CondenseParams& p, int64_t w, const Entries& e, int n, const int* off, uint32_t* bits, int max_words,
                                             int64_t begin, int64_t end) {
    __shared__ long long scratch[32];
    constexpr int T = kBitmapThreads;
    uint32_t* prefix = bits + max_words;
    int found = 0;                           // condensed columns before c0
    for (int64_t c0 = begin; c0 < end; c0 += int64_t{32} * max_words) {
        const int words = static_cast<int>(min(static_cast<int64_t>(max_words), (end - c0 + 31) / 32));
        __syncthreads();
        for (int i = threadIdx.x; i < words; i += T) bits[i] = 0u;
        __syncthreads();
        for (int j = threadIdx.x; j < n; j += T) {
            const int r = row_in_window<WH>(off, j);
            const int64_t at = e.at(r, j), c = checked_column(p, at, e.row_start(r)) - c0;
            if (c0 == begin) p.row_of[at] = static_cast<int32_t>(w * WH + r);
            if (c >= 0 && c < int64_t{32} * words) atomicOr(&bits[c >> 5], 1u << (c & 31));
        }
        __syncthreads();
        long long carry = found;
        for (int base = 0; base < words; base += T) {
            const int i = base + threadIdx.x;
            long long total;
            const long long before = carry + block_exclusive_sum<T>(i < words ? __popc(bits[i]) : 0, scratch, &total);
            if (i < words) prefix[i] = static_cast<uint32_t>(before);
            carry += total;
        }
        __syncthreads();
        found = static_cast<int>(carry);
        for (int j = threadIdx.x; j < n; j += T) {
            const int r = row_in_window<WH>(off, j);
            const int64_t at = e.at(r, j), c = checked_column(p, at, e.row_start(r)) - c0;
            if (c < 0 || c >= int64_t{32} * words) continue;
            p.pos_of[at] = static_cast<int32_t>(prefix[c >> 5] + __popc(bits[c >> 5] & ((1u << (c & 31)) - 1u)));
        }
        for (int i = threadIdx.x; i < words; i += T)
            for (uint32_t x = bits[i]; x; x &= x - 1) atomicAdd(p.refs + c0 + 32 * int64_t{i} + (__ffs(x) - 1), 1);
    }
    return found;
}

template <int WH>
__global__ void __launch_bounds__(kBitmapThreads) wcsr_bitmap_windows_kernel(const CondenseParams p, int max_words) {
    extern __shared__ int32_t dyn[];
    __shared__ int off[WH + 1];
    grid_trigger();
    const int64_t w = p.list[blockIdx.x];
    load_offsets<WH, kBitmapThreads>(p, w, off);
    const int found = bitmap_window<WH>(p, w, WholeWindow{p.row_ptr[w * WH], off}, off[WH], off, reinterpret_cast<uint32_t*>(dyn), max_words, 0, p.k);
    if (threadIdx.x == 0) p.ucount[w] = found;
    grid_wait();
}

// ---- windows cut into pieces
// A CTA to a piece; with one to a whole window a dense row was one SM's work.  ms to build a handle (in brackets the builder
// before that one, which sorted all entries): 16 x 1,000,000, full 72 (4.6) -> 0.52; 16 rows of 1,000,000 entries among
// 5 x 10^7 columns 1530 (25) -> 8.4; 1,000,000 rows of 8 and a full one 8.4 (9.2) -> 3.9; R-MAT 2^21, 16 a row 16.8 (22.7) -> 15.9.
struct LongWindows {
    int windows, pieces;
    const int32_t *window, *first;           // [windows]: see WindowLists
    int32_t* cut_at;                         // [pieces + windows][WH]: where the rows are cut, counted from their starts
    int32_t* cut_col;                        // [pieces + windows]: and the column
    int32_t* found;                          // [pieces]: distinct columns, then those in the pieces of the window before
    // the window that piece q belongs to (its place in the lists); its cuts are cut q + its place and the one behind
    __device__ __forceinline__ int of_piece(int q) const {
        int lo = 0, hi = windows - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first[mid] <= q) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
    __device__ __forceinline__ int of_cut(int g) const {
        int lo = 0, hi = windows - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first[mid] + mid <= g) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
};

// A warp per cut: cut i lies at a column before which there are from i * n / pieces to kPieceSlack entries more than that,
// or, a column holding at most WH of them, at the smallest one with that many.  Found by bisection, which narrows every row's
// part with the columns'; where the rows are cut is looked up in the whole rows, so that whatever they hold the cuts do
// not go back as long as the columns do not (checked by the pieces).
template <int WH>
__global__ void __launch_bounds__(128) wcsr_cut_windows_kernel(const CondenseParams p, const LongWindows lw) {
    constexpr int R = (WH + 31) / 32;        // rows of a lane
    grid_trigger();
    const int lane = threadIdx.x & 31;
    const int g = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (g >= lw.pieces + lw.windows) return;
    const int l = lw.of_cut(g), i = g - lw.first[l] - l;
    const int64_t r0 = int64_t{lw.window[l]} * WH, n = p.row_ptr[min(r0 + WH, p.m)] - p.row_ptr[r0], pieces = pieces_of(n);
    const int32_t* row[R];
    int len[R], a[R], b[R], x[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int64_t r = r0 + lane + 32 * j;
        const bool mine = lane + 32 * j < WH && r < p.m;
        const int64_t start = mine ? p.row_ptr[r] : 0;
        row[j] = p.col_idx + start;
        len[j] = mine ? static_cast<int>(p.row_ptr[r + 1] - start) : 0;
        a[j] = 0;
        b[j] = len[j];
    }
    auto before = [&](int j, int64_t c, int lo, int hi) {        // entries of the row in columns before c, known to be lo .. hi
        while (lo < hi) {
            const int mid = lo + ((hi - lo) >> 1);
            if (row[j][mid] < c) lo = mid + 1; else hi = mid;
        }
        return lo;
    };
    int64_t col = i == 0 ? 0 : p.k;
    if (i > 0 && i < pieces) {
        const unsigned target = static_cast<unsigned>(n * i / pieces);
        int64_t clo = 0;
        while (col - clo > 1) {
            const int64_t mid = (clo + col) >> 1;
            unsigned sum = 0;
#pragma unroll
            for (int j = 0; j < R; ++j) sum += static_cast<unsigned>(x[j] = before(j, mid, a[j], b[j]));
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (sum >= target) {
                col = mid;
                if (sum < target + kPieceSlack) break;
            } else {
                clo = mid;
            }
#pragma unroll
            for (int j = 0; j < R; ++j) (sum >= target ? b[j] : a[j]) = x[j];
        }
    }
    if (lane == 0) lw.cut_col[g] = static_cast<int32_t>(col);
#pragma unroll
    for (int j = 0; j < R; ++j)
        if (lane + 32 * j < WH) lw.cut_at[int64_t{g} * WH + lane + 32 * j] = i == 0 ? 0 : (i == pieces ? len[j] : before(j, col, 0, len[j]));
}

// One CTA per piece: by bitmap where its columns fit one, merged otherwise.
constexpr int kPieceSmem = kPieceCap * 12, kPieceWords = kPieceSmem / 8;
template <int WH>
__global__ void __launch_bounds__(kBitmapThreads) wcsr_pieces_kernel(const CondenseParams p, const LongWindows lw) {
    extern __shared__ int32_t dyn[];
    __shared__ int off[WH + 1];
    __shared__ int64_t base[WH], start[WH];
    __shared__ bool bad;
    grid_trigger();
    grid_wait();                             // the cuts
    const int q = blockIdx.x, l = lw.of_piece(q), g = q + l;
    const int64_t w = lw.window[l];
    const int32_t *lo = lw.cut_at + int64_t{g} * WH, *hi = lo + WH;
    for (int r = threadIdx.x; r < WH; r += kBitmapThreads) {
        start[r] = p.row_ptr[min(w * WH + r, p.m)];
        base[r] = start[r] + lo[r];
        off[r + 1] = hi[r] - lo[r];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t n = 0;
        bad = false;
        off[0] = 0;
        for (int r = 0; r < WH; ++r) {
            base[r] -= n;
            n += off[r + 1];
            // (only rows that do not ascend, or hold columns the matrix does not have)
            if (off[r + 1] < 0 || n > kPieceCap) { bad = true; break; }
            off[r + 1] = static_cast<int>(n);
        }
        if (bad) {
            *p.bad = 1;
            lw.found[q] = 0;
        }
    }
    __syncthreads();
    if (bad) return;
    const int n = off[WH];
    const int64_t begin = lw.cut_col[g], end = lw.cut_col[g + 1];
    const WindowPiece e = {base, start};
    const int found = end - begin <= int64_t{32} * kPieceWords
                          ? bitmap_window<WH>(p, w, e, n, off, reinterpret_cast<uint32_t*>(dyn), kPieceWords, begin, end)
                          : merge_window<WH, kBitmapThreads>(p, w, e, n, off, dyn, kPieceCap, reinterpret_cast<uint32_t*>(dyn + 2 * kPieceCap));
    if (threadIdx.x == 0) lw.found[q] = found;
}

// One CTA per window: its distinct columns, and in found those of the pieces before each.
__global__ void __launch_bounds__(1024) wcsr_piece_sums_kernel(const CondenseParams p, const LongWindows lw) {
    __shared__ long long scratch[32];
    const int q1 = blockIdx.x + 1 < lw.windows ? lw.first[blockIdx.x + 1] : lw.pieces;
    long long carry = 0, total;
    for (int q0 = lw.first[blockIdx.x]; q0 < q1; q0 += 1024) {
        const int q = q0 + threadIdx.x;
        const long long before = block_exclusive_sum(q < q1 ? lw.found[q] : 0, scratch, &total);
        if (q < q1) lw.found[q] = static_cast<int32_t>(carry + before);
        carry += total;
    }
    if (threadIdx.x == 0) p.ucount[lw.window[blockIdx.x]] = static_cast<int32_t>(carry);
}

// One CTA per piece, a warp per row: places in the piece become places in the window.
template <int WH>
__global__ void __launch_bounds__(256) wcsr_piece_places_kernel(const CondenseParams p, const LongWindows lw) {
    const int q = blockIdx.x, l = lw.of_piece(q), lane = threadIdx.x & 31;
    const int32_t first = lw.found[q];
    if (first == 0) return;
    const int32_t *lo = lw.cut_at + int64_t{q + l} * WH, *hi = lo + WH;
    for (int r = threadIdx.x >> 5; r < WH; r += 8) {
        const int64_t start = p.row_ptr[min(int64_t{lw.window[l]} * WH + r, p.m)];
        for (int64_t j = lo[r] + lane; j < hi[r]; j += 32) p.pos_of[start + j] += first;
    }
}

// CTA 0: window_row_ptr; the others: how many columns are referenced at all
__global__ void __launch_bounds__(1024) wcsr_row_ptr_kernel(const int32_t* ucount, int64_t nwin, int b_col, int32_t* window_row_ptr, int* overflow,
                                                            const int32_t* __restrict__ refs, int64_t k, unsigned long long* distinct) {
    if (blockIdx.x == 0) {
        scan_counts(ucount, nwin, b_col, window_row_ptr, overflow);
        return;
    }
    unsigned long long n = 0;
    for (int64_t c = (blockIdx.x - 1) * int64_t{1024} + threadIdx.x; c < k; c += (gridDim.x - 1) * int64_t{1024}) n += refs[c] > 0;
    for (int o = 16; o > 0; o >>= 1) n += __shfl_down_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(distinct, n);
}

// One thread per entry: its column and its value to their places (entries that share a condensed column write the same).
template <int ES>
__global__ void wcsr_place_kernel(int64_t nnz, int wh, int b_col, const int32_t* __restrict__ row_of, const int32_t* __restrict__ pos_of,
                                  const int32_t* __restrict__ col_idx, const uint8_t* __restrict__ vals, const int32_t* __restrict__ window_row_ptr,
                                  int32_t* __restrict__ window_col_idx, uint8_t* __restrict__ packed) {
    for (int64_t p = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; p < nnz; p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int i = row_of[p];
        const int w = i / wh, r = i - w * wh;
        const int64_t at = static_cast<int64_t>(window_row_ptr[w]) + pos_of[p];
        window_col_idx[at] = col_idx[p];
        uint8_t* dst = packed + wcsr_packed_offset(wh, b_col, ES, r, at);
        const uint8_t* src = vals + static_cast<size_t>(p) * ES;
        if constexpr (ES == 1) *dst = *src;
        else if constexpr (ES == 2) *reinterpret_cast<uint16_t*>(dst) = *reinterpret_cast<const uint16_t*>(src);
        else *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(src);
    }
}

// eight lanes per item
__global__ void wcsr_fills_kernel(int64_t n_items, const WcsrDevTask* __restrict__ tasks, const int32_t* __restrict__ bin_tasks,
                                  const int32_t* __restrict__ item_fill, int kt, int2* __restrict__ fills) {
    for (int64_t i = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 3; i < n_items;
         i += (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 3) {
        const WcsrDevTask t = tasks[bin_tasks[i]];
        const int f0 = item_fill[i], n = item_fill[i + 1] - f0;
        for (int j = threadIdx.x & 7; j < n; j += 8) {
            const int done = j * kt;
            fills[f0 + j] = make_int2(t.col_begin + done, min(kt, t.count - done) | (j == 0) << 16 | (j == n - 1) << 17);
        }
    }
}

// ---- reuse classes of the column groups (gather hints; the host rule of wcsr_reuse_classes)
// The class of a row of B is its rank by gather count (ties: the lower index first) against the limits 16 Ki, 32 Ki, ...,
// so no sort is needed: a histogram of the counts says at which count each limit falls and how many of the rows with just
// that count are still inside; only those rows' order among themselves has to be found.

constexpr int kLimits = 7;                   // classes 7 .. 1
struct ClassCut { int32_t count[kLimits]; int32_t quota[kLimits]; };   // inside limit i: more than count[i] gathers, or one of the first quota[i] rows with just as many

constexpr int kSmallCounts = 1024;
__global__ void __launch_bounds__(256) wcsr_count_hist_kernel(const int32_t* __restrict__ refs, int64_t k, int32_t* __restrict__ hist) {
    __shared__ int32_t small[kSmallCounts];
    for (int i = threadIdx.x; i < kSmallCounts; i += 256) small[i] = 0;
    __syncthreads();
    for (int64_t c = blockIdx.x * int64_t{256} + threadIdx.x; c < k; c += gridDim.x * int64_t{256}) {
        const int n = refs[c];
        if (n > 1) atomicAdd(n < kSmallCounts ? &small[n] : hist + n, 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kSmallCounts; i += 256)
        if (small[i]) atomicAdd(hist + i, small[i]);
}

// one CTA: from the highest count down; top = the highest one possible
__global__ void __launch_bounds__(1024) wcsr_class_cut_kernel(const int32_t* __restrict__ hist, int64_t top, ClassCut* cut) {
    __shared__ long long scratch[32];
    if (threadIdx.x < kLimits) {             // (a limit that is not reached: every row gathered more than once is inside)
        cut->count[threadIdx.x] = 1;
        cut->quota[threadIdx.x] = 0;
    }
    long long above = 0;
    for (int64_t base = top; base >= 2 && above < (static_cast<long long>(kWcsrTopClassRows) << (kLimits - 1)); base -= 1024) {
        const int64_t v = base - threadIdx.x;
        const long long h = v >= 2 ? hist[v] : 0;
        long long total;
        const long long before = above + block_exclusive_sum(h, scratch, &total);
#pragma unroll
        for (int i = 0; i < kLimits; ++i) {
            const long long lim = static_cast<long long>(kWcsrTopClassRows) << i;
            if (before < lim && lim <= before + h) {
                cut->count[i] = static_cast<int32_t>(v);
                cut->quota[i] = static_cast<int32_t>(lim - before);
            }
        }
        above += total;
    }
}

// rows whose count is the one of limit i, per chunk of columns: at [block][i]
__global__ void __launch_bounds__(256) wcsr_cut_rows_kernel(const int32_t* __restrict__ refs, int64_t k, int64_t chunk, const ClassCut* __restrict__ cut,
                                                            int32_t* __restrict__ n_rows) {
    __shared__ int n[kLimits];
    if (threadIdx.x < kLimits) n[threadIdx.x] = 0;
    __syncthreads();
    const int64_t c1 = min(k, (blockIdx.x + 1) * chunk);
    for (int64_t c = blockIdx.x * chunk + threadIdx.x; c < c1; c += 256) {
        const int x = refs[c];
        if (x > 1)
#pragma unroll
            for (int i = 0; i < kLimits; ++i)
                if (x == cut->count[i]) atomicAdd(&n[i], 1);
    }
    __syncthreads();
    if (threadIdx.x < kLimits) n_rows[blockIdx.x * kLimits + threadIdx.x] = n[threadIdx.x];
}

__global__ void __launch_bounds__(256) wcsr_class_kernel(const int32_t* __restrict__ refs, int64_t k, int64_t chunk, const ClassCut* __restrict__ cut,
                                                         const int32_t* __restrict__ n_rows, uint8_t* __restrict__ cls) {
    __shared__ int before[kLimits];          // rows with the count of limit i in the columns before this step's
    __shared__ int in_warp[8][kLimits];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < kLimits) before[threadIdx.x] = 0;
    __syncthreads();
    for (int j = threadIdx.x; j < static_cast<int>(blockIdx.x) * kLimits; j += 256)
        if (n_rows[j]) atomicAdd(&before[j % kLimits], n_rows[j]);
    __syncthreads();
    const int64_t c1 = min(k, (blockIdx.x + 1) * chunk);
    for (int64_t base = blockIdx.x * chunk; base < c1; base += 256) {
        const int64_t c = base + threadIdx.x;
        const int x = c < c1 ? refs[c] : 0;
        unsigned at_limit = 0;
        int ordinal[kLimits];
#pragma unroll
        for (int i = 0; i < kLimits; ++i) {
            const unsigned b = __ballot_sync(0xffffffffu, x > 1 && x == cut->count[i]);
            ordinal[i] = __popc(b & ((1u << lane) - 1u));
            if (b >> lane & 1u) at_limit |= 1u << i;
            if (lane == 0) in_warp[warp][i] = __popc(b);
        }
        __syncthreads();
        int level = 0;
        if (x > 1)
#pragma unroll
            for (int i = kLimits - 1; i >= 0; --i) {
                bool inside = x > cut->count[i];
                if (at_limit >> i & 1u) {
                    int n = before[i] + ordinal[i];
                    for (int v = 0; v < warp; ++v) n += in_warp[v][i];
                    inside = n < cut->quota[i];
                }
                if (inside) level = kLimits - i;
            }
        if (c < c1) cls[c] = static_cast<uint8_t>(level);
        __syncthreads();
        if (threadIdx.x < kLimits)
            for (int v = 0; v < 8; ++v) before[threadIdx.x] += in_warp[v][threadIdx.x];
        __syncthreads();
    }
}

__global__ void wcsr_group_class_kernel(const int32_t* __restrict__ col_idx, int64_t n_groups, const uint8_t* __restrict__ cls,
                                        uint8_t* __restrict__ grp_class) {
    for (int64_t g = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; g < n_groups; g += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int4 c = reinterpret_cast<const int4*>(col_idx)[g];
        int best = 0;
        if (c.x >= 0) best = max(best, static_cast<int>(cls[c.x]));
        if (c.y >= 0) best = max(best, static_cast<int>(cls[c.y]));
        if (c.z >= 0) best = max(best, static_cast<int>(cls[c.z]));
        if (c.w >= 0) best = max(best, static_cast<int>(cls[c.w]));
        grp_class[g] = static_cast<uint8_t>(best);
    }
}

// Allocates and fills *d_grp_class [P / 4] from the device copy of window_col_idx and the gather counts refs [k] (each at
// most nwin), in the order of `st`.
int wcsr_reuse_classes_device(const int32_t* d_window_col_idx, int64_t P, const int32_t* refs, int64_t k, int64_t nwin, cudaStream_t st,
                              uint8_t** d_grp_class) {
    *d_grp_class = nullptr;
    if (P <= 0 || k <= 0) return SPMM_OK;
    const int64_t chunk = std::max<int64_t>(256, (k + 1023) / 1024);          // at most 1024 of them
    const unsigned chunks = static_cast<unsigned>((k + chunk - 1) / chunk);
    const int64_t counts = std::max<int64_t>(nwin + 1, kSmallCounts);
    auto up = [](int64_t bytes) { return (bytes + 255) / 256 * 256; };
    const int64_t o_hist = up(k), o_cut = o_hist + up(counts * 4), o_rows = o_cut + 256, bytes = o_rows + int64_t{chunks} * kLimits * 4;
    uint8_t* block = nullptr;                 // classes | histogram of the counts | cuts | rows at the cuts
    if (!dev_alloc_ok(&block, static_cast<size_t>(bytes), st) || !dev_alloc_ok(d_grp_class, static_cast<size_t>(P / 4), st)) {
        dev_free(block, st);
        dev_free(*d_grp_class, st);
        *d_grp_class = nullptr;
        return SPMM_ERR_ALLOC;
    }
    int32_t* hist = reinterpret_cast<int32_t*>(block + o_hist);
    ClassCut* cut = reinterpret_cast<ClassCut*>(block + o_cut);
    int32_t* n_rows = reinterpret_cast<int32_t*>(block + o_rows);
    cudaMemsetAsync(hist, 0, static_cast<size_t>(counts) * 4, st);
    wcsr_count_hist_kernel<<<static_cast<unsigned>(std::min<int64_t>((k + 1023) / 1024, 1024)), 256, 0, st>>>(refs, k, hist);
    wcsr_class_cut_kernel<<<1, 1024, 0, st>>>(hist, nwin, cut);
    wcsr_cut_rows_kernel<<<chunks, 256, 0, st>>>(refs, k, chunk, cut, n_rows);
    wcsr_class_kernel<<<chunks, 256, 0, st>>>(refs, k, chunk, cut, n_rows, block);
    wcsr_group_class_kernel<<<static_cast<unsigned>(std::min<int64_t>((P / 4 + 255) / 256, 2048)), 256, 0, st>>>(d_window_col_idx, P / 4, block, *d_grp_class);
    const bool ok = cudaGetLastError() == cudaSuccess;
    dev_free(block, st);
    if (!ok) {
        dev_free(*d_grp_class, st);
        *d_grp_class = nullptr;
        return SPMM_ERR_CUDA;
    }
    return SPMM_OK;
}

}  // namespace

cudaError_t expand_wcsr_fills(int64_t n_items, const void* d_tasks, const int32_t* d_bin_tasks, const int32_t* d_item_fill, int kt,
                              int32_t* d_fills, cudaStream_t stream) {
    if (n_items <= 0) return cudaSuccess;
    wcsr_fills_kernel<<<static_cast<unsigned>(std::min<int64_t>((n_items + 31) / 32, 4096)), 256, 0, stream>>>(
        n_items, static_cast<const WcsrDevTask*>(d_tasks), d_bin_tasks, d_item_fill, kt, reinterpret_cast<int2*>(d_fills));
    return cudaGetLastError();
}

namespace {

// Every window by its kernel.  The launches touch disjoint data and run side by side, each ending behind the one before
// it (grid_wait); the first starts when the stream gets there.  What follows from the pieces' counts comes behind them all.
template <int WH>
bool condense(CondenseParams p, const WindowLists& lists, const int* count, const LongWindows& lw, cudaStream_t st) {
    const unsigned pieces = static_cast<unsigned>(lw.pieces);
    if (lw.windows > 0) {
        wcsr_cut_windows_kernel<WH><<<(pieces + static_cast<unsigned>(lw.windows) + 3) / 4, 128, 0, st>>>(p, lw);
        if (cudaGetLastError() != cudaSuccess) return false;
        if (cudaFuncSetAttribute(wcsr_pieces_kernel<WH>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPieceSmem) != cudaSuccess) return false;
        if (launch_dependent(wcsr_pieces_kernel<WH>, dim3(pieces), kBitmapThreads, kPieceSmem, st, p, lw) != cudaSuccess) return false;
    }
    bool first = lw.windows == 0;
    auto launch = [&](auto kernel, int64_t grid, int threads, size_t smem, const auto&... args) {
        // (the most there may be: threads that build for other widths set it too)
        if (smem > 48 * 1024 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostBitmap) != cudaSuccess) return false;
        if (!first) return launch_dependent(kernel, dim3(static_cast<unsigned>(grid)), threads, smem, st, p, args...) == cudaSuccess;
        first = false;
        kernel<<<static_cast<unsigned>(grid), threads, smem, st>>>(p, args...);
        return cudaGetLastError() == cudaSuccess;
    };
    auto list = [&](int which, auto kernel, int threads, size_t smem, const auto&... args) {
        p.list = which == kListBitmap ? lists.list[which] : lists.list[which] + 1 - count[which];
        return count[which] == 0 || launch(kernel, count[which], threads, smem, args...);
    };
    const int words = static_cast<int>(std::min<int64_t>((p.k + 31) / 32, kBitmapColumns / 32));
    return list(kListBitmap, wcsr_bitmap_windows_kernel<WH>, kBitmapThreads, static_cast<size_t>(words) * 8, words) &&
           list(kListLarge, wcsr_merge_windows_kernel<WH, 1024>, 1024, size_t{kLargeWindow} * 12) &&
           list(kListMerge, wcsr_merge_windows_kernel<WH, 256>, 256, size_t{kMergeWindow} * 12) &&
           launch(wcsr_sort_windows_kernel<WH>, (p.nwin + kSortWarps - 1) / kSortWarps, 32 * kSortWarps, 0) && [&]() {
               if (lw.windows == 0) return true;
               wcsr_piece_sums_kernel<<<static_cast<unsigned>(lw.windows), 1024, 0, st>>>(p, lw);
               wcsr_piece_places_kernel<WH><<<pieces, 256, 0, st>>>(p, lw);
               return cudaGetLastError() == cudaSuccess;
           }();
}

}  // namespace

int build_wcsr_device(int64_t m, int64_t k, const int64_t* d_row_ptr, const int32_t* d_col_idx, const uint8_t* d_vals,
                      int es, int wh, int b_col, int T, int n_bins, int sms, cudaStream_t st, WcsrHost* out, int64_t* nnz_out,
                      int32_t** d_window_row_ptr, int32_t** d_window_col_idx, uint8_t** d_packed, uint8_t** d_grp_class,
                      WcsrRowStream* rows) {
    *d_grp_class = nullptr;
    if (wh != 16 && wh != 64) return SPMM_ERR_UNSUPPORTED;
    if ((es != 1 && es != 2 && es != 4) || b_col * es != 32) return SPMM_ERR_UNSUPPORTED;
    if (T < 0 || T % b_col != 0 || n_bins <= 0) return SPMM_ERR_INVALID_ARG;
    if (m < 0 || k < 0 || !d_row_ptr) return SPMM_ERR_INVALID_ARG;
    const int64_t nwin = (m + wh - 1) / wh;
    out->wh = wh;
    out->b_col = b_col;
    out->nwin = nwin;
    out->window_row_ptr.assign(static_cast<size_t>(nwin) + 1, 0);      // (may throw: before anything is held on the device)
    *d_window_row_ptr = nullptr;
    *d_window_col_idx = nullptr;
    *d_packed = nullptr;

    // what the GPU tells the host, read with one copy at a time
    struct Flags {
        int err;                              // CSR error code
        int overflow;                         // of the scan
        int n_listed[kLists];                 // windows of the condensation kernels that go by lists
        int bad;                              // an entry out of range or not ascending
        int64_t nnz;
        unsigned long long long_count;        // windows that are cut into pieces, and the pieces
        unsigned long long distinct;          // columns that are referenced
    } flags = {};
    Flags* d_flags = nullptr;
    int32_t* d_lists = nullptr;               // those windows
    uint8_t* d_work = nullptr;                // the entries' rows and places, window lengths, gather counts
    int32_t* d_cuts = nullptr;                // LongWindows' arrays
    auto release = [&]() { dev_free(d_flags, st); dev_free(d_lists, st); dev_free(d_work, st); dev_free(d_cuts, st); };
    auto fail = [&](int code) {
        cudaGetLastError();                  // (of a call that failed: not for a later check to find)
        release();
        dev_free(*d_window_row_ptr, st); dev_free(*d_window_col_idx, st); dev_free(*d_packed, st);
        *d_window_row_ptr = nullptr; *d_window_col_idx = nullptr; *d_packed = nullptr;
        return code;
    };
    auto alloc = [&](void** ptr, size_t bytes) { return dev_alloc(ptr, bytes, st) == cudaSuccess; };

    const int64_t max_long = std::min(nwin, kMostLong);
    if (!alloc(reinterpret_cast<void**>(&d_flags), sizeof(Flags)) || !alloc(reinterpret_cast<void**>(&d_lists), static_cast<size_t>(2 * nwin + max_long + 1) * 4))
        return fail(SPMM_ERR_ALLOC);
    if (cudaMemsetAsync(d_flags, 0, sizeof(Flags), st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    auto read_flags = [&]() {
        return cudaMemcpyAsync(&flags, d_flags, sizeof(Flags), cudaMemcpyDeviceToHost, st) == cudaSuccess && cudaStreamSynchronize(st) == cudaSuccess;
    };
    const unsigned check_grid = static_cast<unsigned>(std::min<int64_t>((m + 255) / 256, 2048));
    // a window is cut where a bitmap would read more than kBitmapReads entries, once per kBitmapColumns
    const int64_t long_from = std::max<int64_t>(kLargeWindow, kBitmapReads / std::max<int64_t>(1, (k + kBitmapColumns - 1) / kBitmapColumns)) + 1;
    // (no window is in two lists: two of them share nwin places, one from either end)
    const WindowLists lists = {wh, k, {d_lists, d_lists + nwin - 1, d_lists + 2 * nwin - 1}, d_flags->n_listed,
                               d_lists + nwin, d_lists + 2 * nwin, &d_flags->long_count, max_long, long_from};
    if (m > 0) csr_check_rows_kernel<<<check_grid, 256, 0, st>>>(m, d_row_ptr, &d_flags->err, &d_flags->nnz, lists);
    if (!read_flags()) return fail(SPMM_ERR_CUDA);
    if (flags.err != 0) return fail(flags.err);
    const int64_t nnz = flags.nnz;
    if (nnz < 0 || (nnz > 0 && (!d_col_idx || !d_vals))) return fail(SPMM_ERR_INVALID_ARG);
    if (nnz >= (int64_t{1} << 31)) return fail(SPMM_ERR_TOO_LARGE);
    *nnz_out = nnz;

    size_t work_bytes = 256;
    auto section = [&](size_t bytes) {
        const size_t at = work_bytes;
        work_bytes += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t o_row_of = section(static_cast<size_t>(nnz) * 4), o_pos_of = section(static_cast<size_t>(nnz) * 4);
    const size_t o_ucount = section(static_cast<size_t>(nwin) * 4), o_refs = section(static_cast<size_t>(k) * 4);
    if (!alloc(reinterpret_cast<void**>(&d_work), work_bytes) ||
        !alloc(reinterpret_cast<void**>(d_window_row_ptr), static_cast<size_t>(nwin + 1) * 4))
        return fail(SPMM_ERR_ALLOC);
    CondenseParams cp;
    cp.m = m;
    cp.k = k;
    cp.nwin = nwin;
    cp.row_ptr = d_row_ptr;
    cp.col_idx = d_col_idx;
    cp.row_of = reinterpret_cast<int32_t*>(d_work + o_row_of);
    cp.pos_of = reinterpret_cast<int32_t*>(d_work + o_pos_of);
    cp.ucount = reinterpret_cast<int32_t*>(d_work + o_ucount);
    cp.refs = reinterpret_cast<int32_t*>(d_work + o_refs);
    cp.bad = &d_flags->bad;
    cp.list = nullptr;
    const unsigned entry_grid = static_cast<unsigned>(std::min<int64_t>((nnz + 255) / 256, 16384));
    if (cudaMemsetAsync(cp.ucount, 0, work_bytes - o_ucount, st) != cudaSuccess) return fail(SPMM_ERR_CUDA);     // and the gather counts behind it
    if (nnz > 0 && k == 0) return fail(SPMM_ERR_OUT_OF_RANGE);
    LongWindows lw = {};
    lw.windows = static_cast<int>(flags.long_count >> kLongShift);
    lw.pieces = static_cast<int>(flags.long_count & ((1ull << kLongShift) - 1));
    if (lw.windows > 0) {
        const int64_t cuts = int64_t{lw.pieces} + lw.windows;
        if (!alloc(reinterpret_cast<void**>(&d_cuts), static_cast<size_t>(cuts * (wh + 1) + lw.pieces) * 4)) return fail(SPMM_ERR_ALLOC);
        lw.window = lists.long_window;
        lw.first = lists.long_first;
        lw.cut_at = d_cuts;
        lw.cut_col = d_cuts + cuts * wh;
        lw.found = lw.cut_col + cuts;
    }
    if (nnz > 0 && !(wh == 16 ? condense<16>(cp, lists, flags.n_listed, lw, st) : condense<64>(cp, lists, flags.n_listed, lw, st))) return fail(SPMM_ERR_CUDA);
    wcsr_row_ptr_kernel<<<1 + static_cast<unsigned>(std::min<int64_t>((k + 1023) / 1024, 128)), 1024, 0, st>>>(
        cp.ucount, nwin, b_col, *d_window_row_ptr, &d_flags->overflow, cp.refs, k, &d_flags->distinct);
    if (cudaMemcpyAsync(out->window_row_ptr.data(), *d_window_row_ptr, static_cast<size_t>(nwin + 1) * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        !read_flags())
        return fail(SPMM_ERR_CUDA);
    if (flags.bad) {
        // (an entry that broke a rule was taken as column 0, so nothing above left its arrays)
        csr_check_cols_kernel<<<check_grid, 256, 0, st>>>(m, k, d_row_ptr, d_col_idx, &d_flags->err);
        if (!read_flags()) return fail(SPMM_ERR_CUDA);
        return fail(flags.err != 0 ? flags.err : SPMM_ERR_INVALID_ARG);
    }
    if (flags.overflow) return fail(SPMM_ERR_TOO_LARGE);
    const int64_t P = out->window_row_ptr[static_cast<size_t>(nwin)];
    out->P = P;
    out->distinct_cols = static_cast<int64_t>(flags.distinct);

    // window_col_idx over a -1 fill, values into the zero-filled packed tiles
    const size_t packed_bytes = static_cast<size_t>(P) * wh * es;
    if (!alloc(reinterpret_cast<void**>(d_window_col_idx), static_cast<size_t>(P) * 4) ||
        !alloc(reinterpret_cast<void**>(d_packed), packed_bytes))
        return fail(SPMM_ERR_ALLOC);
    if (P > 0) {
        cudaMemsetAsync(*d_window_col_idx, 0xFF, static_cast<size_t>(P) * 4, st);
        cudaMemsetAsync(*d_packed, 0, packed_bytes, st);
    }
    if (nnz > 0) {
        if (es == 1)
            wcsr_place_kernel<1><<<entry_grid, 256, 0, st>>>(nnz, wh, b_col, cp.row_of, cp.pos_of, d_col_idx, d_vals, *d_window_row_ptr, *d_window_col_idx, *d_packed);
        else if (es == 2)
            wcsr_place_kernel<2><<<entry_grid, 256, 0, st>>>(nnz, wh, b_col, cp.row_of, cp.pos_of, d_col_idx, d_vals, *d_window_row_ptr, *d_window_col_idx, *d_packed);
        else
            wcsr_place_kernel<4><<<entry_grid, 256, 0, st>>>(nnz, wh, b_col, cp.row_of, cp.pos_of, d_col_idx, d_vals, *d_window_row_ptr, *d_window_col_idx, *d_packed);
    }
    int rc = cudaGetLastError() == cudaSuccess ? wcsr_reuse_classes_device(*d_window_col_idx, P, cp.refs, k, nwin, st, d_grp_class) : SPMM_ERR_CUDA;
    if (!rc && rows && wcsr_wants_rows(es, m, nnz, P)) {
        rc = build_wcsr_rows_device(m, nnz, d_row_ptr, d_col_idx, d_vals, es, sms, cp.row_of, st, rows);
        if (rc == SPMM_ERR_ALLOC) rc = SPMM_OK;          // no room for it: the window kernel serves the handle
    }
    release();                                // (ordered behind the kernels that use them)
    // the split plan needs the window lengths only: the host makes it while the kernels above run
    if (!rc) {
        try {
            rc = plan_wcsr(out, T, n_bins, es);
        } catch (const std::bad_alloc&) {
            rc = SPMM_ERR_ALLOC;
        }
    }
    if (rc) {
        if (rows) free_wcsr_rows(rows, st);
        dev_free(*d_window_row_ptr, st); dev_free(*d_window_col_idx, st); dev_free(*d_packed, st); dev_free(*d_grp_class, st);
        *d_window_row_ptr = nullptr; *d_window_col_idx = nullptr; *d_packed = nullptr; *d_grp_class = nullptr;
    }
    return rc;
}

// ----------------------------------------------------------------------------- row stream

namespace {

constexpr int kRowClasses = 8;

// length class of a row: 0 = longer than task_max, then one class per factor of two down to `pack`, last = packed
__device__ __forceinline__ int row_class(int64_t len, int pack, int task_max) {
    if (len > task_max) return 0;
    int c = 1;
    for (int lim = task_max / 2; lim >= pack; lim /= 2, ++c)
        if (len > lim) return c;
    return c;
}

// Rows are put in the order of their classes (stable) in three passes over chunks of kRowsChunk rows: what each chunk
// has of every class, exclusive sums of that over (class, chunk), and every row to its place.
constexpr int kRowsChunk = 1024;

// What a row adds to the sums over rows in order: x entries (an empty row counts one; a long row none here), y padded
// entries of a long row, z its parts, w its partial slots.
__device__ __forceinline__ int4 row_size(int64_t len, int task_max, int part_len) {
    if (len <= task_max) return make_int4(len > 0 ? static_cast<int>(len) : 1, 0, 0, 0);
    const int parts = static_cast<int>((len + part_len - 1) / part_len);
    return make_int4(0, static_cast<int>((len + 7) / 8 * 8), parts, parts > 1 ? parts : 0);
}

struct ClassSum { int rows, x, y, z, w; };
__device__ __forceinline__ void add_sum(ClassSum* to, const ClassSum& v) {
    if (v.rows) atomicAdd(&to->rows, v.rows);
    if (v.x) atomicAdd(&to->x, v.x);
    if (v.y) atomicAdd(&to->y, v.y);
    if (v.z) atomicAdd(&to->z, v.z);
    if (v.w) atomicAdd(&to->w, v.w);
}

__global__ void __launch_bounds__(256) rows_count_kernel(int64_t m, const int64_t* __restrict__ row_ptr, int pack, int task_max, int part_len, int chunks,
                                                         ClassSum* __restrict__ sums) {
    __shared__ ClassSum n[kRowClasses];
    if (threadIdx.x < kRowClasses) n[threadIdx.x] = ClassSum{0, 0, 0, 0, 0};
    __syncthreads();
    for (int j = threadIdx.x; j < kRowsChunk; j += 256) {
        const int64_t i = static_cast<int64_t>(blockIdx.x) * kRowsChunk + j;
        if (i >= m) break;
        const int64_t len = row_ptr[i + 1] - row_ptr[i];
        const int4 s = row_size(len, task_max, part_len);
        add_sum(&n[row_class(len, pack, task_max)], ClassSum{1, s.x, s.y, s.z, s.w});
    }
    __syncthreads();
    if (threadIdx.x < kRowClasses) sums[threadIdx.x * chunks + blockIdx.x] = n[threadIdx.x];
}

// One CTA: exclusive sums in place, class by class and chunk by chunk; the classes' rows; the sums over all rows behind the last.
__global__ void __launch_bounds__(1024) rows_sums_kernel(int chunks, ClassSum* __restrict__ sums, int32_t* __restrict__ counts) {
    __shared__ ClassSum warp_sum[32];
    __shared__ int class_start[kRowClasses + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = chunks * kRowClasses;
    ClassSum carry = {0, 0, 0, 0, 0};
    auto plus = [](ClassSum a, const ClassSum& b) { a.rows += b.rows; a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; return a; };
    auto scan = [&](ClassSum v) {            // inclusive, over a warp
        for (int o = 1; o < 32; o <<= 1) {
            const ClassSum u = {__shfl_up_sync(0xffffffffu, v.rows, o), __shfl_up_sync(0xffffffffu, v.x, o), __shfl_up_sync(0xffffffffu, v.y, o),
                                __shfl_up_sync(0xffffffffu, v.z, o), __shfl_up_sync(0xffffffffu, v.w, o)};
            if (lane >= o) v = plus(v, u);
        }
        return v;
    };
    for (int base = 0; base < n; base += 1024) {
        const int i = base + threadIdx.x;
        const ClassSum v = i < n ? sums[i] : ClassSum{0, 0, 0, 0, 0};
        const ClassSum in = scan(v);
        if (lane == 31) warp_sum[warp] = in;
        __syncthreads();
        if (warp == 0) warp_sum[lane] = scan(warp_sum[lane]);
        __syncthreads();
        ClassSum ex = {in.rows - v.rows, in.x - v.x, in.y - v.y, in.z - v.z, in.w - v.w};
        ex = plus(ex, carry);
        if (warp) ex = plus(ex, warp_sum[warp - 1]);
        if (i < n) sums[i] = ex;
        if (i < n && i % chunks == 0) class_start[i / chunks] = ex.rows;
        carry = plus(carry, warp_sum[31]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        sums[n] = carry;
        class_start[kRowClasses] = carry.rows;
    }
    __syncthreads();
    if (threadIdx.x < kRowClasses) counts[threadIdx.x] = class_start[threadIdx.x + 1] - class_start[threadIdx.x];
}

// order[position] = row, start[position] = sums over the rows before it; position m closes both.
__global__ void __launch_bounds__(256) rows_order_kernel(int64_t m, const int64_t* __restrict__ row_ptr, int pack, int task_max, int part_len, int chunks,
                                                         const ClassSum* __restrict__ sums, int32_t* __restrict__ order, int4* __restrict__ start) {
    __shared__ ClassSum before[kRowClasses];              // of the rows of the class before this step's
    __shared__ ClassSum in_warp[8][kRowClasses];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < kRowClasses) before[threadIdx.x] = sums[threadIdx.x * chunks + blockIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const ClassSum& t = sums[chunks * kRowClasses];
        order[m] = 0;
        start[m] = make_int4(t.x, t.y, t.z, t.w);
    }
    for (int j = 0; j < kRowsChunk; j += 256) {
        const int64_t i = static_cast<int64_t>(blockIdx.x) * kRowsChunk + j + threadIdx.x;
        const bool on = i < m;
        const int64_t len = on ? row_ptr[i + 1] - row_ptr[i] : 0;
        const int c = on ? row_class(len, pack, task_max) : -1;
        const int4 s = on ? row_size(len, task_max, part_len) : make_int4(0, 0, 0, 0);
        ClassSum mine = {0, 0, 0, 0, 0};                  // of the rows of this class before this one in the warp
#pragma unroll
        for (int q = 0; q < kRowClasses; ++q) {
            const unsigned same = __ballot_sync(0xffffffffu, c == q);
            ClassSum all = {__popc(same), 0, 0, 0, 0}, ex = {__popc(same & ((1u << lane) - 1u)), 0, 0, 0, 0};
            auto field = [&](int v, int* a, int* e) {
                int x = c == q ? v : 0;
                const int own = x;
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                *a = __shfl_sync(0xffffffffu, x, 31);
                *e = x - own;
            };
            if (same) {                                   // (uniform)
                if (q == 0) {
                    field(s.y, &all.y, &ex.y);
                    field(s.z, &all.z, &ex.z);
                    field(s.w, &all.w, &ex.w);
                } else {
                    field(s.x, &all.x, &ex.x);
                }
            }
            if (c == q) mine = ex;
            if (lane == 0) in_warp[warp][q] = all;
        }
        __syncthreads();
        if (on) {
            ClassSum at = before[c];
            for (int v = 0; v < warp; ++v) {
                const ClassSum& u = in_warp[v][c];
                at.rows += u.rows; at.x += u.x; at.y += u.y; at.z += u.z; at.w += u.w;
            }
            at.rows += mine.rows; at.x += mine.x; at.y += mine.y; at.z += mine.z; at.w += mine.w;
            order[at.rows] = static_cast<int32_t>(i);
            start[at.rows] = make_int4(at.x, at.y, at.z, at.w);
        }
        __syncthreads();
        if (threadIdx.x < kRowClasses)
            for (int v = 0; v < 8; ++v) {
                const ClassSum& u = in_warp[v][threadIdx.x];
                ClassSum& t = before[threadIdx.x];
                t.rows += u.rows; t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
            }
        __syncthreads();
    }
}

// What the later passes need of a plan: positions below n_long are long rows, then n_single tasks of one row, then
// packed rows.
struct RowsPlan {
    int64_t m;
    int pack, part_len;
    const int32_t* counts;
    const int4* start;                   // exclusive sums of row_size's fields
    int n_classes;
    __device__ __forceinline__ int n_long() const { return counts[0]; }
    __device__ __forceinline__ int n_single() const {
        int s = 0;
        for (int c = 1; c + 1 < n_classes; ++c) s += counts[c];
        return s;
    }
    // task of position i (not a long row)
    __device__ __forceinline__ int task(int64_t i, int nl, int ns) const {
        const int64_t p0 = static_cast<int64_t>(nl) + ns;
        return i < p0 ? static_cast<int>(i) - nl : ns + (start[i].x - start[p0].x) / pack;
    }
    __device__ __forceinline__ int begin(int task, int first_entry) const { return (first_entry + 3 * task + 3) / 4 * 4; }
    __device__ __forceinline__ int n_tasks(int nl, int ns) const { return nl < m ? task(m - 1, nl, ns) + 1 : 0; }
    // the long rows' first entry: behind the last task
    __device__ __forceinline__ int long_base(int nl, int ns) const { return (begin(n_tasks(nl, ns), start[m].x) + 7) / 8 * 8; }
};

template <int ES> struct RowsValue { using type = uint16_t; };
template <> struct RowsValue<4> { using type = uint32_t; };

// By position: where the row's entries go (at[row]) and what is not an entry of the matrix (the empty rows, the padding);
// the tasks, the long rows and their parts; totals {tasks, parts, long rows, slots}.
template <int ES>
__global__ void rows_plan_kernel(const RowsPlan p, const int32_t* __restrict__ order, const int64_t* __restrict__ row_ptr, int32_t* __restrict__ at,
                                 int4* __restrict__ tasks, int4* __restrict__ parts, int4* __restrict__ longs, int4* __restrict__ total,
                                 int32_t* __restrict__ col, uint8_t* __restrict__ val) {
    using T = typename RowsValue<ES>::type;
    T* dst = reinterpret_cast<T*>(val);
    const int nl = p.n_long(), ns = p.n_single();
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i <= p.m; i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        if (i == p.m) {
            *total = make_int4(p.n_tasks(nl, ns), p.start[p.m].z, nl, p.start[p.m].w);
            continue;
        }
        const int32_t r = order[i];
        const int n = static_cast<int>(row_ptr[r + 1] - row_ptr[r]);
        if (i < nl) {
            const int4 s = p.start[i];
            const int np = p.start[i + 1].z - s.z;
            const int base = p.long_base(nl, ns) + s.y;
            at[r] = base;
            longs[i] = make_int4(r, s.w, np, 0);
            for (int j = 0; j < np; ++j)
                parts[s.z + j] = make_int4(base + j * p.part_len, min(p.part_len, n - j * p.part_len), static_cast<int>(i), j);
            for (int j = n; j < (n + 7) / 8 * 8; ++j) {
                col[base + j] = 0x7fffffff;
                dst[base + j] = 0;
            }
        } else {
            // (a task of packed rows holds at most `pack` of them: the steps to its first one are few)
            const int t = p.task(i, nl, ns);
            int64_t h = i;
            while (h > nl && p.task(h - 1, nl, ns) == t) --h;
            const int first = p.start[h].x;
            const int base = p.begin(t, first);
            const int to = base + (p.start[i].x - first);
            at[r] = to;
            if (n == 0) {
                col[to] = -1;                              // the sign bit and no gather
                dst[to] = 0;
            }
            if (i == h) {
                int64_t h1 = i + 1;
                while (h1 < p.m && p.task(h1, nl, ns) == t) ++h1;
                const int len = p.start[h1].x - first;
                tasks[t] = make_int4(base, len, static_cast<int>(i), 0);
                for (int j = len; j < (len + 3) / 4 * 4; ++j) {
                    col[base + j] = 0x7fffffff;
                    dst[base + j] = 0;
                }
            }
        }
    }
}

// One thread per entry of the matrix (a CTA per long row took 19 us for 60,000 power-law rows, this 6 for all rows).
template <int ES>
__global__ void rows_fill_kernel(int64_t nnz, int task_max, const int32_t* __restrict__ row_of, const int64_t* __restrict__ row_ptr,
                                 const int32_t* __restrict__ at, const int32_t* __restrict__ col_idx, const uint8_t* __restrict__ vals,
                                 int32_t* __restrict__ col, uint8_t* __restrict__ val) {
    using T = typename RowsValue<ES>::type;
    for (int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < nnz; p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int32_t r = row_of[p];
        const int64_t s = row_ptr[r], e = row_ptr[r + 1];
        const int64_t to = at[r] + (p - s);
        const bool last = p == e - 1 && e - s <= task_max;
        col[to] = col_idx[p] | (last ? static_cast<int32_t>(0x80000000u) : 0);
        reinterpret_cast<T*>(val)[to] = reinterpret_cast<const T*>(vals)[p];
    }
}

// the row of every entry, looked up in row_ptr
__global__ void rows_of_entries_kernel(int64_t m, int64_t nnz, const int64_t* __restrict__ row_ptr, int32_t* __restrict__ row_of) {
    for (int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < nnz; p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int64_t lo = 0, hi = m - 1;                       // last row that starts at or before p
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (row_ptr[mid] <= p) lo = mid; else hi = mid - 1;
        }
        row_of[p] = static_cast<int32_t>(lo);
    }
}

unsigned grid_for(int64_t n, int per) { return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, 4096))); }

}  // namespace

void free_wcsr_rows(WcsrRowStream* s, cudaStream_t st) {
    dev_free(s->d_block, st);
    *s = WcsrRowStream();
}

int finish_wcsr_rows(WcsrRowStream* s, cudaStream_t st) {
    if (!s->d_total) return SPMM_OK;
    int32_t total[4] = {0, 0, 0, 0};
    if (cudaMemcpyAsync(total, s->d_total, sizeof(total), cudaMemcpyDeviceToHost, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return SPMM_ERR_CUDA;
    s->d_total = nullptr;
    s->n_tasks = total[0];
    s->n_parts = total[1];
    s->n_long = total[2];
    s->n_slots = total[3];
    return SPMM_OK;
}

int build_wcsr_rows_device(int64_t m, int64_t nnz, const int64_t* d_row_ptr, const int32_t* d_col_idx, const uint8_t* d_vals,
                           int es, int sms, const int32_t* d_row_of, cudaStream_t st, WcsrRowStream* out) {
    *out = WcsrRowStream();
    if (m <= 0 || (es != 2 && es != 4)) return SPMM_OK;
    // Task sizes by the entries there are per SM and 128 groups: small matrices need short tasks and parts to fill
    // the GPU; in large ones a CTA's start and the reduction at its end weigh more (a part of 512 entries is eight
    // steps of a group).  task_max is pack times a power of two, so that the last length class holds the rows of
    // at most `pack` entries and no others.  Measured (us), {pack, task_max, part_len}, fp16 N = 128 / 320:
    //                                        {16,32,256}  {16,64,512}  {16,64,1024}  {16,128,1024}  {32,128,512}  {32,128,2048}
    //   4000 rows TF32 N = 36 (2 entries)        8.7          13.7                                      23.2
    //   R-MAT 2^15, 16 a row (28)                              21.2 / 39    20.8 / 47     23.7 / 43      24.5 / 40     23.7 / 68
    //   60,000 rows (66)                                      37.8 / 93    34.3 / 98     40.8 / 89      45.7 / 94     39.4 / 118
    //   200,000 rows (137)                                    83.4 / 242   78.4 / 237    75.6 / 237     84.7 / 241    76.4 / 235
    //   R-MAT 2^17 (160)                                      82.0 / 193   77.3 / 187    67.3 / 182     76.1 / 190    71.3 / 183
    //   R-MAT 2^20 (1320)                                     623 / 1694   593 / 1652    527 / 1615     560 / 1648    518 / 1590
    // Below 16, {8, 32, 256} / {16, 32, 256} / {8, 32, 128} / {16, 64, 512}, fp16 N = 64 / 320: 45,000 rows (6)
    // 8.2 / 26.0, 12.5 / 26.5, 8.2 / 23.1, 12.6 / 34.3; R-MAT 2^13, 24 a row (10) 7.1 / 18.6, 7.7 / 18.5, 8.1 / 18.4,
    // 8.0 / 21.3; TF32 N = 64: 7.9, 9.6, 7.8, 11.8 and 8.6, 9.1, 9.4, 14.1.
    const int64_t per = wcsr_rows_load(m, nnz, sms);
    if (per >= 500) { out->pack = 32; out->task_max = 128; out->part_len = 2048; }
    else if (per >= 100) { out->pack = 16; out->task_max = 128; out->part_len = 1024; }
    else if (per >= 50) { out->pack = 16; out->task_max = 64; out->part_len = 1024; }
    else if (per >= 16) { out->pack = 16; out->task_max = 64; out->part_len = 512; }
    else { out->pack = 8; out->task_max = 32; out->part_len = 256; }
    // rows of more than one part have more than part_len nonzeros: at most kRowsMaxSlots parts
    out->part_len = static_cast<int>(std::max<int64_t>(out->part_len, (2 * nnz / kRowsMaxSlots + 127) / 128 * 128));
    // Upper bounds for the arrays, so that nothing has to be read back before the end.  An entry is in a task or in a
    // long row; a task of one row has more than `pack` entries, and the packed rows make a run per `pack` of theirs,
    // the last one begun.
    const int64_t max_tasks = (nnz + m) / out->pack + 2;
    const int64_t max_long = nnz / out->task_max + 1;
    const int64_t max_parts = max_long + nnz / out->part_len + 1;
    const int64_t entries = nnz + m + 3 * max_tasks + 8 * max_long + 16;
    if (entries >= (int64_t{1} << 31) || m >= (int64_t{1} << 31) - 1) return SPMM_OK;

    const int64_t chunks = (m + kRowsChunk - 1) / kRowsChunk;
    auto up = [](int64_t bytes) { return (bytes + 255) / 256 * 256; };
    // places by row | sums by position | sums by class and chunk | rows by class | rows of the entries, where not given
    const int64_t o_start = up(m * 4), o_sums = o_start + up((m + 1) * 16), o_counts = o_sums + up((chunks * kRowClasses + 1) * sizeof(ClassSum));
    const int64_t o_row_of = o_counts + 256, work_bytes = o_row_of + (d_row_of ? 0 : nnz * 4);
    uint8_t* d_work = nullptr;
    auto done = [&](int code) {
        if (code) cudaGetLastError();
        dev_free(d_work, st);
        if (code) free_wcsr_rows(out, st);
        return code;
    };
    const int64_t counter_bytes = 32 + max_long * kRowsMaxTiles * 4;
    const int64_t o_order = 0, o_tasks = o_order + up((m + 1) * 4), o_parts = o_tasks + up(max_tasks * 16), o_longs = o_parts + up(max_parts * 16);
    const int64_t o_col = o_longs + up(max_long * 16), o_val = o_col + up(entries * 4), o_counters = o_val + up(entries * es);
    const int64_t o_total = o_counters + up(counter_bytes);
    if (!dev_alloc_ok(&d_work, static_cast<size_t>(work_bytes), st) || !dev_alloc_ok(&out->d_block, static_cast<size_t>(o_total + 16), st))
        return done(SPMM_ERR_ALLOC);
    out->d_order = reinterpret_cast<int32_t*>(out->d_block + o_order);
    out->d_tasks = reinterpret_cast<int32_t*>(out->d_block + o_tasks);
    out->d_parts = reinterpret_cast<int32_t*>(out->d_block + o_parts);
    out->d_longs = reinterpret_cast<int32_t*>(out->d_block + o_longs);
    out->d_col = reinterpret_cast<int32_t*>(out->d_block + o_col);
    out->d_val = out->d_block + o_val;
    out->d_counters = reinterpret_cast<unsigned*>(out->d_block + o_counters);
    out->d_total = reinterpret_cast<int32_t*>(out->d_block + o_total);
    int32_t* d_at = reinterpret_cast<int32_t*>(d_work);
    int4* d_start = reinterpret_cast<int4*>(d_work + o_start);
    ClassSum* d_sums = reinterpret_cast<ClassSum*>(d_work + o_sums);
    int32_t* d_counts = reinterpret_cast<int32_t*>(d_work + o_counts);
    cudaMemsetAsync(out->d_counters, 0, static_cast<size_t>(counter_bytes), st);
    if (!d_row_of && nnz > 0) {
        int32_t* own = reinterpret_cast<int32_t*>(d_work + o_row_of);
        rows_of_entries_kernel<<<grid_for(nnz, 256), 256, 0, st>>>(m, nnz, d_row_ptr, own);
        d_row_of = own;
    }
    const int nc = static_cast<int>(chunks);
    rows_count_kernel<<<static_cast<unsigned>(chunks), 256, 0, st>>>(m, d_row_ptr, out->pack, out->task_max, out->part_len, nc, d_sums);
    rows_sums_kernel<<<1, 1024, 0, st>>>(nc, d_sums, d_counts);
    rows_order_kernel<<<static_cast<unsigned>(chunks), 256, 0, st>>>(m, d_row_ptr, out->pack, out->task_max, out->part_len, nc, d_sums, out->d_order, d_start);
    RowsPlan p;
    p.m = m;
    p.pack = out->pack;
    p.part_len = out->part_len;
    p.counts = d_counts;
    p.start = d_start;
    p.n_classes = 2;                                         // long, packed, and the classes between
    for (int lim = out->task_max / 2; lim >= out->pack; lim /= 2) ++p.n_classes;
    int4* tasks = reinterpret_cast<int4*>(out->d_tasks);
    int4* parts = reinterpret_cast<int4*>(out->d_parts);
    int4* longs = reinterpret_cast<int4*>(out->d_longs);
    int4* total = reinterpret_cast<int4*>(out->d_total);
    auto plan = [&](auto bytes) {
        constexpr int ES = decltype(bytes)::value;
        rows_plan_kernel<ES><<<grid_for(m + 1, 256), 256, 0, st>>>(p, out->d_order, d_row_ptr, d_at, tasks, parts, longs, total, out->d_col, out->d_val);
        if (nnz > 0)
            rows_fill_kernel<ES><<<grid_for(nnz, 256), 256, 0, st>>>(nnz, out->task_max, d_row_of, d_row_ptr, d_at, d_col_idx, d_vals, out->d_col, out->d_val);
    };
    if (es == 2) plan(std::integral_constant<int, 2>());
    else plan(std::integral_constant<int, 4>());
    return done(cudaGetLastError() == cudaSuccess ? SPMM_OK : SPMM_ERR_CUDA);
}

}  // namespace spmm
