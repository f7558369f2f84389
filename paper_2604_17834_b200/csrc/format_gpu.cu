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
// WCSR (window condensation of Sec. 2.3): every stored entry becomes the 64-bit key
// (window << 32 | column); a radix sort and a unique pass (CUB primitives) leave, window after
// window, the ascending union of each window's columns; where the window changes gives each window's
// place in the key list, a prefix sum window_row_ptr (lengths padded to b_col);
// window_col_idx is those columns over a -1 fill, and every value finds its condensed column by
// binary search in its window's list and goes straight into the packed tile layout.
#include <cub/cub.cuh>

#include <cstring>
#include <numeric>
#include <algorithm>
#include <new>

#include "device_memory.h"
#include "format.h"
#include "kernels.h"
#include "spmm_b200.h"

namespace spmm {

namespace {

constexpr int kThreads = 256;

// Validation in two passes, so that the second one never reads past the arrays: once row_ptr is
// known to start at 0 and to be monotone, every position below row_ptr[m] lies inside col_idx.
// (nnz: receives row_ptr[m] where the caller reads it together with *err; may be null)
__global__ void csr_check_rows_kernel(int64_t m, const int64_t* row_ptr, int* err, int64_t* nnz) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (row_ptr[0] != 0) atomicMin(err, SPMM_ERR_INVALID_ARG);
        if (nnz) *nnz = row_ptr[m];
    }
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < m;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        if (row_ptr[i + 1] < row_ptr[i]) atomicMin(err, SPMM_ERR_INVALID_ARG);
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

// out[0] = 0, out[i + 1] = counts[0] + ... + counts[i]; *overflow set if the total passes int32.
__global__ void __launch_bounds__(1024)
exclusive_scan_kernel(const int32_t* counts, int64_t n, int32_t* out, int* overflow) {
    __shared__ long long warp_sum[32];
    __shared__ long long carry;
    if (threadIdx.x == 0) { carry = 0; out[0] = 0; }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t base = 0; base < n; base += blockDim.x) {
        const int64_t i = base + threadIdx.x;
        long long v = i < n ? counts[i] : 0;
        long long x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        if (warp == 0) {
            long long s = warp_sum[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += y;
            }
            warp_sum[lane] = s;
        }
        __syncthreads();
        const long long incl = carry + (warp ? warp_sum[warp - 1] : 0) + x;
        if (i < n) {
            if (incl >= (1ll << 31)) *overflow = 1;
            out[i + 1] = static_cast<int32_t>(incl);
        }
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = incl;
        __syncthreads();
    }
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
    if (smem > 200 * 1024) return SPMM_ERR_TOO_LARGE;
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
        csr_check_rows_kernel<<<check_grid, 256, 0, st>>>(m, d_row_ptr, d_flags, nullptr);
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
    if (smem > 48 * 1024) {
        cudaFuncSetAttribute(bcsr_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        cudaFuncSetAttribute(bcsr_fill_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        cudaFuncSetAttribute(bcsr_fill_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        cudaFuncSetAttribute(bcsr_fill_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
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

// Entry by entry (a warp per row took four times as long: a row of 5000 entries was one warp's work): the row of
// every entry, looked up in row_ptr, and its key = window << cb | column, cb = bits of a column: no empty bits for
// the radix sort to pass over.
// An entry out of range or not ascending in its row sets *bad and counts as column 0.
__global__ void wcsr_keys_kernel(int64_t m, int64_t k, int wh, int cb, const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx,
                                 uint64_t* __restrict__ keys, int32_t* __restrict__ row_of, int* bad) {
    const int64_t nnz = row_ptr[m];
    for (int64_t p = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; p < nnz; p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int64_t lo = 0, hi = m - 1;                       // last row that starts at or before p
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (row_ptr[mid] <= p) lo = mid; else hi = mid - 1;
        }
        int64_t c = col_idx[p];
        if (c < 0 || c >= k || (p > row_ptr[lo] && col_idx[p - 1] >= c)) {
            *bad = 1;
            c = 0;
        }
        row_of[p] = static_cast<int32_t>(lo);
        keys[p] = static_cast<uint64_t>(lo / wh) << cb | static_cast<uint64_t>(c);
    }
}

// The unique keys ascend, so a window's keys are a run: where each run starts (ustart[nwin] = their number);
// per column: is it referenced at all
__global__ void wcsr_starts_kernel(const uint64_t* __restrict__ ukeys, const int* __restrict__ n_unique, int64_t nwin, int cb,
                                   int32_t* __restrict__ ustart, uint8_t* __restrict__ used) {
    const int64_t n = *n_unique;
    const uint64_t col_mask = (uint64_t{1} << cb) - 1;
    for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j <= n; j += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t w = j < n ? static_cast<int64_t>(ukeys[j] >> cb) : nwin;
        const int64_t before = j > 0 ? static_cast<int64_t>(ukeys[j - 1] >> cb) : -1;
        for (int64_t x = before + 1; x <= w; ++x) ustart[x] = static_cast<int32_t>(j);
        if (j < n) used[ukeys[j] & col_mask] = 1;
    }
}

__global__ void wcsr_pad_kernel(const int32_t* __restrict__ ustart, int64_t nwin, int b_col, int32_t* __restrict__ len) {
    for (int64_t w = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; w < nwin;
         w += static_cast<int64_t>(gridDim.x) * blockDim.x)
        len[w] = (ustart[w + 1] - ustart[w] + b_col - 1) / b_col * b_col;
}

__global__ void wcsr_sum_used_kernel(const uint8_t* used, int64_t k, unsigned long long* total) {
    unsigned long long n = 0;
    for (int64_t c = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; c < k;
         c += static_cast<int64_t>(gridDim.x) * blockDim.x)
        n += used[c];
    for (int o = 16; o > 0; o >>= 1) n += __shfl_down_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(total, n);
}

__global__ void wcsr_cols_kernel(const uint64_t* ukeys, const int* n_unique, int cb, const int32_t* ustart,
                                 const int32_t* window_row_ptr, int32_t* window_col_idx) {
    const int64_t n = *n_unique;
    const uint64_t col_mask = (uint64_t{1} << cb) - 1;
    for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j < n;
         j += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const uint64_t key = ukeys[j];
        const int64_t w = static_cast<int64_t>(key >> cb);
        window_col_idx[window_row_ptr[w] + (j - ustart[w])] = static_cast<int32_t>(key & col_mask);
    }
}

// One thread per entry: its column's place in its window's list, by binary search.
template <int ES>
__global__ void wcsr_values_kernel(int64_t nnz, int wh, int b_col, const int32_t* __restrict__ row_of, const int32_t* __restrict__ col_idx,
                                   const uint8_t* __restrict__ vals, const int32_t* __restrict__ ustart, const int32_t* __restrict__ window_row_ptr,
                                   const int32_t* __restrict__ window_col_idx, uint8_t* __restrict__ packed) {
    for (int64_t p = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; p < nnz; p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int i = row_of[p];
        const int w = i / wh, r = i - w * wh;
        const int64_t base = window_row_ptr[w];
        const int32_t* seg = window_col_idx + base;
        const int32_t c = col_idx[p];
        int lo = 0, hi = ustart[w + 1] - ustart[w];      // first position with seg[pos] >= c; c is in the list
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (seg[mid] < c) lo = mid + 1; else hi = mid;
        }
        uint8_t* dst = packed + wcsr_packed_offset(wh, b_col, ES, r, base + lo);
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

__global__ void wcsr_refs_kernel(const int32_t* __restrict__ col_idx, int64_t P, int32_t* __restrict__ refs) {
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < P; q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int32_t c = col_idx[q];
        if (c >= 0) atomicAdd(refs + c, 1);
    }
}

__global__ void iota_kernel(int32_t* __restrict__ x, int64_t n) {
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        x[i] = static_cast<int32_t>(i);
}

// rows in descending order of their gather count (stable: ties by index): rank r -> class
__global__ void wcsr_class_kernel(const int32_t* __restrict__ sorted_refs, const int32_t* __restrict__ order, int64_t k,
                                  uint8_t* __restrict__ cls) {
    for (int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; r < k; r += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int level = 0;
        if (sorted_refs[r] > 1) {
            level = 7;
            for (int64_t lim = kWcsrTopClassRows; level > 0 && r >= lim; lim *= 2) --level;
        }
        cls[order[r]] = static_cast<uint8_t>(level);
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

// Allocates and fills *d_grp_class [P / 4] from the device copy of window_col_idx, in the order of `st`.
int wcsr_reuse_classes_device(const int32_t* d_window_col_idx, int64_t P, int64_t k, int64_t nwin, cudaStream_t st, uint8_t** d_grp_class) {
    *d_grp_class = nullptr;
    if (P <= 0 || k <= 0) return SPMM_OK;
    int count_bits = 1;                       // a row of B is gathered by nwin windows at most
    while (count_bits < 31 && (int64_t{1} << count_bits) <= nwin) ++count_bits;
    int32_t *refs = nullptr, *refs_sorted = nullptr, *ids = nullptr, *order = nullptr;
    size_t tb = 0;
    cub::DeviceRadixSort::SortPairsDescending(nullptr, tb, refs, refs_sorted, ids, order, static_cast<int>(k), 0, count_bits, st);
    const size_t kb = static_cast<size_t>(k) * 4, step = (kb + 255) / 256 * 256;
    uint8_t* block = nullptr;                 // refs | sorted refs | ids | order | classes | CUB's
    if (!dev_alloc_ok(&block, 5 * step + tb, st) || !dev_alloc_ok(d_grp_class, static_cast<size_t>(P / 4), st)) {
        dev_free(block, st);
        dev_free(*d_grp_class, st);
        *d_grp_class = nullptr;
        return SPMM_ERR_ALLOC;
    }
    refs = reinterpret_cast<int32_t*>(block);
    refs_sorted = reinterpret_cast<int32_t*>(block + step);
    ids = reinterpret_cast<int32_t*>(block + 2 * step);
    order = reinterpret_cast<int32_t*>(block + 3 * step);
    uint8_t* cls = block + 4 * step;
    void* temp = block + 5 * step;
    cudaMemsetAsync(refs, 0, kb, st);
    wcsr_refs_kernel<<<2048, 256, 0, st>>>(d_window_col_idx, P, refs);
    iota_kernel<<<static_cast<unsigned>(std::min<int64_t>((k + 255) / 256, 2048)), 256, 0, st>>>(ids, k);
    bool ok = cub::DeviceRadixSort::SortPairsDescending(temp, tb, refs, refs_sorted, ids, order, static_cast<int>(k), 0, count_bits, st) == cudaSuccess;
    if (ok) {
        wcsr_class_kernel<<<static_cast<unsigned>(std::min<int64_t>((k + 255) / 256, 2048)), 256, 0, st>>>(refs_sorted, order, k, cls);
        wcsr_group_class_kernel<<<2048, 256, 0, st>>>(d_window_col_idx, P / 4, cls, *d_grp_class);
        ok = cudaGetLastError() == cudaSuccess;
    }
    dev_free(block, st);
    if (!ok) {
        cudaGetLastError();
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
        int n_unique;                         // unique keys
        int bad;                              // an entry out of range or not ascending
        int64_t nnz;
        unsigned long long distinct;          // columns that are referenced
    } flags = {};
    Flags* d_flags = nullptr;
    uint8_t* d_work = nullptr;                // keys, sorted keys, rows of the entries, window lengths and starts, column marks, CUB's
    auto release = [&]() { dev_free(d_flags, st); dev_free(d_work, st); };
    auto fail = [&](int code) {
        cudaGetLastError();                  // (of a call that failed: not for a later check to find)
        release();
        dev_free(*d_window_row_ptr, st); dev_free(*d_window_col_idx, st); dev_free(*d_packed, st);
        *d_window_row_ptr = nullptr; *d_window_col_idx = nullptr; *d_packed = nullptr;
        return code;
    };
    auto alloc = [&](void** ptr, size_t bytes) { return dev_alloc(ptr, bytes, st) == cudaSuccess; };

    if (!alloc(reinterpret_cast<void**>(&d_flags), sizeof(Flags))) return fail(SPMM_ERR_ALLOC);
    if (cudaMemsetAsync(d_flags, 0, sizeof(Flags), st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
    auto read_flags = [&]() {
        return cudaMemcpyAsync(&flags, d_flags, sizeof(Flags), cudaMemcpyDeviceToHost, st) == cudaSuccess && cudaStreamSynchronize(st) == cudaSuccess;
    };
    const unsigned check_grid = static_cast<unsigned>(std::min<int64_t>((m + 255) / 256, 2048));
    if (m > 0) csr_check_rows_kernel<<<check_grid, 256, 0, st>>>(m, d_row_ptr, &d_flags->err, &d_flags->nnz);
    if (!read_flags()) return fail(SPMM_ERR_CUDA);
    if (flags.err != 0) return fail(flags.err);
    const int64_t nnz = flags.nnz;
    if (nnz < 0 || (nnz > 0 && (!d_col_idx || !d_vals))) return fail(SPMM_ERR_INVALID_ARG);
    if (nnz >= (int64_t{1} << 31)) return fail(SPMM_ERR_TOO_LARGE);
    *nnz_out = nnz;

    // keys -> sorted -> unique
    const int n = static_cast<int>(nnz);
    const unsigned entry_grid = static_cast<unsigned>(std::min<int64_t>((nnz + 255) / 256, 16384));
    int cb = 1;
    while ((int64_t{1} << cb) < k) ++cb;
    int end_bit = cb + 1;
    while ((int64_t{1} << (end_bit - cb)) < nwin) ++end_bit;
    uint64_t *d_keys = nullptr, *d_keys2 = nullptr;
    size_t t1 = 0, t2 = 0;
    if (n > 0) {
        cub::DeviceRadixSort::SortKeys(nullptr, t1, d_keys, d_keys2, n, 0, end_bit, st);
        cub::DeviceSelect::Unique(nullptr, t2, d_keys2, d_keys, &d_flags->n_unique, n, st);
    }
    size_t work_bytes = 0, tb = std::max(t1, t2);
    auto section = [&](size_t bytes) {
        const size_t at = work_bytes;
        work_bytes += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t o_keys = section(static_cast<size_t>(nnz) * 8), o_keys2 = section(static_cast<size_t>(nnz) * 8);
    const size_t o_row_of = section(static_cast<size_t>(nnz) * 4), o_len = section(static_cast<size_t>(nwin + 1) * 4);
    const size_t o_ustart = section(static_cast<size_t>(nwin + 1) * 4), o_used = section(static_cast<size_t>(k)), o_temp = section(tb);
    if (!alloc(reinterpret_cast<void**>(&d_work), work_bytes) ||
        !alloc(reinterpret_cast<void**>(d_window_row_ptr), static_cast<size_t>(nwin + 1) * 4))
        return fail(SPMM_ERR_ALLOC);
    d_keys = reinterpret_cast<uint64_t*>(d_work + o_keys);
    d_keys2 = reinterpret_cast<uint64_t*>(d_work + o_keys2);
    int32_t* d_row_of = reinterpret_cast<int32_t*>(d_work + o_row_of);
    int32_t* d_len = reinterpret_cast<int32_t*>(d_work + o_len);
    int32_t* d_ustart = reinterpret_cast<int32_t*>(d_work + o_ustart);
    uint8_t* d_used = d_work + o_used;
    void* d_temp = d_work + o_temp;
    cudaMemsetAsync(d_ustart, 0, o_temp - o_ustart, st);       // the starts and the marks behind them
    if (n > 0) {
        wcsr_keys_kernel<<<entry_grid, 256, 0, st>>>(m, k, wh, cb, d_row_ptr, d_col_idx, d_keys, d_row_of, &d_flags->bad);
        if (cub::DeviceRadixSort::SortKeys(d_temp, tb, d_keys, d_keys2, n, 0, end_bit, st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
        if (cub::DeviceSelect::Unique(d_temp, tb, d_keys2, d_keys, &d_flags->n_unique, n, st) != cudaSuccess) return fail(SPMM_ERR_CUDA);
        // d_keys now holds the unique keys
        wcsr_starts_kernel<<<2048, 256, 0, st>>>(d_keys, &d_flags->n_unique, nwin, cb, d_ustart, d_used);
    }
    wcsr_pad_kernel<<<static_cast<unsigned>(std::min<int64_t>((nwin + 255) / 256 + 1, 2048)), 256, 0, st>>>(d_ustart, nwin, b_col, d_len);
    exclusive_scan_kernel<<<1, 1024, 0, st>>>(d_len, nwin, *d_window_row_ptr, &d_flags->overflow);
    if (k > 0) wcsr_sum_used_kernel<<<static_cast<unsigned>(std::min<int64_t>((k + 255) / 256, 1024)), 256, 0, st>>>(d_used, k, &d_flags->distinct);
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
    if (n > 0) {
        wcsr_cols_kernel<<<2048, 256, 0, st>>>(d_keys, &d_flags->n_unique, cb, d_ustart, *d_window_row_ptr, *d_window_col_idx);
        if (es == 1)
            wcsr_values_kernel<1><<<entry_grid, 256, 0, st>>>(nnz, wh, b_col, d_row_of, d_col_idx, d_vals, d_ustart, *d_window_row_ptr, *d_window_col_idx, *d_packed);
        else if (es == 2)
            wcsr_values_kernel<2><<<entry_grid, 256, 0, st>>>(nnz, wh, b_col, d_row_of, d_col_idx, d_vals, d_ustart, *d_window_row_ptr, *d_window_col_idx, *d_packed);
        else
            wcsr_values_kernel<4><<<entry_grid, 256, 0, st>>>(nnz, wh, b_col, d_row_of, d_col_idx, d_vals, d_ustart, *d_window_row_ptr, *d_window_col_idx, *d_packed);
    }
    release();                                // (ordered behind the kernels that use them)
    int rc = cudaGetLastError() == cudaSuccess ? wcsr_reuse_classes_device(*d_window_col_idx, P, k, nwin, st, d_grp_class) : SPMM_ERR_CUDA;
    if (!rc && rows && wcsr_wants_rows(es, m, nnz, P)) {
        rc = build_wcsr_rows_device(m, nnz, d_row_ptr, d_col_idx, d_vals, es, sms, st, rows);
        if (rc == SPMM_ERR_ALLOC) rc = SPMM_OK;          // no room for it: the window kernel serves the handle
    }
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

__global__ void rows_class_kernel(int64_t m, const int64_t* __restrict__ row_ptr, int pack, int task_max, uint8_t* __restrict__ cls,
                                  int32_t* __restrict__ ids, int32_t* __restrict__ counts) {
    __shared__ int n[kRowClasses];
    if (threadIdx.x < kRowClasses) n[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < m; i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int c = row_class(row_ptr[i + 1] - row_ptr[i], pack, task_max);
        cls[i] = static_cast<uint8_t>(c);
        ids[i] = static_cast<int32_t>(i);
        atomicAdd(&n[c], 1);
    }
    __syncthreads();
    if (threadIdx.x < kRowClasses && n[threadIdx.x]) atomicAdd(&counts[threadIdx.x], n[threadIdx.x]);
}

struct Int4Sum {
    __host__ __device__ int4 operator()(const int4& a, const int4& b) const { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
};

// Per position of `order`: {entries (an empty row counts one; a long row none here), padded entries of a long row,
// its parts, its partial slots}; position m closes the scan.
__global__ void rows_size_kernel(int64_t m, const int32_t* __restrict__ order, const int64_t* __restrict__ row_ptr, int task_max, int part_len,
                                 int4* __restrict__ size) {
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i <= m; i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int4 s = make_int4(0, 0, 0, 0);
        if (i < m) {
            const int32_t r = order[i];
            const int n = static_cast<int>(row_ptr[r + 1] - row_ptr[r]);
            if (n <= task_max) {
                s.x = n > 0 ? n : 1;
            } else {
                s.y = (n + 7) / 8 * 8;
                s.z = (n + part_len - 1) / part_len;
                s.w = s.z > 1 ? s.z : 0;
            }
        }
        size[i] = s;
    }
}

// What the later passes need of a plan: positions below n_long are long rows, then n_single tasks of one row, then
// packed rows.
struct RowsPlan {
    int64_t m;
    int pack, part_len;
    const int32_t* counts;
    const int4* start;                   // exclusive sums of rows_size_kernel's fields
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

// task heads; descriptors of the long rows and their parts; totals {tasks, parts, long rows, slots}
__global__ void rows_plan_kernel(const RowsPlan p, const int32_t* __restrict__ order, const int64_t* __restrict__ row_ptr, int32_t* __restrict__ head,
                                 int4* __restrict__ parts, int4* __restrict__ longs, int4* __restrict__ total) {
    const int nl = p.n_long(), ns = p.n_single();
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i <= p.m; i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        if (i == p.m) {
            const int tasks = p.n_tasks(nl, ns);
            head[tasks] = static_cast<int32_t>(p.m);
            *total = make_int4(tasks, p.start[p.m].z, nl, p.start[p.m].w);
        } else if (i < nl) {
            const int4 s = p.start[i];
            const int np = p.start[i + 1].z - s.z;
            const int32_t r = order[i];
            const int n = static_cast<int>(row_ptr[r + 1] - row_ptr[r]);
            const int base = p.long_base(nl, ns);
            longs[i] = make_int4(r, s.w, np, 0);
            for (int j = 0; j < np; ++j)
                parts[s.z + j] = make_int4(base + s.y + j * p.part_len, min(p.part_len, n - j * p.part_len), static_cast<int>(i), j);
        } else {
            const int t = p.task(i, nl, ns);
            if (i == nl || t != p.task(i - 1, nl, ns)) head[t] = static_cast<int32_t>(i);
        }
    }
}

template <int ES> struct RowsValue { using type = uint16_t; };
template <> struct RowsValue<4> { using type = uint32_t; };

// eight lanes per position: a row's nonzeros to their place in its task, the task's descriptor and padding
template <int ES>
__global__ void rows_fill_kernel(const RowsPlan p, const int32_t* __restrict__ order, const int32_t* __restrict__ head,
                                 const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx, const uint8_t* __restrict__ vals,
                                 int4* __restrict__ tasks, int32_t* __restrict__ col, uint8_t* __restrict__ val) {
    using T = typename RowsValue<ES>::type;
    const T* src = reinterpret_cast<const T*>(vals);
    T* dst = reinterpret_cast<T*>(val);
    const int nl = p.n_long(), ns = p.n_single();
    const int sub = threadIdx.x & 7;
    for (int64_t i = nl + ((static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 3); i < p.m;
         i += (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 3) {
        const int t = p.task(i, nl, ns);
        const int h = head[t], h1 = head[t + 1];
        const int first = p.start[h].x;
        const int64_t base = p.begin(t, first);
        const int64_t at = base + (p.start[i].x - first);
        const int32_t r = order[i];
        const int64_t s = row_ptr[r];
        const int n = static_cast<int>(row_ptr[r + 1] - s);
        if (n == 0 && sub == 0) {
            col[at] = -1;                                  // the sign bit and no gather
            dst[at] = 0;
        }
        for (int j = sub; j < n; j += 8) {
            col[at + j] = col_idx[s + j] | (j == n - 1 ? static_cast<int32_t>(0x80000000u) : 0);
            dst[at + j] = src[s + j];
        }
        if (i == h) {
            const int len = p.start[h1].x - first;
            if (sub == 0) tasks[t] = make_int4(static_cast<int>(base), len, h, 0);
            if (sub < 4 && len + sub < (len + 3) / 4 * 4) {
                col[base + len + sub] = 0x7fffffff;
                dst[base + len + sub] = 0;
            }
        }
    }
}

// one CTA per long row
template <int ES>
__global__ void rows_fill_long_kernel(const RowsPlan p, const int32_t* __restrict__ order, const int64_t* __restrict__ row_ptr,
                                      const int32_t* __restrict__ col_idx, const uint8_t* __restrict__ vals, int32_t* __restrict__ col,
                                      uint8_t* __restrict__ val) {
    using T = typename RowsValue<ES>::type;
    const T* src = reinterpret_cast<const T*>(vals);
    T* dst = reinterpret_cast<T*>(val);
    const int nl = p.n_long();
    if (static_cast<int>(blockIdx.x) >= nl) return;
    const int base = p.long_base(nl, p.n_single());
    for (int i = blockIdx.x; i < nl; i += gridDim.x) {
        const int32_t r = order[i];
        const int64_t s = row_ptr[r], n = row_ptr[r + 1] - s, at = base + p.start[i].y;
        for (int64_t j = threadIdx.x; j < (n + 7) / 8 * 8; j += blockDim.x) {
            col[at + j] = j < n ? col_idx[s + j] : 0x7fffffff;
            dst[at + j] = j < n ? src[s + j] : T(0);
        }
    }
}

unsigned grid_for(int64_t n, int per) { return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, 4096))); }

}  // namespace

void free_wcsr_rows(WcsrRowStream* s, cudaStream_t st) {
    void* const arrays[] = {s->d_order, s->d_tasks, s->d_parts, s->d_longs, s->d_col, s->d_val, s->d_counters, s->d_total};
    for (void* ptr : arrays) dev_free(ptr, st);
    *s = WcsrRowStream();
}

int finish_wcsr_rows(WcsrRowStream* s, cudaStream_t st) {
    if (!s->d_total) return SPMM_OK;
    int32_t total[4] = {0, 0, 0, 0};
    if (cudaMemcpyAsync(total, s->d_total, sizeof(total), cudaMemcpyDeviceToHost, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return SPMM_ERR_CUDA;
    dev_free(s->d_total, st);
    s->d_total = nullptr;
    s->n_tasks = total[0];
    s->n_parts = total[1];
    s->n_long = total[2];
    s->n_slots = total[3];
    return SPMM_OK;
}

int build_wcsr_rows_device(int64_t m, int64_t nnz, const int64_t* d_row_ptr, const int32_t* d_col_idx, const uint8_t* d_vals,
                           int es, int sms, cudaStream_t st, WcsrRowStream* out) {
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

    uint8_t *d_cls = nullptr, *d_cls2 = nullptr;
    int32_t *d_ids = nullptr, *d_counts = nullptr, *d_head = nullptr;
    int4 *d_size = nullptr, *d_start = nullptr;
    void* d_temp = nullptr;
    auto done = [&](int code) {
        if (code) cudaGetLastError();
        void* const arrays[] = {d_cls, d_cls2, d_ids, d_counts, d_head, d_size, d_start, d_temp};
        for (void* ptr : arrays) dev_free(ptr, st);
        if (code) free_wcsr_rows(out, st);
        return code;
    };
    auto alloc = [&](auto** ptr, int64_t bytes) { return dev_alloc_ok(ptr, static_cast<size_t>(bytes), st); };
    size_t t1 = 0, t2 = 0;
    const int4 zero = make_int4(0, 0, 0, 0);
    cub::DeviceRadixSort::SortPairs(nullptr, t1, d_cls, d_cls2, d_ids, out->d_order, static_cast<int>(m), 0, 3, st);
    cub::DeviceScan::ExclusiveScan(nullptr, t2, d_size, d_start, Int4Sum(), zero, static_cast<int>(m + 1), st);
    size_t tb = std::max(t1, t2);
    const int64_t counter_bytes = 32 + max_long * kRowsMaxTiles * 4;
    if (!alloc(&d_cls, m) || !alloc(&d_cls2, m) || !alloc(&d_ids, m * 4) || !alloc(&d_counts, kRowClasses * 4) || !alloc(&d_head, (max_tasks + 1) * 4) ||
        !alloc(&d_size, (m + 1) * 16) || !alloc(&d_start, (m + 1) * 16) || !alloc(&d_temp, static_cast<int64_t>(tb)) ||
        !alloc(&out->d_order, (m + 1) * 4) || !alloc(&out->d_tasks, max_tasks * 16) || !alloc(&out->d_parts, max_parts * 16) ||
        !alloc(&out->d_longs, max_long * 16) || !alloc(&out->d_col, entries * 4) || !alloc(&out->d_val, entries * es) ||
        !alloc(&out->d_counters, counter_bytes) || !alloc(&out->d_total, 16))
        return done(SPMM_ERR_ALLOC);
    cudaMemsetAsync(d_counts, 0, kRowClasses * 4, st);
    cudaMemsetAsync(out->d_order + m, 0, 4, st);
    cudaMemsetAsync(out->d_counters, 0, static_cast<size_t>(counter_bytes), st);
    rows_class_kernel<<<grid_for(m, 256), 256, 0, st>>>(m, d_row_ptr, out->pack, out->task_max, d_cls, d_ids, d_counts);
    if (cub::DeviceRadixSort::SortPairs(d_temp, tb, d_cls, d_cls2, d_ids, out->d_order, static_cast<int>(m), 0, 3, st) != cudaSuccess)
        return done(SPMM_ERR_CUDA);
    rows_size_kernel<<<grid_for(m + 1, 256), 256, 0, st>>>(m, out->d_order, d_row_ptr, out->task_max, out->part_len, d_size);
    if (cub::DeviceScan::ExclusiveScan(d_temp, tb, d_size, d_start, Int4Sum(), zero, static_cast<int>(m + 1), st) != cudaSuccess)
        return done(SPMM_ERR_CUDA);
    RowsPlan p;
    p.m = m;
    p.pack = out->pack;
    p.part_len = out->part_len;
    p.counts = d_counts;
    p.start = d_start;
    p.n_classes = 2;                                         // long, packed, and the classes between
    for (int lim = out->task_max / 2; lim >= out->pack; lim /= 2) ++p.n_classes;
    int4* tasks = reinterpret_cast<int4*>(out->d_tasks);
    rows_plan_kernel<<<grid_for(m + 1, 256), 256, 0, st>>>(p, out->d_order, d_row_ptr, d_head, reinterpret_cast<int4*>(out->d_parts),
                                                          reinterpret_cast<int4*>(out->d_longs), reinterpret_cast<int4*>(out->d_total));
    const unsigned lg = static_cast<unsigned>(std::min<int64_t>(max_long, 8192));
    if (es == 2) {
        rows_fill_kernel<2><<<grid_for(m * 8, 256), 256, 0, st>>>(p, out->d_order, d_head, d_row_ptr, d_col_idx, d_vals, tasks, out->d_col, out->d_val);
        rows_fill_long_kernel<2><<<lg, 256, 0, st>>>(p, out->d_order, d_row_ptr, d_col_idx, d_vals, out->d_col, out->d_val);
    } else {
        rows_fill_kernel<4><<<grid_for(m * 8, 256), 256, 0, st>>>(p, out->d_order, d_head, d_row_ptr, d_col_idx, d_vals, tasks, out->d_col, out->d_val);
        rows_fill_long_kernel<4><<<lg, 256, 0, st>>>(p, out->d_order, d_row_ptr, d_col_idx, d_vals, out->d_col, out->d_val);
    }
    return done(cudaGetLastError() == cudaSuccess ? SPMM_OK : SPMM_ERR_CUDA);
}

}  // namespace spmm
