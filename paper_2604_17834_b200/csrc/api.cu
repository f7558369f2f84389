// C-ABI layer: handles, format upload, tensor maps, launches (see include/spmm_b200.h).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <memory>
#include <new>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "device_memory.h"
#include "format.h"
#include "kernels.h"
#include "spmm_b200.h"

using namespace spmm;

namespace {

// NVTX range around an entry point (a no-op unless a profiler is attached).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// A CUDA call of this library has failed: its error must not be found again by a later call's check of its launches.
int cuda_error() {
    cudaGetLastError();
    return SPMM_ERR_CUDA;
}

std::atomic<uint64_t> g_wait_limit_ns{2000000000ull};

inline int elem_size(int dtype) { return dtype == SPMM_TF32 ? 4 : (dtype == SPMM_FP8_E4M3 ? 1 : 2); }

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

inline CUtensorMapDataType tmap_dtype(int dtype) {
    return dtype == SPMM_FP8_E4M3 ? CU_TENSOR_MAP_DATA_TYPE_UINT8
         : (dtype == SPMM_TF32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
         : (dtype == SPMM_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16));
}

// 2-D row-major tensor [rows][cols] of the handle's value type, box [box_rows][box_cols].
int encode_2d(CUtensorMap* map, int dtype, const void* base, uint64_t rows, uint64_t cols,
                    uint32_t box_rows, uint32_t box_cols, CUtensorMapSwizzle swz) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return cuda_error();
    const uint64_t es = static_cast<uint64_t>(elem_size(dtype));
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * es};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUtensorMapDataType dt = tmap_dtype(dtype);
    CUresult r = fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? SPMM_OK : cuda_error();
}

// In the order of the default stream: finish_uploads makes what was uploaded ready for every stream (a copy from
// pageable memory may still be on its way when cudaMemcpy returns).
template <class T>
int upload(T** dptr, const void* src, size_t bytes) {
    *dptr = nullptr;
    if (!dev_alloc_ok(dptr, bytes, nullptr)) return SPMM_ERR_ALLOC;
    if (bytes && cudaMemcpy(*dptr, src, bytes, cudaMemcpyHostToDevice) != cudaSuccess) return cuda_error();
    return SPMM_OK;
}
int finish_uploads() { return cudaStreamSynchronize(nullptr) == cudaSuccess ? SPMM_OK : cuda_error(); }

}  // namespace

struct spmm_handle_s {
    int format = 0;      // 0 BCSR, 1 WCSR
    int dtype = 0;
    int es = 2;
    int64_t m = 0, k = 0, nnz = 0;
    bool host_only = false;
    bool c16 = false;        // C in the input's 16-bit type (never with TF32, whose input type is fp32)
    bool col_major = false;  // BCSR: B given as X[N][k], C as Y[N][m]
    bool dynamic = false;    // BCSR: tiles handed out at run time through Cluster Launch Control
    bool want_rows = false;  // WCSR: no option asks for the window kernel or describes its plan
    bool lsu_gather = false; // WCSR: B rows gathered by the load/store units (comparison variant) instead of TMA
    int cs = 4;              // bytes per C element
    int n_ctas = 148;
    int sms = 148;
    int device = 0;

    BcsrHost bcsr;       // index arrays kept; value array dropped after upload unless host_only
    WcsrHost wcsr;

    // device copies
    int32_t* d_ptr = nullptr;        // block_row_ptr / window_row_ptr
    int32_t* d_idx = nullptr;        // block_col_idx / window_col_idx
    uint8_t* d_vals = nullptr;       // blocks / packed values
    int32_t* d_order = nullptr;      // BCSR row order
    BcsrSchedule sched;              // BCSR tile schedule of the most recent dense width
    // BCSR row groups (stacked 128-row blocks): plan, device arrays and their own tile schedule
    BcsrStack stack;
    int stack_min_fill = 0;          // opts.stack_min_fill
    BcsrSchedule sched_stack;
    int32_t* d_sidx = nullptr;       // block columns of the stacked blocks
    int32_t* d_srows = nullptr;      // [groups][R] member block-rows
    uint8_t* d_svals = nullptr;      // [stacked blocks][128][b]
    int32_t* d_stile_recs = nullptr; // {group, token tile, first stacked block, end}
    int32_t* d_scta_ptr = nullptr;
    CUtensorMap tmAs;                // map of d_svals
    int stack_groups = 0;            // token groups of the stacked launch's tile (2, or 1: see ensure_schedule)
    // launches by half tiles (see ensure_schedule; a function of the handle and N), and their maps: boxes of 64 rows of stacked
    // blocks, and, where split, of 64 tokens of X and of 16 tokens of C or Y
    bool split = false, stack_split = false;
    CUtensorMap tmAsh, tmBh, tmCh;
    CUtensorMap tmB3s;               // whole-tile map of B for the stacked launch's token tile
    bool tmB3s_ok = false;
    int k_split = 0;                 // opts.k_split (1: cut outlier block-rows into parts)
    int32_t* d_kmerge = nullptr;     // K-split merge lists: row | first slot | parts, each [n_kmerge]
    int n_kmerge = 0;
    CUtensorMap tmP;                 // store map of the K-split partial tiles
    bool tmP_ok = false;
    int32_t* d_tiles = nullptr;      // {block-row, token tile} pairs (the exported schedule)
    int32_t* d_tile_recs = nullptr;  // the kernel's records: {block-row, token tile, first block, end block}
    int32_t* d_cta_ptr = nullptr;
    // WCSR schedule: sections of d_plan (d_grp_class: or an array of its own, d_class, from the GPU builder)
    int32_t* d_plan = nullptr;
    const WcsrDevTask* d_tasks = nullptr;
    const int32_t* d_bin_ptr = nullptr;
    const int32_t* d_bin_tasks = nullptr;
    const int32_t* d_items = nullptr;
    const int32_t* d_fills = nullptr;
    const int32_t* d_bin_fill = nullptr;
    const int32_t* d_fills_narrow = nullptr;    // WCSR narrow-operand variant (2-byte types, height 16)
    const int32_t* d_bin_fill_narrow = nullptr;
    uint8_t* d_class = nullptr;
    const uint8_t* d_grp_class = nullptr;  // WCSR: reuse class per group of four padded columns (gather hints)
    const int32_t* d_merge = nullptr;      // window | first | nparts, each [n_merge]
    int n_merge = 0;
    int* d_status = nullptr;
    WcsrRowStream rows;              // WCSR: the nonzeros for the row kernel (empty: the window kernel serves the handle)

    float* d_partial = nullptr;      // WCSR workspace
    size_t partial_bytes = 0;
    bool partial_pooled = true;      // false: from cudaMalloc (see ensure_wcsr_workspace)

    // BCSR tensor maps
    CUtensorMap tmA, tmA1;           // (tmA1: for tiles of 128 tokens, whose stages hold more blocks)
    bool tmA_ok = false;
    CUtensorMap tmB;
    CUtensorMap tmB3;                // BCSR: B as [N / 64][k][64] for whole-tile loads
    bool tmB3_ok = false;
    int tmB_groups = 0;
    const void* tmB_ptr = nullptr;
    int64_t tmB_N = -1;
    CUtensorMap tmC;                 // BCSR: the store map of C (or of Y, column-major)
    const void* tmC_ptr = nullptr;
    int64_t tmC_N = -1;

    // staging for spmm_run_host
    void* d_Bstage = nullptr;
    size_t Bstage_bytes = 0;
    float* d_Cstage = nullptr;
    size_t Cstage_bytes = 0;
    // spmm_run_host in column chunks: the copy streams and the events that order them
    static constexpr int kMaxHostChunks = 8;
    cudaStream_t s_in = nullptr, s_out = nullptr;
    cudaEvent_t ev_start = nullptr, ev_in[kMaxHostChunks] = {}, ev_run[kMaxHostChunks] = {};
};

namespace {

void free_partial(spmm_handle_s* h) {
    if (h->partial_pooled) dev_free(h->d_partial, nullptr);
    else cudaFree(h->d_partial);
    h->d_partial = nullptr;
    h->partial_bytes = 0;
    h->partial_pooled = true;
}

void free_handle(spmm_handle_s* h) {
    if (!h) return;
    if (!h->host_only) {
        // the handle's last run may still be on the GPU; its memory goes back to the pool of its own device
        int dev = -1;
        const bool other = cudaGetDevice(&dev) == cudaSuccess && dev != h->device && cudaSetDevice(h->device) == cudaSuccess;
        cudaDeviceSynchronize();
        void* const arrays[] = {
            h->d_ptr, h->d_idx, h->d_vals, h->d_order, h->d_tiles, h->d_tile_recs, h->d_cta_ptr, h->d_kmerge,
            h->d_sidx, h->d_srows, h->d_svals, h->d_stile_recs, h->d_scta_ptr, h->d_status,
            h->d_plan, h->d_class};
        for (void* ptr : arrays) dev_free(ptr, nullptr);
        free_partial(h);
        free_wcsr_rows(&h->rows, nullptr);
        dev_give_back();
        if (other) cudaSetDevice(dev);
        cudaFree(h->d_Bstage);
        cudaFree(h->d_Cstage);
        if (h->s_in) cudaStreamDestroy(h->s_in);
        if (h->s_out) cudaStreamDestroy(h->s_out);
        if (h->ev_start) cudaEventDestroy(h->ev_start);
        for (int i = 0; i < spmm_handle_s::kMaxHostChunks; ++i) {
            if (h->ev_in[i]) cudaEventDestroy(h->ev_in[i]);
            if (h->ev_run[i]) cudaEventDestroy(h->ev_run[i]);
        }
    }
    delete h;
}

// `stream`: the creation's own, which it synchronises before it returns the handle.
int device_setup(spmm_handle_s* h, const spmm_opts_t* opts, cudaStream_t stream) {
    if (h->host_only) {
        h->sms = 148;
        h->n_ctas = (opts && opts->n_ctas > 0) ? opts->n_ctas : 148;
        return SPMM_OK;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cuda_error();
    int major = 0, sms = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return cuda_error();
    if (major != 10) return SPMM_ERR_UNSUPPORTED;   // sm_100a code only
    h->device = dev;
    h->sms = sms;
    h->n_ctas = (opts && opts->n_ctas > 0) ? opts->n_ctas : h->sms;
    if (!dev_alloc_ok(&h->d_status, 4 * sizeof(int), stream)) return SPMM_ERR_ALLOC;
    if (cudaMemsetAsync(h->d_status, 0, 4 * sizeof(int), stream) != cudaSuccess) return cuda_error();
    return SPMM_OK;
}

int check_opts(const spmm_opts_t* opts) {
    if (!opts) return SPMM_OK;
    if (opts->c_type != SPMM_C_FP32 && opts->c_type != SPMM_C_SAME_AS_INPUT) return SPMM_ERR_INVALID_ARG;
    if (opts->layout != SPMM_ROWMAJOR && opts->layout != SPMM_COLMAJOR) return SPMM_ERR_INVALID_ARG;
    if (opts->schedule != SPMM_SCHED_STATIC && opts->schedule != SPMM_SCHED_DYNAMIC) return SPMM_ERR_INVALID_ARG;
    if (opts->gather < SPMM_GATHER_AUTO || opts->gather > SPMM_GATHER_TMA) return SPMM_ERR_INVALID_ARG;
    return SPMM_OK;
}

// Option checks shared by the host and the device builder; on success *hp is a fresh handle.
int new_bcsr_handle(spmm_handle_s** hp, int64_t m, int64_t k, int dtype, int block, const spmm_opts_t* opts) {
    if (dtype != SPMM_BF16 && dtype != SPMM_FP16 && dtype != SPMM_FP8_E4M3 && dtype != SPMM_TF32) return SPMM_ERR_UNSUPPORTED;
    if (int orc = check_opts(opts)) return orc;
    // TF32 (Sec. 3.1's k8 shape, the type of Sec. 4.1's BCSR evaluation): static schedule only
    if (dtype == SPMM_TF32 && opts && opts->schedule != SPMM_SCHED_STATIC) return SPMM_ERR_UNSUPPORTED;
    if (dtype == SPMM_FP8_E4M3) {
        // 8-bit inputs: fp32 C, static schedule; a block row must hold a whole 32-element K step;
        // with column-major operands the rows of X are k bytes and must be multiples of 16
        if (opts && (opts->c_type != SPMM_C_FP32 || opts->schedule != SPMM_SCHED_STATIC)) return SPMM_ERR_UNSUPPORTED;
        if (block < 32) return SPMM_ERR_UNSUPPORTED;
        if (opts && opts->layout == SPMM_COLMAJOR && k % 16 != 0) return SPMM_ERR_UNSUPPORTED;
    }
    spmm_handle_s* h = new (std::nothrow) spmm_handle_s;
    if (!h) return SPMM_ERR_ALLOC;
    h->format = 0;
    h->dtype = dtype;
    h->es = elem_size(dtype);
    h->m = m;
    h->k = k;
    h->host_only = opts && opts->host_only;
    h->c16 = opts && opts->c_type == SPMM_C_SAME_AS_INPUT && dtype != SPMM_TF32;   // TF32's own type is fp32
    h->cs = h->c16 ? 2 : 4;
    h->col_major = opts && opts->layout == SPMM_COLMAJOR;
    h->dynamic = opts && opts->schedule == SPMM_SCHED_DYNAMIC;
    h->stack_min_fill = opts ? opts->stack_min_fill : 0;
    h->k_split = opts ? opts->k_split : 0;
    if (h->stack_min_fill > 100) { delete h; return SPMM_ERR_INVALID_ARG; }
    if (h->dynamic && (h->c16 || h->col_major)) { delete h; return SPMM_ERR_UNSUPPORTED; }
    // column-major operands: rows of X (k elements) and of Y (m elements) must be multiples of
    // 16 bytes for the tensor map and for the 16-byte pieces the epilogue writes
    if (h->col_major && (m % 8 != 0 || (k * h->es) % 16 != 0)) { delete h; return SPMM_ERR_UNSUPPORTED; }
    *hp = h;
    return SPMM_OK;
}

// Map of stored blocks: box of `rows` rows of min(b * es, 128) bytes (a stage unit's: the whole block row, or one column
// slice of it, at most 128 bytes per piece), swizzle = the row bytes.
int encode_blocks(const spmm_handle_s* h, CUtensorMap* map, const void* blocks, int64_t total_rows, int rows) {
    const int b = h->bcsr.b;
    const int unit_bytes = b / bcsr_k_split(b, h->es) * h->es;
    const int row_bytes = unit_bytes < 128 ? unit_bytes : 128;
    const CUtensorMapSwizzle swz = row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                  : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    return encode_2d(map, h->dtype, blocks, static_cast<uint64_t>(total_rows), b, static_cast<uint32_t>(rows), row_bytes / h->es, swz);
}

// Tensor maps of the stored blocks.
int encode_tmA(spmm_handle_s* h) {
    const BcsrHost& f = h->bcsr;
    if (f.nnzb <= 0) return SPMM_OK;
    if (static_cast<int64_t>(f.nnzb) * f.b >= (int64_t{1} << 31)) return SPMM_ERR_TOO_LARGE;
    int rc = encode_blocks(h, &h->tmA, h->d_vals, f.nnzb * f.b, f.b * bcsr_blocks_per_stage(f.b, h->es, 2));
    if (!rc) rc = encode_blocks(h, &h->tmA1, h->d_vals, f.nnzb * f.b, f.b * bcsr_blocks_per_stage(f.b, h->es, 1));
    h->tmA_ok = rc == SPMM_OK;
    return rc;
}

// Row groups: the plan from the index arrays, then (unless host_only) the stacked values built on
// the device from the uploaded blocks, the groups' index arrays and the map of the stacked values.
int setup_stack(spmm_handle_s* h) {
    const BcsrHost& f = h->bcsr;
    // static schedule only; b = 128 blocks already are 128 rows high
    // (row groups exist for the 16-bit types, for TF32 with block rows of up to 128 bytes, and for E4M3 with column-major operands)
    const bool eligible = !h->dynamic && f.b < 128 && h->stack_min_fill >= 0 && !(h->dtype == SPMM_TF32 && f.b > 32) &&
                          !(h->dtype == SPMM_FP8_E4M3 && !h->col_major);
    int rc = build_bcsr_stack(f, eligible ? h->stack_min_fill : -1, &h->stack);
    if (rc || h->host_only || h->stack.ng == 0) return rc;
    const BcsrStack& st = h->stack;
    rc = stack_bcsr_device(h->d_vals, st, f.b, h->es, &h->d_svals);
    if (!rc) rc = upload(&h->d_sidx, st.col_idx.data(), st.col_idx.size() * 4);
    if (!rc) rc = upload(&h->d_srows, st.rows.data(), st.rows.size() * 4);
    if (rc) return rc;
    std::vector<int32_t>().swap(h->stack.src);        // only needed to build the values
    rc = encode_blocks(h, &h->tmAs, h->d_svals, st.ns * kStackRows, kStackRows);         // (block rows of at most 128 bytes)
    return rc ? rc : encode_blocks(h, &h->tmAsh, h->d_svals, st.ns * kStackRows, kStackRows / 2);
}

int create_bcsr(spmm_handle_t* out, const CsrView& a, int dtype, int block, const spmm_opts_t* opts) {
    spmm_handle_s* h = nullptr;
    int rc = new_bcsr_handle(&h, a.m, a.k, dtype, block, opts);
    if (rc) return rc;
    rc = validate_csr(a);
    if (rc) { delete h; return rc; }
    h->nnz = a.nnz;
    rc = device_setup(h, opts, nullptr);
    if (rc) { free_handle(h); return rc; }
    try {
        rc = build_bcsr(a, block, &h->bcsr);
    } catch (const std::bad_alloc&) {
        rc = SPMM_ERR_ALLOC;
    }
    if (rc) { free_handle(h); return rc; }
    if (!h->host_only) {
        const BcsrHost& f = h->bcsr;
        if (static_cast<int64_t>(f.nnzb) * f.b >= (int64_t{1} << 31)) { free_handle(h); return SPMM_ERR_TOO_LARGE; }
        rc = upload(&h->d_ptr, f.block_row_ptr.data(), f.block_row_ptr.size() * 4);
        if (!rc) rc = upload(&h->d_idx, f.block_col_idx.data(), f.block_col_idx.size() * 4);
        if (!rc) rc = upload(&h->d_vals, f.blocks.data(), f.blocks.size());
        if (!rc) rc = upload(&h->d_order, f.row_order.data(), f.row_order.size() * 4);
        if (!rc) rc = encode_tmA(h);
        if (rc) { free_handle(h); return rc; }
        std::vector<uint8_t>().swap(h->bcsr.blocks);   // the device copy is the one that counts
    }
    try {
        rc = setup_stack(h);
    } catch (const std::bad_alloc&) {
        rc = SPMM_ERR_ALLOC;
    }
    if (!rc && !h->host_only) rc = finish_uploads();
    if (rc) { free_handle(h); return rc; }
    *out = h;
    return SPMM_OK;
}

// The same handle from a CSR matrix in device memory: the format is built by GPU kernels.
int create_bcsr_device(spmm_handle_t* out, int64_t m, int64_t k, const int64_t* d_row_ptr, const int32_t* d_col_idx,
                       const void* d_vals, int dtype, int block, const spmm_opts_t* opts, cudaStream_t stream) {
    if (opts && opts->host_only) return SPMM_ERR_INVALID_ARG;
    spmm_handle_s* h = nullptr;
    int rc = new_bcsr_handle(&h, m, k, dtype, block, opts);
    if (rc) return rc;
    rc = device_setup(h, opts, stream);
    if (rc) { free_handle(h); return rc; }
    try {
        rc = build_bcsr_device(m, k, d_row_ptr, d_col_idx, static_cast<const uint8_t*>(d_vals), h->es, block, stream,
                               &h->bcsr, &h->nnz, &h->d_ptr, &h->d_idx, &h->d_vals);
    } catch (const std::bad_alloc&) {
        rc = SPMM_ERR_ALLOC;
    }
    if (!rc) rc = upload(&h->d_order, h->bcsr.row_order.data(), h->bcsr.row_order.size() * 4);
    if (!rc) rc = encode_tmA(h);
    if (!rc) {
        try {
            rc = setup_stack(h);
        } catch (const std::bad_alloc&) {
            rc = SPMM_ERR_ALLOC;
        }
    }
    if (!rc) rc = finish_uploads();
    if (rc) { free_handle(h); return rc; }
    *out = h;
    return SPMM_OK;
}

// Uploads the schedule arrays of a WCSR handle (everything but the three format arrays): one allocation, one copy.
// In the order of `stream` (the host arrays have been read when it returns).
int upload_wcsr_plan(spmm_handle_s* h, cudaStream_t stream) {
    const WcsrHost& f = h->wcsr;
    const size_t nt = f.tasks.size(), nm = f.merge_window.size(), ni = f.bin_tasks.size();
    const bool narrow = !f.bin_fill_narrow.empty();
    // sections in 4-byte words, each on a 16-byte boundary
    size_t words = 0;
    auto section = [&](size_t n) {
        const size_t at = words;
        words += (n + 3) / 4 * 4;
        return at;
    };
    const size_t o_tasks = section(4 * nt), o_bin_ptr = section(f.bin_ptr.size()), o_bin_tasks = section(ni), o_items = section(4 * ni);
    const size_t o_item_fill = section(f.item_fill.size()), o_bin_fill = section(f.bin_fill.size());
    const size_t o_item_fill_n = section(f.item_fill_narrow.size()), o_bin_fill_n = section(f.bin_fill_narrow.size());
    const size_t o_merge = section(3 * nm), o_class = section((f.grp_class.size() + 3) / 4);
    const size_t n_words = words;
    const std::unique_ptr<int32_t[]> w(new int32_t[n_words]);          // (what lies between the sections is never read)
    // the fills themselves are written on the GPU, behind what is copied
    const size_t o_fills = section(2 * static_cast<size_t>(f.item_fill.empty() ? 0 : f.item_fill.back()));
    const size_t o_fills_n = section(2 * static_cast<size_t>(narrow ? f.item_fill_narrow.back() : 0));
    static_assert(sizeof(WcsrDevTask) == 16, "four words per task");
    for (size_t i = 0; i < nt; ++i) {
        const WcsrTask& t = f.tasks[i];
        const WcsrDevTask d = {f.window_row_ptr[t.window] + t.q0, t.count, t.window, t.slot};
        std::memcpy(&w[o_tasks + 4 * i], &d, 16);
    }
    for (size_t i = 0; i < ni; ++i) {
        const WcsrTask& t = f.tasks[f.bin_tasks[i]];
        w[o_items + 4 * i] = t.window;
        w[o_items + 4 * i + 1] = t.slot;
        w[o_items + 4 * i + 2] = t.count;
        w[o_items + 4 * i + 3] = 0;
    }
    auto put = [&](size_t at, const void* src, size_t bytes) {
        if (bytes) std::memcpy(&w[at], src, bytes);
    };
    put(o_bin_ptr, f.bin_ptr.data(), f.bin_ptr.size() * 4);
    put(o_bin_tasks, f.bin_tasks.data(), ni * 4);
    put(o_item_fill, f.item_fill.data(), f.item_fill.size() * 4);
    put(o_bin_fill, f.bin_fill.data(), f.bin_fill.size() * 4);
    put(o_item_fill_n, f.item_fill_narrow.data(), f.item_fill_narrow.size() * 4);
    put(o_bin_fill_n, f.bin_fill_narrow.data(), f.bin_fill_narrow.size() * 4);
    put(o_merge, f.merge_window.data(), nm * 4);
    put(o_merge + nm, f.merge_first.data(), nm * 4);
    put(o_merge + 2 * nm, f.merge_nparts.data(), nm * 4);
    put(o_class, f.grp_class.data(), f.grp_class.size());
    if (!dev_alloc_ok(&h->d_plan, words * 4, stream)) return SPMM_ERR_ALLOC;
    if (cudaMemcpyAsync(h->d_plan, w.get(), n_words * 4, cudaMemcpyHostToDevice, stream) != cudaSuccess) return cuda_error();
    int32_t* fills = h->d_plan + o_fills;
    int32_t* fills_n = h->d_plan + o_fills_n;
    if (expand_wcsr_fills(static_cast<int64_t>(ni), h->d_plan + o_tasks, h->d_plan + o_bin_tasks, h->d_plan + o_item_fill, f.kt, fills, stream) != cudaSuccess ||
        (narrow && expand_wcsr_fills(static_cast<int64_t>(ni), h->d_plan + o_tasks, h->d_plan + o_bin_tasks, h->d_plan + o_item_fill_n,
                                     kWcsrNarrowCols, fills_n, stream) != cudaSuccess))
        return cuda_error();
    h->n_merge = static_cast<int>(nm);
    h->d_tasks = reinterpret_cast<WcsrDevTask*>(h->d_plan + o_tasks);
    h->d_bin_ptr = h->d_plan + o_bin_ptr;
    h->d_bin_tasks = h->d_plan + o_bin_tasks;
    h->d_items = h->d_plan + o_items;
    h->d_fills = fills;
    h->d_bin_fill = h->d_plan + o_bin_fill;
    if (narrow) {
        h->d_fills_narrow = fills_n;
        h->d_bin_fill_narrow = h->d_plan + o_bin_fill_n;
    }
    h->d_merge = h->d_plan + o_merge;
    if (!f.grp_class.empty()) {
        h->d_grp_class = reinterpret_cast<const uint8_t*>(h->d_plan + o_class);
        std::vector<uint8_t>().swap(h->wcsr.grp_class);
    }
    return SPMM_OK;
}

// Option and size checks shared by the host and the device builder; on success *hp is a fresh handle.
int new_wcsr_handle(spmm_handle_s** hp, int64_t m, int64_t k, int dtype, const spmm_opts_t* opts, int* b_col_out, int* T_out) {
    if (dtype != SPMM_BF16 && dtype != SPMM_FP16 && dtype != SPMM_TF32 && dtype != SPMM_FP8_E4M3) return SPMM_ERR_UNSUPPORTED;
    if (int orc = check_opts(opts)) return orc;
    if (opts && opts->layout == SPMM_COLMAJOR) return SPMM_ERR_UNSUPPORTED;   // BCSR only
    // 8-bit inputs: fp32 C, the TMA gather
    if (dtype == SPMM_FP8_E4M3 && opts && (opts->c_type != SPMM_C_FP32 || opts->gather == SPMM_GATHER_LSU)) return SPMM_ERR_UNSUPPORTED;
    if (opts && opts->schedule == SPMM_SCHED_DYNAMIC) return SPMM_ERR_UNSUPPORTED;
    const int es = elem_size(dtype);
    const int b_col_default = 32 / es;
    const int b_col = (opts && opts->b_col > 0) ? opts->b_col : b_col_default;
    if (b_col != b_col_default) return SPMM_ERR_UNSUPPORTED;
    const int T = (opts && opts->split_cols > 0) ? opts->split_cols : 0;   // 0: chosen from the matrix
    if (T % b_col != 0) return SPMM_ERR_INVALID_ARG;
    spmm_handle_s* h = new (std::nothrow) spmm_handle_s;
    if (!h) return SPMM_ERR_ALLOC;
    h->format = 1;
    h->dtype = dtype;
    h->es = es;
    h->m = m;
    h->k = k;
    h->host_only = opts && opts->host_only;
    h->c16 = opts && opts->c_type == SPMM_C_SAME_AS_INPUT && dtype != SPMM_TF32;
    h->cs = h->c16 ? 2 : 4;
    h->lsu_gather = opts && opts->gather == SPMM_GATHER_LSU;
    h->want_rows = !opts || (opts->gather == SPMM_GATHER_AUTO && opts->split_cols <= 0 && opts->n_ctas <= 0);
    if (h->lsu_gather && h->c16) { delete h; return SPMM_ERR_UNSUPPORTED; }   // the comparison variant writes fp32 C
    *hp = h;
    *b_col_out = b_col;
    *T_out = T;
    return SPMM_OK;
}

int create_wcsr(spmm_handle_t* out, const CsrView& a, int dtype, int wh, const spmm_opts_t* opts) {
    spmm_handle_s* h = nullptr;
    int b_col = 0, T = 0;
    int rc = new_wcsr_handle(&h, a.m, a.k, dtype, opts, &b_col, &T);
    if (rc) return rc;
    if (h->lsu_gather && wh != 16) { delete h; return SPMM_ERR_UNSUPPORTED; }
    rc = validate_csr(a);
    if (rc) { delete h; return rc; }
    h->nnz = a.nnz;
    rc = device_setup(h, opts, nullptr);
    if (rc) { free_handle(h); return rc; }
    try {
        rc = build_wcsr(a, wh, b_col, T, h->n_ctas * wcsr_bins_per_sm(h->es, wh), &h->wcsr);
    } catch (const std::bad_alloc&) {
        rc = SPMM_ERR_ALLOC;
    }
    if (rc) { free_handle(h); return rc; }
    if (!h->host_only) {
        const WcsrHost& f = h->wcsr;
        rc = upload(&h->d_ptr, f.window_row_ptr.data(), f.window_row_ptr.size() * 4);
        if (!rc) rc = upload(&h->d_idx, f.window_col_idx.data(), f.window_col_idx.size() * 4);
        if (!rc) rc = upload(&h->d_vals, f.packed.data(), f.packed.size());
        try {
            if (!rc) rc = upload_wcsr_plan(h, nullptr);
        } catch (const std::bad_alloc&) {
            rc = SPMM_ERR_ALLOC;
        }
        if (!rc && h->want_rows && wcsr_wants_rows(a.es, a.m, a.nnz, f.P)) {
            int64_t* d_rp = nullptr;
            int32_t* d_ci = nullptr;
            uint8_t* d_va = nullptr;
            rc = upload(&d_rp, a.row_ptr, static_cast<size_t>(a.m + 1) * 8);
            if (!rc) rc = upload(&d_ci, a.col_idx, static_cast<size_t>(a.nnz) * 4);
            if (!rc) rc = upload(&d_va, a.vals, static_cast<size_t>(a.nnz) * a.es);
            if (!rc) rc = build_wcsr_rows_device(a.m, a.nnz, d_rp, d_ci, d_va, a.es, h->sms, nullptr, nullptr, &h->rows);
            if (!rc) rc = finish_wcsr_rows(&h->rows, nullptr);
            dev_free(d_rp, nullptr);
            dev_free(d_ci, nullptr);
            dev_free(d_va, nullptr);
            if (rc == SPMM_ERR_ALLOC) {          // no room for the row stream: the window kernel serves the handle
                free_wcsr_rows(&h->rows, nullptr);
                rc = SPMM_OK;
            }
        }
        if (!rc) rc = finish_uploads();
        if (rc) { free_handle(h); return rc; }
        std::vector<uint8_t>().swap(h->wcsr.packed);
    }
    *out = h;
    return SPMM_OK;
}

// The same handle from a CSR matrix in device memory: the format arrays are built by GPU kernels.
int create_wcsr_device(spmm_handle_t* out, int64_t m, int64_t k, const int64_t* d_row_ptr, const int32_t* d_col_idx,
                       const void* d_vals, int dtype, int wh, const spmm_opts_t* opts, cudaStream_t stream) {
    if (opts && opts->host_only) return SPMM_ERR_INVALID_ARG;
    spmm_handle_s* h = nullptr;
    int b_col = 0, T = 0;
    int rc = new_wcsr_handle(&h, m, k, dtype, opts, &b_col, &T);
    if (rc) return rc;
    if (h->lsu_gather && wh != 16) { delete h; return SPMM_ERR_UNSUPPORTED; }
    rc = device_setup(h, opts, stream);
    if (rc) { free_handle(h); return rc; }
    try {
        rc = build_wcsr_device(m, k, d_row_ptr, d_col_idx, static_cast<const uint8_t*>(d_vals), h->es, wh, b_col, T,
                               h->n_ctas * wcsr_bins_per_sm(h->es, wh), h->sms, stream, &h->wcsr, &h->nnz, &h->d_ptr, &h->d_idx,
                               &h->d_vals, &h->d_class, h->want_rows ? &h->rows : nullptr);
        h->d_grp_class = h->d_class;
        if (!rc) rc = upload_wcsr_plan(h, stream);
        if (!rc) rc = finish_wcsr_rows(&h->rows, stream);
    } catch (const std::bad_alloc&) {
        rc = SPMM_ERR_ALLOC;
    }
    if (!rc && cudaStreamSynchronize(stream) != cudaSuccess) rc = cuda_error();
    if (rc) { free_handle(h); return rc; }
    *out = h;
    return SPMM_OK;
}

int make_view(CsrView* v, int64_t m, int64_t k, const int64_t* row_ptr, const int32_t* col_idx, const void* vals,
              int dtype) {
    if (dtype < 0 || dtype > 3) return SPMM_ERR_INVALID_ARG;
    if (m < 0 || k < 0 || !row_ptr) return SPMM_ERR_INVALID_ARG;
    if (m >= (int64_t{1} << 31) || k >= (int64_t{1} << 31)) return SPMM_ERR_TOO_LARGE;
    v->m = m;
    v->k = k;
    v->row_ptr = row_ptr;
    v->nnz = row_ptr[m];
    v->col_idx = col_idx;
    v->vals = static_cast<const uint8_t*>(vals);
    v->es = elem_size(dtype);
    return SPMM_OK;
}

// Map of B for the WCSR row gather: box = one row x 128 bytes.
int encode_gather_map(CUtensorMap* map, int dtype, const void* base, uint64_t rows, uint64_t cols) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return cuda_error();
    const uint32_t es = static_cast<uint32_t>(elem_size(dtype));
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * es};
    const cuuint32_t box[2] = {128 / es, 1};
    const cuuint32_t estr[2] = {1, 1};
    const CUtensorMapDataType dt = tmap_dtype(dtype);
    const CUtensorMapSwizzle swz = dtype == SPMM_TF32 ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : CU_TENSOR_MAP_SWIZZLE_128B;
    const CUtensorMapL2promotion promo = cols * es >= 128 ? CU_TENSOR_MAP_L2_PROMOTION_L2_128B : CU_TENSOR_MAP_L2_PROMOTION_NONE;
    CUresult r = fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                    promo, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? SPMM_OK : cuda_error();
}

int ensure_tmB(spmm_handle_s* h, const void* B, int64_t N, int groups) {
    if (h->tmB_ptr == B && h->tmB_N == N && h->tmB_groups == groups) return SPMM_OK;
    int rc;
    if (h->format == 1) {
        rc = encode_gather_map(&h->tmB, h->dtype, B, static_cast<uint64_t>(h->k), static_cast<uint64_t>(N));
    } else if (h->col_major) {
        // X as [N][k]: box = 128 tokens x min(b, 64) elements, swizzle = the box's row bytes;
        // and the same memory as [N / 128][128][k] so that one request brings all token groups
        // of a tile (whole groups only; a ragged last tile uses the 2-D map, zero filled)
        // (per stage unit: the block's k extent, or one column slice of it -- bcsr_k_split)
        const uint32_t unit_bytes = h->bcsr.b / bcsr_k_split(h->bcsr.b, h->es) * h->es;
        const uint32_t row_bytes = unit_bytes < 128 ? unit_bytes : 128;
        const uint32_t bw = row_bytes / h->es;
        const CUtensorMapSwizzle swz = row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                      : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
        rc = encode_2d(&h->tmB, h->dtype, B, static_cast<uint64_t>(N), static_cast<uint64_t>(h->k), 128, bw, swz);
        if (!rc && h->split) rc = encode_2d(&h->tmBh, h->dtype, B, static_cast<uint64_t>(N), static_cast<uint64_t>(h->k), 64, bw, swz);
        EncodeTiledFn fn = get_encode_fn();
        auto whole_tile_map = [&](int g, CUtensorMap* out, bool* ok) {
            *ok = false;
            *out = h->tmB;
            if (rc || !fn || N < 128) return;
            const cuuint64_t dims[3] = {static_cast<cuuint64_t>(h->k), 128, static_cast<cuuint64_t>(N / 128)};
            const cuuint64_t strides[2] = {static_cast<cuuint64_t>(h->k) * h->es, static_cast<cuuint64_t>(h->k) * 128 * h->es};
            const cuuint32_t box[3] = {bw, 128, static_cast<cuuint32_t>(g)};
            const cuuint32_t estr[3] = {1, 1, 1};
            const CUtensorMapDataType dt = tmap_dtype(h->dtype);
            CUresult r = fn(out, dt, 3, const_cast<void*>(B), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            *ok = r == CUDA_SUCCESS;
            if (!*ok) *out = h->tmB;
        };
        whole_tile_map(groups, &h->tmB3, &h->tmB3_ok);
        if (h->stack.ng > 0 && h->stack_groups > 0) whole_tile_map(h->stack_groups, &h->tmB3s, &h->tmB3s_ok);
    } else {
        // B as [k][N]: box = kb rows (the block's k extent, or one column slice of A's block:
        // bcsr_k_split) x 128 bytes of tokens; 4-byte elements take the 128-byte swizzle with
        // 32-byte atoms, which is what a token-major (MN-major) tensor-core operand of that
        // width reads
        const uint32_t tok = 128u / static_cast<uint32_t>(h->es);          // tokens per box row
        const uint32_t kb = static_cast<uint32_t>(h->bcsr.b / bcsr_k_split(h->bcsr.b, h->es));
        const CUtensorMapSwizzle swz = h->es == 4 ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : CU_TENSOR_MAP_SWIZZLE_128B;
        rc = encode_2d(&h->tmB, h->dtype, B, static_cast<uint64_t>(h->k), static_cast<uint64_t>(N), kb, tok, swz);
        h->tmBh = h->tmB;
        // the same memory as [N / tok][k][tok]: one request then brings a whole token tile
        // (es * groups boxes); only full groups of tok tokens are covered, a ragged tail uses tmB
        EncodeTiledFn fn = get_encode_fn();
        auto whole_tile_map = [&](int g, CUtensorMap* out, bool* ok) {
            *ok = false;
            *out = h->tmB;
            if (rc || !fn || N < static_cast<int64_t>(tok)) return;
            const cuuint64_t dims[3] = {tok, static_cast<cuuint64_t>(h->k), static_cast<cuuint64_t>(N / tok)};
            const cuuint64_t strides[2] = {static_cast<cuuint64_t>(N) * h->es, 128};
            const cuuint32_t box[3] = {tok, kb, static_cast<cuuint32_t>(h->es * g)};
            const cuuint32_t estr[3] = {1, 1, 1};
            CUresult r = fn(out, tmap_dtype(h->dtype), 3, const_cast<void*>(B), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            *ok = r == CUDA_SUCCESS;
            if (!*ok) *out = h->tmB;
        };
        whole_tile_map(groups, &h->tmB3, &h->tmB3_ok);
        if (h->stack.ng > 0 && h->stack_groups > 0) whole_tile_map(h->stack_groups, &h->tmB3s, &h->tmB3s_ok);
    }
    if (rc) return rc;
    h->tmB_ptr = B;
    h->tmB_N = N;
    h->tmB_groups = groups;
    return SPMM_OK;
}

// Store map of C for the BCSR epilogue (shared-memory staging tile -> TMA store).
int ensure_tmC(spmm_handle_s* h, void* C, int64_t N) {
    if (h->tmC_ptr == C && h->tmC_N == N) return SPMM_OK;
    if (h->col_major && h->c16) return SPMM_OK;          // stored without a map
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return cuda_error();
    const uint32_t w = static_cast<uint32_t>(bcsr_epi_cols(h->bcsr.b, h->c16, h->col_major));
    const CUtensorMapDataType dt = !h->c16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                 : (h->dtype == SPMM_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16);
    const cuuint32_t estr[2] = {1, 1};
    auto encode = [&](CUtensorMap* map, cuuint32_t tokens) {
        if (h->col_major) {                  // (fp32: box rows of 64 bytes)
            const cuuint64_t dims[2] = {static_cast<cuuint64_t>(h->m), static_cast<cuuint64_t>(N)};
            const cuuint64_t strides[1] = {static_cast<cuuint64_t>(h->m) * h->cs};
            const cuuint32_t box[2] = {w, tokens};
            return fn(map, dt, 2, C, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                      CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        }
        const cuuint64_t dims[2] = {static_cast<cuuint64_t>(N), static_cast<cuuint64_t>(h->m)};
        const cuuint64_t strides[1] = {static_cast<cuuint64_t>(N) * h->cs};
        const cuuint32_t box[2] = {tokens, w};
        return fn(map, dt, 2, C, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult r = encode(&h->tmC, 32);
    if (r == CUDA_SUCCESS && h->split) r = encode(&h->tmCh, 16);
    if (r != CUDA_SUCCESS) return cuda_error();
    h->tmC_ptr = C;
    h->tmC_N = N;
    return SPMM_OK;
}

// Gives the device arrays of the schedule back; no run may be using them.
void drop_schedule(spmm_handle_s* h) {
    int32_t** const arrays[] = {&h->d_tiles, &h->d_tile_recs, &h->d_cta_ptr, &h->d_stile_recs, &h->d_scta_ptr, &h->d_kmerge};
    for (int32_t** a : arrays) {
        dev_free(*a, nullptr);
        *a = nullptr;
    }
    h->n_kmerge = 0;
    h->tmP_ok = false;
    h->sched.N = -1;
}

// The device arrays of a schedule (and of its row groups', where it has any).
int upload_schedule(spmm_handle_s* h, const BcsrSchedule& sc, const BcsrSchedule& ss, int64_t N) {
    const BcsrHost& f = h->bcsr;
    const BcsrStack& st = h->stack;
    int rc = upload(&h->d_tiles, sc.tiles.data(), sc.tiles.size() * 4);
    if (!rc) {
        // self-contained records, so that a role needs one load per tile (and can fetch it a tile ahead)
        const size_t nt = sc.tiles.size() / 2;
        std::vector<int32_t> recs(4 * nt);
        for (size_t i = 0; i < nt; ++i) {
            recs[4 * i + 1] = sc.tiles[2 * i + 1];
            if (sc.units.empty()) {
                const int32_t I = sc.tiles[2 * i];
                recs[4 * i] = I;
                recs[4 * i + 2] = f.block_row_ptr[I];
                recs[4 * i + 3] = f.block_row_ptr[I + 1];
            } else {
                // K-split: the tile names a unit {block-row, first block, end block, slot}; a part
                // carries -1 - slot in place of the block-row
                const int32_t* u = &sc.units[4 * static_cast<size_t>(sc.tiles[2 * i])];
                recs[4 * i] = u[3] < 0 ? u[0] : -1 - u[3];
                recs[4 * i + 2] = u[1];
                recs[4 * i + 3] = u[2];
            }
        }
        rc = upload(&h->d_tile_recs, recs.data(), recs.size() * 4);
    }
    if (!rc && sc.n_slots > 0) {
        // merge lists (split block-rows in ascending order: their slots are consecutive), the
        // partial tiles' workspace and its store map
        // (the parts of a block-row are consecutive units, in part order)
        std::vector<int32_t> rows, firsts, parts;
        for (size_t u = 0; u < sc.units.size() / 4; ++u) {
            const int32_t I = sc.units[4 * u], slot = sc.units[4 * u + 3];
            if (slot < 0) continue;
            if (rows.empty() || rows.back() != I) { rows.push_back(I); firsts.push_back(slot); parts.push_back(0); }
            parts.back()++;
        }
        std::vector<int32_t> mg;
        mg.insert(mg.end(), rows.begin(), rows.end());
        mg.insert(mg.end(), firsts.begin(), firsts.end());
        mg.insert(mg.end(), parts.begin(), parts.end());
        h->n_kmerge = static_cast<int>(rows.size());
        rc = upload(&h->d_kmerge, mg.data(), mg.size() * 4);
        const size_t need = static_cast<size_t>(sc.n_slots) * f.b * static_cast<size_t>(N) * 4;
        if (!rc && need > h->partial_bytes) {
            if (h->d_partial) {
                if (cudaDeviceSynchronize() != cudaSuccess) rc = cuda_error();
                else free_partial(h);
            }
            if (!rc && !dev_alloc_ok(&h->d_partial, need, nullptr)) rc = SPMM_ERR_ALLOC;
            if (!rc) h->partial_bytes = need;
        }
        if (!rc) {
            EncodeTiledFn fn = get_encode_fn();
            const cuuint64_t dims[2] = {static_cast<cuuint64_t>(N), static_cast<cuuint64_t>(sc.n_slots) * f.b};
            const cuuint64_t strides[1] = {static_cast<cuuint64_t>(N) * 4};
            const cuuint32_t box[2] = {32, static_cast<cuuint32_t>(bcsr_epi_cols(f.b, false, false))};
            const cuuint32_t estr[2] = {1, 1};
            if (!fn || fn(&h->tmP, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, h->d_partial, dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                rc = cuda_error();
            else
                h->tmP_ok = true;
        }
    }
    if (!rc) rc = upload(&h->d_cta_ptr, sc.cta_ptr.data(), sc.cta_ptr.size() * 4);
    if (!rc && !ss.tiles.empty()) {
        const size_t nt = ss.tiles.size() / 2;
        std::vector<int32_t> recs(4 * nt);
        for (size_t i = 0; i < nt; ++i) {
            const int32_t g = ss.tiles[2 * i];
            recs[4 * i] = g;
            recs[4 * i + 1] = ss.tiles[2 * i + 1];
            recs[4 * i + 2] = st.ptr[g];
            recs[4 * i + 3] = st.ptr[g + 1];
        }
        rc = upload(&h->d_stile_recs, recs.data(), recs.size() * 4);
        if (!rc) rc = upload(&h->d_scta_ptr, ss.cta_ptr.data(), ss.cta_ptr.size() * 4);
    }
    return rc ? rc : finish_uploads();
}

// Bytes that the longest tile of a launch brings into shared memory, from which on it runs by half tiles.
constexpr int64_t kSplitMinBytes = 768 << 10;

// Tile width, slab width and the tile schedule for dense width N (cached for the last N).
int ensure_schedule(spmm_handle_s* h, int64_t N) {
    if (h->sched.N == N) return SPMM_OK;
    const BcsrHost& f = h->bcsr;
    // token tile: the largest of 512 / 256 / 128 columns that divides N (Sec. 4.3: pick a tile
    // width that divides the dense width so that no padded columns are computed); otherwise
    // the largest tile, whose ragged last tile is predicated.
    const int gmax = bcsr_token_groups_max(h->dtype, f.b, h->c16 ? 1 : 0, h->col_major ? 1 : 0);
    int groups = 0;
    for (int g = gmax; g >= 1; g >>= 1)
        if (N % (128 * g) == 0) { groups = g; break; }
    if (!groups) groups = N >= 128 * gmax ? gmax : (N > 128 ? 2 : 1);
    // keep at least ~8 tiles per CTA so that the schedule has something to balance
    while (groups > 1 && f.nbr * ((N + 128 * groups - 1) / (128 * groups)) < 8 * h->n_ctas) groups >>= 1;
    const int bnt = 128 * groups;
    const int n_tt = static_cast<int>((N + bnt - 1) / bnt);
    // slab: token tiles whose B rows (k x slab columns) stay within ~16 MB of L2 (C streams through the same cache)
    const int64_t slab_cols = (int64_t{16} << 20) / (h->k * h->es > 0 ? h->k * h->es : 1);
    int64_t sw = slab_cols / bnt;
    if (sw < 1) sw = 1;
    if (sw > n_tt) sw = n_tt;
    BcsrSchedule sc, ss;
    const BcsrStack& st = h->stack;
    int rc;
    // Where the 128-token tiles of a launch are half as many as the CTAs or fewer, each is computed by two CTAs: half of
    // its tokens in either, or, where 128-row stacked blocks are multiplied, half of their rows.  An SM's load rate and its
    // tensor core bound such a launch; an SM then loads (64 + b) / (128 + b) as much (0.56 / 0.60 / 0.67 / 0.75; stacked blocks
    // 0.75).  The sums are the same.  Only from kSplitMinBytes in the longest tile on (shorter ones are latencies, and two CTAs
    // fetch the blocks, or the tokens, twice); row groups only where their longest tile, not the work as a whole, decides when
    // the last CTA ends.  us:
    //   1500 x 9000, b = 64, 10 % full rows, fp16, N = 200 (3.4 MB a tile)   35.0 -> 22.5
    //   3000 x 16000, b = 16, 10 % full rows, bf16, N = 256 (8 MB, grouped)  93.2 -> 67.9
    //   600 x 6000, b = 16, 10 % full rows, TF32, N = 200 (6 MB, grouped)    55.2 -> 41.6
    //   3000 x 6000, b = 32, 10 % full rows, fp16, N = 512 (3 MB, grouped)   25.9 -> 26.6: left alone
    //   1024 x 4096 and back, b = 64, density 0.2, N = 300 (0.3 MB)          10.7 -> 11.0: left alone
    //   6000 x 5000, b = 32, TF32, N = 1500 (5 MB; 3.7 MB of work per CTA)   48.8 -> 60.7: left alone
    // Row groups of 150 random skewed products: 1.02 to 1.66 of the speed with whole tiles, none slower.  Plain blocks, speed
    // over that with whole tiles, at 0.8 - 1 / 2 - 2.5 MB a tile and 8 to 66 tiles; with 74 (148 CTAs):
    //   bf16  b = 16   row-major 1.00 - 1.01 / 1.01 - 1.02; 1.01    column-major 1.20 - 1.23 / 1.24 - 1.25; 1.20
    //         b = 32             0.98 - 1.01 / 0.99 - 1.02; 1.02                 1.14 - 1.18 / 1.22 - 1.24; 1.16
    //         b = 64             1.07 - 1.15 / 1.14 - 1.17; 1.11 - 1.29          1.09 - 1.20 / 1.18 - 1.20; 1.14 - 1.31
    //         b = 128            0.99 - 1.09 / 1.05 - 1.14; 1.04 - 1.16          1.05 - 1.14 / 1.08 - 1.17; 1.10 - 1.20
    //   E4M3  b = 32 / 64 / 128                                                  1.27 - 1.32 / 1.05 - 1.12 / 0.98 - 1.05; 1.06 - 1.33
    //   TF32  b = 16   row-major 0.97 - 0.99 / 0.99 - 1.00; 0.97 - 1.00                column-major 1.08 - 1.10 / 1.14; 1.08
    //         b = 32             1.00 - 1.05 / 1.04 - 1.07; 1.07 - 1.17          1.00 - 1.07 / 1.03 - 1.07; 1.09 - 1.17
    //         b = 64             0.95 - 1.00 / 0.95 - 0.97; 0.99 - 1.07          0.95 - 1.03 / 0.94 - 1.02; 0.99 - 1.06
    //         b = 128            0.94 - 1.01 / 0.96 - 1.03; 0.97 - 1.19          0.98 - 1.04 / 0.99 - 1.03; 1.01 - 1.20
    // so that TF32 blocks of 64, and row-major ones of 128 of less than 4 MB a tile, are halved only where that fills the grid
    // (66 tiles of 5 MB, b = 64: 1.04).
    // Those are widths of whole tiles of whole 128-byte lines.  A ragged or misaligned row-major tile takes a request per 32
    // tokens, fewer in a half: TF32, N = 72 / 120 / 200 / 248 / 500, b = 64 1.04 - 1.07 / 1.09 - 1.12 / 1.04 - 1.07 / 1.10 - 1.13 / 1.48,
    // b = 128 1.00 - 1.04 / 1.15 - 1.25 / 1.10 - 1.18 / 1.15 - 1.24 / 1.31 - 1.39, b = 16 1.03 / 1.13 / 1.03 / 1.12 / 1.51; whole
    // lines, N = 160 / 320: b = 64 0.98 / 1.03, others 0.97; N = 96, b = 64 1.03 - 1.07.
    // (One MMA of two CTAs, cta_group::2, in their place: 16.3 for the fourth, 70 for the last: with N = 64 or 128 its
    // exchange of the other half's block rows takes longer than the product.)
    bool split = false, stack_split = false;
    auto split_fits = [&](int64_t n_tiles, int64_t longest, int64_t rows) {
        const int64_t bytes = longest * (128 + rows) * f.b * h->es;
        if (rows == f.b && h->es == 4) {
            const bool very_long = bytes >= int64_t{4} << 20, fills = 32 * n_tiles > (very_long ? 14 : 15) * h->n_ctas;
            const bool even = N % 32 == 0 && !(f.b == 64 && N % 128 >= 64);
            if (h->col_major ? f.b == 64 && !fills
                             : even && (f.b == 16 || (!fills && (f.b == 64 || (f.b == 128 && !very_long))))) return false;
        }
        return N > 64 && 2 * n_tiles <= h->n_ctas && bytes >= kSplitMinBytes && !h->dynamic && !(h->dtype == SPMM_FP8_E4M3 && !h->col_major);
    };
    // Such a launch has two CTAs to each of the first lists, as many as there are tiles: they hold all of them (tiles are dealt to
    // the least loaded CTA, the first of several), or it is none.
    auto in_first_lists = [](const BcsrSchedule& s) {
        const size_t n = s.tiles.size() / 2;
        return n < s.cta_ptr.size() && static_cast<size_t>(s.cta_ptr[n]) == n;
    };
    try {
        // dynamic scheduling: one list in the global order (slab by slab, longest block-row first)
        // b = 64 gains little per stacked block (its MMAs, not the operand traffic, bound it), so
        // its row groups are used only when they make at least one tile per CTA
        const int64_t n_tt_groups = (N + 128 * kStackGroups - 1) / (128 * kStackGroups);
        const bool use_groups = st.ng > 0 && (f.b <= 32 || st.ng * n_tt_groups >= h->n_ctas);
        if (!use_groups) {
            // K-split of outlier block-rows: static schedule, fp32 row-major C (the parts' partial
            // tiles are fp32 and go through the same epilogue as C)
            rc = SPMM_OK;
            // (opt-in: measured 2 - 7 % slower than the uncut plan on the skewed sweep -- the parts'
            // extra epilogues and the merge launch cost more than the better balance returns)
            if (!h->dynamic && !h->c16 && !h->col_major && h->k_split > 0)
                rc = build_bcsr_ksplit(f, n_tt, h->n_ctas, &sc.units, &sc.n_slots, &sc.cap);
            if (!rc && !sc.units.empty()) {
                const int32_t nu = static_cast<int32_t>(sc.units.size() / 4);
                std::vector<int32_t> order(static_cast<size_t>(nu)), lens(static_cast<size_t>(nu));
                for (int32_t u = 0; u < nu; ++u) order[u] = u;
                auto ulen = [&](int32_t u) { return sc.units[4 * u + 2] - sc.units[4 * u + 1]; };
                std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return ulen(x) > ulen(y); });
                for (int32_t r = 0; r < nu; ++r) lens[r] = ulen(order[r]);
                rc = build_tile_schedule(order, lens, kTileFixedCost, n_tt, static_cast<int>(sw), h->n_ctas, &sc);
            } else if (!rc) {
                rc = build_bcsr_schedule(f, n_tt, static_cast<int>(sw), h->dynamic ? 1 : h->n_ctas, &sc);
                const int32_t I = f.nbr > 0 ? f.row_order[0] : 0;
                split = !rc && groups == 1 && f.nbr > 0 && split_fits(f.nbr * n_tt, f.block_row_ptr[I + 1] - f.block_row_ptr[I], f.b) && in_first_lists(sc);
            }
        } else {
            // The row groups get a launch and a schedule of their own; the launch of the remaining
            // block-rows starts on the SMs the first one leaves idle, CTA after CTA as they free up.
            // CTAs are dispatched in index order, so CTA j of the second launch starts when the
            // j-th lightest CTA of the first one is done: its list is dealt with that head start.
            const int bnt_s = 128 * kStackGroups;
            const int n_tt_s = static_cast<int>((N + bnt_s - 1) / bnt_s);
            int64_t sws = slab_cols / bnt_s;
            if (sws < 1) sws = 1;
            if (sws > n_tt_s) sws = n_tt_s;
            std::vector<int32_t> units, lens;
            for (int64_t g = 0; g < st.ng; ++g) {
                units.push_back(static_cast<int32_t>(g));
                lens.push_back(st.ptr[g + 1] - st.ptr[g]);
            }
            std::vector<int64_t> loads;
            rc = build_tile_schedule(units, lens, kStackTileFixedCost, n_tt_s, static_cast<int>(sws), h->n_ctas, &ss,
                                     bcsr_stack_block_cost(kStackGroups), nullptr, &loads);
            ss.groups = kStackGroups;
            ss.N = N;
            if (!rc) {
                std::sort(loads.begin(), loads.end());
                units.clear();
                lens.clear();
                for (int64_t r = 0; r < f.nbr; ++r) {
                    const int32_t I = f.row_order[r];
                    if (st.stacked[I]) continue;
                    units.push_back(I);
                    lens.push_back(f.block_row_ptr[I + 1] - f.block_row_ptr[I]);
                }
                std::vector<int64_t> totals;
                rc = build_tile_schedule(units, lens, kTileFixedCost, n_tt, static_cast<int>(sw), h->n_ctas, &sc,
                                         bcsr_block_cost(f.b, groups), &loads, &totals);
                // Where the longest tile of a row group alone exceeds a CTA's share of the whole work by half (few groups,
                // a narrow dense operand), its launch is a handful of CTAs working while the others are done: the
                // groups then run with 128-token tiles, twice as many and less than half as long.  Results are the
                // same bits (a token's sums do not depend on its tile).  10 % full block-rows, us: 6000 x 5000 TF32,
                // b = 32, N = 1500 (24 tiles of 157 stacked blocks, an 80 us launch whose CTAs were busy for 18 us on
                // average) 79.6 -> 50.4; 8192 x 8192 fp16, b = 32, N = 504 78.7 -> 53.0; with the share exceeded by
                // 15 % only (b = 16, N = 1000) 99.7 -> 103.6, the stacked blocks being fetched twice as often.
                int64_t work = 0, rest = 0, most = 0;
                for (int64_t x : totals) work += x;
                rest = work;
                for (int64_t x : loads) rest -= x;
                for (int64_t g = 0; g < st.ng; ++g) most = std::max<int64_t>(most, st.ptr[g + 1] - st.ptr[g]);
                const int64_t longest = (most + kStackTileFixedCost) * bcsr_stack_block_cost(kStackGroups);
                if (!rc && N > 64 && 2 * longest * h->n_ctas > 3 * work) {
                    BcsrSchedule kc, ks;
                    std::vector<int32_t> gu, gl;
                    for (int64_t g = 0; g < st.ng; ++g) {
                        gu.push_back(static_cast<int32_t>(g));
                        gl.push_back(st.ptr[g + 1] - st.ptr[g]);
                    }
                    rc = build_tile_schedule(gu, gl, kStackTileFixedCost, static_cast<int>((N + 127) / 128), static_cast<int>(2 * sws), h->n_ctas, &ks,
                                             bcsr_stack_block_cost(1), nullptr, &loads);
                    // (in halves of 64 rows a stacked block costs 2 (128 + 64) instead of 2 (128 + 128); the other launch is
                    // dealt for one CTA per tile, so that some of its lists start when the halves are done and count twice)
                    const int64_t n_tiles = static_cast<int64_t>(ks.tiles.size() / 2);
                    const int64_t whole = (most + kStackTileFixedCost) * bcsr_stack_block_cost(1);
                    stack_split = !rc && split_fits(n_tiles, most, kStackRows) && (whole * 3 / 4 + 2 * rest / (h->n_ctas - n_tiles)) * 10 < whole * 9 &&
                                  in_first_lists(ks);
                    // (a narrow operand fills half of either tile: 16-bit blocks of 16 then lose 2 to 5 % with the smaller one's
                    // stages unless it is halved; 4848 x 6768, bf16, N = 72 58.1 -> 60.2, 8000 x 12000, N = 96 82 -> 86)
                    const bool narrow = h->es == 2 && f.b == 16 && N <= 96 && !stack_split;
                    if (!rc && !narrow) {
                        std::sort(loads.begin(), loads.end());
                        rc = build_tile_schedule(units, lens, kTileFixedCost, n_tt, static_cast<int>(sw), h->n_ctas, &kc,
                                                 bcsr_block_cost(f.b, groups), &loads);
                    }
                    if (!rc && !narrow) {
                        sc = std::move(kc);
                        ss = std::move(ks);
                        ss.groups = 1;
                        ss.N = N;
                    }
                }
            }
        }
    } catch (const std::bad_alloc&) {
        rc = SPMM_ERR_ALLOC;
    }
    if (rc) return rc;
    sc.groups = groups;
    sc.N = N;
    if (!h->host_only) {
        if (h->d_tiles) {   // a previous schedule may still be in use by a running kernel
            if (cudaDeviceSynchronize() != cudaSuccess) return cuda_error();
            drop_schedule(h);
        }
        try {
            rc = upload_schedule(h, sc, ss, N);
        } catch (const std::bad_alloc&) {
            rc = SPMM_ERR_ALLOC;
        }
        if (rc) {
            drop_schedule(h);            // the handle holds no schedule rather than half of one
            return rc;
        }
    }
    h->stack_groups = ss.tiles.empty() ? 0 : ss.groups;
    h->split = split;
    h->stack_split = stack_split;
    h->tmB_N = -1;                   // (the stacked launch's map of B depends on its tile)
    h->sched_stack = std::move(ss);
    h->sched = std::move(sc);
    return SPMM_OK;
}

// Which request of a stage goes first, its stored blocks or its B tiles: the one that is longer on its way.  Many
// block-rows share a token tile, which is then close by in L2, and the blocks go first; where few do, the tiles do.  The line, by
// block-rows (148 CTAs), from the speed with the tiles first over that with the blocks first, geometric means over products
// of random sizes, row-major, N = 300 - 50,000 (single ones are within 0.94 and 1.06, and so are two runs of one with
// other buffers, now and then):
//   block-rows    under 10   10 - 20   20 - 30   30 - 50   60 - 100   100 - 200
//   b = 128 TF32  1.016      1.011     1.008     1.003     0.983      0.951
//           bf16  1.015      1.014     1.005     0.997     0.961      0.977
//   b = 64  TF32  1.014      1.006     1.007     1.007     1.000      0.995, under 16 blocks a row
//           bf16  1.007      1.006     1.002     0.998     0.996      0.99
// b <= 32 and stacked blocks do not gain on either side, nor do short stages (b = 64 in tiles of 128 tokens), narrow operands
// (under 1000 columns 0.997: their weights are what comes from afar) or column-major ones (b = 128, under 30 block-rows: 16-bit
// 1.002, TF32 0.99, E4M3 0.988).  TF32 at b = 64
// has the longest B tiles beside its blocks (32 KB to 8): long tiles, 32 blocks a row and more, gain at any number of
// block-rows.  us, blocks first and tiles first: 8192 x 8192, b = 64, density 0.4, TF32, N = 16,384 2225 and 2134; 5000 x 7000,
// 10 % full rows, N = 16,384 947 and 927; 1819 x 5601, b = 128, 10 % full rows, N = 9288 105.1 and 103.2; 3584 x 18944, b = 128,
// bf16, N = 2048 87.5 and 82.3.
bool bcsr_tiles_first(const spmm_handle_s* h, int64_t N, int groups) {
    const BcsrHost& f = h->bcsr;
    if (f.b < 64 || (f.b == 64 && groups == 1) || N < 1024 || h->col_major) return false;
    if (h->es == 4 && f.b == 64) return 3 * f.nbr < h->n_ctas || f.nnzb >= 32 * f.nbr;
    return 5 * f.nbr < h->n_ctas;
}

int run_bcsr(spmm_handle_s* h, const void* B, void* C, int64_t N, cudaStream_t stream) {
    const BcsrHost& f = h->bcsr;
    // the box of the dense operand is 64 tokens wide (128 with column-major operands or 1-byte values)
    if (N < ((h->col_major || h->es == 1) ? 128 : 64)) return SPMM_ERR_UNSUPPORTED;
    if (f.nbr == 0) return SPMM_OK;
    int rc = ensure_schedule(h, N);
    if (rc) return rc;
    BcsrParams p;
    p.block_row_ptr = h->d_ptr;
    p.block_col_idx = h->d_idx;
    p.tiles = reinterpret_cast<const int4*>(h->d_tile_recs);
    p.cta_ptr = h->d_cta_ptr;
    p.C = C;
    p.m = h->m;
    p.N = N;
    p.status = h->d_status;
    p.wait_limit_ns = g_wait_limit_ns.load();
    p.stack_rows = nullptr;
    p.plain_col_idx = nullptr;
    p.plain_vals = nullptr;
    p.B = nullptr;
    p.k = h->k;
    p.overlap = 0;
    p.tiles_first = bcsr_tiles_first(h, N, h->sched.groups) ? 1 : 0;
    BcsrMaps tm;
    tm.A = h->sched.groups <= 1 ? h->tmA1 : h->tmA;
    tm.A0 = h->tmA;
    if (!h->tmA_ok) {
        // no stored block at all: the kernel never touches A, any valid map will do
        rc = encode_2d(&tm.A, h->dtype, h->d_vals, 8, 8, 8, 8, CU_TENSOR_MAP_SWIZZLE_NONE);
        if (rc) return rc;
        tm.A0 = tm.A;
    }
    rc = ensure_tmB(h, B, N, h->sched.groups);
    if (rc) return rc;
    p.use_3d = h->tmB3_ok ? 1 : 0;
    rc = ensure_tmC(h, C, N);
    if (rc) return rc;
    if (!h->sched_stack.tiles.empty()) {
        // the row groups first (the longest block-rows are among them), then everything else
        BcsrParams ps = p;
        ps.block_col_idx = h->d_sidx;
        ps.tiles = reinterpret_cast<const int4*>(h->d_stile_recs);
        ps.cta_ptr = h->d_scta_ptr;
        ps.stack_rows = h->d_srows;
        if (h->dtype == SPMM_TF32) {
            ps.plain_col_idx = h->d_idx;
            ps.plain_vals = reinterpret_cast<const float*>(h->d_vals);
            ps.B = static_cast<const float*>(B);
        }
        ps.use_3d = h->tmB3s_ok ? 1 : 0;
        ps.overlap = 1;
        p.overlap = 2;
        const int n_tiles = static_cast<int>(h->sched_stack.tiles.size() / 2);
        const BcsrMaps ts = {h->stack_split ? h->tmAsh : h->tmAs, {}, h->tmB, h->tmB3s, h->tmC, {}};
        cudaError_t es = launch_bcsr_stacked(h->dtype, f.b, h->stack_split ? kSplitGroups : h->stack_groups, h->c16, h->col_major, ts, ps,
                                             h->stack_split ? n_tiles : h->n_ctas, stream);
        if (es != cudaSuccess) return cuda_error();
        if (h->sched.tiles.empty()) return SPMM_OK;
    }
    // dynamic: one CTA per tile, the schedule was built as a single list in the global order
    const int grid = h->dynamic ? static_cast<int>(h->sched.tiles.size() / 2) : h->n_ctas;
    if (grid <= 0) return SPMM_OK;
    tm.B = h->split ? h->tmBh : h->tmB;
    tm.B3 = h->tmB3;
    tm.C = h->split ? h->tmCh : h->tmC;
    if (h->split) {
        const cudaError_t eh = launch_bcsr(h->dtype, f.b, kSplitGroups, h->c16, h->col_major, 0, tm, p, static_cast<int>(h->sched.tiles.size() / 2), stream);
        return eh == cudaSuccess ? SPMM_OK : cuda_error();
    }
    const bool ksplit = h->sched.n_slots > 0 && h->tmP_ok;
    if (ksplit) p.overlap = 1;          // the merge kernel's CTAs may be placed while this grid runs
    tm.P = ksplit ? h->tmP : h->tmC;
    cudaError_t e = launch_bcsr(h->dtype, f.b, h->sched.groups, h->c16, h->col_major, h->dynamic, tm, p, grid, stream);
    if (e != cudaSuccess) return cuda_error();
    if (ksplit) {
        BcsrMergeParams mp;
        mp.row = h->d_kmerge;
        mp.first = h->d_kmerge + h->n_kmerge;
        mp.nparts = h->d_kmerge + 2 * h->n_kmerge;
        mp.partial = h->d_partial;
        mp.C = static_cast<float*>(C);
        mp.m = h->m;
        mp.N = N;
        mp.n = h->n_kmerge;
        mp.b = f.b;
        if (launch_bcsr_merge(mp, stream) != cudaSuccess) return cuda_error();
    }
    return SPMM_OK;
}

int64_t wcsr_workspace_bytes(const spmm_handle_s* h, int64_t N) {
    return h->wcsr.n_slots * int64_t{h->wcsr.wh} * N * 4;
}

// Stored values per padded column up to which the row kernel is the faster one at dense width N.  The window kernel
// takes 128-token tiles whose row of B is 256 (2-byte types; from 64 tokens on it has a variant for half of that) or
// 512 bytes, so it is at its best from N = 64 / 128 on; a launch the row kernel's short tasks alone can spread over
// the GPU (load < 16) is latency, which condensing does not help.  Row / window kernel, us, 16 entries a row in a
// band, at 1.2 / 1.4 / 1.9 values per column:
//   100,000 rows  fp16 N = 32   0.62 / 0.81 / 0.97 of the window kernel's time    TF32 N = 64    0.64 / 0.79 / 1.10
//                 fp16 N = 128  1.05 / 1.29 / 1.70                                TF32 N = 128   0.95 / 1.13 / 1.56
//   8000 rows     fp16 N = 128  0.60 / 0.84 / 1.43                                TF32 N = 128   0.72 / 0.85 / 1.03
// Where a row of B leaves more than a quarter of a warp's lanes idle, the large launches of the 2-byte types (load
// >= 100) are the window kernel's as well: N = 320 on R-MAT 2^20, 24 a row, 1450 us against 1600, on 200,000 rows of
// power-law length 285 against 344; with the lanes full, N = 256, 1046 against 998 and 209 against 214.
double wcsr_rows_limit(const spmm_handle_s* h, int64_t N) {
    const int64_t load = wcsr_rows_load(h->m, h->nnz, h->sms);
    const int es = h->es;
    if (load < 16 || N < (es == 4 ? 128 : 64)) return kRowsMaxPerCol;
    if (es == 4) return 1.4;
    if (load < 100) return 1.22;
    const RowsShape s = wcsr_rows_shape(N, es, (N * es) % 32 == 0);
    const int64_t busy = int64_t{32 / s.lanes} * s.lanes * (N * es), all = int64_t{32} * s.lanes * s.tiles * s.vec;
    return busy * 4 < all * 3 ? 0.0 : 1.22;
}

// Whether a run takes the row kernel: the handle has a row stream and it is the faster one.  A function of the handle
// and the dense width alone.
bool use_rows(const spmm_handle_s* h, int64_t N) {
    return (h->rows.n_tasks > 0 || h->rows.n_parts > 0) && N * h->es < (int64_t{1} << 32) &&
           static_cast<double>(h->nnz) <= wcsr_rows_limit(h, N) * static_cast<double>(h->wcsr.P);
}

// Bytes of partial rows one launch of the row kernel wants for `tiles` column tiles.
size_t rows_partial_bytes(const spmm_handle_s* h, const RowsShape& s, int tiles) {
    return static_cast<size_t>(h->rows.n_slots) * s.tile_cols * 4 * tiles;
}

RowsShape rows_shape(const spmm_handle_s* h, const void* B, const void* C, int64_t N) {
    // (N * es % 32 == 0 makes C's rows multiples of 32 bytes as well: its elements are at least as wide)
    const bool aligned32 = (N * h->es) % 32 == 0 && ((reinterpret_cast<uintptr_t>(B) | reinterpret_cast<uintptr_t>(C)) & 31) == 0;
    return wcsr_rows_shape(N, h->es, aligned32);
}

// Threads of a CTA of the row kernel.  A long row's part is 16 strands, which the CTA's groups sum one after the other
// where there are fewer groups than that.  A launch that is over when its slowest part is gains from twice the warps (512
// threads: 0.6 - 1.07 of the speed of 256); in larger ones, and where the parts themselves take turns, a CTA then holds its slot
// for its slowest warp.  Speed with 256 over 128 threads, TF32, by entries per SM and 128 groups (load) and parts (N = 320 is
// three tiles, a CTA for every part in each):
//                          load  parts  N = 36 (3 groups)  128 (2)  256 (1)  320 (2)
//   power-law rows, 2000    2    189                       1.37     1.58     1.06
//                   4000    3    240    1.22               1.40     1.73     0.95
//                   9000    6    536    1.08               1.13     1.47     0.91
//                   12,000  5    455    1.14               1.18     1.51     0.96
//                   16,000  3     95    1.20               1.34     1.77     1.17
//   R-MAT 2^11, 16 a row    1    241    1.27               1.29     1.81     1.03
//         2^12, 24 a row    4    640    1.04               1.10     1.51     0.87
//         2^13, 16 a row    6    960    0.83               0.90     1.28     0.81
//         2^14, 8 a row     7    662    0.98                        1.27
int wcsr_rows_threads(const spmm_handle_s* h, const RowsShape& s) {
    const int groups = 32 / s.lanes;
    if (h->rows.n_parts == 0 || groups > 3 || wcsr_rows_load(h->m, h->nnz, h->sms) >= (groups == 1 ? 8 : 7)) return kRowsThreads;
    return int64_t{3} * h->rows.n_parts * s.tiles <= (groups == 1 ? 21 : 13) * h->sms ? 256 : kRowsThreads;
}

// fp32 sums of one column per instruction and strands without padding, for TF32 in 16-byte vectors (rows of B that are no
// multiple of 32 bytes, or narrow): where the rows are short, the operand is narrow or the launch large, it is chains of
// gathers, and what two columns per instruction and the padding save in issue slots they cost in latency and L1.  Speed over
// that with both, by entries a row and entries per SM and 128 groups (load):
//                              row  load   N = 16   36     52     76     252
//   power-law rows, 300,000     3    70    1.01     1.07   1.11   1.12   1.08
//                    50,000     6    20    1.15     1.00   1.00   1.02   1.01
//   R-MAT 2^20                  4   280    1.04     1.03   1.04   1.03   1.03
//         2^20                 16   900    1.01     1.02          1.02
//   power-law rows, 400,000    17   390    1.00     1.03          1.06
//   R-MAT 2^15                  7    15    1.05     1.00   0.99   0.99   0.93
//         2^16                 21    80    1.03     0.98   1.00   0.98   0.98
//   power-law rows, 100,000    14    78    1.06     0.98   1.00   0.96   1.00
//                    20,000    12    14    1.02     1.00   0.98   0.96   0.96
//                    6000      12     4    0.98     1.00   1.01   1.00   0.99
bool wcsr_rows_plain(const spmm_handle_s* h, const RowsShape& s) {
    if (h->es != 4 || s.vec != 16) return false;
    const int64_t load = wcsr_rows_load(h->m, h->nnz, h->sms);
    return load >= 128 || (load >= 8 && (s.tiles * s.lanes <= 8 || h->nnz < 6 * h->m));
}

// partial: room for cap bytes of partial rows; the column tiles go in as few launches as that and the counters allow,
// and are made narrower where it does not hold one (sums do not depend on the cut).  A tile of one vector takes
// kRowsMaxSlots * 32 bytes at most, which the built-in scratch holds.
int launch_wcsr_rows_all(spmm_handle_s* h, const void* B, void* C, float* partial, size_t cap, int64_t N, cudaStream_t stream) {
    if (g_wait_limit_ns.load() == 0) return launch_wcsr_rows_give_up(h->d_status, stream) == cudaSuccess ? SPMM_OK : cuda_error();
    const WcsrRowStream& r = h->rows;
    RowsShape s = rows_shape(h, B, C, N);
    if (rows_partial_bytes(h, s, 1) > cap) {
        const int64_t ve = s.vec / h->es, lanes = static_cast<int64_t>(cap / 4) / (static_cast<int64_t>(r.n_slots) * ve);
        if (lanes < 1) return SPMM_ERR_TOO_LARGE;
        s.lanes = static_cast<int>(std::min<int64_t>(lanes, s.lanes));
        s.tiles = static_cast<int>((N + s.lanes * ve - 1) / (s.lanes * ve));
        s.tile_cols = static_cast<int>(s.lanes * ve);
    }
    WcsrRowsParams p;
    p.tasks = reinterpret_cast<const int4*>(r.d_tasks);
    p.parts = reinterpret_cast<const int4*>(r.d_parts);
    p.longs = reinterpret_cast<const int4*>(r.d_longs);
    p.order = r.d_order;
    p.col = r.d_col;
    p.val = r.d_val;
    p.zeros = reinterpret_cast<const uint8_t*>(r.d_counters);
    p.counters = r.d_counters + 8;
    p.partial = partial;
    p.B = B;
    p.C = C;
    p.N = N;
    p.n_tasks = r.n_tasks;
    p.n_parts = r.n_parts;
    const int threads = wcsr_rows_threads(h, s);
    const bool plain = wcsr_rows_plain(h, s);
    int step = std::min(s.tiles, kRowsMaxTiles);
    while (step > 1 && rows_partial_bytes(h, s, step) > cap) --step;
    for (int t = 0; t < s.tiles; t += step)
        if (launch_wcsr_rows(h->dtype, h->c16 ? 1 : 0, s, p, t, std::min(step, s.tiles - t), threads, plain, stream) != cudaSuccess)
            return cuda_error();
    return SPMM_OK;
}

// What a run of the row kernel wants at any dense width up to N, whatever the alignment of its operands: the columns
// that one launch covers, at most kRowsMaxTiles tiles of 32 lanes, and at most N and the lanes that the last vector and
// an even cut into tiles leave over.  (The sum itself does not grow with N: 3976 columns take eight tiles of 31 lanes,
// 4104 nine of 29.)
size_t rows_workspace_bytes(const spmm_handle_s* h, int64_t N) {
    const int64_t ve = 32 / h->es;
    return static_cast<size_t>(h->rows.n_slots) * 4 * static_cast<size_t>(std::min<int64_t>(kRowsMaxTiles * 32 * ve, N + (kRowsMaxTiles + 1) * ve));
}

// The workspace of a run at dense width N, by the kernel it takes.
size_t wcsr_run_bytes(const spmm_handle_s* h, int64_t N, bool rows) {
    return rows ? rows_workspace_bytes(h, N) : static_cast<size_t>(wcsr_workspace_bytes(h, N));
}

int launch_wcsr_all(spmm_handle_s* h, const void* B, void* C, float* partial, int64_t N, cudaStream_t stream) {
    const WcsrHost& f = h->wcsr;
    const int bnt = 128;                    // tokens per tile; wider B takes one pass per tile
    WcsrParams p;
    p.bin_ptr = h->d_bin_ptr;
    p.items = reinterpret_cast<const int4*>(h->d_items);
    // narrow dense operand: the variant whose stages hold more columns
    const bool narrow = h->d_bin_fill_narrow != nullptr && N <= kWcsrNarrowMaxN && !h->lsu_gather;
    p.fills = reinterpret_cast<const int2*>(narrow ? h->d_fills_narrow : h->d_fills);
    p.bin_fill = narrow ? h->d_bin_fill_narrow : h->d_bin_fill;
    p.col_idx = h->d_idx;
    // Gather hints: B rows whose reuse class fits half of a 126 MB L2 at this dense width are
    // fetched evict-last, everything else evict-first.  Class c holds at most
    // kWcsrTopClassRows << (7 - c) rows of N * es bytes each.
    p.grp_class = h->lsu_gather ? nullptr : h->d_grp_class;
    p.hot_min = 8;
    for (int c = 1; c <= 7; ++c)
        if ((static_cast<int64_t>(kWcsrTopClassRows) << (7 - c)) * N * h->es <= (int64_t{64} << 20)) { p.hot_min = c; break; }
    // (measured on the R-MAT configuration at N = 128: DRAM reads 2.84 -> 2.53 GB, L2 sector hit rate
    // 50 -> 53 %, time unchanged -- the kernel is bound by the latency of its gathers, not by DRAM
    // bytes; storing C evict-first as well measured 1 - 5 % slower and is left off)
    p.hint_flags = 1;
    p.packed = h->d_vals;
    p.B = B;
    p.C = C;
    p.partial = partial;
    p.m = h->m;
    p.N = N;
    p.n_bins = static_cast<int32_t>(f.bin_ptr.size()) - 1;
    p.n_tt = static_cast<int32_t>((N + bnt - 1) / bnt);
    p.status = h->d_status;
    p.wait_limit_ns = g_wait_limit_ns.load();
    if (!f.tasks.empty()) {
        int rc = ensure_tmB(h, B, N, 1);
        if (rc) return rc;
        cudaError_t e = launch_wcsr(h->dtype, f.wh, h->c16, narrow ? 1 : 0, h->lsu_gather ? 1 : 0, h->tmB, p, h->sms, stream);
        if (e != cudaSuccess) return cuda_error();
    }
    MergeParams mp;
    mp.window = h->d_merge;
    mp.first = h->d_merge + h->n_merge;
    mp.nparts = h->d_merge + 2 * h->n_merge;
    mp.partial = partial;
    mp.C = C;
    mp.m = h->m;
    mp.N = N;
    mp.n = h->n_merge;
    cudaError_t e = launch_wcsr_merge(mp, f.wh, h->c16 ? (h->dtype == SPMM_FP16 ? 1 : 2) : 0, stream);
    return e == cudaSuccess ? SPMM_OK : cuda_error();
}

// The handle's workspace for partial tiles or partial rows (grown, never shrunk).  It outlives the run and serves runs
// on any stream, so it is ready for all of them when this returns, and never an allocation on a stream that is
// captured: that would be a node of the graph, whose memory exists while the graph runs only.  A run that needs to grow
// it under capture asks for memory outside the pool instead: refused (SPMM_ERR_ALLOC, nothing launched) in the capture
// modes that forbid an allocation, lasting in the relaxed one.
int ensure_wcsr_workspace(spmm_handle_s* h, size_t need, cudaStream_t stream) {
    if (need <= h->partial_bytes) return SPMM_OK;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess) {    // (the legacy stream while a blocking one is captured)
        cudaGetLastError();
        capture = cudaStreamCaptureStatusActive;
    }
    if (h->d_partial) {
        if (cudaDeviceSynchronize() != cudaSuccess) return cuda_error();
        free_partial(h);
    }
    if (capture == cudaStreamCaptureStatusNone) {
        if (!dev_alloc_ready_ok(&h->d_partial, need, stream)) return SPMM_ERR_ALLOC;
    } else {
        if (cudaMalloc(reinterpret_cast<void**>(&h->d_partial), need) != cudaSuccess) {
            cudaGetLastError();
            h->d_partial = nullptr;
            return SPMM_ERR_ALLOC;
        }
        h->partial_pooled = false;
    }
    h->partial_bytes = need;
    return SPMM_OK;
}

// rows: use_rows for the whole operand of which these are N columns (the kernels add in different orders)
int run_wcsr(spmm_handle_s* h, const void* B, void* C, int64_t N, bool rows, cudaStream_t stream) {
    if (int rc = ensure_wcsr_workspace(h, wcsr_run_bytes(h, N, rows), stream)) return rc;
    if (rows) return launch_wcsr_rows_all(h, B, C, h->d_partial, h->partial_bytes, N, stream);
    return launch_wcsr_all(h, B, C, h->d_partial, N, stream);
}

int check_run_args(spmm_handle_s* h, const void* B, const void* C, int64_t N) {
    if (!h || !B || !C || N <= 0) return SPMM_ERR_INVALID_ARG;
    if (h->host_only) return SPMM_ERR_HOST_ONLY;
    // the handle's arrays, tensor maps and kernel attributes belong to the device it was created on
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return cuda_error();
    if (dev != h->device) return SPMM_ERR_INVALID_ARG;
    // row-major B and C have N elements per row: rows must stay 16-byte aligned (column-major
    // operands have k and m elements per row, checked at creation)
    if (!h->col_major && (N * h->es) % 16 != 0) return SPMM_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(B) & 15) || (reinterpret_cast<uintptr_t>(C) & 15)) return SPMM_ERR_UNSUPPORTED;
    if (N >= (int64_t{1} << 31)) return SPMM_ERR_TOO_LARGE;
    return SPMM_OK;
}

}  // namespace

// ============================================================================= C ABI

extern "C" {

int spmm_bcsr_create_csr(spmm_handle_t* out, int64_t m, int64_t k, const int64_t* row_ptr, const int32_t* col_idx,
                         const void* vals, int dtype, int block, const spmm_opts_t* opts) {
    NvtxRange nvtx_range("spmm_bcsr_create_csr");
    if (!out) return SPMM_ERR_INVALID_ARG;
    *out = nullptr;
    CsrView v;
    int rc = make_view(&v, m, k, row_ptr, col_idx, vals, dtype);
    if (rc) return rc;
    return create_bcsr(out, v, dtype, block, opts);
}

int spmm_bcsr_create_csr_device(spmm_handle_t* out, int64_t m, int64_t k, const int64_t* row_ptr_dev,
                                const int32_t* col_idx_dev, const void* vals_dev, int dtype, int block,
                                const spmm_opts_t* opts, void* stream) {
    NvtxRange nvtx_range("spmm_bcsr_create_csr_device");
    if (!out) return SPMM_ERR_INVALID_ARG;
    *out = nullptr;
    if (dtype < 0 || dtype > 3 || m < 0 || k < 0 || !row_ptr_dev) return SPMM_ERR_INVALID_ARG;
    if (m >= (int64_t{1} << 31) || k >= (int64_t{1} << 31)) return SPMM_ERR_TOO_LARGE;
    return create_bcsr_device(out, m, k, row_ptr_dev, col_idx_dev, vals_dev, dtype, block, opts, static_cast<cudaStream_t>(stream));
}

int spmm_wcsr_create_csr_device(spmm_handle_t* out, int64_t m, int64_t k, const int64_t* row_ptr_dev,
                                const int32_t* col_idx_dev, const void* vals_dev, int dtype, int window_height,
                                const spmm_opts_t* opts, void* stream) {
    NvtxRange nvtx_range("spmm_wcsr_create_csr_device");
    if (!out) return SPMM_ERR_INVALID_ARG;
    *out = nullptr;
    if (dtype < 0 || dtype > 3 || m < 0 || k < 0 || !row_ptr_dev) return SPMM_ERR_INVALID_ARG;
    if (m >= (int64_t{1} << 31) || k >= (int64_t{1} << 31)) return SPMM_ERR_TOO_LARGE;
    return create_wcsr_device(out, m, k, row_ptr_dev, col_idx_dev, vals_dev, dtype, window_height, opts, static_cast<cudaStream_t>(stream));
}

int spmm_bcsr_create_coo(spmm_handle_t* out, int64_t m, int64_t k, int64_t nnz, const int32_t* rows,
                         const int32_t* cols, const void* vals, int dtype, int block, const spmm_opts_t* opts) {
    NvtxRange nvtx_range("spmm_bcsr_create_coo");
    if (!out) return SPMM_ERR_INVALID_ARG;
    *out = nullptr;
    if (dtype < 0 || dtype > 3) return SPMM_ERR_INVALID_ARG;
    CsrOwned o;
    int rc;
    try {
        rc = coo_to_csr(m, k, nnz, rows, cols, static_cast<const uint8_t*>(vals), elem_size(dtype), &o);
    } catch (const std::bad_alloc&) {
        rc = SPMM_ERR_ALLOC;
    }
    if (rc) return rc;
    return spmm_bcsr_create_csr(out, m, k, o.row_ptr.data(), o.col_idx.data(), o.vals.data(), dtype, block, opts);
}

int spmm_wcsr_create_csr(spmm_handle_t* out, int64_t m, int64_t k, const int64_t* row_ptr, const int32_t* col_idx,
                         const void* vals, int dtype, int window_height, const spmm_opts_t* opts) {
    NvtxRange nvtx_range("spmm_wcsr_create_csr");
    if (!out) return SPMM_ERR_INVALID_ARG;
    *out = nullptr;
    CsrView v;
    int rc = make_view(&v, m, k, row_ptr, col_idx, vals, dtype);
    if (rc) return rc;
    return create_wcsr(out, v, dtype, window_height, opts);
}

int spmm_wcsr_create_coo(spmm_handle_t* out, int64_t m, int64_t k, int64_t nnz, const int32_t* rows,
                         const int32_t* cols, const void* vals, int dtype, int window_height,
                         const spmm_opts_t* opts) {
    NvtxRange nvtx_range("spmm_wcsr_create_coo");
    if (!out) return SPMM_ERR_INVALID_ARG;
    *out = nullptr;
    if (dtype < 0 || dtype > 3) return SPMM_ERR_INVALID_ARG;
    CsrOwned o;
    int rc;
    try {
        rc = coo_to_csr(m, k, nnz, rows, cols, static_cast<const uint8_t*>(vals), elem_size(dtype), &o);
    } catch (const std::bad_alloc&) {
        rc = SPMM_ERR_ALLOC;
    }
    if (rc) return rc;
    return spmm_wcsr_create_csr(out, m, k, o.row_ptr.data(), o.col_idx.data(), o.vals.data(), dtype, window_height,
                                opts);
}

int spmm_run(spmm_handle_t h, const void* B_dev, void* C_dev, int64_t N, void* stream) {
    NvtxRange nvtx_range("spmm_run");
    int rc = check_run_args(h, B_dev, C_dev, N);
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (h->format == 0) return run_bcsr(h, B_dev, C_dev, N, st);
    return run_wcsr(h, B_dev, C_dev, N, use_rows(h, N), st);
}

int spmm_bcsr_plan(spmm_handle_t h, int64_t N) {
    NvtxRange nvtx_range("spmm_bcsr_plan");
    if (!h || N <= 0) return SPMM_ERR_INVALID_ARG;
    if (h->format != 0) return SPMM_ERR_INVALID_ARG;
    if (N < ((h->col_major || h->es == 1) ? 128 : 64) || (!h->col_major && (N * h->es) % 16 != 0)) return SPMM_ERR_UNSUPPORTED;
    return ensure_schedule(h, N);
}

int spmm_prepare(spmm_handle_t h, int64_t N) {
    NvtxRange nvtx_range("spmm_prepare");
    if (!h || N <= 0) return SPMM_ERR_INVALID_ARG;
    if (h->format == 0) return spmm_bcsr_plan(h, N);
    if ((N * h->es) % 16 != 0) return SPMM_ERR_UNSUPPORTED;
    if (N >= (int64_t{1} << 31)) return SPMM_ERR_TOO_LARGE;
    if (h->host_only) return SPMM_OK;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return cuda_error();
    if (dev != h->device) return SPMM_ERR_INVALID_ARG;
    // for every width up to N: a handle with a row stream may take either kernel there
    const size_t need = std::max(wcsr_run_bytes(h, N, false), wcsr_run_bytes(h, N, true));
    return ensure_wcsr_workspace(h, need, nullptr);
}

int spmm_wcsr_run_static(spmm_handle_t h, const void* B_dev, void* C_dev, int64_t N, void* stream) {
    NvtxRange nvtx_range("spmm_wcsr_run_static");
    int rc = check_run_args(h, B_dev, C_dev, N);
    if (rc) return rc;
    if (h->format != 1) return SPMM_ERR_INVALID_ARG;
    float* scratch = nullptr;
    size_t cap = 0;
    if (wcsr_static_scratch(&scratch, &cap) != cudaSuccess) return cuda_error();
    if (static_cast<size_t>(wcsr_workspace_bytes(h, N)) > cap) return SPMM_ERR_TOO_LARGE;
    if (use_rows(h, N))
        return launch_wcsr_rows_all(h, B_dev, C_dev, scratch, cap, N, static_cast<cudaStream_t>(stream));
    return launch_wcsr_all(h, B_dev, C_dev, scratch, N, static_cast<cudaStream_t>(stream));
}

int spmm_run_host(spmm_handle_t h, const void* B_host, void* C_host, int64_t N, void* stream) {
    NvtxRange nvtx_range("spmm_run_host");
    if (!h || !B_host || !C_host || N <= 0) return SPMM_ERR_INVALID_ARG;
    if (h->host_only) return SPMM_ERR_HOST_ONLY;
    {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess) return cuda_error();
        if (dev != h->device) return SPMM_ERR_INVALID_ARG;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t bbytes = static_cast<size_t>(h->k) * N * h->es;
    const size_t cbytes = static_cast<size_t>(h->m) * N * h->cs;
    if (bbytes > h->Bstage_bytes) {
        cudaFree(h->d_Bstage);
        h->d_Bstage = nullptr;
        h->Bstage_bytes = 0;
        if (dev_malloc(&h->d_Bstage, bbytes) != cudaSuccess) return SPMM_ERR_ALLOC;
        h->Bstage_bytes = bbytes;
    }
    if (cbytes > h->Cstage_bytes) {
        cudaFree(h->d_Cstage);
        h->d_Cstage = nullptr;
        h->Cstage_bytes = 0;
        if (dev_malloc(reinterpret_cast<void**>(&h->d_Cstage), cbytes) != cudaSuccess) return SPMM_ERR_ALLOC;
        h->Cstage_bytes = cbytes;
    }
    // Large operands go in column chunks (token chunks), so that the copy of one chunk's result to
    // the host overlaps the copy of the next chunk's operand to the device (the two directions of
    // the link are independent) and the kernels in between.  Chunks are whole slices of N that the
    // kernels accept by themselves; each is staged as its own contiguous array, so the kernels
    // run unchanged on it.  Row-major operands: a chunk is a column range, copied with 2-D
    // copies whose rows are at least 256 bytes; column-major: a contiguous range of tokens.
    int nchunks = 1;
    if (bbytes + cbytes >= (size_t{8} << 20)) {
        for (int c = spmm_handle_s::kMaxHostChunks; c >= 2; c >>= 1) {
            if (N % c != 0) continue;
            const int64_t nc = N / c;
            const bool ok = h->col_major ? (nc >= 128)
                                         : (nc * h->es >= 256 && (nc * h->es) % 16 == 0 && (nc * h->cs) % 16 == 0 &&
                                            (h->format == 1 || nc >= 64));
            if (ok) { nchunks = c; break; }
        }
    }
    if (nchunks == 1) {
        if (cudaMemcpyAsync(h->d_Bstage, B_host, bbytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return cuda_error();
        int rc = spmm_run(h, h->d_Bstage, h->d_Cstage, N, stream);
        if (rc) return rc;
        if (cudaMemcpyAsync(C_host, h->d_Cstage, cbytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) return cuda_error();
        if (cudaStreamSynchronize(st) != cudaSuccess) return cuda_error();
        return SPMM_OK;
    }
    if (!h->s_in) {
        if (cudaStreamCreateWithFlags(&h->s_in, cudaStreamNonBlocking) != cudaSuccess ||
            cudaStreamCreateWithFlags(&h->s_out, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&h->ev_start, cudaEventDisableTiming) != cudaSuccess)
            return cuda_error();
        for (int i = 0; i < spmm_handle_s::kMaxHostChunks; ++i)
            if (cudaEventCreateWithFlags(&h->ev_in[i], cudaEventDisableTiming) != cudaSuccess ||
                cudaEventCreateWithFlags(&h->ev_run[i], cudaEventDisableTiming) != cudaSuccess)
                return cuda_error();
    }
    const int64_t nc = N / nchunks;
    const bool rows = h->format == 1 && use_rows(h, N);
    const size_t bchunk = bbytes / nchunks, cchunk = cbytes / nchunks;
    const uint8_t* Bh = static_cast<const uint8_t*>(B_host);
    uint8_t* Chost = static_cast<uint8_t*>(C_host);
    uint8_t* dB = static_cast<uint8_t*>(h->d_Bstage);
    uint8_t* dC = reinterpret_cast<uint8_t*>(h->d_Cstage);
    bool bad = false;
    // the staging buffers may still be read by work queued on `stream` earlier
    bad |= cudaEventRecord(h->ev_start, st) != cudaSuccess;
    bad |= cudaStreamWaitEvent(h->s_in, h->ev_start, 0) != cudaSuccess;
    for (int c = 0; c < nchunks && !bad; ++c) {
        if (h->col_major)
            bad |= cudaMemcpyAsync(dB + c * bchunk, Bh + c * bchunk, bchunk, cudaMemcpyHostToDevice, h->s_in) != cudaSuccess;
        else
            bad |= cudaMemcpy2DAsync(dB + c * bchunk, nc * h->es, Bh + static_cast<size_t>(c) * nc * h->es, N * h->es, nc * h->es,
                                     static_cast<size_t>(h->k), cudaMemcpyHostToDevice, h->s_in) != cudaSuccess;
        bad |= cudaEventRecord(h->ev_in[c], h->s_in) != cudaSuccess;
    }
    int rc = SPMM_OK;
    for (int c = 0; c < nchunks && !bad && !rc; ++c) {
        bad |= cudaStreamWaitEvent(st, h->ev_in[c], 0) != cudaSuccess;
        if (bad) break;
        rc = check_run_args(h, dB + c * bchunk, dC + c * cchunk, nc);
        if (!rc) rc = h->format == 0 ? run_bcsr(h, dB + c * bchunk, dC + c * cchunk, nc, st) : run_wcsr(h, dB + c * bchunk, dC + c * cchunk, nc, rows, st);
        if (rc) break;
        bad |= cudaEventRecord(h->ev_run[c], st) != cudaSuccess;
        bad |= cudaStreamWaitEvent(h->s_out, h->ev_run[c], 0) != cudaSuccess;
        if (h->col_major)
            bad |= cudaMemcpyAsync(Chost + c * cchunk, dC + c * cchunk, cchunk, cudaMemcpyDeviceToHost, h->s_out) != cudaSuccess;
        else
            bad |= cudaMemcpy2DAsync(Chost + static_cast<size_t>(c) * nc * h->cs, N * h->cs, dC + c * cchunk, nc * h->cs, nc * h->cs,
                                     static_cast<size_t>(h->m), cudaMemcpyDeviceToHost, h->s_out) != cudaSuccess;
    }
    // nothing of this call may still be in flight when it returns, whatever happened above
    const bool s1 = cudaStreamSynchronize(h->s_in) == cudaSuccess;
    const bool s2 = cudaStreamSynchronize(st) == cudaSuccess;
    const bool s3 = cudaStreamSynchronize(h->s_out) == cudaSuccess;
    if (rc) return rc;
    return (bad || !s1 || !s2 || !s3) ? cuda_error() : SPMM_OK;
}

int spmm_check(spmm_handle_t h) {
    if (!h) return SPMM_ERR_INVALID_ARG;
    if (h->host_only) return SPMM_ERR_HOST_ONLY;
    int st[4] = {0, 0, 0, 0};
    if (cudaMemcpy(st, h->d_status, sizeof(st), cudaMemcpyDeviceToHost) != cudaSuccess) return cuda_error();
    if (st[0] != 0) {
        cudaMemset(h->d_status, 0, sizeof(st));
        cudaStreamSynchronize(nullptr);          // (the next run may come on a stream that does not wait for this one)
        if (st[0] == 2) return SPMM_ERR_DEV_BOUNDS;
        return st[3] != 0 ? SPMM_ERR_DEV_UNDRAINED : SPMM_ERR_DEV_TIMEOUT;
    }
    return SPMM_OK;
}

int spmm_get_info(spmm_handle_t h, int64_t N, spmm_info_t* info) {
    if (!h || !info || N < 0) return SPMM_ERR_INVALID_ARG;
    std::memset(info, 0, sizeof(*info));
    info->format = h->format;
    info->dtype = h->dtype;
    info->m = h->m;
    info->k = h->k;
    info->nnz = h->nnz;
    info->n_ctas = h->n_ctas;
    const double s = h->es, n = static_cast<double>(N);
    if (h->format == 0) {
        const BcsrHost& f = h->bcsr;
        info->block = f.b;
        info->n_units = f.nnzb;
        info->stored_values = f.nnzb * f.b * f.b;
        info->n_rows_units = f.nbr;
        info->n_empty = f.n_empty;
        int64_t rows_touched = f.distinct_bcols * f.b;
        if (rows_touched > h->k) rows_touched = h->k;
        info->distinct_b_rows = rows_touched;
        info->bytes_a = static_cast<double>(info->stored_values) * s;
        info->bytes_idx = static_cast<double>(f.nbr + 1 + f.nnzb) * 4.0;
        info->bytes_gather = static_cast<double>(f.nnzb) * f.b * n * s;
        info->n_stacked_rows = static_cast<int32_t>(h->stack.rows.size());
        info->n_stack_blocks = h->stack.ns;
        if (h->sched.N >= 0) {
            info->n_slots = h->sched.n_slots;
            info->n_split = h->n_kmerge;
            if (h->host_only && h->sched.n_slots > 0) {
                int64_t ns = 0, last = -1;
                for (size_t u = 0; u < h->sched.units.size() / 4; ++u)
                    if (h->sched.units[4 * u + 3] >= 0 && h->sched.units[4 * u] != last) { last = h->sched.units[4 * u]; ++ns; }
                info->n_split = ns;
            }
            info->n_tasks = static_cast<int64_t>(h->sched.units.size() / 4);
            info->split_cols = h->sched.cap;
            info->workspace_bytes = h->sched.n_slots * f.b * h->sched.N * 4;
            info->plan_n = h->sched.N;
            info->plan_token_tile = 128 * h->sched.groups;
            info->plan_slab_tiles = h->sched.slab_w;
        }
    } else {
        const WcsrHost& f = h->wcsr;
        info->block = f.wh;
        info->b_col = f.b_col;
        info->n_units = f.P;
        info->stored_values = f.P * f.wh;
        info->n_rows_units = f.nwin;
        info->n_empty = f.n_empty;
        info->n_tasks = static_cast<int64_t>(f.tasks.size());
        info->n_split = f.n_split;
        info->n_slots = f.n_slots;
        info->split_cols = f.T;
        info->n_bins = static_cast<int32_t>(f.bin_ptr.size()) - 1;
        info->distinct_b_rows = f.distinct_cols;
        info->bytes_a = static_cast<double>(info->stored_values) * s;
        info->bytes_idx = static_cast<double>(f.nwin + 1 + f.P) * 4.0;
        info->bytes_gather = static_cast<double>(f.P) * n * s;
        info->workspace_bytes = N > 0 ? static_cast<int64_t>(wcsr_run_bytes(h, N, use_rows(h, N))) : 0;
    }
    info->fill_ratio = info->stored_values ? static_cast<double>(h->nnz) / static_cast<double>(info->stored_values) : 0.0;
    info->bytes_b_touched = static_cast<double>(info->distinct_b_rows) * n * s;
    info->bytes_c = static_cast<double>(h->m) * n * h->cs;
    info->flops_stored = 2.0 * static_cast<double>(info->stored_values) * n;
    return SPMM_OK;
}

int spmm_export(spmm_handle_t h, int which, void* host_dst, size_t cap, size_t* need) {
    if (!h || !need) return SPMM_ERR_INVALID_ARG;
    const void* dev_src = nullptr;    // device array in canonical layout, or
    const void* host_src = nullptr;   // host array in canonical layout
    size_t bytes = 0;
    bool unpack_wcsr = false;
    bool host_copy = false;           // the array is kept on the host even when the handle is on the device
    std::vector<int32_t> tmp;
    if (h->format == 0) {
        const BcsrHost& f = h->bcsr;
        switch (which) {
            case SPMM_X_BCSR_BLOCK_ROW_PTR: bytes = f.block_row_ptr.size() * 4; dev_src = h->d_ptr; host_src = f.block_row_ptr.data(); break;
            case SPMM_X_BCSR_BLOCK_COL_IDX: bytes = f.block_col_idx.size() * 4; dev_src = h->d_idx; host_src = f.block_col_idx.data(); break;
            case SPMM_X_BCSR_BLOCKS: bytes = static_cast<size_t>(f.nnzb) * f.b * f.b * h->es; dev_src = h->d_vals; host_src = f.blocks.data(); break;
            case SPMM_X_BCSR_ROW_ORDER: bytes = f.row_order.size() * 4; dev_src = h->d_order; host_src = f.row_order.data(); break;
            case SPMM_X_BCSR_TILE_PTR:
                if (h->sched.N < 0) return SPMM_ERR_INVALID_ARG;
                bytes = h->sched.cta_ptr.size() * 4; dev_src = h->d_cta_ptr; host_src = h->sched.cta_ptr.data(); break;
            case SPMM_X_BCSR_TILES:
                if (h->sched.N < 0) return SPMM_ERR_INVALID_ARG;
                bytes = h->sched.tiles.size() * 4; dev_src = h->d_tiles; host_src = h->sched.tiles.data(); break;
            case SPMM_X_BCSR_UNITS:
                if (h->sched.N < 0) return SPMM_ERR_INVALID_ARG;
                bytes = h->sched.units.size() * 4; host_src = h->sched.units.data(); host_copy = true; break;
            // the row-group plan lives on the host in every mode
            case SPMM_X_BCSR_STACK_ROWS: bytes = h->stack.rows.size() * 4; host_src = h->stack.rows.data(); host_copy = true; break;
            case SPMM_X_BCSR_STACK_PTR: bytes = h->stack.ptr.size() * 4; host_src = h->stack.ptr.data(); host_copy = true; break;
            case SPMM_X_BCSR_STACK_COL_IDX: bytes = h->stack.col_idx.size() * 4; host_src = h->stack.col_idx.data(); host_copy = true; break;
            case SPMM_X_BCSR_STACK_TILE_PTR:
                if (h->sched.N < 0) return SPMM_ERR_INVALID_ARG;
                bytes = h->sched_stack.cta_ptr.size() * 4; host_src = h->sched_stack.cta_ptr.data(); host_copy = true; break;
            case SPMM_X_BCSR_STACK_TILES:
                if (h->sched.N < 0) return SPMM_ERR_INVALID_ARG;
                bytes = h->sched_stack.tiles.size() * 4; host_src = h->sched_stack.tiles.data(); host_copy = true; break;
            default: return SPMM_ERR_INVALID_ARG;
        }
    } else {
        const WcsrHost& f = h->wcsr;
        switch (which) {
            case SPMM_X_WCSR_WINDOW_ROW_PTR: bytes = f.window_row_ptr.size() * 4; dev_src = h->d_ptr; host_src = f.window_row_ptr.data(); break;
            case SPMM_X_WCSR_WINDOW_COL_IDX: bytes = static_cast<size_t>(f.P) * 4; dev_src = h->d_idx; host_src = f.window_col_idx.data(); break;
            case SPMM_X_WCSR_VALUES: bytes = static_cast<size_t>(f.P) * f.wh * h->es; unpack_wcsr = true; break;
            case SPMM_X_WCSR_TASKS: bytes = f.tasks.size() * 16; break;
            case SPMM_X_WCSR_BIN_PTR: bytes = f.bin_ptr.size() * 4; dev_src = h->d_bin_ptr; host_src = f.bin_ptr.data(); break;
            case SPMM_X_WCSR_BIN_TASKS: bytes = f.bin_tasks.size() * 4; dev_src = h->d_bin_tasks; host_src = f.bin_tasks.data(); break;
            case SPMM_X_WCSR_GROUP_CLASS: bytes = static_cast<size_t>(f.P / 4); dev_src = h->d_grp_class; host_src = f.grp_class.data(); break;
            default: return SPMM_ERR_INVALID_ARG;
        }
    }
    *need = bytes;
    if (!host_dst) return SPMM_OK;
    if (cap < bytes) return SPMM_ERR_INVALID_ARG;
    if (bytes == 0) return SPMM_OK;
    if (unpack_wcsr) {
        const WcsrHost& f = h->wcsr;
        std::vector<uint8_t> packed_dl;
        const uint8_t* packed = f.packed.data();
        if (!h->host_only) {
            packed_dl.resize(bytes);
            if (cudaMemcpy(packed_dl.data(), h->d_vals, bytes, cudaMemcpyDeviceToHost) != cudaSuccess) return cuda_error();
            packed = packed_dl.data();
        }
        uint8_t* dst = static_cast<uint8_t*>(host_dst);
        for (int r = 0; r < f.wh; ++r)
            for (int64_t q = 0; q < f.P; ++q)
                std::memcpy(dst + (static_cast<size_t>(r) * f.P + q) * h->es,
                            packed + wcsr_packed_offset(f.wh, f.b_col, h->es, r, q), h->es);
        return SPMM_OK;
    }
    if (h->format == 1 && which == SPMM_X_WCSR_TASKS) {
        const WcsrHost& f = h->wcsr;
        int32_t* dst = static_cast<int32_t*>(host_dst);
        if (h->host_only) {
            for (size_t i = 0; i < f.tasks.size(); ++i) {
                dst[4 * i + 0] = f.tasks[i].window;
                dst[4 * i + 1] = f.tasks[i].q0;
                dst[4 * i + 2] = f.tasks[i].count;
                dst[4 * i + 3] = f.tasks[i].slot;
            }
        } else {
            std::vector<WcsrDevTask> dt(f.tasks.size());
            if (cudaMemcpy(dt.data(), h->d_tasks, bytes, cudaMemcpyDeviceToHost) != cudaSuccess) return cuda_error();
            for (size_t i = 0; i < dt.size(); ++i) {
                dst[4 * i + 0] = dt[i].window;
                dst[4 * i + 1] = dt[i].col_begin - f.window_row_ptr[dt[i].window];
                dst[4 * i + 2] = dt[i].count;
                dst[4 * i + 3] = dt[i].slot;
            }
        }
        return SPMM_OK;
    }
    if (h->host_only || host_copy) {
        std::memcpy(host_dst, host_src, bytes);
        return SPMM_OK;
    }
    return cudaMemcpy(host_dst, dev_src, bytes, cudaMemcpyDeviceToHost) == cudaSuccess ? SPMM_OK : cuda_error();
}

int spmm_destroy(spmm_handle_t h) {
    free_handle(h);
    return SPMM_OK;
}

const char* spmm_status_string(int code) {
    switch (code) {
        case SPMM_OK: return "ok";
        case SPMM_ERR_INVALID_ARG: return "invalid argument";
        case SPMM_ERR_UNSORTED: return "unsorted or duplicate entries";
        case SPMM_ERR_OUT_OF_RANGE: return "index out of range";
        case SPMM_ERR_UNSUPPORTED: return "unsupported size, dtype, alignment or device";
        case SPMM_ERR_ALLOC: return "allocation failed";
        case SPMM_ERR_CUDA: return "CUDA call failed (is there a B200 and a usable context?)";
        case SPMM_ERR_DEV_TIMEOUT: return "a bounded wait inside a kernel ran out";
        case SPMM_ERR_HOST_ONLY: return "handle was created host_only";
        case SPMM_ERR_TOO_LARGE: return "size exceeds a fixed capacity";
        case SPMM_ERR_DEV_BOUNDS: return "a kernel met an index outside its range";
        case SPMM_ERR_DEV_UNDRAINED: return "a bounded wait inside a kernel ran out and so did the wait for its work in flight";
        default: return "unknown status";
    }
}


int spmm_set_wait_limit_ns(uint64_t ns) {
    g_wait_limit_ns.store(ns);
    return SPMM_OK;
}

}  // extern "C"
