// WCSR product for windows that condense almost nothing (about one stored value per padded column):
// C rows are summed on the CUDA cores straight from a private copy of the nonzeros, the "row stream"
// (see WcsrRowStream in format.h).
//
// Why not the tensor cores here: the window kernel stages every (window, column) row of B through
// shared memory and multiplies it with a packed 16-row tile that holds one nonzero; the packed
// tiles (16 stored values per column) are the largest stream from HBM after C, and its time is the
// round trip of a stage.  With about one nonzero per column the same gathers can go straight into
// registers: no stage, no hand-shake, no padded values, and a product of a row of B with one scalar.
// What bounds this kernel is the latency and the L1 data path of the gathered rows (long-scoreboard
// stalls, L1 data pipe 67 % busy on an R-MAT graph of 2^19 rows, fp16, N = 128; DRAM 23 %).
//
// Work split.  A column tile is `lanes` vectors of VB bytes of B; a warp holds 32 / lanes groups.
// One group takes one task (whole rows) and walks its nonzeros four at a time: the columns and
// values of a step come with one vector load each (the group's lanes read the same address), all
// four gathers are in flight together, and the next step's columns are requested behind them.  An
// entry with the sign bit set ends a row: the sums are stored (C is written once, rows without
// nonzeros included) and start again at zero.
// A row longer than the task limit is cut into parts, one CTA each: 16 strands take every 16th run
// of eight nonzeros, their sums are added in strand order through shared memory, and where a row has
// several parts the last CTA to finish adds the partial rows in part order.  The order of every sum
// is fixed by the plan alone, so results are identical from run to run and for every cut of N.
//
// Measured and not kept (R-MAT 2^21, fp16, N = 128; this form 805 us in the same run): eight gathers
// in flight per lane (1197 us: registers), a register ring that refills each slot as it is consumed
// (869), rows brought through shared memory with cp.async (1227) or TMA row gathers (1244), and
// mma.sync with the gathered rows as operand, from registers (1332) or from TMA gathers (1635).
#include "kernels.h"
#include "ptx.cuh"

namespace spmm {

namespace {

constexpr int kStrands = 16;            // partial sums of a part: strand = (entry / 8) % kStrands, whatever the dense width
constexpr int kNoCol = 0x7fffffff;      // an entry without a gather: row without nonzeros, or padding

template <int VB> struct Vec { uint32_t w[VB / 4]; };

// read-only vector loads / stores of 16 or 32 bytes (the address is a multiple of the size)
template <int VB>
__device__ __forceinline__ Vec<VB> ld_row(const uint8_t* p) {
    Vec<VB> r;
    if constexpr (VB == 32)
        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
                     : "l"(p));
    else
        asm volatile("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]) : "l"(p));
    return r;
}

// acc[e] += a * b[e] over one vector of B.  16-bit types: the product of two 16-bit values is exact in
// fp32, so the mixed-precision FMA rounds once, like an FMA of the widened values.  (Widening first and
// a packed fma.rn.f32x2 measured 9 % slower.)  fp32 goes two columns at a time: R-MAT 2^17, 16 a row, N = 200
// 120.9 -> 118.6 us, 200,000 power-law rows N = 64 47.2 -> 46.2.  PLAIN: one column at a time
// (wcsr_rows_plain in api.cu).
template <int FMT, bool PLAIN, int VB, int VE>
__device__ __forceinline__ void fma_vec(float (&acc)[VE], uint32_t a, const Vec<VB>& b) {
    if constexpr (FMT == 2 && PLAIN) {
#pragma unroll
        for (int i = 0; i < VE; ++i) acc[i] = fmaf(__uint_as_float(a), __uint_as_float(b.w[i]), acc[i]);
        return;
    }
    if constexpr (FMT == 2) {
#pragma unroll
        for (int i = 0; i < VE; i += 2)
            asm("{\n\t"
                ".reg .b64 d, x, y;\n\t"
                "mov.b64 d, {%0, %1};\n\t"
                "mov.b64 x, {%3, %4};\n\t"
                "mov.b64 y, {%2, %2};\n\t"
                "fma.rn.f32x2 d, x, y, d;\n\t"
                "mov.b64 {%0, %1}, d;\n\t"
                "}\n"
                : "+f"(acc[i]), "+f"(acc[i + 1])
                : "r"(a), "r"(b.w[i]), "r"(b.w[i + 1]));
        return;
    }
#pragma unroll
    for (int i = 0; i < VB / 4; ++i) {
        const unsigned short av = static_cast<unsigned short>(a);
        const unsigned short lo = static_cast<unsigned short>(b.w[i]), hi = static_cast<unsigned short>(b.w[i] >> 16);
        if constexpr (FMT == 0) {
            asm("fma.rn.f32.f16 %0, %1, %2, %0;" : "+f"(acc[2 * i]) : "h"(av), "h"(lo));
            asm("fma.rn.f32.f16 %0, %1, %2, %0;" : "+f"(acc[2 * i + 1]) : "h"(av), "h"(hi));
        } else if constexpr (FMT == 1) {
            asm("fma.rn.f32.bf16 %0, %1, %2, %0;" : "+f"(acc[2 * i]) : "h"(av), "h"(lo));
            asm("fma.rn.f32.bf16 %0, %1, %2, %0;" : "+f"(acc[2 * i + 1]) : "h"(av), "h"(hi));
        }
    }
}

// Four consecutive entries of the stream.
template <int ES>
struct Ent4 {
    int c[4];
    uint32_t v[ES];
    __device__ __forceinline__ uint32_t val(int u) const {
        if constexpr (ES == 4) return v[u];
        else return (u & 1) ? (v[u >> 1] >> 16) : (v[u >> 1] & 0xffffu);
    }
};
template <int ES>
__device__ __forceinline__ Ent4<ES> ld_ent4(const int32_t* col, const uint8_t* val, int e, bool ok) {
    Ent4<ES> r;
    if (ok) {
        const int4 c = __ldg(reinterpret_cast<const int4*>(col + e));
        r.c[0] = c.x; r.c[1] = c.y; r.c[2] = c.z; r.c[3] = c.w;
        if constexpr (ES == 4) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(val) + (e >> 2));
            r.v[0] = v.x; r.v[1] = v.y; r.v[2] = v.z; r.v[3] = v.w;
        } else {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(val) + (e >> 2));
            r.v[0] = v.x; r.v[1] = v.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) r.c[i] = kNoCol;
#pragma unroll
        for (int i = 0; i < ES; ++i) r.v[i] = 0u;
    }
    return r;
}

template <int FMT, int CT, int VB, int VE>
__device__ __forceinline__ void store_c(uint8_t* dst, const float (&acc)[VE]) {
    using CElem = typename CType<FMT, CT>::type;
    if constexpr (sizeof(CElem) == 4) {
        constexpr int kPer = VB == 32 ? 8 : 4;           // the wide variant's rows of C are 32-byte aligned as well
#pragma unroll
        for (int i = 0; i < VE; i += kPer) {
            uint32_t w[kPer];
#pragma unroll
            for (int j = 0; j < kPer; ++j) w[j] = __float_as_uint(acc[i + j]);
            st_global_vec<kPer * 4>(dst + i * 4, w);
        }
    } else {
        uint32_t w[VE / 2];
#pragma unroll
        for (int j = 0; j < VE / 2; ++j) {
            const CElem lo = from_f32<CElem>(acc[2 * j]), hi = from_f32<CElem>(acc[2 * j + 1]);
            w[j] = static_cast<uint32_t>(*reinterpret_cast<const unsigned short*>(&lo)) |
                   (static_cast<uint32_t>(*reinterpret_cast<const unsigned short*>(&hi)) << 16);
        }
        st_global_vec<VE * 2>(dst, w);
    }
}

// Resident CTAs per SM: registers cap the bytes in flight.  Wide vectors: 7 (72 registers) measured 805 us
// on R-MAT 2^21 fp16 N = 128, 5 CTAs 858, 8 CTAs 893; 16-byte vectors: 8 (with 6: R-MAT 2^20 TF32 N = 76 645 -> 703, 2^17 bf16
// N = 40 38.4 -> 40.2, of 45,000 rows fp16 N = 48 12.9 -> 11.5; with 10: 30,000 rows fp16 N = 48 8.8 -> 9.3).
// THREADS: kRowsThreads, or 256 (wcsr_rows_threads in api.cu).
template <int FMT, int CT, int VB, int THREADS, bool PLAIN = false>
__global__ void __launch_bounds__(THREADS, THREADS > kRowsThreads ? 3 : (VB == 32 ? 7 : 8))
wcsr_rows_kernel(const WcsrRowsParams p) {
    constexpr int kWarps = THREADS / 32;
    constexpr int ES = FMT == 2 ? 4 : 2;
    constexpr int VE = VB / ES;                           // dense columns per lane
    using CElem = typename CType<FMT, CT>::type;
    // long rows' strands: [kStrands][lanes][VE + 1]; with a pitch of VE (or of lanes, transposed) the strands of a
    // warp and the columns of the adding threads met in a quarter of the banks: 11 of 41 million wavefronts of the L1 data
    // path on R-MAT 2^19, fp16, N = 128; on 2^21 812 -> 794 us.  PLAIN: [kStrands][VE][lanes], which takes less from L1
    extern __shared__ float red[];
    __shared__ unsigned arrived;

    grid_trigger();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane / p.lanes, l = lane - g * p.lanes;
    const int tile = p.tile0 + blockIdx.y;
    const int64_t n = (static_cast<int64_t>(tile) * p.lanes + l) * VE;         // first dense column of this lane
    const bool on = g < p.groups && n < p.N;
    const uint8_t* B = static_cast<const uint8_t*>(p.B) + n * ES;
    const uint32_t pitch = static_cast<uint32_t>(p.N) * ES;
    const int64_t c_pitch = p.N * static_cast<int64_t>(sizeof(CElem));

    float acc[VE];
#pragma unroll
    for (int i = 0; i < VE; ++i) acc[i] = 0.f;

    // an entry without a gather reads zeros of the library's own
    auto gather = [&](int c) -> Vec<VB> {
        const uint32_t j = static_cast<uint32_t>(c) & 0x7fffffffu;
        const uint8_t* src = B + static_cast<uint64_t>(j) * pitch;
        return ld_row<VB>(j != static_cast<uint32_t>(kNoCol) ? src : p.zeros);
    };

    if (static_cast<int>(blockIdx.x) >= p.n_parts) {
        // ------------------------------------------------------------------ whole rows, one task per group
        const int id = ((static_cast<int>(blockIdx.x) - p.n_parts) * kWarps + warp) * p.groups + g;
        if (!on || id >= p.n_tasks) {
            grid_wait();                                  // (a CTA of this grid has always waited: the next launch relies on it)
            return;
        }
        const int4 d = __ldg(p.tasks + id);               // first entry, entries, position in order
        const int32_t* order = p.order + d.z;
        uint8_t* C = static_cast<uint8_t*>(p.C) + n * sizeof(CElem);
        Ent4<ES> cur = ld_ent4<ES>(p.col, p.val, d.x, d.y > 0);
        int row = __ldg(order);
        grid_wait();
        for (int e = 0; e < d.y; e += 4) {
            Vec<VB> b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) b[u] = gather(cur.c[u]);
            const Ent4<ES> nxt = ld_ent4<ES>(p.col, p.val, d.x + e + 4, e + 4 < d.y);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                fma_vec<FMT, PLAIN, VB, VE>(acc, cur.val(u), b[u]);
                if (cur.c[u] < 0) {                       // the row's last entry
                    store_c<FMT, CT, VB, VE>(C + row * c_pitch, acc);
#pragma unroll
                    for (int i = 0; i < VE; ++i) acc[i] = 0.f;
                    row = __ldg(++order);                 // (order has one element more than there are rows)
                }
            }
            cur = nxt;
        }
        return;
    }

    // ---------------------------------------------------------------------- one part of a long row
    const int4 d = __ldg(p.parts + blockIdx.x);           // first entry, entries, long row, part
    const int4 lr = __ldg(p.longs + d.z);                 // row, first slot, parts
    grid_wait();
    const int n_groups = kWarps * p.groups;
    const int tile_cols = p.lanes * VE;
    if (g < p.groups) {
        for (int strand = warp * p.groups + g; strand < kStrands; strand += n_groups) {
#pragma unroll
            for (int i = 0; i < VE; ++i) acc[i] = 0.f;
            if (on) {
                Ent4<ES> cur = ld_ent4<ES>(p.col, p.val, d.x + strand * 8, strand * 8 < d.y);
                for (int e = strand * 8; e < d.y;) {
                    Vec<VB> b[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) b[u] = gather(cur.c[u]);
                    const int en = (e & 4) ? e + kStrands * 8 - 4 : e + 4;      // the strand's next four entries
                    const Ent4<ES> nxt = ld_ent4<ES>(p.col, p.val, d.x + en, en < d.y);
#pragma unroll
                    for (int u = 0; u < 4; ++u) fma_vec<FMT, PLAIN, VB, VE>(acc, cur.val(u), b[u]);
                    cur = nxt;
                    e = en;
                }
            }
#pragma unroll
            for (int i = 0; i < VE; ++i) red[PLAIN ? strand * tile_cols + i * p.lanes + l : (strand * p.lanes + l) * (VE + 1) + i] = acc[i];
        }
    }
    __syncthreads();
    const int64_t n_tile = static_cast<int64_t>(tile) * tile_cols;
    CElem* Crow = static_cast<CElem*>(p.C) + lr.x * p.N + n_tile;
    const int64_t slot_pitch = static_cast<int64_t>(gridDim.y) * tile_cols;
    float* part0 = p.partial + static_cast<int64_t>(lr.y) * slot_pitch + static_cast<int64_t>(blockIdx.y) * tile_cols;
    for (int t = threadIdx.x; t < tile_cols; t += THREADS) {
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < kStrands; ++i) s += red[PLAIN ? i * tile_cols + (t % VE) * p.lanes + t / VE : i * (p.lanes * (VE + 1)) + t + t / VE];
        if (lr.z == 1) {
            if (n_tile + t < p.N) Crow[t] = from_f32<CElem>(s);
        } else {
            part0[d.w * slot_pitch + t] = s;
        }
    }
    if (lr.z == 1) return;
    // several parts: the CTA that arrives last adds them in part order.  The counter wraps to zero, so
    // it is ready for the next launch.
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) arrived = atomicInc(p.counters + d.z * kRowsMaxTiles + blockIdx.y, static_cast<unsigned>(lr.z) - 1u);
    __syncthreads();
    if (arrived != static_cast<unsigned>(lr.z) - 1u) return;
    __threadfence();
    for (int t = threadIdx.x; t < tile_cols; t += THREADS) {
        if (n_tile + t >= p.N) break;
        float s = 0.f;
        int i = 0;
        for (; i + 8 <= lr.z; i += 8) {
            float x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = __ldcg(part0 + (i + j) * slot_pitch + t);
#pragma unroll
            for (int j = 0; j < 8; ++j) s += x[j];
        }
        for (; i < lr.z; ++i) s += __ldcg(part0 + i * slot_pitch + t);
        Crow[t] = from_f32<CElem>(s);
    }
}

__global__ void wcsr_rows_give_up_kernel(int* status) {
    grid_trigger();
    grid_wait();
    if (atomicCAS(status, 0, 1) == 0) {
        status[1] = 31;                                   // (where other kernels name the wait that ran out)
        status[2] = 0;
    }
}

template <int VB, int THREADS>
cudaError_t launch_vb(int dtype, int c16, bool plain, const WcsrRowsParams& p, dim3 grid, size_t smem, cudaStream_t stream) {
    auto go = [&](auto kfn) { return launch_dependent(kfn, grid, THREADS, smem, stream, p); };
    if (dtype == 2) {
        if constexpr (VB == 16) {
            if (plain) return go(wcsr_rows_kernel<2, 0, VB, THREADS, true>);
        }
        return go(wcsr_rows_kernel<2, 0, VB, THREADS>);
    }
    if (dtype == 1) return c16 ? go(wcsr_rows_kernel<0, 1, VB, THREADS>) : go(wcsr_rows_kernel<0, 0, VB, THREADS>);
    if (dtype == 0) return c16 ? go(wcsr_rows_kernel<1, 1, VB, THREADS>) : go(wcsr_rows_kernel<1, 0, VB, THREADS>);
    return cudaErrorInvalidValue;
}

}  // namespace

// 32-byte vectors for rows of more than 128 bytes (R-MAT 2^21 fp16 N = 128: 805 against 864 us with 16 bytes;
// 192-byte rows, R-MAT 2^20, fp16 / TF32: 518 / 454 against 592 / 537); up to there 16-byte vectors: fewer rows
// share a warp, and its store at a row's end stops the others less often (128 bytes, 200,000 rows, fp16 / TF32:
// 52 / 45 against 75 / 58).  Rows that are cut anyhow get one column tile more where that fills the lanes (1280
// bytes, three tiles of 14 lanes instead of two of 20, R-MAT 2^20 TF32 N = 320: 2577 against 2819; two tiles for
// one of 20 lanes read the entries twice: 1655 against 1661 there, 41 against 39 on R-MAT 2^15).
RowsShape wcsr_rows_shape(int64_t N, int es, bool aligned32) {
    RowsShape s;
    s.vec = aligned32 && N * es > 128 ? 32 : 16;
    const int64_t vecs = (N * es + s.vec - 1) / s.vec;
    int64_t tiles = (vecs + 31) / 32;               // a group is part of one warp
    auto used = [&](int64_t t) { const int64_t l = (vecs + t - 1) / t; return 32 / l * l * vecs * 100 / (l * t); };
    if (tiles > 1 && used(tiles + 1) > used(tiles) * 5 / 4) ++tiles;
    s.lanes = static_cast<int>((vecs + tiles - 1) / tiles);
    s.tiles = static_cast<int>((vecs + s.lanes - 1) / s.lanes);
    s.tile_cols = s.lanes * (s.vec / es);
    return s;
}

cudaError_t launch_wcsr_rows_give_up(int* status, cudaStream_t stream) {
    return launch_dependent(wcsr_rows_give_up_kernel, dim3(1), 1, 0, stream, status);
}

cudaError_t launch_wcsr_rows(int dtype, int c16, const RowsShape& s, WcsrRowsParams p, int tile0, int tiles, int threads, bool plain, cudaStream_t stream) {
    p.lanes = s.lanes;
    p.groups = 32 / s.lanes;
    p.tile0 = tile0;
    const int per_cta = threads / 32 * p.groups;
    const int64_t ctas = p.n_parts + (static_cast<int64_t>(p.n_tasks) + per_cta - 1) / per_cta;
    if (ctas <= 0 || tiles <= 0) return cudaSuccess;
    const dim3 grid(static_cast<unsigned>(ctas), static_cast<unsigned>(tiles));
    const size_t smem = p.n_parts > 0 ? static_cast<size_t>(kStrands) * (s.tile_cols + (plain ? 0 : s.lanes)) * 4 : 0;     // at most 34 KB
    if (threads == 256) return s.vec == 32 ? launch_vb<32, 256>(dtype, c16, plain, p, grid, smem, stream) : launch_vb<16, 256>(dtype, c16, plain, p, grid, smem, stream);
    return s.vec == 32 ? launch_vb<32, kRowsThreads>(dtype, c16, plain, p, grid, smem, stream) : launch_vb<16, kRowsThreads>(dtype, c16, plain, p, grid, smem, stream);
}

}  // namespace spmm
