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
// stalls, L1 data pipe 65 % busy on an R-MAT graph of 2^19 rows, fp16, N = 128; DRAM 23 %).
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

constexpr int kWarps = kRowsThreads / 32;
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
template <int BYTES>
__device__ __forceinline__ void st_vec(uint8_t* p, const uint32_t* w) {
    if constexpr (BYTES == 32)
        asm volatile("st.global.v8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
                     ::"r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "l"(p) : "memory");
    else
        asm volatile("st.global.v4.b32 [%4], {%0, %1, %2, %3};" ::"r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "l"(p) : "memory");
}

// acc[e] += a * b[e] over one vector of B.  16-bit types: the product of two 16-bit values is exact in
// fp32, so the mixed-precision FMA rounds once, like an FMA of the widened values.  (Widening first and
// a packed fma.rn.f32x2 measured 9 % slower.)
template <int FMT, int VB, int VE>
__device__ __forceinline__ void fma_vec(float (&acc)[VE], uint32_t a, const Vec<VB>& b) {
#pragma unroll
    for (int i = 0; i < VB / 4; ++i) {
        if constexpr (FMT == 2) {
            acc[i] = fmaf(__uint_as_float(a), __uint_as_float(b.w[i]), acc[i]);
        } else {
            const unsigned short av = static_cast<unsigned short>(a);
            const unsigned short lo = static_cast<unsigned short>(b.w[i]), hi = static_cast<unsigned short>(b.w[i] >> 16);
            if constexpr (FMT == 0) {
                asm("fma.rn.f32.f16 %0, %1, %2, %0;" : "+f"(acc[2 * i]) : "h"(av), "h"(lo));
                asm("fma.rn.f32.f16 %0, %1, %2, %0;" : "+f"(acc[2 * i + 1]) : "h"(av), "h"(hi));
            } else {
                asm("fma.rn.f32.bf16 %0, %1, %2, %0;" : "+f"(acc[2 * i]) : "h"(av), "h"(lo));
                asm("fma.rn.f32.bf16 %0, %1, %2, %0;" : "+f"(acc[2 * i + 1]) : "h"(av), "h"(hi));
            }
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
            st_vec<kPer * 4>(dst + i * 4, w);
        }
    } else {
        uint32_t w[VE / 2];
#pragma unroll
        for (int j = 0; j < VE / 2; ++j) {
            const CElem lo = from_f32<CElem>(acc[2 * j]), hi = from_f32<CElem>(acc[2 * j + 1]);
            w[j] = static_cast<uint32_t>(*reinterpret_cast<const unsigned short*>(&lo)) |
                   (static_cast<uint32_t>(*reinterpret_cast<const unsigned short*>(&hi)) << 16);
        }
        st_vec<VE * 2>(dst, w);
    }
}
