// tbe_internal.cuh -- device-side structures and steps shared by the forward
// gather-pool and the backward segmented reduce.
//
// Both hot loops have the same shape: a run of items in position order, grouped
// into consecutive segments (forward: the bags of a table, delimited by the
// jagged offsets; backward: runs of equal sorted row ids), where each item names
// a row to gather and a scalar coefficient, and each segment's output is the
// coefficient-weighted sum of its rows. The pooled bag of the paper's sparse_arch
// (Sec. IV.A.2) and its de-duplicated adjoint are both this shape.
//
// Work is cut into chunks of item positions of one size per call, so every warp
// does the same amount of gathering whatever the bag-length distribution (heavy tails,
// empty bags, one-hot bags). A segment that straddles chunk boundaries is summed
// piecewise; its pieces are combined afterwards in one fixed order, in fp64, by a
// fix-up pass (tbe_fixup.cuh), so results are deterministic.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <type_traits>

#include "cb_tbe.h"

namespace cbtbe {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarpThreads = 256;  // block size of the warp-per-chunk kernels
#ifndef CB_WALK_MIN_BLOCKS
#define CB_WALK_MIN_BLOCKS 4  // resident blocks per SM the walker kernels are compiled for
#endif
#ifndef CB_WALK_ROWS
#define CB_WALK_ROWS 4  // 16-byte rows in flight per lane in the walker (with one vector per lane)
#endif
// The backward reduce's own targets, and those of its form with the optimizer
// step fused (measured beside reduce_min_blocks).
#ifndef CB_REDUCE_MIN_BLOCKS
#define CB_REDUCE_MIN_BLOCKS 3
#endif
#ifndef CB_REDUCE_ROWS
#define CB_REDUCE_ROWS 8
#endif
#ifndef CB_REDUCE_APPLY_MIN_BLOCKS
#define CB_REDUCE_APPLY_MIN_BLOCKS 3
#endif
#ifndef CB_REDUCE_APPLY_ROWS
#define CB_REDUCE_APPLY_ROWS 4
#endif

// Per-table facts the kernels need, built once at create time.
struct TableDev {
    const void* data;   // row-major [rows, dim] of dtype
    int64_t rows;
    int64_t row_base;   // rows of all tables before this one (global row id base)
    // Backward sort key of row r: key_base + r, with key_base = row_base + t.
    // Each table owns rows + 1 keys; key_base + rows marks a lookup whose index
    // is out of range, which sorts after the table's rows into a run of its own
    // that the reduce drops.
    int64_t key_base;
    int32_t dim;
    int32_t doff;       // column offset of this table in the [B, sum dims] output
    int32_t dtype;      // cb_dtype
    int32_t row_vecs;   // 16-byte vectors per stored row
    int32_t grad_vecs;  // 16-byte vectors per grad_out row, in the output's type
};

// Consecutive item positions of one table. A boundary that is not moved has chunk_len
// positions on each side; the forward moves it by up to snap_cap, so its chunks hold up
// to chunk_len + snap_cap, and the reduce's, cut at run ends, less than 2 * chunk_len.
struct Chunk {
    int64_t k0;     // first item position
    int64_t first;  // forward: first bag touching k0; backward: first run of the table
                    // that begins at or after k0
    int32_t table;
    uint32_t len;   // bits 0..30: item count; bit 31: last chunk of its table (forward),
                    // or k0 lies inside a run begun earlier (backward)
};

struct Problem {
    const TableDev* tables;
    const uint4* zero_row;  // 2 KB of zeros: the row an invalid or padding item reads
    const void* indices;
    const void* offsets;
    const float* weights;
    int* error;
    int64_t n;
    int32_t T;
    int32_t B;
    int32_t sum_d;
    int32_t is32;
    int32_t mean;
    int32_t dmax;  // largest dim (row stride of the carry buffers)
    int32_t out_dtype;  // cb_dtype of the pooled output and of grad_out
};

struct Plan {
    int32_t chunk_len;
    int32_t snap_cap;                  // segments up to this long are never split (0: no snapping)
    int32_t num_classes;
    const int32_t* class_tables;       // [T] table ids grouped by kernel class
    const int32_t* class_table_start;  // [num_classes + 1]
    int64_t* table_pos;                // [T + 1] first item position of each table
    int64_t* ord_chunk_base;           // [T + 1] first chunk of class_tables[i]
    int64_t* class_chunk_base;         // [num_classes + 1]
    int64_t* table_chunk;              // [T] first chunk of each table
    Chunk* chunks;                     // [max_chunks]
    int64_t max_chunks;
    float* carry_head;                 // [max_chunks, dmax] piece of a segment begun earlier
    float* carry_tail;                 // [max_chunks, dmax] piece of a segment begun here
    unsigned long long* split;         // [max_chunks] kSplit... : segments cut by the chunk's edges
    uint32_t* chunk_next;              // [num_classes + 1] next chunk to hand out per class, and
                                       // over all classes (zeroed by the plan)
};

// A chunk's split word: in the low half the segment begun in it that runs past its
// end, if kSplitBegins; kSplitGoesOn if it begins inside a segment. The fix-up counts
// the blocks that are done with their share of the begun segment above.
constexpr unsigned long long kSplitBegins = 1ull << 32;
constexpr unsigned long long kSplitGoesOn = 1ull << 33;
constexpr unsigned long long kSplitArrival = 1ull << 34;

__host__ __device__ __forceinline__ int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }
__host__ __device__ __forceinline__ int64_t max64(int64_t a, int64_t b) { return a > b ? a : b; }

__device__ __forceinline__ void set_error(int* err, int code) { atomicCAS(err, 0, code); }

__device__ __forceinline__ int64_t load_index(const void* p, int64_t i, int is32) {
    return is32 ? static_cast<int64_t>(__ldg(static_cast<const int*>(p) + i))
                : static_cast<int64_t>(__ldg(static_cast<const long long*>(p) + i));
}

__device__ __forceinline__ int64_t warp_id_global() {
    return (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
}
__device__ __forceinline__ int64_t warps_in_grid() {
    return (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
}

// Every kernel of the lookups, the cross term and the replication (not the gather rate
// probes) is launched with programmatic stream serialization and begins with
// begin_kernel(): its launch overlaps the end of the kernel before
// it, whose results it then waits for (the wait covers everything earlier on the
// stream too, since that kernel began with the same wait). A call is a chain of 3 to
// 20 short kernels: a serving request's forward 22 -> 15 us, fp32 step of 330 K
// lookups 239 -> 220 us, one-hot step 210 -> 188 us, uniform bf16 step 2.07 -> 2.03 ms.
__device__ __forceinline__ void begin_kernel() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... Params, class... Args>
inline void launch(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const Args&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// Blocks of `threads` that one SM holds, and the grid of a persistent kernel
// whose warps take `chunk_bound` chunks.
template <class KernelT>
inline int resident_blocks(KernelT kernel, int threads) {
    int per_sm = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    return per_sm;
}
inline int warp_grid(int64_t chunk_bound, int64_t cap) {
    const int64_t need = (chunk_bound + (kWarpThreads / 32) - 1) / (kWarpThreads / 32);
    return static_cast<int>(max64(1, min64(need, cap)));
}

// The walkers' chunk order: a warp takes the next chunk of its class from a
// counter (lane 0 fetches the one after while the warp walks the current one),
// so chunks start in order and cheap chunks do not leave warps idle.
__device__ __forceinline__ int64_t first_chunk(const Plan& Q, int cls, int64_t cb, int lane) {
    const int64_t j = lane == 0 ? cb + atomicAdd(Q.chunk_next + cls, 1u) : 0;
    return __shfl_sync(kFull, j, 0);
}
__device__ __forceinline__ int64_t fetch_next_chunk(const Plan& Q, int cls, int64_t cb, int lane) {
    return lane == 0 ? cb + atomicAdd(Q.chunk_next + cls, 1u) : 0;
}

// ---------------------------------------------------------------- bags of positions

// The bag of each lookup, from a window of 32 bag ends held one per lane, in
// positions relative to the chunk start: every position is below 2^30, so these
// are exact in 32 bits (saturated, for malformed offsets, well inside the
// sentinel kPastTable that marks ends past the table's last bag).
constexpr int32_t kPastTable = INT32_MAX;

__device__ __forceinline__ int32_t rel32(int64_t x, int64_t k0) {
    const int64_t r = x - k0;
    return static_cast<int32_t>(r < -(int64_t(1) << 30) ? -(int64_t(1) << 30)
                                                        : (r > (int64_t(1) << 30) ? (int64_t(1) << 30) : r));
}

struct BagWindow32 {
    int64_t win;        // first bag of the window
    int32_t win_start;  // start of bag win
    int32_t my_end;     // end of bag win + lane
};

__device__ __forceinline__ BagWindow32 bag_window32(const Problem& P, int64_t first, int64_t bag_hi,
                                                    int64_t k0, int lane) {
    BagWindow32 W;
    W.win = first;
    W.win_start = first < bag_hi ? rel32(load_index(P.offsets, first, P.is32), k0) : kPastTable;
    W.my_end = first + lane < bag_hi ? rel32(load_index(P.offsets, first + lane + 1, P.is32), k0) : kPastTable;
    return W;
}

// Every lane calls this with its relative position q; the window moves forward
// 32 bags at a time until every valid lane has its bag (bag = -1 otherwise).
__device__ __forceinline__ void find_bag32(const Problem& P, BagWindow32& W, int64_t bag_hi, int64_t k0,
                                           int32_t q, bool valid, int lane, int64_t& bag, int32_t& s,
                                           int32_t& e) {
    bag = -1;
    s = e = 0;
    while (true) {
        int cnt = 0;  // ends at or before q in the window
#pragma unroll
        for (int b = 16; b >= 1; b >>= 1)
            if (__shfl_sync(kFull, W.my_end, cnt + b - 1) <= q) cnt += b;
        if (__shfl_sync(kFull, W.my_end, 31) <= q) cnt = 32;
        const int32_t e_sel = __shfl_sync(kFull, W.my_end, cnt < 32 ? cnt : 31);
        const int32_t s_sel = __shfl_sync(kFull, W.my_end, cnt > 0 ? cnt - 1 : 0);
        if (valid && bag < 0 && cnt < 32) {
            bag = W.win + cnt;
            e = e_sel;
            s = cnt > 0 ? s_sel : W.win_start;
        }
        if (!__any_sync(kFull, valid && bag < 0)) break;
        W.win_start = __shfl_sync(kFull, W.my_end, 31);
        W.win += 32;
        W.my_end = W.win + lane < bag_hi ? rel32(load_index(P.offsets, W.win + lane + 1, P.is32), k0) : kPastTable;
    }
}

// The bags of 32 consecutive positions p0 .. p0 + 31 without shuffles when
// possible: the window's ends inside the step become bits of a mask (one warp
// OR), and lane l's bag is the window's first bag plus the ends at or before
// p0 + l. Returns false (nothing written) when two ends coincide (an empty bag)
// or the step reaches past the window's last end; the caller then bisects.
__device__ __forceinline__ bool bags_by_mask(const BagWindow32& W, int32_t p0, int lane, bool want_range,
                                             int64_t& bag, int32_t& s, int32_t& e) {
    const bool before = W.my_end < p0;
    const bool inside = W.my_end >= p0 && W.my_end <= p0 + 31;
    const uint32_t nbefore = __popc(__ballot_sync(kFull, before));
    const uint32_t nin = __popc(__ballot_sync(kFull, inside));
    const uint32_t mask = __reduce_or_sync(kFull, inside ? 1u << (W.my_end - p0) : 0u);
    if (__popc(mask) != static_cast<int>(nin) || nbefore + nin >= 32) return false;  // warp-uniform
    const uint32_t le = lane == 31 ? kFull : (2u << lane) - 1u;
    const int cnt = static_cast<int>(nbefore) + __popc(mask & le);
    bag = W.win + cnt;
    if (want_range) {
        e = __shfl_sync(kFull, W.my_end, cnt);
        const int32_t prev = __shfl_sync(kFull, W.my_end, cnt > 0 ? cnt - 1 : 0);
        s = cnt > 0 ? prev : W.win_start;
    }
    return true;
}

// ---------------------------------------------------------------- storage types

template <int DT> struct Storage;
template <> struct Storage<CB_F32> { static constexpr int kElems = 4; };
template <> struct Storage<CB_F16> { static constexpr int kElems = 8; };
template <> struct Storage<CB_BF16> { static constexpr int kElems = 8; };

template <int DT>
__device__ __forceinline__ void unpack(const uint4& r, float (&f)[Storage<DT>::kElems]);

template <>
__device__ __forceinline__ void unpack<CB_F32>(const uint4& r, float (&f)[4]) {
    f[0] = __uint_as_float(r.x);
    f[1] = __uint_as_float(r.y);
    f[2] = __uint_as_float(r.z);
    f[3] = __uint_as_float(r.w);
}

template <>
__device__ __forceinline__ void unpack<CB_F16>(const uint4& r, float (&f)[8]) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        __half2 h;
        memcpy(&h, &w[i], 4);
        const float2 p = __half22float2(h);
        f[2 * i] = p.x;
        f[2 * i + 1] = p.y;
    }
}

// bfloat16 is the upper half of a binary32 word, so widening is a shift.
template <>
__device__ __forceinline__ void unpack<CB_BF16>(const uint4& r, float (&f)[8]) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}

// ---------------------------------------------------------------- output rows

// Cache hints for data touched once per call (CB_STREAM_HINTS): outputs
// stored with evict-first (st.global.cs), so that they leave L2 before the
// rows the walkers gather again, and one-pass payload streams loaded with it.
#ifndef CB_STREAM_HINTS
#define CB_STREAM_HINTS 1
#endif
__device__ __forceinline__ void store_stream(float4* p, float4 v) {
    if (CB_STREAM_HINTS) __stcs(p, v);
    else *p = v;
}
__device__ __forceinline__ void store_stream(uint2* p, uint2 v) {
    if (CB_STREAM_HINTS) __stcs(p, v);
    else *p = v;
}
__device__ __forceinline__ uint32_t load_stream(const uint32_t* p) { return CB_STREAM_HINTS ? __ldcs(p) : __ldg(p); }

// Four consecutive columns of an output row, stored as fp32 or rounded to
// fp16 / bf16 (round to nearest even).
__device__ __forceinline__ void store_out4(void* row, int64_t col, float a, float b, float c, float d,
                                           int dtype) {
    if (dtype == CB_F32) {
        store_stream(reinterpret_cast<float4*>(static_cast<float*>(row) + col), make_float4(a, b, c, d));
        return;
    }
    uint2 w;
    if (dtype == CB_F16) {
        const __half2 lo = __floats2half2_rn(a, b), hi = __floats2half2_rn(c, d);
        memcpy(&w.x, &lo, 4);
        memcpy(&w.y, &hi, 4);
    } else {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
        memcpy(&w.x, &lo, 4);
        memcpy(&w.y, &hi, 4);
    }
    store_stream(reinterpret_cast<uint2*>(static_cast<uint16_t*>(row) + col), w);
}

__host__ __device__ __forceinline__ int dtype_bytes(int dtype) { return dtype == CB_F32 ? 4 : 2; }

// ---------------------------------------------------------------- accumulation

// acc += w * row (WEIGHTED) or acc += row. Half-precision rows use the
// mixed-precision add of sm_100+ (f16/bf16 operand widened exactly, fp32 sum),
// which is the same arithmetic as widening first and then adding.
// (Measured on cfg5: widening fp16 pairs first and adding in fp32 took 29 %
// more instructions and 11 % more time; widening them and adding with one
// packed fp32x2 add, 16 % more instructions and 12 % more time.)
template <int DT, bool WEIGHTED>
__device__ __forceinline__ void accumulate(float (&a)[Storage<DT>::kElems], const uint4& x, float w) {
    const uint32_t word[4] = {x.x, x.y, x.z, x.w};
    if constexpr (DT == CB_F32) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float f = __uint_as_float(word[i]);
            a[i] = WEIGHTED ? fmaf(w, f, a[i]) : a[i] + f;
        }
    } else if constexpr (WEIGHTED) {
        float f[8];
        unpack<DT>(x, f);
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = fmaf(w, f[i], a[i]);
    } else if constexpr (DT == CB_F16) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm("{ .reg .b16 lo, hi;\n\t mov.b32 {lo, hi}, %2;\n\t"
                " add.rn.f32.f16 %0, lo, %0;\n\t add.rn.f32.f16 %1, hi, %1; }"
                : "+f"(a[2 * i]), "+f"(a[2 * i + 1]) : "r"(word[i]));
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm("{ .reg .b16 lo, hi;\n\t mov.b32 {lo, hi}, %2;\n\t"
                " add.rn.f32.bf16 %0, lo, %0;\n\t add.rn.f32.bf16 %1, hi, %1; }"
                : "+f"(a[2 * i]), "+f"(a[2 * i + 1]) : "r"(word[i]));
    }
}

// ---------------------------------------------------------------- the walkers
//
// A warp walks one chunk of item positions in batches of 32 (forward: Gather in
// tbe_forward.cuh; backward: Reduce in tbe_reduce.cuh). A row is spread over
// V = 32 / G lanes, 16 bytes per lane and vector, VPL vectors per lane (G = 1 for
// more than one), so a warp step gathers G rows; V is the smallest power of two
// that holds the row. Lanes past a row that is not a power of two of vectors load
// one of the row's own vectors again (the same cache lines, no branch) and never
// store what they sum. Several steps' rows are loaded together, then added
// segment by segment.

// Forward positions are relative to the chunk start and clamped to
// [kRelLo, kRelHi], which keeps every comparison with [0, len] exact in 32 bits.
constexpr int32_t kRelLo = -1;
constexpr int32_t kRelHi = 1 << 30;

__device__ __forceinline__ int32_t rel_pos(int64_t x, int64_t k0) {
    const int64_t r = x - k0;
    return r < kRelLo ? kRelLo : (r > kRelHi ? kRelHi : static_cast<int32_t>(r));
}

// Number of a row's layout: 0..5 for 32, 16, .., 1 rows per step (1, 2, 4, .., 32
// lanes per row), 6 and 7 for 2 and 4 vectors per lane.
__device__ __forceinline__ int row_layout(int row_vecs) { return 32 - __clz(row_vecs - 1); }

struct EndSlot {
    int32_t seg;
    int32_t len;  // segment length; -1 when it began in an earlier chunk, 0 for the
                  // piece of one that runs past the chunk end
};

// A cache line requested into L1 ahead of its load, without a register.
__device__ __forceinline__ void prefetch_l1(const void* p) {
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// ---------------------------------------------------------------- small scans

// Inclusive warp scan.
__device__ __forceinline__ int64_t warp_incl_scan(int64_t x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Exclusive block scan for blockDim.x a multiple of 32 (<= 1024). `sh` needs
// 33 int64 slots. Returns the exclusive prefix; *total receives the block sum.
__device__ __forceinline__ int64_t block_excl_scan(int64_t x, int64_t* sh, int64_t* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t inc = warp_incl_scan(x, lane);
    if (lane == 31) sh[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int64_t s = lane < nw ? sh[lane] : 0;
        const int64_t si = warp_incl_scan(s, lane);
        if (lane < nw) sh[lane] = si - s;
        if (lane == 31) sh[32] = si;
    }
    __syncthreads();
    const int64_t r = sh[wid] + inc - x;
    *total = sh[32];
    __syncthreads();
    return r;
}

}  // namespace cbtbe
