// tbe_reduce.cuh -- the backward segmented reduce (runs of equal sorted row
// ids; per run the coefficient-weighted sum of the gathered grad_out slices,
// the de-duplicated adjoint of the pooled bag of Sec. IV.A.2), and the
// optimizer step that can be fused where a run's sum ends. Included by
// tbe_reduce_{f32,f16,bf16}.cu and tbe_backward_apply.cu (instantiations) and by
// tbe_backward.cu (the step of split runs and of the second pass).
#pragma once

#include <cuda_bf16.h>

#include "tbe_internal.cuh"
#include "tbe_launch.h"

namespace cbtbe {

// ---------------------------------------------------------------- optimizer step

// Start of a stored row.
__device__ __forceinline__ char* row_ptr(const TableDev& td, int64_t row) {
    return static_cast<char*>(const_cast<void*>(td.data)) + row * td.dim * dtype_bytes(td.dtype);
}

// The stored bits of four consecutive columns of a row: 16 bytes (fp32) or
// 8 bytes in .x, .y (fp16 / bf16).
__device__ __forceinline__ uint4 load_cols(const char* rowp, int dtype, int col) {
    if (dtype == CB_F32) return *reinterpret_cast<const uint4*>(rowp + 4 * col);
    const uint2 x = *reinterpret_cast<const uint2*>(rowp + 2 * col);
    return make_uint4(x.x, x.y, 0u, 0u);
}

// new = E - scale * g for the four columns whose stored bits are `x`, rounded
// once from fp32 to the storage type (round to nearest even), and stored.
__device__ __forceinline__ void store_step(char* rowp, int dtype, int col, uint4 x, float4 g, float scale) {
    if (dtype == CB_F32) {
        float4 v = make_float4(__uint_as_float(x.x), __uint_as_float(x.y), __uint_as_float(x.z),
                               __uint_as_float(x.w));
        v.x = fmaf(-scale, g.x, v.x);
        v.y = fmaf(-scale, g.y, v.y);
        v.z = fmaf(-scale, g.z, v.z);
        v.w = fmaf(-scale, g.w, v.w);
        *reinterpret_cast<float4*>(rowp + 4 * col) = v;
        return;
    }
    uint2 y;
    if (dtype == CB_F16) {
        __half2 a, b;
        memcpy(&a, &x.x, 4);
        memcpy(&b, &x.y, 4);
        const float2 fa = __half22float2(a), fb = __half22float2(b);
        a = __floats2half2_rn(fmaf(-scale, g.x, fa.x), fmaf(-scale, g.y, fa.y));
        b = __floats2half2_rn(fmaf(-scale, g.z, fb.x), fmaf(-scale, g.w, fb.y));
        memcpy(&y.x, &a, 4);
        memcpy(&y.y, &b, 4);
    } else {
        const float f0 = __uint_as_float(x.x << 16), f1 = __uint_as_float(x.x & 0xffff0000u);
        const float f2 = __uint_as_float(x.y << 16), f3 = __uint_as_float(x.y & 0xffff0000u);
        const __nv_bfloat162 a = __floats2bfloat162_rn(fmaf(-scale, g.x, f0), fmaf(-scale, g.y, f1));
        const __nv_bfloat162 b = __floats2bfloat162_rn(fmaf(-scale, g.z, f2), fmaf(-scale, g.w, f3));
        memcpy(&y.x, &a, 4);
        memcpy(&y.y, &b, 4);
    }
    *reinterpret_cast<uint2*>(rowp + 2 * col) = y;
}

__device__ __forceinline__ void step_cols(const TableDev& td, int64_t row, int col, float4 g, float scale) {
    char* p = row_ptr(td, row);
    store_step(p, td.dtype, col, load_cols(p, td.dtype, col), g, scale);
}

// This lane's share of sum g^2 over four columns, in one fixed order of
// roundings (an explicit product and three fused multiply-adds): written as a
// plain sum of products, the compiler may fuse either product of a pair, and
// may choose differently in the fused and the two-pass step, which must give
// the same Adagrad state bit for bit.
__device__ __forceinline__ float sq4(float4 g) {
    return fmaf(g.w, g.w, fmaf(g.z, g.z, fmaf(g.y, g.y, __fmul_rn(g.x, g.x))));
}

// The Adagrad scale of a row spread over V lanes (a warp's lane groups may hold
// different rows) from each lane's share `sq` of the summed squares and the row's
// previous state `m0` (meaningful in the group's first lane, which stores the new
// state if `active`).
__device__ __forceinline__ float adagrad_scale(const BwdOut& O, float* st, int dim, float sq, float m0, int V,
                                               bool active) {
    const int lane = threadIdx.x & 31;
    for (int off = V / 2; off >= 1; off >>= 1) sq += __shfl_xor_sync(kFull, sq, off);
    float m = 0.f;
    if ((lane & (V - 1)) == 0 && active) {
        m = m0 + sq / static_cast<float>(dim);
        *st = m;
    }
    m = __shfl_sync(kFull, m, lane & ~(V - 1));
    return O.lr / (sqrtf(m) + O.eps);
}

// The step's scale for one row: lr (SGD), or lr / (sqrt(m) + eps) after
// m += mean of the squared gradient (row-wise Adagrad). `sq` is this lane's
// share of sum g^2; the whole warp calls this, lane 0 owns the state word.
__device__ __forceinline__ float step_scale(const BwdOut& O, int t, int64_t row, int dim, float sq) {
    if (O.apply != kApplyAdagrad) return O.lr;
    float* st = O.state[t] + row;
    return adagrad_scale(O, st, dim, sq, (threadIdx.x & 31) == 0 ? *st : 0.f, 32, true);
}

// The fused step on complete runs' rows, as the walker holds them: a lane group of
// V lanes holds one row, lane v of it vectors v + 32k. Either every group holds the
// same totals and one of them is `active`, or each holds a run of its own. `m0`:
// the row's previous Adagrad state (in the group's first lane). The row's loads are
// issued before the scale is summed. Out of line: the walker ends runs in many
// places, and a copy of the step in each of them overflowed the instruction cache.
template <int N>
struct GradRow {
    float4 v[N];   // four gradient columns each
    int col[N];    // first column of each, or -1 past the row
};

template <int N, int V>
__device__ __noinline__ void apply_row(const Problem& P, const BwdOut& O, int t, uint32_t row,
                                       const GradRow<N> g, float m0, bool active) {
    const TableDev& td = P.tables[t];
    char* p = row_ptr(td, row);
    const int dtype = td.dtype;
    uint4 x[N];
#pragma unroll
    for (int k = 0; k < N; ++k)
        if (active && g.col[k] >= 0) x[k] = load_cols(p, dtype, g.col[k]);
    float scale = O.lr;
    if (O.apply == kApplyAdagrad) {
        float sq = 0.f;
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (g.col[k] >= 0)
                sq += sq4(g.v[k]);
        scale = adagrad_scale(O, O.state[t] + row, td.dim, sq, m0, V, active);
    }
    if (!active) return;
#pragma unroll
    for (int k = 0; k < N; ++k)
        if (g.col[k] >= 0) store_step(p, dtype, g.col[k], x[k], g.v[k], scale);
}

// ---------------------------------------------------------------- (5) reduce

// One chunk of a table's sorted positions, walked by one warp in batches of 32.
// The kernel that counted the run heads left a flag per position: 32 of them are
// the mask of a batch's run ends, and runs are output in order, so the row a run
// goes to follows from the chunk's first run by counting; only the keys at run
// ends are read. (Taking the ends
// from a list of run starts took a window scan per batch, a list in shared
// memory, and two more passes over the keys to write the run keys and starts: on
// the three batches below 1102 / 1294 / 3162 us, and 65 / 65 / 120 us more for the
// runs; comparing the keys here, read twice, 1133 / 946 / 2585; with the flags 1116 /
// 946 / 2543.)
// The end of a run is a few instructions, repeated in every step of a load
// group: add, store, advance the output row. Runs cut by the chunk's edges leave
// their piece in the carry rows. Out-of-range lookups sort to the table's end
// under its spare key: their run is summed (of some row of the table) and dropped.
// APPLY: the optimizer step is fused where a run's sum ends (compiled as its
// own kernels, so the gradient-writing reduce carries none of its code).
template <int GO, int VPL, bool PACKED, bool APPLY, int G>
struct Reduce {
    static constexpr int E = Storage<GO>::kElems;  // grad_out storage: fp32, or fp16 / bf16 (mixed precision)
    static constexpr int V = 32 / G;
    static constexpr int kRows = APPLY ? CB_REDUCE_APPLY_ROWS : CB_REDUCE_ROWS;
    static constexpr int kWide = kRows > VPL ? kRows / VPL : 1;
    static constexpr int UG = kWide < V ? kWide : V;  // row steps per load group
    static constexpr int kItems = UG * G;
    static constexpr uint32_t kItemMask = kItems == 32 ? kFull : (1u << (kItems & 31)) - 1u;
    static constexpr uint32_t kStepMask = G == 32 ? kFull : (1u << (G & 31)) - 1u;
    static constexpr bool kFastBatch = VPL == 1;
    static_assert(VPL == 1 || G == 1, "several vectors per lane: one row per step");

    const Problem& P;  // kernel parameters: read in place, not held in registers
    const Plan& Q;
    const BwdOut& O;
    int32_t j;  // the chunk
    int32_t t;
    int lane, g, v;
    int32_t row_vecs, dim;
    bool at_head;   // the open run began in an earlier chunk
    float* dst;     // this lane's columns of the open run's output row
    float* next;    // and of the run after it
    float ain[VPL][E], aout[VPL][E];

    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int k = 0; k < VPL; ++k)
#pragma unroll
            for (int x = 0; x < E; ++x) ain[k][x] = aout[k][x] = 0.f;
    }
    __device__ __forceinline__ void add(const uint4 (&x)[VPL], float w) {
#pragma unroll
        for (int k = 0; k < VPL; ++k) accumulate<GO, PACKED>(ain[k], x[k], w);
    }
    __device__ __forceinline__ void store(float* at, const float (&t4)[VPL][E]) const {
#pragma unroll
        for (int k = 0; k < VPL; ++k)
            if (v + 32 * k < row_vecs)
#pragma unroll
                for (int x = 0; x < E; x += 4)
                    store_stream(reinterpret_cast<float4*>(at + 32 * k * E + x),
                                 make_float4(t4[k][x], t4[k][x + 1], t4[k][x + 2], t4[k][x + 3]));
    }
    __device__ __forceinline__ float* carry(float* rows) const {
        return rows + static_cast<int64_t>(j) * P.dmax + v * E;
    }
    // The sums of the open run over the lane groups, and a clean start.
    __device__ __forceinline__ void total(float (&tot)[VPL][E]) {
#pragma unroll
        for (int k = 0; k < VPL; ++k)
#pragma unroll
            for (int x = 0; x < E; ++x) tot[k][x] = aout[k][x] + ain[k][x];
#pragma unroll
        for (int off = V; off < 32; off <<= 1)
#pragma unroll
            for (int x = 0; x < E; ++x) tot[0][x] += __shfl_xor_sync(kFull, tot[0][x], off);
        zero();
    }
    // The fused step of the run that this lane's group holds.
    __device__ __forceinline__ void step(uint32_t key, const float (&tot)[VPL][E], float m0, bool active) const {
        GradRow<VPL * E / 4> r;
#pragma unroll
        for (int k = 0; k < VPL; ++k)
#pragma unroll
            for (int x = 0; x < E / 4; ++x) {
                const int col = (v + 32 * k) * E + 4 * x;
                r.v[k * (E / 4) + x] = make_float4(tot[k][4 * x], tot[k][4 * x + 1], tot[k][4 * x + 2],
                                                   tot[k][4 * x + 3]);
                r.col[k * (E / 4) + x] = col < dim ? col : -1;
            }
        apply_row<VPL * E / 4, V>(P, O, t, key - static_cast<uint32_t>(P.tables[t].key_base), r, m0, active);
    }
    // The end of a run (fused step: its key, and its row's previous state).
    __device__ __forceinline__ void flush(uint32_t key, float m0) {
        float tot[VPL][E];
        total(tot);
        if constexpr (APPLY) {
            if (!at_head) {
                step(key, tot, m0, g == 0);
                return;
            }
            if (g == 0) store(dst, tot);
            at_head = false;
        } else {
            if (g == 0) store(dst, tot);
            at_head = false;
            dst = next;
            next += dim;
        }
    }

    struct Walk {
        const uint32_t* keys;
        const uint32_t* vals;
        const uint32_t* bits;    // head flags from the chunk's cell on
        int32_t shift;           // of the chunk's first position within them
        int32_t len, table_end;  // items of the chunk; end of the table, relative to the chunk
    };
    __device__ __forceinline__ uint32_t fetch(const Walk& w, int32_t q) const {
        return q < w.len ? load_stream(w.vals + q) : 0u;
    }
    // (bag, bits of w_i * s_b) of a sorted item.
    __device__ __forceinline__ uint2 coefficient(uint32_t val) const {
        if constexpr (PACKED) return __ldg(O.packed + min(val, static_cast<uint32_t>(P.n - 1)));
        return make_uint2(val, 0u);
    }

    // grad_out rows of this table's bags start at `rows`, `stride` bytes apart.
    __device__ __forceinline__ void walk(const Walk& w, const char* rows, uint32_t stride, bool piece, int64_t out_row,
                                         int64_t out_float) {
        const TableDev& td = P.tables[t];
        const uint32_t dead = static_cast<uint32_t>(td.key_base + td.rows);
        const uint32_t bag_lo = static_cast<uint32_t>(t) * static_cast<uint32_t>(P.B);
        rows += (v < row_vecs ? v : 0) * 16;
        int voff[VPL];  // lanes past the row load one of its vectors again and never store what they sum
#pragma unroll
        for (int k = 0; k < VPL; ++k) voff[k] = k > 0 && v + 32 * k < row_vecs ? 512 * k : 0;
        zero();
        at_head = piece;
        if constexpr (APPLY) {
            dst = carry(Q.carry_head);
        } else {
            next = O.grads + out_float + v * E;
            dst = piece ? carry(Q.carry_head) : next;
            if (piece) out_row -= 1, out_float -= dim;  // the first end is that of the run before
            else next += dim;
        }
        bool open = piece;  // the run of the next item began before it
        uint32_t nxt = fetch(w, lane), far = 0u;
        uint2 npk = coefficient(nxt);
        if (PACKED) far = fetch(w, 32 + lane);
        // Item q ends its run where the flag of position q + 1 is set: a batch's mask
        // is 32 flags from bit shift + 1 + base on, across two words.
        const uint32_t* word = w.bits + ((w.shift + 1) >> 5);
        const int skew = (w.shift + 1) & 31;
        uint32_t lo = __ldg(word), hi = __ldg(word + 1);
        bool dead_run = false;  // the open run is the one of out-of-range lookups
        for (int32_t base = 0; base < w.len; base += 32) {
            // The next batch's items are loaded while this batch's rows are in
            // flight (with coefficients, which depend on them: one batch further).
            const uint2 pk = npk;
            if (PACKED) {
                nxt = far;
                far = fetch(w, base + 64 + lane);
            } else {
                nxt = fetch(w, base + 32 + lane);
            }
            npk = coefficient(nxt);
            const int nb = min(32, w.len - base);
            uint32_t mask = __funnelshift_r(lo, hi, skew) & (nb == 32 ? kFull : (1u << nb) - 1u);
            lo = hi;
            hi = __ldg(word + (base >> 5) + 2);
            if (base + nb == w.table_end) {
                // The table's last run ends here. It is not output if it holds the
                // out-of-range lookups.
                dead_run = __ldg(w.keys + w.table_end - 1) == dead;
                const uint32_t last = 1u << (nb - 1);
                mask = dead_run ? mask & ~last : mask | last;
            }
            const bool have = lane < nb;
            const bool end = (mask >> lane) & 1u;
            const uint32_t key = end ? __ldg(w.keys + base + lane) : 0u;
            float state = 0.f;
            if constexpr (!APPLY) {
                // Row id (row_base_t + r = key - t) and float offset of a run.
                if (end) {
                    const int r = __popc(mask & ((1u << lane) - 1u));
                    O.unique_ids[out_row + r] = static_cast<int64_t>(key) - t;
                    O.grad_offsets[out_row + r] = out_float + static_cast<int64_t>(r) * dim;
                }
                out_row += __popc(mask);
                out_float += static_cast<int64_t>(__popc(mask)) * dim;
            } else if (end) {
                // The table rows that this batch steps start moving into L1, and
                // their states into the lanes that hold the runs' ends.
                const uint32_t r = key - static_cast<uint32_t>(td.key_base);
                const char* row = static_cast<const char*>(td.data) + static_cast<uint64_t>(r) * td.row_vecs * 16u;
                for (int x = 0; x < td.row_vecs * 16; x += 128) prefetch_l1(row + x);
                if (O.apply == kApplyAdagrad) state = O.state[t][r];
            }
            // Row of the bag within the table's (kept inside it whatever the payload).
            const uint32_t my_a = have ? min(pk.x - bag_lo, static_cast<uint32_t>(P.B - 1)) : 0u;
            // runs of one lookup, begun in this chunk
            const uint32_t singles = mask & ((mask << 1) | (open ? 0u : 1u));
            if (kFastBatch && mask == 0 && nb == 32) {
                // The whole batch adds into the open run: every load group
                // unrolled, so loads of later groups overlap the adds of earlier ones.
#pragma unroll
                for (int i = 0; i < 32; i += G) {
                    const uint32_t a = __shfl_sync(kFull, my_a, i + g);
                    const float c = PACKED ? __uint_as_float(__shfl_sync(kFull, pk.y, i + g)) : 1.f;
                    const char* p = rows + static_cast<uint64_t>(a) * stride;
                    uint4 x[VPL];
#pragma unroll
                    for (int k = 0; k < VPL; ++k) x[k] = __ldg(reinterpret_cast<const uint4*>(p + voff[k]));
                    add(x, c);
                }
            } else
#pragma unroll 1
            for (int i0 = 0; i0 < nb; i0 += kItems) {
                uint4 buf[UG][VPL];
                float wt[UG];
#pragma unroll
                for (int u = 0; u < UG; ++u) {
                    const int src = i0 + u * G + g;
                    const uint32_t a = __shfl_sync(kFull, my_a, src);
                    wt[u] = PACKED ? __uint_as_float(__shfl_sync(kFull, pk.y, src)) : 1.f;
                    const char* p = rows + static_cast<uint64_t>(a) * stride;
#pragma unroll
                    for (int k = 0; k < VPL; ++k) buf[u][k] = __ldg(reinterpret_cast<const uint4*>(p + voff[k]));
                }
                const uint32_t m = (mask >> i0) & kItemMask;
                if (m == 0 && i0 + kItems <= nb) {
#pragma unroll
                    for (int u = 0; u < UG; ++u) add(buf[u], wt[u]);
                    continue;
                }
#pragma unroll
                for (int u = 0; u < UG; ++u) {
                    const int left = nb - (i0 + u * G);  // items from this step on
                    if (left <= 0) break;
                    uint32_t mu = (m >> (u * G)) & kStepMask;
                    if (mu == 0) {
                        if (G == 1 || g < left) add(buf[u], wt[u]);
                        continue;
                    }
                    if (((singles >> (i0 + u * G)) & kStepMask) == kStepMask) {
                        // Every lane group's item is a whole run: each stores (or steps) its own.
                        float one[VPL][E] = {};
#pragma unroll
                        for (int k = 0; k < VPL; ++k) accumulate<GO, PACKED>(one[k], buf[u][k], wt[u]);
                        if constexpr (APPLY) {
                            step(__shfl_sync(kFull, key, i0 + u * G + g), one,
                                 __shfl_sync(kFull, state, i0 + u * G + g), true);
                        } else {
                            store(dst + g * dim, one);
                            dst += G * dim;
                            next += G * dim;
                        }
                        continue;
                    }
                    if constexpr (G == 1) {
                        add(buf[u], wt[u]);
                        flush(APPLY ? __shfl_sync(kFull, key, i0 + u) : 0u,
                              APPLY ? __shfl_sync(kFull, state, i0 + u) : 0.f);
                    } else {
                        // Runs end after item i0 + u*G + p for each set bit p; this lane
                        // group's item (p index g) belongs to the first of them with g <= p.
                        bool added = g >= left;
                        do {
                            const int p = __ffs(mu) - 1;
                            if (!added && g <= p) {
                                add(buf[u], wt[u]);
                                added = true;
                            }
                            flush(APPLY ? __shfl_sync(kFull, key, i0 + u * G + p) : 0u,
                                  APPLY ? __shfl_sync(kFull, state, i0 + u * G + p) : 0.f);
                            mu &= mu - 1;
                        } while (mu);
                        if (!added) add(buf[u], wt[u]);
                    }
                }
            }
            open = !((mask >> (nb - 1)) & 1u);
            // Two-level summation: at most 32 / G terms per lane enter `ain`
            // before it is folded into `aout`, which bounds the rounding error.
#pragma unroll
            for (int k = 0; k < VPL; ++k)
#pragma unroll
                for (int x = 0; x < E; ++x) {
                    aout[k][x] += ain[k][x];
                    ain[k][x] = 0.f;
                }
        }
        if (open && !dead_run && __ldg(w.keys + w.len - 1) != dead) {
            // The run goes on in the next chunk: this chunk's piece of it.
            float tot[VPL][E];
            total(tot);
            if (!at_head && lane == 0) {
                // its number in the table, for the fix-up
                // (a chunk with a run begun in it begins inside none)
                Q.split[j] = kSplitBegins | (APPLY ? 0u : static_cast<uint32_t>(out_row - O.out_first[t]));
            }
            if (g == 0) store(carry(at_head ? Q.carry_head : Q.carry_tail), tot);
        }
    }
};

// Resident blocks per SM the reduce is compiled for: 3 with 8 rows in flight per
// lane, so that slices that come from DRAM or a distant L2 have the bytes in
// flight; 3 with 4 rows when the optimizer step is fused, which carries the table
// row too; 2 for four vectors per lane (16 columns in two levels). Measured, reduce
// of 41 M lookups on skewed indices (fp32 grad_out) / 12 M uniform (bf16) / 26 M
// weighted uniform (fp32), us: 8 rows at 3 blocks 1140 / 952 / 2675; 4 at 4 1133 /
// 1167 (4 at 5) / 2925; 12 at 2 1331 / - / 2613; 16 at 2 - / 1017 / -. Fused Adagrad
// step of 1.3 M lookups (Adagrad) / 41 M (SGD): 4 rows at 3 blocks 174 / 1928, 4 at 4
// 180 / 2051; without the batches with no run end unrolled - / 2154; without the runs
// of one lookup stepped by a lane group each 223 / 2140; with a row's state and
// stored values loaded only where its run ends 244 / -.
template <int VPL, bool APPLY>
constexpr int reduce_min_blocks() {
    return VPL == 4 ? 2 : (APPLY && VPL == 1 ? CB_REDUCE_APPLY_MIN_BLOCKS : CB_REDUCE_MIN_BLOCKS);
}

template <int GO, int VPL, bool PACKED, int GC, bool APPLY>
__device__ __forceinline__ void reduce_chunk(const Problem& P, const Plan& Q, const BwdOut& O, const void* grad_out,
                                             int64_t j, const Chunk& ch, const TableDev& td, int lane) {
    constexpr int eb = GO == CB_F32 ? 4 : 2;
    const int t = ch.table;
    Reduce<GO, VPL, PACKED, APPLY, GC> r{P, Q, O};
    r.j = static_cast<int32_t>(j);
    r.t = t;
    r.lane = lane;
    r.g = lane / r.V;
    r.v = lane - r.g * r.V;
    r.row_vecs = td.grad_vecs;
    r.dim = td.dim;
    typename Reduce<GO, VPL, PACKED, APPLY, GC>::Walk w;
    w.keys = O.keys_sorted + ch.k0;
    w.vals = O.vals_sorted + ch.k0;
    // the chunk's cell: positions [x0, x0 + chunk_len) of the table
    w.bits = O.head_bits + j * (Q.chunk_len / 32);
    w.shift = static_cast<int32_t>(ch.k0 - Q.table_pos[t] - (j - Q.table_chunk[t]) * Q.chunk_len);
    w.len = static_cast<int32_t>(ch.len & 0x7fffffffu);
    w.table_end = static_cast<int32_t>(Q.table_pos[t + 1] - ch.k0);
    if (lane == 0) Q.split[j] = ch.len >> 31 ? kSplitGoesOn : 0;
    if (w.len == 0) return;
    // ch.first: the chunk's first run that begins in it (the one after the piece)
    r.walk(w, static_cast<const char*>(grad_out) + static_cast<int64_t>(td.doff) * eb, P.sum_d * eb, (ch.len >> 31) != 0,
           O.out_first[t] + ch.first, O.float_base[t] + ch.first * td.dim);
}

template <int GO, int VPL, bool PACKED, int GC, bool APPLY>
__global__ void __launch_bounds__(kWarpThreads, reduce_min_blocks<VPL, APPLY>())
    bwd_reduce_kernel(const __grid_constant__ Problem P, const __grid_constant__ Plan Q,
                      const __grid_constant__ BwdOut O, const void* grad_out, int cls) {
    begin_kernel();
    if (*O.cap_fail) return;
    const int lane = threadIdx.x & 31;
    const int64_t cb = Q.class_chunk_base[cls];
    const int64_t ce = min64(Q.class_chunk_base[cls + 1], Q.max_chunks);
    for (int64_t j = first_chunk(Q, cls, cb, lane); j < ce;) {
        const int64_t nxt = fetch_next_chunk(Q, cls, cb, lane);
        const Chunk ch = Q.chunks[j];
        reduce_chunk<GO, VPL, PACKED, GC, APPLY>(P, Q, O, grad_out, j, ch, P.tables[ch.table], lane);
        j = __shfl_sync(kFull, nxt, 0);
    }
}

// Tables of several row layouts in one launch, as in the forward. 2 blocks per SM:
// at 3 the compiler spills 100 to 160 bytes (26 M weighted lookups, dims 64/128/256:
// 2672 us at 3, 2581 at 2; fused Adagrad of 490 K: 162 and 129; fp32 gradients of
// 330 K: 47 and 48).
constexpr int kMixedReduceBlocks = 2;
template <int GO, bool PACKED, bool APPLY>
__global__ void __launch_bounds__(kWarpThreads, kMixedReduceBlocks)
    bwd_reduce_mixed_kernel(const __grid_constant__ Problem P, const __grid_constant__ Plan Q,
                            const __grid_constant__ BwdOut O, const void* grad_out) {
    begin_kernel();
    if (*O.cap_fail) return;
    const int lane = threadIdx.x & 31;
    const int64_t ce = min64(Q.class_chunk_base[Q.num_classes], Q.max_chunks);
    for (int64_t j = first_chunk(Q, Q.num_classes, 0, lane); j < ce;) {
        const int64_t nxt = fetch_next_chunk(Q, Q.num_classes, 0, lane);
        const Chunk ch = Q.chunks[j];
        const TableDev& td = P.tables[ch.table];
        switch (row_layout(td.grad_vecs)) {
            case 0: reduce_chunk<GO, 1, PACKED, 32, APPLY>(P, Q, O, grad_out, j, ch, td, lane); break;
            case 1: reduce_chunk<GO, 1, PACKED, 16, APPLY>(P, Q, O, grad_out, j, ch, td, lane); break;
            case 2: reduce_chunk<GO, 1, PACKED, 8, APPLY>(P, Q, O, grad_out, j, ch, td, lane); break;
            case 3: reduce_chunk<GO, 1, PACKED, 4, APPLY>(P, Q, O, grad_out, j, ch, td, lane); break;
            case 4: reduce_chunk<GO, 1, PACKED, 2, APPLY>(P, Q, O, grad_out, j, ch, td, lane); break;
            case 5: reduce_chunk<GO, 1, PACKED, 1, APPLY>(P, Q, O, grad_out, j, ch, td, lane); break;
            case 6: reduce_chunk<GO, 2, PACKED, 1, APPLY>(P, Q, O, grad_out, j, ch, td, lane); break;
            default: reduce_chunk<GO, 4, PACKED, 1, APPLY>(P, Q, O, grad_out, j, ch, td, lane); break;
        }
        j = __shfl_sync(kFull, nxt, 0);
    }
}

template <auto Kernel, class... Args>
static void launch_reduce_grid(int64_t chunk_bound, int num_sms, cudaStream_t s, const Args&... args) {
    static const int cap = resident_blocks(Kernel, kWarpThreads);
    launch(Kernel, warp_grid(chunk_bound, static_cast<int64_t>(cap) * num_sms), kWarpThreads, 0, s, args...);
}

// cls < 0: all classes, in one launch.
template <int GO, bool APPLY>
void launch_bwd_reduce_t(const Problem& P, const Plan& Q, const BwdOut& O, const void* grad_out,
                         int cls, int vpl, int gc, bool packed, int64_t chunk_bound, int num_sms,
                         cudaStream_t s) {
    if (cls < 0) {
        if (packed) launch_reduce_grid<bwd_reduce_mixed_kernel<GO, true, APPLY>>(chunk_bound, num_sms, s, P, Q, O, grad_out);
        else launch_reduce_grid<bwd_reduce_mixed_kernel<GO, false, APPLY>>(chunk_bound, num_sms, s, P, Q, O, grad_out);
        return;
    }
#define CB_CASE(V, G, PK)                                                                \
    if (vpl == V && gc == G && packed == PK) {                                            \
        launch_reduce_grid<bwd_reduce_kernel<GO, V, PK, G, APPLY>>(chunk_bound, num_sms, s, P, Q, O, grad_out, cls); \
        return;                                                                          \
    }
    CB_CASE(1, 1, false) CB_CASE(1, 2, false) CB_CASE(1, 4, false) CB_CASE(1, 8, false)
    CB_CASE(1, 16, false) CB_CASE(1, 32, false) CB_CASE(2, 1, false) CB_CASE(4, 1, false)
    CB_CASE(1, 1, true) CB_CASE(1, 2, true) CB_CASE(1, 4, true) CB_CASE(1, 8, true)
    CB_CASE(1, 16, true) CB_CASE(1, 32, true) CB_CASE(2, 1, true) CB_CASE(4, 1, true)
#undef CB_CASE
}

}  // namespace cbtbe
