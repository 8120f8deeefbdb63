// tbe_forward.cuh -- forward gather-pool kernel template of the pooled
// embedding bag (sparse_arch lookups, Sec. IV.A.2; jagged categorical features,
// Abstract):
//   out[b, Doff_t + j] = s_b * sum_{i in bag(t, b)} w_i * E_t[indices[i], j]
//
// One warp per chunk of lookup positions. A stored row is spread over V lanes
// (16 bytes per lane per vector; V the power of two that holds the row, up to
// 32), and a warp step gathers G = 32 / V rows of the chunk at once, each lane keeping several
// 16-byte loads in flight. Rows widen to fp32 in registers; the G per-row
// partial sums of a bag meet through warp shuffles when the bag is emitted.
// Instantiated per storage type in tbe_forward_{f32,f16,bf16}.cu.
#pragma once

#include "tbe_internal.cuh"
#include "tbe_launch.h"
#include "tbe_plan.cuh"

namespace cbtbe {

// One chunk, walked by one warp in batches of 32 lookups. Before a batch's rows
// are loaded, the warp finds every bag ending inside it from a window of 32 bag
// ends (one per lane): their end positions become a 32-bit mask, and their
// numbers go, in order, to a per-warp list in shared memory; empty bags are
// written out during this scan. The rows are loaded a group of warp steps at a
// time and added bag by bag.
//
// The code is kept small: one copy of the end of a bag (combine, mean, output
// type, pieces) in the whole walker, reached by a loop over the ends of a load
// group, and one copy of the loads, whether or not the batch holds padding or
// invalid lookups (those load a valid lookup's row and are left out of the sums).
// With the end of a bag copied into every step of the group, twice, the walker
// overflowed the instruction cache (1.6 M weighted lookups on rows of 3 to 12
// vectors: 24 cycles of waiting for instructions per instruction issued). Gather
// of that call, with the small code: 190 -> 73 us; of 26 M weighted lookups on
// bf16 rows of 64 / 128 / 256: 1.54 -> 1.38 ms; of 41 M unweighted lookups on
// 256-byte fp16 rows: 0.84 ms either way.
template <int DT, int VPL, bool WEIGHTED, int G>
struct Gather {
    static constexpr int E = Storage<DT>::kElems;
    static constexpr int V = 32 / G;                                  // lanes per row
    static constexpr int kRows = CB_WALK_ROWS / VPL > 0 ? CB_WALK_ROWS / VPL : 1;
    static constexpr int UG = kRows < V ? kRows : V;                  // row steps per load group (V steps per batch)
    static constexpr int kItems = UG * G;                             // lookups per load group
    static constexpr uint32_t kItemMask = kItems == 32 ? kFull : (1u << (kItems & 31)) - 1u;
    static constexpr uint32_t kStepMask = G == 32 ? kFull : (1u << (G & 31)) - 1u;
    static constexpr bool kTwoLevel = DT == CB_F32;  // half rows: one fp32 level (registers)
    static_assert(VPL == 1 || G == 1, "several vectors per lane: one row per step");

    const Problem& P;  // kernel parameters: read in place, not held in registers
    const Plan& Q;
    void* out;         // [B, sum D] of P.out_dtype
    int32_t j;         // the chunk
    uint32_t rows;     // of the table (below 2^32)
    int64_t k0;
    int32_t len, bag_lo, doff, row_vecs;
    bool last;         // owns empty bags that start at the chunk end
    bool runs_on;      // the chunk's last bag runs past its end (set by the last scan)
    int lane, g, v;
    EndSlot* slots;
    // window of bag ends, relative to k0: lane i holds the end of bag seg + i
    int32_t seg, s_cur, my_end;
    float ain[VPL][E], aout[VPL][kTwoLevel ? E : 1];

    __device__ __forceinline__ int32_t end_of(int32_t bag) const {
        return bag < bag_lo + P.B ? rel_pos(load_index(P.offsets, bag + 1, P.is32), k0) : kRelHi;
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
#pragma unroll
            for (int x = 0; x < E; ++x) ain[k][x] = 0.f;
#pragma unroll
            for (int x = 0; x < (kTwoLevel ? E : 1); ++x) aout[k][x] = 0.f;
        }
    }
    __device__ __forceinline__ void add(const uint4 (&x)[VPL], float w) {
#pragma unroll
        for (int k = 0; k < VPL; ++k) accumulate<DT, WEIGHTED>(ain[k], x[k], w);
    }
    // N columns from column `col` of a pooled row, in the output's type.
    template <int N>
    __device__ __forceinline__ void store_vec(int64_t col, const float (&t)[N]) const {
        if (P.out_dtype == CB_F32) {
#pragma unroll
            for (int x = 0; x < N; x += 4)
                store_stream(reinterpret_cast<float4*>(static_cast<float*>(out) + col + x),
                             make_float4(t[x], t[x + 1], t[x + 2], t[x + 3]));
        } else {
#pragma unroll
            for (int x = 0; x < N; x += 4) store_out4(out, col + x, t[x], t[x + 1], t[x + 2], t[x + 3], P.out_dtype);
        }
    }
    __device__ __forceinline__ int64_t out_col(int32_t bag, int k) const {
        return static_cast<int64_t>(bag - bag_lo) * P.sum_d + doff + (v + 32 * k) * E;
    }

    // Bags ending at or before `bend` (the batch starts at `base`) leave the
    // window: non-empty ones are listed and marked in the returned mask, empty
    // ones owned by this chunk are written out. Ends are non-decreasing, so the
    // finished bags are a prefix of the window. At the chunk end, the bag that
    // runs past it is listed too, as a piece (`runs_on`).
    __device__ __forceinline__ uint32_t scan(int32_t base, int32_t bend) {
        runs_on = false;
        __syncwarp();  // every lane is done reading the previous batch's list
        uint32_t mask = 0;
        int nend = 0;
        for (;;) {
            int32_t my_beg = __shfl_up_sync(kFull, my_end, 1);
            if (lane == 0) my_beg = s_cur;
            const bool nonempty = my_end > my_beg;
            const bool done = my_end <= bend && (nonempty || my_end < len || last);
            const uint32_t dm = __ballot_sync(kFull, done);
            const uint32_t ne = __ballot_sync(kFull, done && nonempty);
            // (index masked: malformed offsets, which are reported, can break the
            // prefix property but never reach past the list)
            if (done && nonempty)
                slots[(nend + __popc(ne & ((1u << lane) - 1u))) & 31] =
                    EndSlot{seg + lane, my_beg >= 0 ? my_end - my_beg : -1};
            for (uint32_t em = dm & ~ne; em; em &= em - 1) {
                // An empty bag pools to zeros.
                const float z[E] = {};
                if (g == 0)
#pragma unroll
                    for (int k = 0; k < VPL; ++k)
                        if (v + 32 * k < row_vecs) store_vec(out_col(seg + __ffs(em) - 1, k), z);
            }
            mask |= __reduce_or_sync(kFull, (done && nonempty) ? 1u << ((my_end - base - 1) & 31) : 0u);
            nend += __popc(ne);
            const int nd = __popc(dm);
            if (nd == 0) break;
            const int32_t last_end = __shfl_sync(kFull, my_end, nd - 1);
            const int32_t moved = __shfl_down_sync(kFull, my_end, nd & 31);
            s_cur = last_end;
            seg += nd;
            my_end = lane + nd < 32 ? moved : end_of(seg + lane);
            // A full window that finished before `bend` leaves more to find; at
            // the chunk end, so may one that finished exactly there (empty bags
            // at the end of the table's last chunk).
            if (nd < 32 || (last_end >= bend && bend != len)) break;
        }
        if (bend == len && seg < bag_lo + P.B && s_cur < len && len > 0) {
            if (lane == 0) slots[nend & 31] = EndSlot{seg, s_cur >= 0 ? 0 : -1};
            mask |= 1u << ((len - base - 1) & 31);
            runs_on = true;
        }
        __syncwarp();
        return mask;
    }

    // The end of listed bag `s`: its row, or this chunk's piece of it. Half rows on
    // several lane groups: each of the first two groups ends with 4 of the lane's 8
    // columns, so the first round of the combine exchanges half the sums, and both
    // groups store (1.6 M weighted lookups on rows of 3 to 12 vectors: 74 -> 70 us;
    // 41 M on 256-byte rows: 838 -> 834).
    static constexpr bool kSplit = VPL == 1 && E == 8 && G >= 2;
    static constexpr int kOut = kSplit ? 4 : E;  // columns that a lane ends with, per vector
    __device__ __forceinline__ void flush(const EndSlot s) {
        float tot[VPL][kOut];
        const bool up = kSplit && (g & 1) != 0;  // takes the upper 4 columns
        if constexpr (kSplit) {
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float mine = up ? ain[0][x + 4] : ain[0][x], other = up ? ain[0][x] : ain[0][x + 4];
                tot[0][x] = mine + __shfl_xor_sync(kFull, other, V);
            }
        } else {
#pragma unroll
            for (int k = 0; k < VPL; ++k)
#pragma unroll
                for (int x = 0; x < E; ++x) tot[k][x] = kTwoLevel ? aout[k][x] + ain[k][x] : ain[k][x];
        }
#pragma unroll
        for (int off = kSplit ? 2 * V : V; off < 32; off <<= 1)
#pragma unroll
            for (int x = 0; x < kOut; ++x) tot[0][x] += __shfl_xor_sync(kFull, tot[0][x], off);
        zero();
        const bool writes = g < (kSplit ? 2 : 1);
        const int col = up ? 4 : 0;
        // Kept inside the table's bags whatever the list holds.
        const int32_t bag = min(max(s.seg, bag_lo), bag_lo + P.B - 1);
        if (s.len > 0) {  // a complete bag
            if (P.mean) {
                const float scale = static_cast<float>(s.len);
#pragma unroll
                for (int k = 0; k < VPL; ++k)
#pragma unroll
                    for (int x = 0; x < kOut; ++x) tot[k][x] = tot[k][x] / scale;
            }
            if (writes)
#pragma unroll
                for (int k = 0; k < VPL; ++k)
                    if (v + 32 * k < row_vecs) store_vec(out_col(bag, k) + col, tot[k]);
            return;
        }
        // A piece of a bag split across chunks: fp32, for the fix-up.
        const bool started = s.len == 0;
        if (started && lane == 0) Q.split[j] |= kSplitBegins | static_cast<uint32_t>(bag);
        float* dst = (started ? Q.carry_tail : Q.carry_head) + static_cast<int64_t>(j) * P.dmax + col;
        if (writes)
#pragma unroll
            for (int k = 0; k < VPL; ++k)
                if (v + 32 * k < row_vecs)
#pragma unroll
                    for (int x = 0; x < kOut; x += 4)
                        *reinterpret_cast<float4*>(dst + (v + 32 * k) * E + x) =
                            make_float4(tot[k][x], tot[k][x + 1], tot[k][x + 2], tot[k][x + 3]);
    }

    // A load group of one-lookup bags: every lane group's row is a whole bag, so
    // no sums meet and each group stores its own.
    __device__ __forceinline__ void store_singles(const uint4 (&buf)[UG][VPL], const float (&wt)[UG], int ce) {
#pragma unroll
        for (int u = 0; u < UG; ++u) {
            const int32_t bag = min(max(slots[(ce + u * G + g) & 31].seg, bag_lo), bag_lo + P.B - 1);
#pragma unroll
            for (int k = 0; k < VPL; ++k) {
                float t[E] = {};
                accumulate<DT, WEIGHTED>(t, buf[u][k], wt[u]);
                if (v + 32 * k < row_vecs) store_vec(out_col(bag, k), t);
            }
        }
    }

    struct Raw {
        int64_t r;
        float w;
    };
    __device__ __forceinline__ Raw fetch(int32_t q) const {
        Raw x{-1, 0.f};
        if (q < len) {
            x.r = load_index(P.indices, k0 + q, P.is32);
            if (WEIGHTED) x.w = __ldg(P.weights + k0 + q);
        }
        return x;
    }

    __device__ __forceinline__ void walk(const uint4* table) {
        const char* row0 = reinterpret_cast<const char*>(table + (v < row_vecs ? v : 0));
        const uint32_t row_bytes = row_vecs * 16u;
        // Vector v + 32k of the row, relative to the lane's first; lanes past the
        // row load one of its vectors again and never store what they sum.
        int voff[VPL];
#pragma unroll
        for (int k = 0; k < VPL; ++k) voff[k] = k > 0 && v + 32 * k < row_vecs ? 32 * k : 0;
        zero();
        s_cur = seg < bag_lo + P.B ? rel_pos(load_index(P.offsets, seg, P.is32), k0) : kRelHi;
        my_end = end_of(seg + lane);
        bool open = s_cur < 0;  // the sums hold part of a bag
        if (lane == 0) Q.split[j] = open ? kSplitGoesOn : 0;
        Raw nxt = fetch(lane);
        if (len == 0) scan(0, 0);  // a table's chunk without lookups: its empty bags
        for (int32_t base = 0; base < len; base += 32) {
            const int nb = min(32, len - base);
            // The next batch's payload is loaded while this batch's rows are in
            // flight; it is only looked at when its batch comes up.
            const Raw cur = nxt;
            nxt = fetch(base + 32 + lane);
            const uint32_t mask = scan(base, base + nb);
            // Row ids are checked here, once per lookup; an invalid one (and
            // padding) contributes nothing.
            const bool valid = static_cast<uint64_t>(cur.r) < rows;
            if (!valid && lane < nb) set_error(P.error, CB_ERR_INDEX_OOB);
            const uint32_t vm = __ballot_sync(kFull, valid);
            uint32_t my_a = static_cast<uint32_t>(cur.r);
            const uint32_t some = __shfl_sync(kFull, my_a, vm ? __ffs(vm) - 1 : 0);
            if (!valid) my_a = vm ? some : 0u;
            const char* base_row = vm ? row0 : reinterpret_cast<const char*>(P.zero_row + v);
            // lookups that are a bag of their own, begun in this chunk
            uint32_t singles = mask & ((mask << 1) | (open ? 0u : 1u)) & vm;
            if (runs_on) singles &= ~(1u << (nb - 1));
            int ce = 0;  // next entry of the list
#pragma unroll 1
            for (int i0 = 0; i0 < nb; i0 += kItems) {
                uint4 buf[UG][VPL];
                float wt[UG];
#pragma unroll
                for (int u = 0; u < UG; ++u) {
                    const int src = i0 + u * G + g;
                    const uint32_t a = __shfl_sync(kFull, my_a, src);
                    wt[u] = WEIGHTED ? __shfl_sync(kFull, cur.w, src) : 1.f;
                    const uint4* p =
                        reinterpret_cast<const uint4*>(base_row + static_cast<uint64_t>(a) * row_bytes);
#pragma unroll
                    for (int k = 0; k < VPL; ++k) buf[u][k] = __ldg(p + voff[k]);
                }
                uint32_t m = (mask >> i0) & kItemMask;  // bags ending in the group
                const uint32_t live = (vm >> i0) & kItemMask;
                if (m == 0 && live == kItemMask) {
#pragma unroll
                    for (int u = 0; u < UG; ++u) add(buf[u], wt[u]);
                    continue;
                }
                if (((singles >> i0) & kItemMask) == kItemMask) {
                    store_singles(buf, wt, ce);
                    ce += kItems;
                    continue;
                }
                // Bag by bag: the group's lookups up to the next end, then its row.
                uint32_t todo = live;
                for (;;) {
                    const uint32_t upto = m ? (m ^ (m - 1)) : kFull;  // up to the lowest end
                    const uint32_t now = todo & upto;
#pragma unroll
                    for (int u = 0; u < UG; ++u) {
                        const uint32_t step = (now >> (u * G)) & kStepMask;
                        if (step != 0 && ((step >> g) & 1u)) add(buf[u], wt[u]);
                    }
                    if (m == 0) break;
                    flush(slots[ce++]);
                    todo &= ~upto;
                    m &= m - 1;
                }
            }
            open = !(mask >> (nb - 1) & 1u);
            // Two-level summation: at most 32 / G terms per lane enter `ain`
            // before it is folded into `aout`, which bounds the rounding error.
            if constexpr (kTwoLevel) {
#pragma unroll
                for (int k = 0; k < VPL; ++k)
#pragma unroll
                    for (int x = 0; x < E; ++x) {
                        aout[k][x] += ain[k][x];
                        ain[k][x] = 0.f;
                    }
            }
        }
    }
};

// Resident blocks per SM the gather is compiled for. The row walker with one
// vector per lane and no weights fits 5 blocks' registers (48) without
// spilling, and the gather's rate out of L2 grows with the warps resident
// (cfg5: 4.07 -> 3.72 ms from 4 to 5 blocks); the other layouts spill at 48
// registers and keep 4.
#ifndef CB_WALK_MIN_BLOCKS_ROW
#define CB_WALK_MIN_BLOCKS_ROW 5
#endif
#ifndef CB_WALK_ROW_WEIGHTED
#define CB_WALK_ROW_WEIGHTED 0  // 1: weighted row layouts take CB_WALK_MIN_BLOCKS_ROW too
#endif
template <int VPL, bool WEIGHTED, int GC>
constexpr int gather_min_blocks() {
    return VPL == 1 && GC != 4 && (!WEIGHTED || CB_WALK_ROW_WEIGHTED) ? CB_WALK_MIN_BLOCKS_ROW
                                                                                : CB_WALK_MIN_BLOCKS;
}

#ifndef CB_WALK_MIN_BLOCKS_MIXED
#define CB_WALK_MIN_BLOCKS_MIXED 4
#endif

// Chunk j, walked by one warp.
template <int DT, int VPL, bool WEIGHTED, int GC>
__device__ __forceinline__ void gather_chunk(const Problem& P, const Plan& Q, void* out, int64_t j, const Chunk& ch,
                                             const TableDev& td, int lane, EndSlot* slots) {
    Gather<DT, VPL, WEIGHTED, GC> w{P, Q, out};
    w.j = static_cast<int32_t>(j);
    w.k0 = ch.k0;
    w.rows = static_cast<uint32_t>(td.rows);
    w.len = static_cast<int32_t>(ch.len & 0x7fffffffu);
    w.bag_lo = ch.table * P.B;
    w.doff = td.doff;
    w.row_vecs = td.row_vecs;
    w.last = (ch.len >> 31) != 0;
    w.lane = lane;
    w.g = lane / w.V;
    w.v = lane - w.g * w.V;
    w.slots = slots;
    w.seg = static_cast<int32_t>(ch.first);
    w.walk(static_cast<const uint4*>(td.data));
}

template <int DT, int VPL, bool WEIGHTED, int GC>
__global__ void __launch_bounds__(kWarpThreads, gather_min_blocks<VPL, WEIGHTED, GC>())
    fwd_gather_kernel(const __grid_constant__ Problem P, const __grid_constant__ Plan Q, void* out,
                      int cls) {
    __shared__ EndSlot slots[kWarpThreads / 32][32];
    begin_kernel();
    const int lane = threadIdx.x & 31;
    const int64_t cb = Q.class_chunk_base[cls];
    const int64_t ce = min64(Q.class_chunk_base[cls + 1], Q.max_chunks);
    for (int64_t j = first_chunk(Q, cls, cb, lane); j < ce;) {
        const int64_t nxt = fetch_next_chunk(Q, cls, cb, lane);
        const Chunk ch = Q.chunks[j];
        gather_chunk<DT, VPL, WEIGHTED, GC>(P, Q, out, j, ch, P.tables[ch.table], lane, slots[threadIdx.x >> 5]);
        j = __shfl_sync(kFull, nxt, 0);
    }
}

// Chunk j, whatever its table's row layout.
template <int DT, bool WEIGHTED>
__device__ __forceinline__ void gather_any(const Problem& P, const Plan& Q, void* out, int64_t j, const Chunk& ch,
                                           const TableDev& td, int lane, EndSlot* mine) {
    switch (row_layout(td.row_vecs)) {
        case 0: gather_chunk<DT, 1, WEIGHTED, 32>(P, Q, out, j, ch, td, lane, mine); break;
        case 1: gather_chunk<DT, 1, WEIGHTED, 16>(P, Q, out, j, ch, td, lane, mine); break;
        case 2: gather_chunk<DT, 1, WEIGHTED, 8>(P, Q, out, j, ch, td, lane, mine); break;
        case 3: gather_chunk<DT, 1, WEIGHTED, 4>(P, Q, out, j, ch, td, lane, mine); break;
        case 4: gather_chunk<DT, 1, WEIGHTED, 2>(P, Q, out, j, ch, td, lane, mine); break;
        case 5: gather_chunk<DT, 1, WEIGHTED, 1>(P, Q, out, j, ch, td, lane, mine); break;
        case 6: gather_chunk<DT, 2, WEIGHTED, 1>(P, Q, out, j, ch, td, lane, mine); break;
        default: gather_chunk<DT, 4, WEIGHTED, 1>(P, Q, out, j, ch, td, lane, mine); break;
    }
}

// Tables of several row layouts (one storage type) in one launch: every layout's
// walker is compiled in, and a warp takes chunks of all classes in one sequence
// (the counter after the classes' own), so that the GPU does not wait for the last
// warps of each class in turn.
template <int DT, bool WEIGHTED>
__global__ void __launch_bounds__(kWarpThreads, CB_WALK_MIN_BLOCKS_MIXED)
    fwd_gather_mixed_kernel(const __grid_constant__ Problem P, const __grid_constant__ Plan Q, void* out) {
    __shared__ EndSlot slots[kWarpThreads / 32][32];
    begin_kernel();
    const int lane = threadIdx.x & 31;
    EndSlot* mine = slots[threadIdx.x >> 5];
    const int64_t ce = min64(Q.class_chunk_base[Q.num_classes], Q.max_chunks);
    for (int64_t j = first_chunk(Q, Q.num_classes, 0, lane); j < ce;) {
        const int64_t nxt = fetch_next_chunk(Q, Q.num_classes, 0, lane);
        const Chunk ch = Q.chunks[j];
        const TableDev& td = P.tables[ch.table];
        gather_any<DT, WEIGHTED>(P, Q, out, j, ch, td, lane, mine);
        j = __shfl_sync(kFull, nxt, 0);
    }
}

// A small forward in one kernel and its fix-up: the grid holds a warp for every
// chunk, every block scans the tables for itself and every warp places its own chunk,
// all 32 lanes searching. The plan kernel it saves was a third of such a call's
// time on the GPU: serving request of 5 K lookups in 26 tables 15.0 -> 12.2 us, one
// table of 512 lookups 15.1 -> 11.8 (at 3 blocks, 80 registers: 13.3 and 13.1; at 4:
// 14.9 and 11.5). With more chunks than resident warps (here
// kPlannedBlocks blocks of 8 per SM) the searches would come again for each, ahead of its loads.
template <int DT, bool WEIGHTED>
__global__ void __launch_bounds__(kWarpThreads, kPlannedBlocks)
    fwd_planned_kernel(const __grid_constant__ Problem P, const __grid_constant__ Plan Q, void* out) {
    __shared__ int64_t pos[kPlanTables + 1], ord[kPlanTables + 1], sh[33];
    __shared__ EndSlot slots[kWarpThreads / 32][32];
    begin_kernel();
    plan_tables(P, Q, 0, pos, ord, nullptr, sh);
    const int lane = threadIdx.x & 31;
    const int64_t total = min64(ord[P.T], Q.max_chunks);
    if (blockIdx.x == 0 && threadIdx.x == 0) Q.class_chunk_base[Q.num_classes] = total;  // for the fix-up
    for (int64_t j = warp_id_global(); j < total; j += warps_in_grid()) {
        const Chunk ch = plan_chunk<32>(P, Q, pos, ord, j, lane);
        if (lane == 0) Q.chunks[j] = ch;
        gather_any<DT, WEIGHTED>(P, Q, out, j, ch, P.tables[ch.table], lane, slots[threadIdx.x >> 5]);
    }
}

template <auto Kernel, class... Args>
static void launch_gather(int64_t chunk_bound, int num_sms, cudaStream_t s, const Args&... args) {
    static const int cap = resident_blocks(Kernel, kWarpThreads);
    launch(Kernel, warp_grid(chunk_bound, static_cast<int64_t>(cap) * num_sms), kWarpThreads, 0, s, args...);
}

// Row layouts compiled for: one vector per lane with 1 to 32 rows per step, or
// 2 or 4 vectors per lane with one row per step. cls = kAllClasses: all classes, in
// one launch; kPlanned: with their plan.
template <int DT>
void launch_gather_dtype(const Problem& P, const Plan& Q, void* out, int cls, int vpl, int gc,
                         int64_t chunk_bound, int num_sms, cudaStream_t s) {
    if (cls == kPlanned) {
        if (P.weights) launch_gather<fwd_planned_kernel<DT, true>>(chunk_bound, num_sms, s, P, Q, out);
        else launch_gather<fwd_planned_kernel<DT, false>>(chunk_bound, num_sms, s, P, Q, out);
        return;
    }
    if (cls == kAllClasses) {
        if (P.weights) launch_gather<fwd_gather_mixed_kernel<DT, true>>(chunk_bound, num_sms, s, P, Q, out);
        else launch_gather<fwd_gather_mixed_kernel<DT, false>>(chunk_bound, num_sms, s, P, Q, out);
        return;
    }
#define CB_CASE(V, G)                                                                                     \
    if (vpl == V && gc == G) {                                                                             \
        if (P.weights) launch_gather<fwd_gather_kernel<DT, V, true, G>>(chunk_bound, num_sms, s, P, Q, out, cls); \
        else launch_gather<fwd_gather_kernel<DT, V, false, G>>(chunk_bound, num_sms, s, P, Q, out, cls);    \
        return;                                                                                            \
    }
    CB_CASE(1, 1) CB_CASE(1, 2) CB_CASE(1, 4) CB_CASE(1, 8) CB_CASE(1, 16) CB_CASE(1, 32)
    CB_CASE(2, 1) CB_CASE(4, 1)
#undef CB_CASE
}

}  // namespace cbtbe
