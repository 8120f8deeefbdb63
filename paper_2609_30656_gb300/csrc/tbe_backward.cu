// tbe_backward.cu -- de-duplicated backward of the pooled embedding bag with
// respect to the table rows (the adjoint of the sparse_arch lookup, Sec. IV.A.2):
//   G[row_base_t + r] = sum_{i : table t, indices[i] == r} w_i * s_b(i) * grad_out[b(i), Doff_t ..]
//
// Steps: (1) key generation: one warp per chunk of lookups walks the bags and
// writes key_i = key_base_t + indices[i] with a payload (the bag id, or the
// lookup position plus a packed (bag, w_i * s_b) pair when a coefficient is
// needed); (2) radix sort of each table's range; (3) runs of equal sorted keys,
// counted per chunk of sorted positions, and (4) per-table output ranges and
// packed gradient offsets; (5) segmented reduce of the gathered grad_out
// slices, one warp per chunk; (6) fp64 fix-up of runs that straddle chunks.
#include <cuda_bf16.h>

#include "tbe_internal.cuh"
#include "tbe_fixup.cuh"
#include "tbe_launch.h"
#include "tbe_reduce.cuh"

namespace cbtbe {

// ---------------------------------------------------------------- (1) keys

// A warp walks one chunk kKeygenSteps x 32 lookups at a time: the indices (and
// weights) of all the steps are loaded first, so that many loads are in flight
// per warp, then each step finds its lanes' bags and writes.
#ifndef CB_KEYGEN_STEPS
#define CB_KEYGEN_STEPS 12
#endif
constexpr int kKeygenSteps = CB_KEYGEN_STEPS;

// Compiled with no minimum of resident blocks: 48 registers, 5 blocks of 256
// threads per SM. (A minimum of 1 let it take 72 registers, 3 blocks: cfg5
// 0.63 -> 0.75 ms; a minimum of 6, 40 registers: cfg5u 0.63 -> 0.71 ms.)
// COUNT: the first sort pass's digits are counted on the way (few tiles).
template <bool PACKED, bool COUNT>
__global__ void __launch_bounds__(kWarpThreads) keygen_kernel(Problem P, Plan Q, KeyGen K) {
    begin_kernel();
    const int lane = threadIdx.x & 31;
    const int64_t total = min(Q.class_chunk_base[Q.num_classes], Q.max_chunks);
    // all classes' chunks in one sequence: the counter after the classes' own
    for (int64_t j = first_chunk(Q, Q.num_classes, 0, lane); j < total;) {
        const int64_t nxt = fetch_next_chunk(Q, Q.num_classes, 0, lane);
        const Chunk ch = Q.chunks[j];
        const int t = ch.table;
        const TableDev& td = P.tables[t];
        const int64_t rows = td.rows, key_base = td.key_base;
        const int64_t k0 = ch.k0;
        const int32_t len = static_cast<int32_t>(ch.len & 0x7fffffffu);
        const int64_t bag_lo = static_cast<int64_t>(t) * P.B, bag_hi = bag_lo + P.B;
        uint32_t* keys = K.keys + k0;
        uint32_t* vals = K.vals + k0;
        // the chunk's first position within its table, and the table's counts
        const int64_t in_table = k0 - Q.table_pos[t];
        uint32_t* digits = COUNT ? K.tile_digits + K.table_first_tile[t] * 256 : nullptr;
        BagWindow32 W = bag_window32(P, ch.first, bag_hi, k0, lane);
        for (int32_t base = 0; base < len; base += 32 * kKeygenSteps) {
            int64_t idx[kKeygenSteps];
            float wt[kKeygenSteps];
#pragma unroll
            for (int u = 0; u < kKeygenSteps; ++u) {
                const int32_t q = base + 32 * u + lane;
                idx[u] = q < len ? load_index(P.indices, k0 + q, P.is32) : 0;
                wt[u] = PACKED && P.weights && q < len ? __ldg(P.weights + k0 + q) : 1.f;
            }
#pragma unroll
            for (int u = 0; u < kKeygenSteps; ++u) {
                const int32_t q = base + 32 * u + lane;
                if (base + 32 * u >= len) break;  // warp-uniform
                const bool valid = q < len;
                int64_t my_bag;
                int32_t my_s = 0, my_e = 0;
                if (!bags_by_mask(W, base + 32 * u, lane, PACKED && P.mean, my_bag, my_s, my_e))
                    find_bag32(P, W, bag_hi, k0, q, valid, lane, my_bag, my_s, my_e);
                if (!valid) continue;
                if (my_bag >= bag_hi) {  // only reachable with malformed offsets
                    set_error(P.error, CB_ERR_BAD_OFFSETS);
                    my_bag = bag_hi - 1;
                }
                // An out-of-range index takes the table's spare key (it sorts
                // after every row into a run the reduce drops) and a bag outside
                // the table: it contributes to no gradient row.
                int64_t r = idx[u];
                uint32_t bag = static_cast<uint32_t>(my_bag);
                if (r < 0 || r >= rows) {
                    set_error(P.error, CB_ERR_INDEX_OOB);
                    r = rows;
                    bag = kDeadBag;
                }
                keys[q] = static_cast<uint32_t>(key_base + r);
                if (COUNT) atomicAdd(digits + (in_table + q) / kSortTileKeys * 256 + (r & 255), 1u);
                if (PACKED) {
                    float c = wt[u];
                    if (P.mean && my_e > my_s) c = c / static_cast<float>(my_e - my_s);
                    vals[q] = static_cast<uint32_t>(k0 + q);
                    K.packed[k0 + q] = make_uint2(bag, __float_as_uint(c));
                } else {
                    vals[q] = bag;
                }
            }
        }
        j = __shfl_sync(kFull, nxt, 0);
    }
}

// ---------------------------------------------------------------- (3) runs

// A table's sorted positions are cut into cells of chunk_len positions (the last
// one shorter), numbered as its chunks. Per cell: how many runs begin in it (low
// half) and where the first does (high half; kNoHead: none), and a flag per
// position for the reduce. One warp per cell, all of its keys loaded before any is
// compared.
constexpr uint32_t kNoHead = 0xffffu;

__global__ void __launch_bounds__(kWarpThreads) bwd_heads_kernel(const __grid_constant__ Problem P,
                                                                 const __grid_constant__ Plan Q,
                                                                 const __grid_constant__ BwdOut O) {
    begin_kernel();
    constexpr int kBatches = kMaxChunk / 32;
    const int lane = threadIdx.x & 31;
    const int64_t total = min64(Q.class_chunk_base[Q.num_classes], Q.max_chunks);
    const int64_t j = warp_id_global();
    if (j >= total) return;
    const int t = Q.chunks[j].table;
    const int64_t p0 = Q.table_pos[t], p1 = max64(p0, Q.table_pos[t + 1]);
    const int64_t x0 = min64(p0 + (j - Q.table_chunk[t]) * Q.chunk_len, p1);
    const int32_t len = static_cast<int32_t>(min64(Q.chunk_len, p1 - x0));
    const uint32_t* keys = O.keys_sorted + x0;
    uint32_t k[kBatches];
#pragma unroll
    for (int i = 0; i < kBatches; ++i) k[i] = 32 * i + lane < len ? __ldg(keys + 32 * i + lane) : 0u;
    uint32_t before = x0 > p0 ? __ldg(keys - 1) : ~k[0];  // (lane 0) a table's first key starts a run
    uint32_t count = 0, first = kNoHead, flags = 0;
#pragma unroll
    for (int i = 0; i < kBatches; ++i) {
        if (32 * i >= len) break;  // warp-uniform
        uint32_t prev = __shfl_up_sync(kFull, k[i], 1);
        if (lane == 0) prev = before;
        const uint32_t b = __ballot_sync(kFull, 32 * i + lane < len && k[i] != prev);
        count += __popc(b);
        if (first == kNoHead && b) first = 32 * i + __ffs(b) - 1;
        if (lane == i) flags = b;
        before = __shfl_sync(kFull, k[i], 31);
    }
    if (lane < (len + 31) / 32) O.head_bits[j * (Q.chunk_len / 32) + lane] = flags;
    if (lane == 0) O.heads[j] = count | (first << 16);
}

// ---------------------------------------------------------------- (4) ranges

// The output's layout from the tables' run counts (one block): first row and
// first float of every table, the totals, and the capacity check.
__device__ __forceinline__ void output_ranges(const Problem& P, const BwdOut& O, int64_t* sh) {
    const int tid = threadIdx.x;
    int64_t rows = 0, floats = 0;
    for (int t0 = 0; t0 < P.T; t0 += blockDim.x) {
        const int u = t0 + tid;
        const int64_t live = u < P.T ? __ldcg(O.run_count + u) : 0;
        const int64_t dim = u < P.T ? P.tables[u].dim : 0;
        int64_t rows_total, floats_total;
        const int64_t ex_rows = block_excl_scan(live, sh, &rows_total);
        const int64_t ex_floats = block_excl_scan(live * dim, sh, &floats_total);
        if (u < P.T) {
            O.out_first[u] = rows + ex_rows;
            O.float_base[u] = floats + ex_floats;
            if (O.table_offsets) O.table_offsets[u] = rows + ex_rows;
        }
        rows += rows_total;
        floats += floats_total;
    }
    if (tid == 0) {
        O.out_first[P.T] = rows;
        O.float_base[P.T] = floats;
        if (O.table_offsets) O.table_offsets[P.T] = rows;
        *O.num_unique = rows;
        *O.num_floats = floats;
        int fail = 0;
        // After a timed-out sort pass the sorted order is not trustworthy. (The error
        // word does not tell: it keeps an earlier error of the call, and the host may
        // have read and cleared it between a size query and its finish.)
        if (O.timed_out && *O.timed_out) {
            set_error(P.error, CB_ERR_TIMEOUT);
            fail = 1;
        }
        if (O.grads && (rows > O.cap_rows || floats > O.cap_floats)) {
            set_error(P.error, CB_ERR_CAPACITY);
            fail = 1;
        }
        *O.cap_fail = fail;
        if (O.grads && !fail) O.grad_offsets[rows] = floats;
    }
}

// One block per table scans its cells' counts into the reduce's chunks: a cell in
// which a run begins becomes the chunk from that run on (the positions before it
// join the chunk before), a cell without one stays a chunk inside a run, a piece
// for the fix-up. So only runs that cover whole cells are split, and a piece
// holds nothing but its run. The last block to finish lays out the output.
__global__ void __launch_bounds__(1024) bwd_runs_kernel(const __grid_constant__ Problem P,
                                                        const __grid_constant__ Plan Q,
                                                        const __grid_constant__ BwdOut O) {
    begin_kernel();
    constexpr int kPer = 4;
    __shared__ int64_t sh[33];
    __shared__ bool sh_last;
    const int t = blockIdx.x, tid = threadIdx.x;
    if (t == 0)  // the walkers' chunk counters
        for (int c = tid; c <= Q.num_classes; c += blockDim.x) Q.chunk_next[c] = 0;
    const int64_t p0 = Q.table_pos[t], p1 = max64(p0, Q.table_pos[t + 1]);
    const int64_t C = Q.chunk_len;
    const int64_t c0 = Q.table_chunk[t];
    const int64_t cells = min64(max64(1, (p1 - p0 + C - 1) / C), Q.max_chunks - c0);
    int64_t carry = 0;
    for (int64_t i0 = 0; i0 < cells; i0 += static_cast<int64_t>(blockDim.x) * kPer) {
        const int64_t i = i0 + static_cast<int64_t>(tid) * kPer;
        uint32_t h[kPer + 1];
        int64_t sum = 0;
#pragma unroll
        for (int u = 0; u <= kPer; ++u) h[u] = i + u < cells && p1 > p0 ? O.heads[c0 + i + u] : kNoHead << 16;
#pragma unroll
        for (int u = 0; u < kPer; ++u) sum += h[u] & 0xffffu;
        int64_t total;
        int64_t run = carry + block_excl_scan(sum, sh, &total);
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (i + u < cells) {
                const uint32_t f = h[u] >> 16, fn = h[u + 1] >> 16;
                const int64_t x0 = min64(p0 + (i + u) * C, p1);
                const int64_t k0 = f == kNoHead ? x0 : x0 + f;
                int64_t k1 = p1;
                if (i + u + 1 < cells) k1 = min64(p0 + (i + u + 1) * C, p1) + (fn == kNoHead ? 0 : fn);
                Chunk ch;
                ch.k0 = k0;
                ch.first = run;
                ch.table = t;
                ch.len = static_cast<uint32_t>(max64(0, k1 - k0)) | (f == kNoHead && p1 > p0 ? 0x80000000u : 0u);
                Q.chunks[c0 + i + u] = ch;
            }
            run += h[u] & 0xffffu;
        }
        carry += total;
    }
    if (tid == 0) {
        // A table's last run may hold its out-of-range lookups (the spare key):
        // it is not output.
        const TableDev& td = P.tables[t];
        const bool dead = p1 > p0 && static_cast<int64_t>(O.keys_sorted[p1 - 1]) == td.key_base + td.rows;
        O.run_count[t] = carry - (dead ? 1 : 0);
        __threadfence();
        sh_last = atomicAdd(O.tables_done, 1u) == static_cast<uint32_t>(P.T) - 1;
    }
    __syncthreads();
    if (!sh_last) return;
    __threadfence();
    output_ranges(P, O, sh);
    if (tid == 0) *O.tables_done = 0;
}

// The ranges alone, for a call that finishes a size query.
__global__ void __launch_bounds__(1024) bwd_outputs_kernel(const __grid_constant__ Problem P,
                                                           const __grid_constant__ BwdOut O) {
    begin_kernel();
    __shared__ int64_t sh[33];
    output_ranges(P, O, sh);
}

// ---------------------------------------------------------------- (6) fix-up

// Runs split over chunks (hot rows that cover whole cells). With the optimizer step
// fused, the row is stepped as soon as its sum is complete. (With a list of the heavy
// runs for a second kernel, and a third kernel for the step, reduce and fix-up of 330 K
// fp32 lookups took 53 us, in one kernel 44; of 1.3 M with fused Adagrad 256 and 244.)
struct RunSplit {
    static constexpr bool kNarrow = true;
    const Problem& P;
    const Plan& Q;
    const BwdOut& O;
    int total;

    // A run's pieces are consecutive chunks that begin inside a run, and hold nothing but
    // it. How many of the chunks i0, i0 + dir, ... do: kNear are looked at, all at once (a
    // serial look, 32 at a time, was the longest chain of a mid-size call's fix-up).
    static constexpr int kWindows = 4, kNear = 32 * kWindows;
    struct Near {
        uint32_t in[kWindows];
        __device__ __forceinline__ int count() const {
            int n = 0;
#pragma unroll
            for (int u = 0; u < kWindows; ++u)
                if (n == 32 * u) n += __clz(__brev(~in[u]));
            return n;
        }
    };
    __device__ __forceinline__ Near near(int i0, int dir, int lane) const {
        unsigned long long word[kWindows];
#pragma unroll
        for (int u = 0; u < kWindows; ++u) {
            const int i = i0 + dir * (32 * u + lane);
            word[u] = i >= 0 && i < total ? Q.split[i] : 0;
        }
        Near x;
#pragma unroll
        for (int u = 0; u < kWindows; ++u) x.in[u] = __ballot_sync(kFull, (word[u] & kSplitGoesOn) != 0);
        return x;
    }
    // Beyond them, a search by 33 parts a round: the pieces of one run are those of its
    // table with as many runs before them. The last piece of `like`'s run after chunk lo,
    // and the first before chunk hi, which are pieces of it.
    __device__ __forceinline__ bool is_piece(int i, const Chunk& like) const {
        const Chunk& ch = Q.chunks[i];
        return (ch.len >> 31) != 0 && ch.table == like.table && ch.first == like.first;
    }
    __device__ __forceinline__ int last_piece(int lo, int lane) const {
        const Chunk like = Q.chunks[lo];
        int hi = total;  // none
#pragma unroll 1
        while (hi - lo > 1) {
            const int step = (hi - lo + 32) / 33, p = lo + (lane + 1) * step;
            const int c = __clz(__brev(~__ballot_sync(kFull, p < hi && is_piece(p, like))));
            hi = min(hi, lo + (c + 1) * step);
            lo += c * step;
        }
        return lo;
    }
    __device__ __forceinline__ int first_piece(int hi, int lane) const {
        const Chunk like = Q.chunks[hi];
        int lo = -1;  // none
#pragma unroll 1
        while (hi - lo > 1) {
            const int step = (hi - lo + 32) / 33, p = hi - (lane + 1) * step;
            const int c = __clz(__brev(~__ballot_sync(kFull, p > lo && is_piece(p, like))));
            lo = max(lo, hi - (c + 1) * step);
            hi -= c * step;
        }
        return hi;
    }

    __device__ __forceinline__ int pieces(int j, uint32_t, int lane) const {
        const int n = near(j + 1, 1, lane).count();
        return n < kNear ? n : last_piece(j + n, lane) - j;
    }
    __device__ __forceinline__ bool origin(int i, int lane, int& j, int& m) const {
        const Near next = near(i + 1, 1, lane), prev = near(i - 1, -1, lane);
        const int after = next.count(), before = prev.count();
        const int last = after < kNear ? i + after : last_piece(i + after, lane);
        j = (before < kNear ? i - before : first_piece(i - before, lane)) - 1;
        m = last - j;
        // (a run of out-of-range lookups is not summed: no chunk has it as begun)
        return j >= 0 && (Q.split[j] & kSplitBegins) != 0;
    }
    // Where the sum goes: the gradient row, or, for a fused step, the tail slot of the
    // chunk where the run begins.
    using Dest = float*;
    __device__ __forceinline__ Dest dest(int j, uint32_t seg, int t) const {
        return O.apply ? Q.carry_tail + static_cast<int64_t>(j) * P.dmax
                       : O.grads + O.float_base[t] + static_cast<int64_t>(seg) * P.tables[t].dim;
    }
    __device__ __forceinline__ void store(Dest d, int x0, double (&acc)[4]) const {
        *reinterpret_cast<float4*>(d + x0) = make_float4(static_cast<float>(acc[0]), static_cast<float>(acc[1]),
                                                         static_cast<float>(acc[2]), static_cast<float>(acc[3]));
    }
    // The fused step of the row: lane l steps columns [4l + 128k, + 4).
    __device__ __forceinline__ void stored(int j, int t, int lane) const {
        if (!O.apply) return;
        const float* g = dest(j, 0, t);
        const TableDev& td = P.tables[t];
        const Chunk ch = Q.chunks[j];
        // the chunk's last position belongs to the run
        const int64_t r = static_cast<int64_t>(O.keys_sorted[ch.k0 + (ch.len & 0x7fffffffu) - 1]) - td.key_base;
        float sq = 0.f;
#pragma unroll 1
        for (int x0 = lane * 4; x0 < td.dim; x0 += 128) sq += sq4(*reinterpret_cast<const float4*>(g + x0));
        const float scale = step_scale(O, t, r, td.dim, sq);
#pragma unroll 1
        for (int x0 = lane * 4; x0 < td.dim; x0 += 128)
            step_cols(td, r, x0, *reinterpret_cast<const float4*>(g + x0), scale);
    }
};

// BLOCKS per SM: 3 (80 registers), or 5 (48, and spills) for a grid of 2 to 4 blocks per SM,
// which then is resident beside the end of the reduce. Whole backward, us, at 3 and 5: 52 K
// lookups with the fused step (216 blocks) 75.5, 79.8; 106 K one-hot (446 blocks) 78.4,
// 71.6; 158 K (657 blocks) 88.1, 89.9; 330 K (736 blocks) 104.4, 106.0; the fix-up alone of
// 123 M skewed ones 62, 78.
template <int BLOCKS>
__global__ void __launch_bounds__(kWarpThreads, BLOCKS) bwd_fixup_kernel(const __grid_constant__ Problem P,
                                                                         const __grid_constant__ Plan Q,
                                                                         const __grid_constant__ BwdOut O, int span,
                                                                         int group_blocks) {
    begin_kernel();
    if (*O.cap_fail) return;
    const int total = static_cast<int>(min64(Q.class_chunk_base[Q.num_classes], Q.max_chunks));
    fix_split(P, Q, RunSplit{P, Q, O, total}, total, span, group_blocks);
}

// ---------------------------------------------------------------- launchers

template <auto Kernel>
static void launch_keygen_one(const Problem& P, const Plan& Q, const KeyGen& K, int64_t chunk_bound, int num_sms,
                              cudaStream_t s) {
    static const int cap = resident_blocks(Kernel, kWarpThreads);
    launch(Kernel, warp_grid(chunk_bound, static_cast<int64_t>(cap) * num_sms), kWarpThreads, 0, s, P, Q, K);
}

void launch_keygen(const Problem& P, const Plan& Q, const KeyGen& K, bool packed, int64_t chunk_bound,
                   int num_sms, cudaStream_t s) {
    if (packed && K.tile_digits) launch_keygen_one<keygen_kernel<true, true>>(P, Q, K, chunk_bound, num_sms, s);
    else if (packed) launch_keygen_one<keygen_kernel<true, false>>(P, Q, K, chunk_bound, num_sms, s);
    else if (K.tile_digits) launch_keygen_one<keygen_kernel<false, true>>(P, Q, K, chunk_bound, num_sms, s);
    else launch_keygen_one<keygen_kernel<false, false>>(P, Q, K, chunk_bound, num_sms, s);
}

void launch_bwd_runs(const Problem& P, const Plan& Q, const BwdOut& O, int64_t chunk_bound, int num_sms,
                     cudaStream_t s) {
    const int64_t blocks = (chunk_bound + kWarpThreads / 32 - 1) / (kWarpThreads / 32);
    launch(bwd_heads_kernel, static_cast<unsigned>(max64(blocks, 1)), kWarpThreads, 0, s, P, Q, O);
    // A block of 1024 per table while the GPU holds them at once; more tables with few cells
    // (backward of 16 K lookups in 2000 tables 158 -> 133 us, of 74 K in 3000 236 -> 198)
    // take blocks of 256. With many cells the largest table may have most of them.
    const bool small = P.T > 2 * num_sms && chunk_bound - P.T <= 8192;
    launch(bwd_runs_kernel, static_cast<unsigned>(P.T), small ? 256 : 1024, 0, s, P, Q, O);
}

void launch_bwd_outputs(const Problem& P, const BwdOut& O, cudaStream_t s) {
    launch(bwd_outputs_kernel, 1, 1024, 0, s, P, O);
}

void launch_bwd_reduce(const Problem& P, const Plan& Q, const BwdOut& O, const void* grad_out, int cls,
                       int vpl, int gc, bool packed, bool apply, int64_t chunk_bound, int num_sms,
                       cudaStream_t s) {
    if (P.out_dtype == CB_F16) {
        launch_bwd_reduce_f16(P, Q, O, grad_out, cls, vpl, gc, packed, apply, chunk_bound, num_sms, s);
    } else if (P.out_dtype == CB_BF16) {
        launch_bwd_reduce_bf16(P, Q, O, grad_out, cls, vpl, gc, packed, apply, chunk_bound, num_sms, s);
    } else if (apply) {
        launch_bwd_reduce_f32_apply(P, Q, O, grad_out, cls, vpl, gc, packed, chunk_bound, num_sms, s);
    } else {
        launch_bwd_reduce_f32(P, Q, O, grad_out, cls, vpl, gc, packed, chunk_bound, num_sms, s);
    }
}

void launch_bwd_fixup(const Problem& P, const Plan& Q, const BwdOut& O, int64_t chunk_bound,
                      int num_sms, cudaStream_t s) {
    const FixupGrid g(chunk_bound, num_sms);
    auto* kernel = g.blocks > 2 * num_sms && g.blocks <= 4 * num_sms ? bwd_fixup_kernel<5> : bwd_fixup_kernel<3>;
    launch(kernel, g.blocks, kWarpThreads, 0, s, P, Q, O, g.span, g.group_blocks);
}

// ---------------------------------------------------------------- (7) sparse step

// The optimizer step from a row-sparse gradient already in memory (written by
// the backward). Every touched row is independent: a warp takes 32 rows, each
// lane fetches one row's id and gradient offset and finds its table by
// bisection over the per-table ranges (one round trip for all 32), then the
// warp steps the rows R at a time, issuing all their gradient, table and state
// loads before any store. Lane l owns columns 4l + 128m, m < M (the fused
// step's order, so both give the same sums of squares). Nothing is done when
// the gradient buffers were too small (the backward then wrote no rows).
#ifndef CB_APPLY_MIN_BLOCKS
#define CB_APPLY_MIN_BLOCKS 4  // resident blocks per SM for rows of up to 128 columns (wider: 2)
#endif
#ifndef CB_APPLY_ROWS_M1
#define CB_APPLY_ROWS_M1 2  // rows stepped at once for rows of up to 128 columns
#endif
constexpr int kApplyShTables = 1024;  // table offsets staged in shared memory up to this many tables

// One lane's row of a group of 32: where its stored row, gradient and state
// are, its (dim, dtype), and its previous Adagrad state.
struct ApplyRow {
    unsigned long long row;    // start of the stored row
    unsigned long long grad;   // start of its gradient
    unsigned long long state;  // its state word (Adagrad), or 0
    int shape;                 // dim << 2 | dtype (dim 0: nothing loaded or stored)
    float m0;
};

__device__ __forceinline__ ApplyRow apply_row_meta(const Problem& P, const BwdOut& O, const int64_t* toff,
                                                   int64_t u0, int64_t U, int64_t F, int lane, bool adagrad) {
    const int64_t u = min64(u0 + lane, U - 1);
    const int64_t id = __ldg(O.unique_ids + u);
    const int64_t goff = __ldg(O.grad_offsets + u);
    int lo = 0, hi = P.T;  // table_offsets[lo] <= u < table_offsets[lo + 1]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (toff[mid] <= u) lo = mid;
        else hi = mid;
    }
    const TableDev& td = P.tables[lo];
    const int64_t row = id - td.row_base;
    // A gradient this handle's backward wrote always passes; a row that does not
    // (buffers from elsewhere) is skipped and reported, never followed outside
    // a table, the gradient or the state.
    const bool ok = row >= 0 && row < td.rows && goff >= 0 && goff + td.dim <= F;
    if (!ok && u0 + lane < U) set_error(P.error, CB_ERR_INDEX_OOB);
    ApplyRow m;
    m.row = reinterpret_cast<unsigned long long>(row_ptr(td, ok ? row : 0));
    m.grad = reinterpret_cast<unsigned long long>(O.grads + (ok ? goff : 0));
    m.state = adagrad && ok ? reinterpret_cast<unsigned long long>(O.state[lo] + row) : 0ull;
    m.shape = ((ok ? td.dim : 0) << 2) | td.dtype;
    m.m0 = m.state ? *reinterpret_cast<const float*>(m.state) : 0.f;
    return m;
}

template <int M, int R>
__global__ void __launch_bounds__(kWarpThreads, M == 1 ? CB_APPLY_MIN_BLOCKS : 2)
    apply_sparse_kernel(const __grid_constant__ Problem P, const __grid_constant__ BwdOut O) {
    static_assert(32 % R == 0, "rows per step divide the warp's 32");
    begin_kernel();
    // The per-table first rows, for the bisection that finds each row's table.
    __shared__ int64_t sh_toff[kApplyShTables + 1];
    const bool staged = P.T <= kApplyShTables;
    if (staged)
        for (int t = threadIdx.x; t <= P.T; t += blockDim.x) sh_toff[t] = __ldg(O.table_offsets + t);
    __syncthreads();
    const int64_t* toff = staged ? sh_toff : O.table_offsets;
    const int lane = threadIdx.x & 31;
    const int64_t U = *O.num_unique;
    const int64_t F = *O.num_floats;
    if (U > O.cap_rows || F > O.cap_floats) return;
    const bool adagrad = O.apply == kApplyAdagrad;
    // (Loading the next group's ids, offsets and states while this group steps
    // was measured: no faster on cfg5.)
    for (int64_t u0 = warp_id_global() * 32; u0 < U; u0 += warps_in_grid() * 32) {
        const ApplyRow cur = apply_row_meta(P, O, toff, u0, U, F, lane, adagrad);
        const int rows_here = static_cast<int>(min64(32, U - u0));
        for (int r0 = 0; r0 < rows_here; r0 += R) {
            char* rp[R];
            int shape[R];
            float4 g[R][M];
            uint4 x[R][M];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                rp[i] = reinterpret_cast<char*>(__shfl_sync(kFull, cur.row, r0 + i));
                const float* gp = reinterpret_cast<const float*>(__shfl_sync(kFull, cur.grad, r0 + i));
                shape[i] = __shfl_sync(kFull, cur.shape, r0 + i);
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const int x0 = lane * 4 + 128 * m;
                    if (x0 < (shape[i] >> 2)) {
                        g[i][m] = *reinterpret_cast<const float4*>(gp + x0);
                        x[i][m] = load_cols(rp[i], shape[i] & 3, x0);
                    }
                }
            }
            float scale[R];
#pragma unroll
            for (int i = 0; i < R; ++i) scale[i] = O.lr;
            if (adagrad) {
                // The Adagrad scale with the arithmetic of adagrad_scale: the R
                // rows' butterflies interleaved, then lane r0 + i, which holds
                // row r0 + i's state, takes that row's update.
                float sq[R];
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    sq[i] = 0.f;
#pragma unroll
                    for (int m = 0; m < M; ++m)
                        if (lane * 4 + 128 * m < (shape[i] >> 2)) sq[i] += sq4(g[i][m]);
                }
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
                    for (int i = 0; i < R; ++i) sq[i] += __shfl_xor_sync(kFull, sq[i], off);
                float mine = 0.f;
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (lane == r0 + i) mine = sq[i];
                float my_scale = O.lr;
                if (lane >= r0 && lane < r0 + R && lane < rows_here && cur.state) {
                    const float m = cur.m0 + mine / static_cast<float>(cur.shape >> 2);
                    *reinterpret_cast<float*>(cur.state) = m;
                    my_scale = O.lr / (sqrtf(m) + O.eps);
                }
#pragma unroll
                for (int i = 0; i < R; ++i) scale[i] = __shfl_sync(kFull, my_scale, r0 + i);
            }
#pragma unroll
            for (int i = 0; i < R; ++i) {
                if (r0 + i >= rows_here) break;  // warp-uniform
                const int dim = shape[i] >> 2;
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const int x0 = lane * 4 + 128 * m;
                    if (x0 < dim) store_step(rp[i], shape[i] & 3, x0, x[i][m], g[i][m], scale[i]);
                }
            }
        }
    }
}

template <int M, int R>
void launch_apply_sparse_m(const Problem& P, const BwdOut& O, int num_sms, cudaStream_t s) {
    static const int cap = resident_blocks(apply_sparse_kernel<M, R>, kWarpThreads) * num_sms;
    launch(apply_sparse_kernel<M, R>, cap, kWarpThreads, 0, s, P, O);
}

void launch_apply_sparse(const Problem& P, const BwdOut& O, int num_sms, cudaStream_t s) {
    if (P.dmax <= 128) launch_apply_sparse_m<1, CB_APPLY_ROWS_M1>(P, O, num_sms, s);
    else if (P.dmax <= 256) launch_apply_sparse_m<2, 4>(P, O, num_sms, s);
    else launch_apply_sparse_m<4, 2>(P, O, num_sms, s);
}

}  // namespace cbtbe
