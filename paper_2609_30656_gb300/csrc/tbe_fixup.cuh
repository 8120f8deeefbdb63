// tbe_fixup.cuh -- the fix-up of segments (bags, or runs of equal sorted row ids)
// that the walkers split over chunks, shared by the forward and the backward.
//
// A segment that straddles chunks left its tail piece in the chunk j where it
// begins and head pieces in the m chunks after it. The pieces are added in a fixed
// order into fp64, so the result is deterministic. Up to kHeavyPieces: by the warp
// that finds the segment. Up to kGroupedPieces: by its block. More (a bag or a hot row
// of tens of thousands of lookups, cut every 32 to 512 of them): the chunks are cut
// into groups of kPieceGroup, a block adds the segment's pieces in a group, and the
// last block to arrive at the segment adds up its groups. No block waits for another.
//
// Bound by latency: a chain of six or seven dependent loads where nothing is heavy. Its
// code is kept small, with one copy of each loop: a call's kernels are run in turn, and
// what this one brings into the instruction cache the next call's first kernels have to
// fetch again (with the sums written out twice, 95 to 110 KB, the plan after it took 10.3
// us instead of 6.4).
//
// Against one warp per bag (forward), and a block per run that looked for its pieces 32
// at a time (backward), us. One table, 80 % of the lookups in one bag, fp32 rows of 64:
// 20 K lookups 151 -> 38, 300 K 1427 -> 56, 1 M 2362 -> 75, 40 M 12900 -> 582; fp16 rows
// of 128, 1 M: 4630 -> 89. Every lookup of one row, backward, fp32 columns of 64: 300 K
// 290 -> 115, 1 M 482 -> 177, 40 M 3043 -> 1421; of 128, 1 M: 503 -> 195.
#pragma once

#include "tbe_internal.cuh"
#include "tbe_launch.h"

namespace cbtbe {

constexpr int kHeavyPieces = 32;
// About the square root of the pieces of the longest segments, so that a group and the
// sum over the groups take about as long.
constexpr int kPieceGroup = 128;
constexpr int kGroupedPieces = 256;
constexpr int kRowsInFlight = 8;

// One warp or the warps of a block over rows of `dim` columns: V lanes per row (a power
// of two, four columns each; a row of more than 128 columns takes several passes), G rows
// at a time. Lane (g, c) takes rows g, g + G, ...
struct RowLanes {
    int nv, V, G, g, c;
    __device__ __forceinline__ RowLanes(int dim, bool block) {
        const int lane = threadIdx.x & 31;
        nv = dim / 4;
        V = nv >= 32 ? 32 : 1 << (32 - __clz(nv - 1));
        G = (block ? kWarpThreads : 32) / V;
        g = (block ? threadIdx.x : lane) / V;
        c = lane & (V - 1);
    }
    // acc += this lane's share of rows 0 .. n - 1 of fp32, `stride` floats apart, at
    // columns 4v .. 4v + 3. Narrow: eight rows in fp32 first, by halves (3u of their
    // absolute sum; GB300's fp64 adds are scarce: a backward of 330 K lookups 106 us so, 119
    // with every row into fp64), else each row into fp64.
    __device__ __forceinline__ void add(bool narrow, const float* rows, int n, int64_t stride, int v, double (&acc)[4]) const {
        rows += g * stride + 4 * v;
        stride *= G;
#pragma unroll 1
        for (int k = g; k < n; k += kRowsInFlight * G, rows += kRowsInFlight * stride) {
            float4 h[kRowsInFlight];
#pragma unroll
            for (int u = 0; u < kRowsInFlight; ++u)
                h[u] = k + u * G < n ? __ldcg(reinterpret_cast<const float4*>(rows + u * stride))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
            if (narrow) {
#pragma unroll
                for (int w = 1; w < kRowsInFlight; w *= 2)
#pragma unroll
                    for (int u = 0; u < kRowsInFlight; u += 2 * w) {
                        h[u].x += h[u + w].x;
                        h[u].y += h[u + w].y;
                        h[u].z += h[u + w].z;
                        h[u].w += h[u + w].w;
                    }
            } else {
#pragma unroll
                for (int u = 1; u < kRowsInFlight; ++u) {
                    acc[0] += h[u].x;
                    acc[1] += h[u].y;
                    acc[2] += h[u].z;
                    acc[3] += h[u].w;
                }
            }
            acc[0] += h[0].x;
            acc[1] += h[0].y;
            acc[2] += h[0].z;
            acc[3] += h[0].w;
        }
    }
    // The same for n fp64 rows, each the low words in one row of floats and the high
    // words in the next, `next` further; `stride` floats from one to the next.
    __device__ __forceinline__ void add64(const float* rows, int n, int64_t stride, int64_t next, int v,
                                          double (&acc)[4]) const {
        rows += g * stride + 4 * v;
        stride *= G;
        constexpr int kFlight = kRowsInFlight / 2;
#pragma unroll 1
        for (int k = g; k < n; k += kFlight * G, rows += kFlight * stride) {
            int4 lo[kFlight], hi[kFlight];
#pragma unroll
            for (int u = 0; u < kFlight; ++u) {
                const float* p = rows + u * stride;
                const bool in = k + u * G < n;
                lo[u] = in ? __ldcg(reinterpret_cast<const int4*>(p)) : make_int4(0, 0, 0, 0);
                hi[u] = in ? __ldcg(reinterpret_cast<const int4*>(p + next)) : make_int4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < kFlight; ++u) {
                acc[0] += __hiloint2double(hi[u].x, lo[u].x);
                acc[1] += __hiloint2double(hi[u].y, lo[u].y);
                acc[2] += __hiloint2double(hi[u].z, lo[u].z);
                acc[3] += __hiloint2double(hi[u].w, lo[u].w);
            }
        }
    }
    static __device__ __forceinline__ void put64(float* row, int64_t next, int v, const double (&acc)[4]) {
        reinterpret_cast<int4*>(row)[v] = make_int4(__double2loint(acc[0]), __double2loint(acc[1]),
                                                    __double2loint(acc[2]), __double2loint(acc[3]));
        reinterpret_cast<int4*>(row + next)[v] = make_int4(__double2hiint(acc[0]), __double2hiint(acc[1]),
                                                           __double2hiint(acc[2]), __double2hiint(acc[3]));
    }
    // The shares of a warp's lane groups, added up: every lane ends with its columns' sums.
    __device__ __forceinline__ void fold(double (&acc)[4]) const {
#pragma unroll 1
        for (int off = V; off < 32; off *= 2)
#pragma unroll
            for (int x = 0; x < 4; ++x) acc[x] += __shfl_xor_sync(kFull, acc[x], off);
    }
};

// Split states what is split: Split::kNarrow, whether heavy segments are added narrow too
// (the others are); pieces(j, seg, lane), the chunks after
// chunk j that hold the rest of the segment begun there; origin(i, lane, j, m), the
// chunk where the segment that chunk i begins inside was begun, and its pieces
// (false: it has none to add); dest(j, seg, t), where its sum goes, loaded ahead of the
// pieces; store(dest, x0, acc), four columns of it; stored(j, t, lane), after all of them.
// All but store are called by whole warps.
//
// The warps of the first group_blocks blocks look for groups of chunks that begin inside
// a heavy segment, a group each, and leave them to their block (the first chunk of all
// begins inside none); those of the others for segments begun in their chunks, span
// chunks at a time, and leave the heavy ones to their block.
template <class Split>
__device__ __forceinline__ void fix_split(const Problem& P, const Plan& Q, const Split& split, int total, int span,
                                          int group_blocks) {
    constexpr int kWarps = kWarpThreads / 32;
    // Heavy segments of a round: they begin more than kHeavyPieces chunks apart, in the
    // at most kWarps * 32 chunks that the block scans.
    constexpr int kMaxHeavy = kWarps * 32 / kHeavyPieces + 2;
    __shared__ double shares[4][kWarps][32];
    __shared__ int4 heavy[kMaxHeavy];  // first chunk, pieces, table, the group's chunk or the segment
    __shared__ int heavy_count;
    __shared__ bool sh_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool scans = static_cast<int>(blockIdx.x) >= group_blocks;
    const int64_t dmax = P.dmax;
    // Scanning, a block takes the chunks of its warps side by side; groups that follow each
    // other, most likely of one segment, go to different blocks.
    const int blocks = scans ? gridDim.x - group_blocks : group_blocks, me = scans ? blockIdx.x - group_blocks : blockIdx.x;
    const int64_t block_step = scans ? kWarps * span : kPieceGroup, warp_step = scans ? span : blocks * kPieceGroup;
    const int64_t step = scans ? blocks * block_step : kWarps * warp_step;
#pragma unroll 1
    for (int64_t at = (scans ? me : me + 1) * block_step; at < total; at += step) {
        const int64_t base = at + warp * warp_step;
        const unsigned long long mine = lane < (scans ? span : 1) && base + lane < total ? Q.split[base + lane] : 0;
        // Each warp its own light segments, then the block the heavy ones one by one.
        uint32_t found = __ballot_sync(kFull, (mine & (scans ? kSplitBegins : kSplitGoesOn)) != 0);
        if (threadIdx.x == 0) heavy_count = 0;
        if (!__syncthreads_or(found != 0)) continue;
        bool block = false;
        int next = 0;
#pragma unroll 1
        for (;;) {
            int j, m, t, dim, group = 0;
            uint32_t seg = 0;
            typename Split::Dest dest;
            if (!block) {
                if (found == 0) {
                    __syncthreads();
                    block = true;
                    continue;
                }
                const int b = __ffs(found) - 1;
                found &= found - 1;
                j = static_cast<int>(base) + b;
                t = Q.chunks[j].table;
                seg = __shfl_sync(kFull, static_cast<uint32_t>(mine), b);
                // (loads that the sum needs, ahead of those that find its pieces)
                dim = P.tables[t].dim;
                if (scans) dest = split.dest(j, seg, t);
                if (scans) m = split.pieces(j, seg, lane);
                else if (!split.origin(j, lane, j, m) || m <= kGroupedPieces) continue;
                if (m > kHeavyPieces) {
                    if (lane == 0) {
                        const int slot = atomicAdd(&heavy_count, 1);
                        if (slot < kMaxHeavy)
                            heavy[slot] = make_int4(j, m, t, scans ? static_cast<int>(seg) : static_cast<int>(base));
                    }
                    continue;
                }
            } else {
                if (next >= min(heavy_count, kMaxHeavy)) break;
                const int4 h = heavy[next++];
                j = h.x;
                m = h.y;
                t = h.z;
                group = h.w;
                seg = static_cast<uint32_t>(h.w);
                dim = P.tables[t].dim;
                if (scans) dest = split.dest(j, seg, t);
            }
            const RowLanes w(dim, block);
            const bool grouped = m > kGroupedPieces;
            const int first = (j / kPieceGroup + 1) * kPieceGroup;               // of the groups after j's
            const int groups = grouped ? (j + m - first) / kPieceGroup + 1 : 0;
            const int single = grouped && (j + m) % kPieceGroup == 0 ? 1 : 0;    // a last group of one piece
            // A group's share of its segment's pieces first: left in fp64 in place of the
            // first two (a single piece is its own sum). Then the arrival at the segment, and
            // for the last to arrive (or the only one) the sum: the tail, the pieces up to the
            // first group (or all), and the groups.
            bool share = !scans;
#pragma unroll 1
            for (;;) {
                const int row = share ? group : j + 1;
                const int n = share ? min(kPieceGroup, j + m + 1 - group) : (grouped ? first - row : m);
                if (!share && grouped) {
                    __threadfence();
                    __syncthreads();
                    if (threadIdx.x == 0) {
                        sh_last = static_cast<int>(atomicAdd(Q.split + j, kSplitArrival) / kSplitArrival) == groups;
                        __threadfence();
                    }
                    __syncthreads();
                    if (!sh_last) break;
                    if (!scans) {
                        seg = static_cast<uint32_t>(Q.split[j]);
                        dest = split.dest(j, seg, t);
                    }
                }
                float* rows = Q.carry_head + row * dmax;
#pragma unroll 1
                for (int v = w.c; v < w.nv + w.c && !(share && n == 1); v += 32) {  // as often in every lane
                    double acc[4] = {0.0, 0.0, 0.0, 0.0};
                    if (v < w.nv) {
                        if (!share && w.g == 0) {
                            const float4 a = *(reinterpret_cast<const float4*>(Q.carry_tail + j * dmax) + v);
                            acc[0] = a.x;
                            acc[1] = a.y;
                            acc[2] = a.z;
                            acc[3] = a.w;
                        }
                        w.add(Split::kNarrow || !block, rows, n, dmax, v, acc);
                        if (!share && grouped) {
                            w.add64(Q.carry_head + first * dmax, groups - single, kPieceGroup * dmax, dmax, v, acc);
                            if (single && w.g == 0) {
                                const float4 a = __ldcg(reinterpret_cast<const float4*>(Q.carry_head + (j + m) * dmax) + v);
                                acc[0] += a.x;
                                acc[1] += a.y;
                                acc[2] += a.z;
                                acc[3] += a.w;
                            }
                        }
                    }
                    w.fold(acc);
                    if (block) {  // the warps' sums meet in the first warp, in their order
#pragma unroll
                        for (int x = 0; x < 4; ++x) shares[x][warp][lane] = acc[x];
                        __syncthreads();
#pragma unroll 1
                        for (int q = 1; q < kWarps && warp == 0; ++q)
#pragma unroll
                            for (int x = 0; x < 4; ++x) acc[x] += shares[x][q][lane];
                        __syncthreads();
                    }
                    if (w.g == 0 && v < w.nv) {
                        if (share) RowLanes::put64(rows, dmax, v, acc);
                        else split.store(dest, 4 * v, acc);
                    }
                }
                if (!share) {
                    __syncwarp();
                    if (!block || warp == 0) split.stored(j, t, lane);
                    break;
                }
                share = false;
            }
        }
        __syncthreads();
    }
}

// The grid: a block for every group but the first, up to two per SM (then a warp for every
// group), and the scanning blocks.
struct FixupGrid {
    int span, group_blocks, blocks;
    FixupGrid(int64_t chunk_bound, int num_sms) {
        span = fixup_span(chunk_bound, num_sms);
        group_blocks = static_cast<int>(min64((chunk_bound - 1) / kPieceGroup, static_cast<int64_t>(num_sms) * 2));
        blocks = group_blocks + fixup_grid(chunk_bound, span, num_sms);
    }
};

}  // namespace cbtbe
