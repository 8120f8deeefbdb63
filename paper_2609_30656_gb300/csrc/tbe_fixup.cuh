// tbe_fixup.cuh -- the fix-up of segments (bags, or runs of equal sorted row ids)
// that the walkers split over chunks, shared by the forward and the backward.
//
// A segment that straddles chunks left its tail piece in the chunk j where it
// begins and head pieces in the m chunks after it. The pieces are added in a fixed
// order into fp64, so the result is deterministic. Up to kHeavyPieces pieces: one
// warp, lanes owning columns. More (a bag or a hot row of tens of thousands of
// lookups, cut every 32 to 512 of them): the chunks are cut into groups of
// kPieceGroup, a block adds the pieces of a heavy segment in one group, and the
// last block to arrive at the segment adds up its groups. No block waits for
// another. Bound by latency for a few groups, else by L2. Forward of one table with
// 80 % of its lookups in one bag (fp32, 64 columns), one warp per bag against this:
// 20 K lookups 151 -> 40 us, 300 K 1427 -> 56, 1 M 2362 -> 74, 40 M 12900 -> 566; with
// fp16 rows of 128, 1 M: 4630 -> 87.
#pragma once

#include "tbe_internal.cuh"

namespace cbtbe {

constexpr int64_t kHeavyPieces = 32;
// Chunks per group: about the square root of the pieces of the longest segments, so
// that a group and the sum over the groups take about as long.
constexpr int64_t kPieceGroup = 128;

// ---------------------------------------------------------------- one warp

constexpr int kInnerPieces = 16;

// acc (fp64, four columns from x0) += pieces i0, i0 + step, ... below m, each at
// head + piece * dmax. The pieces are summed in fp32 in groups of kInnerPieces,
// each group folded into acc: GB300's fp64 adds are scarce (one per piece and
// column made a heavy-run combine fp64-bound), and an fp32 sum of at most 16
// pieces rounds within 16u of their absolute sum. Four loads in flight.
__device__ __forceinline__ void add_pieces(const float* head, int64_t i0, int64_t step, int64_t m, int dmax,
                                           int x0, double (&acc)[4]) {
    for (int64_t g = i0; g < m; g += kInnerPieces * step) {
        const int64_t gend = min64(m, g + kInnerPieces * step);
        float in[4] = {0.f, 0.f, 0.f, 0.f};
        int64_t i = g;
        for (; i + 3 * step < gend; i += 4 * step) {
            float4 h[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) h[c] = *reinterpret_cast<const float4*>(head + (i + c * step) * dmax + x0);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                in[0] += h[c].x;
                in[1] += h[c].y;
                in[2] += h[c].z;
                in[3] += h[c].w;
            }
        }
        for (; i < gend; i += step) {
            const float4 h = *reinterpret_cast<const float4*>(head + i * dmax + x0);
            in[0] += h.x;
            in[1] += h.y;
            in[2] += h.z;
            in[3] += h.w;
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[x] += in[x];
    }
}

// ---------------------------------------------------------------- one block

// The block as R rows of nv threads: thread (r, c) adds rows r, r + R, ... of four
// columns from 4c.
struct BlockRows {
    int nv, R, r, c;
    bool on;
    __device__ __forceinline__ explicit BlockRows(int dim) {
        nv = dim / 4;
        R = kWarpThreads / nv;
        r = threadIdx.x / nv;
        c = threadIdx.x - r * nv;
        on = r < R;
    }
};

constexpr int kRowsInFlight = 8;

// acc += this thread's share of fp32 rows 0 .. n - 1, `stride` floats apart. NARROW:
// eight rows in fp32 first (3 levels of adds, 3u of their absolute sum), as the
// backward's pieces always were in groups of 16; else each row into fp64.
template <bool NARROW>
__device__ __forceinline__ void add_rows(const BlockRows& b, const float* rows, int64_t n, int64_t stride,
                                         double (&acc)[4]) {
    if (!b.on) return;
    for (int64_t k = b.r; k < n; k += kRowsInFlight * b.R) {
        float4 h[kRowsInFlight];
#pragma unroll
        for (int u = 0; u < kRowsInFlight; ++u)
            h[u] = k + u * b.R < n ? __ldcg(reinterpret_cast<const float4*>(rows + (k + u * b.R) * stride) + b.c)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
        if (NARROW) {
#pragma unroll
            for (int w = 1; w < kRowsInFlight; w *= 2)
#pragma unroll
                for (int u = 0; u < kRowsInFlight; u += 2 * w) {
                    h[u].x += h[u + w].x;
                    h[u].y += h[u + w].y;
                    h[u].z += h[u + w].z;
                    h[u].w += h[u + w].w;
                }
        }
#pragma unroll
        for (int u = 0; u < (NARROW ? 1 : kRowsInFlight); ++u) {
            acc[0] += h[u].x;
            acc[1] += h[u].y;
            acc[2] += h[u].z;
            acc[3] += h[u].w;
        }
    }
}

// The same for fp64 rows 0 .. n - 1, `stride` doubles apart.
__device__ __forceinline__ void add_rows64(const BlockRows& b, const double* rows, int64_t n, int64_t stride,
                                           double (&acc)[4]) {
    if (!b.on) return;
    for (int64_t k = b.r; k < n; k += 4 * b.R) {
        double2 h[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int x = 0; x < 2; ++x)
                h[u][x] = k + u * b.R < n
                              ? __ldcg(reinterpret_cast<const double2*>(rows + (k + u * b.R) * stride) + 2 * b.c + x)
                              : make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            acc[0] += h[u][0].x;
            acc[1] += h[u][0].y;
            acc[2] += h[u][1].x;
            acc[3] += h[u][1].y;
        }
    }
}

// The R shares of every column, added by halves; the sum is in the threads of row 0.
__device__ __forceinline__ void add_shares(const BlockRows& b, double (*sh)[4], double (&acc)[4]) {
    int half = 1;
    while (half < b.R) half *= 2;
    const int i = threadIdx.x;
    if (b.on)
#pragma unroll
        for (int x = 0; x < 4; ++x) sh[i][x] = acc[x];
    __syncthreads();
    for (half /= 2; half >= 1; half /= 2) {
        if (b.r < half && b.r + half < b.R)
#pragma unroll
            for (int x = 0; x < 4; ++x) sh[i][x] += sh[i + half * b.nv][x];
        __syncthreads();
    }
    if (b.r == 0)
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[x] = sh[i][x];
}

// ---------------------------------------------------------------- the fix-up

// Split states what is split: Split::kNarrow; pieces(j, seg, lane), the chunks after
// chunk j that hold the rest of the segment begun there; origin(i, lane, j, m), the
// chunk where the segment that chunk i begins inside was begun, and its pieces
// (false: it has none to add); store(j, seg, t, x0, acc), four columns of a
// segment's sum; stored(j, t, lane), by one warp, after all of them. All but store
// are called by whole warps.
template <class Split>
__device__ __forceinline__ void fix_split(const Problem& P, const Plan& Q, const Split& split, int64_t total, int span) {
    constexpr int kWarps = kWarpThreads / 32;
    // Heavy segments of a round: they begin more than kHeavyPieces chunks apart, in the
    // at most kWarps * 32 chunks that the block scans.
    constexpr int kMaxHeavy = kWarps * 32 / static_cast<int>(kHeavyPieces) + 2;
    __shared__ double shares[kWarpThreads][4];
    __shared__ int4 heavy[kMaxHeavy];
    __shared__ int heavy_count;
    __shared__ int64_t sh_j, sh_m;
    __shared__ bool sh_last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;

    // One block's arrival at the heavy segment begun in chunk j, m pieces after it; the
    // last of its groups' blocks and of the block that found it adds it up.
    auto arrive = [&](int64_t j, int64_t m) {
        const int64_t g0 = j / kPieceGroup, groups = (j + m) / kPieceGroup - g0;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned long long before = atomicAdd(Q.split + j, kSplitArrival);
            sh_last = static_cast<int64_t>(before / kSplitArrival) == groups;
            __threadfence();
        }
        __syncthreads();
        if (!sh_last) return;
        const int t = Q.chunks[j].table;
        const uint32_t seg = static_cast<uint32_t>(Q.split[j]);
        const BlockRows b(P.tables[t].dim);
        const float* head = Q.carry_head;
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        // The pieces up to the first group's start, the whole groups' sums, and a last
        // group of one piece, which is its own sum.
        add_rows<Split::kNarrow>(b, head + (j + 1) * P.dmax, min64(m, (g0 + 1) * kPieceGroup - (j + 1)), P.dmax, acc);
        const int64_t first = (g0 + 1) * kPieceGroup, single = groups > 0 && (j + m) % kPieceGroup == 0 ? 1 : 0;
        add_rows64(b, reinterpret_cast<const double*>(head + first * P.dmax), groups - single, kPieceGroup / 2 * P.dmax,
                   acc);
        add_rows<false>(b, head + (j + m) * P.dmax, single, P.dmax, acc);
        add_shares(b, shares, acc);
        if (b.r == 0) {
            const float4 a = *reinterpret_cast<const float4*>(Q.carry_tail + j * P.dmax + 4 * b.c);
            acc[0] += a.x;
            acc[1] += a.y;
            acc[2] += a.z;
            acc[3] += a.w;
            split.store(j, seg, t, 4 * b.c, acc);
        }
        __syncthreads();
        if (w == 0) split.stored(j, t, lane);
    };

    const int64_t round = static_cast<int64_t>(gridDim.x) * kWarps * span;
    for (int64_t base0 = static_cast<int64_t>(blockIdx.x) * kWarps * span; base0 < total; base0 += round) {
        if (threadIdx.x == 0) heavy_count = 0;
        __syncthreads();
        const int64_t base = base0 + static_cast<int64_t>(w) * span;
        const unsigned long long mine = lane < span && base + lane < total ? Q.split[base + lane] : 0;
        for (uint32_t mask = __ballot_sync(kFull, (mine & kSplitBegins) != 0); mask; mask &= mask - 1) {
            const int b = __ffs(mask) - 1;
            const int64_t j = base + b;
            const uint32_t seg = __shfl_sync(kFull, static_cast<uint32_t>(mine), b);
            const int64_t m = split.pieces(j, seg, lane);
            const int t = Q.chunks[j].table;
            if (m > kHeavyPieces) {
                if (lane == 0) {
                    const int slot = atomicAdd(&heavy_count, 1);
                    if (slot < kMaxHeavy) heavy[slot] = make_int4(static_cast<int>(j), static_cast<int>(m), 0, 0);
                }
                continue;
            }
            const int dim = P.tables[t].dim;
            for (int x0 = lane * 4; x0 < dim; x0 += 128) {
                const float4 a = *reinterpret_cast<const float4*>(Q.carry_tail + j * P.dmax + x0);
                double acc[4] = {a.x, a.y, a.z, a.w};
                add_pieces(Q.carry_head + (j + 1) * P.dmax, 0, 1, m, P.dmax, x0, acc);
                split.store(j, seg, t, x0, acc);
            }
            split.stored(j, t, lane);
        }
        __syncthreads();
        const int count = min(heavy_count, kMaxHeavy);
        for (int h = 0; h < count; ++h) arrive(heavy[h].x, heavy[h].y);
        __syncthreads();
    }

    // Groups that begin inside a segment (the first chunk of all begins none).
    for (int64_t g = 1 + blockIdx.x; g * kPieceGroup < total; g += gridDim.x) {
        const int64_t i = g * kPieceGroup;
        if (!(Q.split[i] & kSplitGoesOn)) continue;  // block-uniform
        if (w == 0) {
            int64_t j = 0, m = 0;
            if (!split.origin(i, lane, j, m)) m = 0;
            if (lane == 0) {
                sh_j = j;
                sh_m = m;
            }
        }
        __syncthreads();
        const int64_t j = sh_j, m = sh_m;
        __syncthreads();
        if (m <= kHeavyPieces) continue;
        const int64_t n = min64(kPieceGroup, j + m + 1 - i);
        if (n > 1) {
            const BlockRows b(P.tables[Q.chunks[i].table].dim);
            float* rows = Q.carry_head + i * P.dmax;
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            add_rows<Split::kNarrow>(b, rows, n, P.dmax, acc);
            add_shares(b, shares, acc);
            // in place of the first two pieces
            if (b.r == 0)
#pragma unroll
                for (int x = 0; x < 2; ++x)
                    *(reinterpret_cast<double2*>(rows) + 2 * b.c + x) = make_double2(acc[2 * x], acc[2 * x + 1]);
        }
        arrive(j, m);
    }
}

}  // namespace cbtbe
