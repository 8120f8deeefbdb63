// tbe_plan.cuh -- the steps of the chunk plan (see tbe_plan.cu), shared by the plan
// kernel and by the small forward, which plans its own chunks.
#pragma once

#include "tbe_internal.cuh"
#include "tbe_launch.h"

namespace cbtbe {

// The tables' part of the plan, by one block: item ranges (pos), and the first
// chunk of every table in class order (ord) and, with tiles, the first sort tile in
// table order (tile_ord), each with the total at the end. Positions never decrease:
// a table whose first offset lies before an earlier table's (malformed, reported
// here) begins where that one does. So the tables' ranges do not overlap, and all
// of them together have no more chunks and tiles than n lookups can (room for the
// workspace, and in the backward a key in a table's range is one of its rows).
__device__ __forceinline__ void plan_tables(const Problem& P, const Plan& Q, int64_t tile_len, int64_t* pos, int64_t* ord,
                                            int64_t* tile_ord, int64_t* sh) {
    const int tid = threadIdx.x;
    auto start = [&](int t) {
        return min64(max64(load_index(P.offsets, static_cast<int64_t>(t) * P.B, P.is32), 0), P.n);
    };
    bool falls = false;
#pragma unroll 1
    for (int t = tid; t <= P.T; t += blockDim.x) {
        const int64_t x = start(t);
        pos[t] = x;
        if (t < P.T) falls = falls || start(t + 1) < x;
    }
    if (__syncthreads_or(falls)) {
        if (tid == 0) {
            set_error(P.error, CB_ERR_BAD_OFFSETS);
#pragma unroll 1
            for (int t = 1; t <= P.T; ++t) pos[t] = max64(pos[t], pos[t - 1]);
        }
        __syncthreads();
    }
    int64_t chunks = 0, tiles = 0;
#pragma unroll 1
    for (int i0 = 0; i0 < P.T; i0 += blockDim.x) {
        const int i = i0 + tid;
        int64_t cnt = 0, tcnt = 0;
        if (i < P.T) {
            const int t = Q.class_tables[i];
            const int64_t nt = max64(0, pos[t + 1] - pos[t]);
            cnt = max64(1, (nt + Q.chunk_len - 1) / Q.chunk_len);
            if (tile_len > 0) tcnt = max64(1, (max64(0, pos[i + 1] - pos[i]) + tile_len - 1) / tile_len);
        }
        int64_t total;
        const int64_t ex = block_excl_scan(cnt, sh, &total);
        if (i < P.T) ord[i] = chunks + ex;
        chunks += total;
        if (tile_len > 0) {
            const int64_t tex = block_excl_scan(tcnt, sh, &total);
            if (i < P.T) tile_ord[i] = tiles + tex;
            tiles += total;
        }
    }
    if (tid == 0) {
        ord[P.T] = chunks;
        if (tile_len > 0) tile_ord[P.T] = tiles;
    }
    __syncthreads();
}

// Largest i in [0, n) with base[i] <= j.
__device__ __forceinline__ int owner_of(const int64_t* base, int n, int64_t j) {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (base[mid] <= j) lo = mid; else hi = mid;
    }
    return lo;
}

// The first bag of table t starting at or after x0, and after x1 (lower bounds
// over the table's offsets, in [t*B, (t+1)*B + 1]), found together by W lanes that
// probe W points of both ranges at a time. A range narrows to the points around the
// first one that is not below x, whatever the later ones say, so that for decreasing
// offsets too the bag found starts at or after x and the one before it before x:
// a boundary that moves (see below) never leaves its table.
template <int W>
__device__ __forceinline__ void bag_lower_bounds(const Problem& P, int t, int64_t x0, int64_t x1, int lane, int64_t& r0,
                                                 int64_t& r1) {
    const uint32_t sub = lane & (W - 1);
    const int shift = lane & ~(W - 1);
    const int64_t blo = static_cast<int64_t>(t) * P.B;
    const int64_t x[2] = {x0, x1};
    uint32_t a[2] = {0u, 0u}, b[2] = {static_cast<uint32_t>(P.B) + 1u, static_cast<uint32_t>(P.B) + 1u};
    while (__any_sync(kFull, a[0] < b[0] || a[1] < b[1])) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const uint32_t R = b[s] - a[s];
            // R / (W + 1), or one less; up to W points left: each is probed
            const uint32_t step = max(1u, __umulhi(R, 0xffffffffu / (W + 1)));
            const uint32_t m = a[s] + (R <= W ? sub : (sub + 1) * step);
            const bool below = m < b[s] && load_index(P.offsets, blo + m, P.is32) < x[s];
            const uint32_t all = (__ballot_sync(kFull, below) >> shift) & (kFull >> (32 - W));
            const uint32_t cnt = __clz(__brev(~all));  // points below x before the first that is not
            if (R <= W) {
                a[s] += cnt;
                b[s] = a[s];
            } else {
                if (cnt < W) b[s] = a[s] + (cnt + 1) * step;
                if (cnt > 0) a[s] += cnt * step + 1;
            }
        }
    }
    r0 = blo + a[0];
    r1 = blo + a[1];
}

// A chunk boundary at x moves to the end of the bag it falls in, unless that bag
// is longer than the cap: short bags are then never split, and only heavy ones
// leave pieces for the fix-up. Monotone in x, so consecutive chunks stay
// contiguous (a chunk may come out empty). `a` is the first bag starting at or
// after x; it also gives the first bag touching the moved boundary (the one
// starting exactly there if any, the first of equal starts; else the one
// containing it).
struct Boundary {
    int64_t k;      // position
    int64_t first;  // first bag of a chunk starting at k
};

__device__ __forceinline__ Boundary boundary(const Problem& P, const Plan& Q, int t, int64_t a, int64_t x, int64_t p0,
                                             int64_t p1) {
    const bool may_move = Q.snap_cap > 0 && x > p0 && x < p1;
    const int64_t blo = static_cast<int64_t>(t) * P.B, bhi = blo + P.B;
    const int64_t e = a <= bhi ? load_index(P.offsets, a, P.is32) : -1;
    const int64_t s0 = a > blo ? load_index(P.offsets, a - 1, P.is32) : 0;
    int64_t k = x;
    if (may_move && a <= bhi && e != x && a != blo && e - s0 <= Q.snap_cap && e <= p1) k = e;
    // Moved to e (= offsets[a], with offsets[a - 1] < x < e): bag a starts
    // there. Else the bag starting exactly at x, or the one containing it.
    const int64_t first = (a <= bhi && e == k) ? a : a - 1;
    return {k, min64(max64(first, blo), bhi)};
}

// Chunk j of the plan, by W lanes (all lanes of the warp call this; each group of W
// with its own j).
template <int W>
__device__ __forceinline__ Chunk plan_chunk(const Problem& P, const Plan& Q, const int64_t* pos, const int64_t* ord,
                                            int64_t j, int lane) {
    const int64_t C = Q.chunk_len;
    const int i = owner_of(ord, P.T, j);
    const int t = Q.class_tables[i];
    const int64_t local = j - ord[i];
    const int64_t p0 = pos[t];
    const int64_t p1 = max64(p0, pos[t + 1]);
    const int64_t nch = max64(1, (p1 - p0 + C - 1) / C);
    const bool last = local >= nch - 1;
    const int64_t x0 = min64(p0 + local * C, p1);
    const int64_t x1 = last ? p1 : min64(p0 + (local + 1) * C, p1);
    int64_t a0, a1;
    bag_lower_bounds<W>(P, t, x0, x1, lane, a0, a1);
    const Boundary b0 = boundary(P, Q, t, a0, x0, p0, p1);
    const int64_t k1 = last ? x1 : boundary(P, Q, t, a1, x1, p0, p1).k;
    Chunk ch;
    ch.k0 = b0.k;
    ch.first = b0.first;
    ch.table = t;
    ch.len = static_cast<uint32_t>(max64(0, k1 - b0.k)) | (last ? 0x80000000u : 0u);
    return ch;
}

}  // namespace cbtbe
