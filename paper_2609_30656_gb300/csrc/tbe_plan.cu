// tbe_plan.cu -- offsets validation and the chunk plan shared by the forward
// gather-pool and the backward key generation / segmented reduce.
//
// A table's items (lookup positions, key-major so each table's lookups are
// contiguous) are cut into chunks of at most chunk_len positions; a table with
// no lookups still gets one (empty) chunk so that its empty bags are written.
// Chunks are numbered class by class (tables grouped by kernel instantiation),
// table by table within a class. The backward's sort tiles are placed with them.
#include "tbe_internal.cuh"
#include "tbe_launch.h"

namespace cbtbe {

__global__ void validate_offsets_kernel(Problem P) {
    begin_kernel();
    const int64_t nb = static_cast<int64_t>(P.T) * P.B;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; k <= nb;
         k += stride) {
        const int64_t o = load_index(P.offsets, k, P.is32);
        bool bad = o < 0 || o > P.n;
        if (k == 0 && o != 0) bad = true;
        if (k == nb && o != P.n) bad = true;
        if (k < nb && load_index(P.offsets, k + 1, P.is32) < o) bad = true;
        if (bad) set_error(P.error, CB_ERR_BAD_OFFSETS);
    }
}

// The tables' part of the plan, by one block: item ranges (pos), and the first
// chunk of every table in class order (ord) and, with tiles, the first sort tile in
// table order (tile_ord), each with the total at the end.
__device__ __forceinline__ void plan_tables(const Problem& P, const Plan& Q, int64_t tile_len, int64_t* pos, int64_t* ord,
                                            int64_t* tile_ord, int64_t* sh) {
    const int tid = threadIdx.x;
    for (int t = tid; t <= P.T; t += blockDim.x) {
        const int64_t x = load_index(P.offsets, static_cast<int64_t>(t) * P.B, P.is32);
        pos[t] = min64(max64(x, 0), P.n);
    }
    __syncthreads();
    int64_t chunks = 0, tiles = 0;
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

// More tables than a block's shared memory holds: the tables' part runs first, as
// a kernel of its own, into global memory.
constexpr int kPlanTables = 1024;

__global__ void __launch_bounds__(1024) plan_tables_kernel(const __grid_constant__ Problem P,
                                                           const __grid_constant__ Plan Q,
                                                           const __grid_constant__ TilePlan S) {
    __shared__ int64_t sh[33];
    begin_kernel();
    plan_tables(P, Q, S.tile_len, Q.table_pos, Q.ord_chunk_base, S.table_first_tile, sh);
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
// probe W points of both ranges at a time.
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
            const uint32_t cnt = __popc((__ballot_sync(kFull, below) >> shift) & ((1u << W) - 1u));
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

// The whole plan in one launch: every block scans the tables for itself in shared
// memory (up to kPlanTables of them), then W lanes place each chunk and one lane each
// sort tile. It also clears what later kernels count in: the walkers' chunk
// counters and S.zero. Latency-bound searches, 6 blocks of 256 threads per SM.
// W = 8 (6 dependent loads for 65536 bags, where a bisection takes 17) while the
// chunks' lanes are all resident, else 1.
// (A one-block kernel for the tables, then a bisection per thread for the chunks,
// and both again for the tiles: forward prep of 8 tables of 41 K lookups in 2048
// bags 19.4 us, now 16.6; of 20 tables of 80 K 20.8, now 14.5; of 20 tables of 2 M
// 28, now 26; with W = 8 there, 51. The sort 8 us less without its own plan.)
template <int W>
__global__ void __launch_bounds__(256, 6) plan_kernel(const __grid_constant__ Problem P, const __grid_constant__ Plan Q,
                                                      const __grid_constant__ TilePlan S) {
    __shared__ int64_t sh_pos[kPlanTables + 1], sh_ord[kPlanTables + 1], sh_tile[kPlanTables + 1];
    __shared__ int64_t sh[33];
    begin_kernel();
    const bool own = P.T <= kPlanTables;
    const int64_t* pos = own ? sh_pos : Q.table_pos;
    const int64_t* ord = own ? sh_ord : Q.ord_chunk_base;
    const int64_t* tile_ord = own ? sh_tile : S.table_first_tile;
    if (own) plan_tables(P, Q, S.tile_len, sh_pos, sh_ord, sh_tile, sh);
    const int tid = threadIdx.x;
    const int64_t total = min64(ord[P.T], Q.max_chunks);
    if (blockIdx.x == 0) {
        for (int i = tid; i <= P.T; i += blockDim.x) {
            if (own) {
                Q.table_pos[i] = pos[i];
                if (S.tile_len > 0) S.table_first_tile[i] = tile_ord[i];
            }
            if (i < P.T) Q.table_chunk[Q.class_tables[i]] = ord[i];
        }
        for (int c = tid; c <= Q.num_classes; c += blockDim.x) {
            Q.class_chunk_base[c] = min64(ord[Q.class_table_start[c]], Q.max_chunks);
            Q.chunk_next[c] = 0;
        }
        if (tid == 0) {
            if (ord[P.T] > Q.max_chunks) set_error(P.error, CB_ERR_BAD_OFFSETS);
            if (S.tile_len > 0) *S.num_tiles = min64(tile_ord[P.T], S.max_tiles);
        }
    }
    const int64_t first = static_cast<int64_t>(blockIdx.x) * blockDim.x + tid;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t C = Q.chunk_len;
    const int lane = tid & 31;
    for (int64_t w = first; (w - lane) / W < total; w += stride) {  // warp-uniform
        const int64_t j = min64(w / W, total - 1);
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
        if ((lane & (W - 1)) != 0 || w / W >= total) continue;
        const Boundary b0 = boundary(P, Q, t, a0, x0, p0, p1);
        const int64_t k1 = last ? x1 : boundary(P, Q, t, a1, x1, p0, p1).k;
        Chunk ch;
        ch.k0 = b0.k;
        ch.first = b0.first;
        ch.table = t;
        ch.len = static_cast<uint32_t>(max64(0, k1 - b0.k)) | (last ? 0x80000000u : 0u);
        Q.chunks[j] = ch;
    }
    if (S.tile_len <= 0) return;
    const int64_t tiles = min64(tile_ord[P.T], S.max_tiles);
    for (int64_t j = first; j < tiles; j += stride) {
        const int t = owner_of(tile_ord, P.T, j);
        const int64_t p0 = pos[t], p1 = max64(p0, pos[t + 1]);
        Chunk ch;
        ch.k0 = min64(p0 + (j - tile_ord[t]) * S.tile_len, p1);
        ch.first = 0;
        ch.table = t;
        ch.len = static_cast<uint32_t>(min64(S.tile_len, p1 - ch.k0));
        S.tiles[j] = ch;
    }
    for (int64_t k = first; k < S.zero_words; k += stride) S.zero[k] = 0;
}

void launch_validate_offsets(const Problem& P, int num_sms, cudaStream_t s) {
    const int64_t nb = static_cast<int64_t>(P.T) * P.B + 1;
    const int blocks = static_cast<int>(min64((nb + 255) / 256, int64_t(num_sms) * 8));
    launch(validate_offsets_kernel, max(blocks, 1), 256, 0, s, P);
}

void launch_plan(const Problem& P, const Plan& Q, const TilePlan* S, int64_t chunk_bound, int num_sms, cudaStream_t s) {
    const TilePlan none{};
    if (P.T > kPlanTables) launch(plan_tables_kernel, 1, 1024, 0, s, P, Q, S ? *S : none);
    const int64_t cap = static_cast<int64_t>(num_sms) * 6;
    if (chunk_bound <= cap * 32)
        launch(plan_kernel<8>, static_cast<unsigned>((chunk_bound + 31) / 32), 256, 0, s, P, Q, S ? *S : none);
    else
        launch(plan_kernel<1>, static_cast<unsigned>(min64((chunk_bound + 255) / 256, cap)), 256, 0, s, P, Q,
               S ? *S : none);
}
int plan_launches(const Problem& P) { return P.T > kPlanTables ? 2 : 1; }

}  // namespace cbtbe
