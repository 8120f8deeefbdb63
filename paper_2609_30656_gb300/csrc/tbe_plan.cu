// tbe_plan.cu -- offsets validation and the chunk plan shared by the forward
// gather-pool and the backward key generation / segmented reduce.
//
// A table's items (lookup positions, key-major so each table's lookups are
// contiguous) are cut every chunk_len positions, and the forward's cuts moved to bag
// ends; a table with no lookups still gets one (empty) chunk so that its empty bags
// are written.
// Chunks are numbered class by class (tables grouped by kernel instantiation),
// table by table within a class. The backward's sort tiles are placed with them.
#include "tbe_internal.cuh"
#include "tbe_launch.h"
#include "tbe_plan.cuh"

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

// More tables than a block's shared memory holds: the tables' part runs first, as
// a kernel of its own, into global memory.
__global__ void __launch_bounds__(1024) plan_tables_kernel(const __grid_constant__ Problem P,
                                                           const __grid_constant__ Plan Q,
                                                           const __grid_constant__ TilePlan S) {
    __shared__ int64_t sh[33];
    begin_kernel();
    plan_tables(P, Q, S.tile_len, Q.table_pos, Q.ord_chunk_base, S.table_first_tile, sh);
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
#pragma unroll 1
        for (int i = tid; i <= P.T; i += blockDim.x) {
            if (own) {
                Q.table_pos[i] = pos[i];
                if (S.tile_len > 0) S.table_first_tile[i] = tile_ord[i];
            }
            if (i < P.T) Q.table_chunk[Q.class_tables[i]] = ord[i];
        }
#pragma unroll 1
        for (int c = tid; c <= Q.num_classes; c += blockDim.x) {
            Q.class_chunk_base[c] = min64(ord[Q.class_table_start[c]], Q.max_chunks);
            Q.chunk_next[c] = 0;
        }
        if (tid == 0 && S.tile_len > 0) *S.num_tiles = min64(tile_ord[P.T], S.max_tiles);
    }
    const int64_t first = static_cast<int64_t>(blockIdx.x) * blockDim.x + tid;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int lane = tid & 31;
#pragma unroll 1
    for (int64_t w = first; (w - lane) / W < total; w += stride) {  // warp-uniform
        const int64_t j = min64(w / W, total - 1);
        const Chunk ch = plan_chunk<W>(P, Q, pos, ord, j, lane);
        if ((lane & (W - 1)) != 0 || w / W >= total) continue;
        Q.chunks[j] = ch;
    }
    if (S.tile_len <= 0) return;
    const int64_t tiles = min64(tile_ord[P.T], S.max_tiles);
#pragma unroll 1
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
#pragma unroll 1
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
