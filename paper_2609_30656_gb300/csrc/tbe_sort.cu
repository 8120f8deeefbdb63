// tbe_sort.cu -- stable LSD radix sort of (row id, payload) pairs for the
// de-duplicated backward of the pooled embedding bag.
//
// A table's lookups are contiguous and its sort keys are key_base_t + r with
// r <= rows_t (r = rows_t: an out-of-range index), so each table's range is
// sorted on its own, on the bits of r only (3 passes of 8 bits for tables of
// fewer than 16M rows), in tiles of at most 4096
// positions that never straddle tables. A block ranks its tile's keys by digit
// (warp match + per-warp counters, stable by position), lays them out by digit
// in shared memory and writes each digit's run to that digit's slots of the
// output. The first output slot of each (tile, digit) is found one of two ways:
//   reduce-then-scan (default): one kernel counts every tile's digits, one
//     scans the counts per table, and the scatter reads its slots; no block
//     waits on another. With few tiles the scatter sums the counts itself, and
//     the counts come from the kernel that wrote the keys (key generation, or
//     the pass before).
//   single sweep (CB_SORT_LOOKBACK): one streaming kernel counts every pass's
//     digit histogram per table; each pass then reads and writes every pair
//     once, a block publishing its per-digit counts and finding those of the
//     table's earlier tiles by a decoupled look-back over their published
//     words. The look-back wait is bounded in time: when it runs out the kernel
//     records CB_ERR_TIMEOUT, publishes anyway so later tiles finish, and
//     writes nothing.
#include "tbe_internal.cuh"
#include "tbe_launch.h"

namespace cbtbe {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;  // 4096 keys
static_assert(kSortTile == kSortTileKeys, "tile size shared with the host plan");
constexpr int kRadix = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr uint32_t kFlagAgg = 1u << 30;
constexpr uint32_t kFlagIncl = 2u << 30;
constexpr uint32_t kCountMask = (1u << 30) - 1;

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t load_volatile(const uint32_t* p) {
    return *reinterpret_cast<const volatile uint32_t*>(p);
}
__device__ __forceinline__ void store_volatile(uint32_t* p, uint32_t v) {
    *reinterpret_cast<volatile uint32_t*>(p) = v;
}

constexpr int kLookbackWindow = 8;  // predecessor tiles inspected per look-back round

__device__ __forceinline__ uint32_t sort_digit(uint32_t key, uint32_t key_base, int shift) {
    return ((key - key_base) >> shift) & (kRadix - 1);
}

// *p += v in the lanes where `on`, returning the old value there (0 elsewhere):
// one predicated shared-memory atomic, with no branch around it.
__device__ __forceinline__ uint32_t shared_add_if(uint32_t* p, uint32_t v, bool on) {
    uint32_t old = 0;
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t@q atom.shared.add.u32 %0, [%2], %3;\n\t}"
        : "+r"(old)
        : "r"(static_cast<uint32_t>(on)), "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(v)
        : "memory");
    return old;
}

// Stable rank of a tile's keys within each warp; item j of lane l of warp w is
// tile position w*512 + j*32 + l. The lanes holding one digit in item j find
// each other (match), their lowest lane adds their number to the warp's
// counter of that digit and shares the old value. A warp's shared-memory
// atomics take effect in issue order, so item j's lanes count before item
// j + 1's, and lanes of one item by lane: the rank follows the position.
// Positions past the tile count under the extra digit kRadix. The matches of
// kRankBatch items are found before their atomics are issued (in item order),
// so that independent match, atomic and shuffle latencies overlap.
#ifndef CB_RANK_BATCH
#define CB_RANK_BATCH 2
#endif
constexpr int kRankBatch = CB_RANK_BATCH;
// NT threads per block rank a tile of kSortTile keys, NI = kSortTile / NT per thread.
template <int NT>
__device__ __forceinline__ void rank_tile(const uint32_t (&key)[kSortTile / NT], int tile_count, uint32_t key_base,
                                          int shift, uint32_t (*sh_warp)[kRadix + 1],
                                          uint32_t (&rank2)[kSortTile / NT / 2]) {
    constexpr int NI = kSortTile / NT;
    static_assert(NI % kRankBatch == 0, "rank batches divide the items");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
    for (int j0 = 0; j0 < NI; j0 += kRankBatch) {
        uint32_t d[kRankBatch], peers[kRankBatch], before[kRankBatch];
#pragma unroll
        for (int i = 0; i < kRankBatch; ++i) {
            const int j = j0 + i;
            const int local = wid * (32 * NI) + j * 32 + lane;
            d[i] = local < tile_count ? sort_digit(key[j], key_base, shift) : kRadix;
            peers[i] = __match_any_sync(kFull, d[i]);
        }
#pragma unroll
        for (int i = 0; i < kRankBatch; ++i) {
            const int leader = __ffs(peers[i]) - 1;
            before[i] = shared_add_if(&sh_warp[wid][d[i]], static_cast<uint32_t>(__popc(peers[i])), lane == leader);
        }
#pragma unroll
        for (int i = 0; i < kRankBatch; ++i) {
            const int j = j0 + i;
            const int leader = __ffs(peers[i]) - 1;
            const uint32_t r = __shfl_sync(kFull, before[i], leader) + __popc(peers[i] & lt_mask);
            if (j & 1) rank2[j >> 1] |= r << 16; else rank2[j >> 1] = r;  // two 16-bit ranks per register
        }
    }
}

// The tile laid out by digit in shared memory (slot = the warp's start of the
// digit, which holds the digit's tile-local start plus the counts of earlier
// warps, + the rank): every slot first (the counters are read-only here), then
// the stores.
template <int NT>
__device__ __forceinline__ void scatter_tile(const uint32_t (&key)[kSortTile / NT], const uint32_t (&val)[kSortTile / NT],
                                             uint32_t (&rank2)[kSortTile / NT / 2], int tile_count, uint32_t key_base,
                                             int shift, const uint32_t (*sh_warp)[kRadix + 1],
                                             uint32_t* sh_keys, uint32_t* sh_vals) {
    constexpr int NI = kSortTile / NT;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < NI; ++j) {
        const uint32_t dd = sort_digit(key[j], key_base, shift);
        const uint32_t r = (j & 1) ? (rank2[j >> 1] >> 16) : (rank2[j >> 1] & 0xffffu);
        const uint32_t pos = (sh_warp[wid][dd] + r) & 0xffffu;  // < 4096 for real items
        rank2[j >> 1] = (j & 1) ? ((rank2[j >> 1] & 0xffffu) | (pos << 16))
                                : ((rank2[j >> 1] & 0xffff0000u) | pos);
    }
#pragma unroll
    for (int j = 0; j < NI; ++j) {
        const int local = wid * (32 * NI) + j * 32 + lane;
        if (local < tile_count) {
            const uint32_t pos = (j & 1) ? (rank2[j >> 1] >> 16) : (rank2[j >> 1] & 0xffffu);
            sh_keys[pos] = key[j];
            sh_vals[pos] = val[j];
        }
    }
}

// Consecutive shared slots of one digit go to consecutive global slots
// (destination = sh_goff[digit] + slot). Half a tile at a time: its shared
// reads, its destinations, its stores.
// NEXT: the digits of the next pass are counted for the tile that each pair lands
// in (tile first + (destination - p0) / kSortTile, at most last).
template <int NT, bool NEXT = false>
__device__ __forceinline__ void write_tile(const SortPass& S, int tile_count, uint32_t key_base,
                                           const int32_t* sh_goff, const uint32_t* sh_keys,
                                           const uint32_t* sh_vals, int32_t p0 = 0, int32_t first = 0, int32_t last = 0) {
    const int tid = threadIdx.x;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        constexpr int kHalf = kSortTile / NT / 2;
        uint32_t key[kHalf], val[kHalf];
        int32_t dst[kHalf];
#pragma unroll
        for (int j = 0; j < kHalf; ++j) {
            const int i = tid + (h * kHalf + j) * NT;
            key[j] = i < tile_count ? sh_keys[i] : 0u;
            val[j] = i < tile_count ? sh_vals[i] : 0u;
        }
#pragma unroll
        for (int j = 0; j < kHalf; ++j)
            dst[j] = sh_goff[sort_digit(key[j], key_base, S.shift)] + tid + (h * kHalf + j) * NT;
#pragma unroll
        for (int j = 0; j < kHalf; ++j) {
            const int i = tid + (h * kHalf + j) * NT;
            const bool in = i < tile_count && dst[j] >= 0 && dst[j] < S.n;
            if (in) {
                S.keys_out[dst[j]] = key[j];
                S.vals_out[dst[j]] = val[j];
            }
            if (NEXT) {
                // The lanes that count where the first counting lane does are added by
                // it together: a hot row's pairs are neighbours here, and would queue
                // up at one counter.
                const int32_t tile = min(first + max(dst[j] - p0, 0) / kSortTile, last);
                const uint32_t at = static_cast<uint32_t>(tile) * kRadix + sort_digit(key[j], key_base, S.shift + 8);
                const uint32_t active = __ballot_sync(kFull, in);
                const int lead = active ? __ffs(active) - 1 : 0;
                const uint32_t lead_at = __shfl_sync(kFull, at, lead);
                const uint32_t same = __ballot_sync(kFull, in && at == lead_at);
                const int lane = tid & 31;
                if (in && (lane == lead || !((same >> lane) & 1u)))
                    atomicAdd(S.next_digits + at, lane == lead ? static_cast<uint32_t>(__popc(same)) : 1u);
            }
        }
    }
}

__global__ void __launch_bounds__(kSortThreads, 3) onesweep_kernel(SortPass S) {
    extern __shared__ __align__(16) uint32_t sh_dyn[];
    uint32_t* sh_keys = sh_dyn;                            // tile-sorted keys
    uint32_t* sh_vals = sh_dyn + kSortTile;                // tile-sorted payloads
    __shared__ uint32_t sh_warp[kSortWarps][kRadix + 1];   // per-warp counts, then prefixes
                                                           // (slot kRadix: positions past the tile)
    __shared__ int32_t sh_goff[kRadix];                    // global destination - local index
    __shared__ int64_t sh_scan[33];
    __shared__ uint32_t sh_tile;
    __shared__ int sh_abort;
    begin_kernel();

    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) {
        sh_tile = atomicAdd(S.tile_counter, 1u);
        sh_abort = 0;
    }
    for (int i = tid; i < kSortWarps * (kRadix + 1); i += kSortThreads) (&sh_warp[0][0])[i] = 0;
    __syncthreads();
    const uint32_t tile = sh_tile;
    if (tile >= *S.num_tiles) return;  // the grid is an upper bound on the tiles
    const Chunk tc = S.tiles[tile];
    const int t = tc.table;
    const int64_t tile_base = tc.k0;
    const int tile_count = static_cast<int>(min64(tc.len & 0x7fffffffu, S.n - tile_base));
    const uint32_t key_base = static_cast<uint32_t>(S.tables[t].key_base);
    const int64_t first_tile = S.table_first_tile[t];

    // Warp-striped load: item j of lane l is position tile_base + wid*512 + j*32 + l.
    // Keys, payloads and ranks stay in registers until the shared scatter.
    uint32_t key[kSortItems], val[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int local = wid * (32 * kSortItems) + j * 32 + lane;
        const bool valid = local < tile_count;
        key[j] = valid ? __ldg(S.keys_in + tile_base + local) : 0u;
        val[j] = valid ? __ldg(S.vals_in + tile_base + local) : 0u;
    }
    uint32_t rank2[kSortItems / 2];
    rank_tile<kSortThreads>(key, tile_count, key_base, S.shift, sh_warp, rank2);
    __syncthreads();

    // Thread d: per-warp exclusive prefix and the tile's count of digit d.
    const int d = tid;
    uint32_t count = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t c = sh_warp[w][d];
        sh_warp[w][d] = count;
        count += c;
    }
    uint32_t* my_status = S.status + static_cast<int64_t>(tile) * kRadix + d;
    store_volatile(my_status, (tile == first_tile ? kFlagIncl : kFlagAgg) | count);
    int64_t total;
    const int64_t start = block_excl_scan(count, sh_scan, &total);
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) sh_warp[w][d] += static_cast<uint32_t>(start);

    // Decoupled look-back over earlier tiles for digit d, kLookbackWindow
    // predecessors per round (independent loads), bounded in time.
    uint32_t excl = 0;
    if (tile > first_tile) {
        int64_t k = static_cast<int64_t>(tile) - 1;
        const uint64_t t0 = global_ns();
        uint32_t spins = 0;
        bool done = false;
        while (!done) {
            uint32_t word[kLookbackWindow];
#pragma unroll
            for (int w = 0; w < kLookbackWindow; ++w) {
                const int64_t kk = k - w;
                const uint32_t* src = (S.force_timeout && tile == 1) ? S.never_set
                                                                      : S.status + kk * kRadix + d;
                word[w] = kk >= first_tile ? load_volatile(src) : kFlagIncl;
            }
            int used = 0;
#pragma unroll
            for (int w = 0; w < kLookbackWindow; ++w) {
                if (done || used < w) continue;      // stopped earlier in this round
                const uint32_t flag = word[w] & ~kCountMask;
                if (flag == 0) continue;             // not published yet: poll it again
                excl += word[w] & kCountMask;
                used = w + 1;
                if (flag == kFlagIncl || k - w <= first_tile) done = true;
            }
            k -= used;
            if (!done && used == 0) {
                // The nearest predecessor has not published yet: poll that one
                // word alone, backing off, then read the window again.
                const uint32_t* src = (S.force_timeout && tile == 1) ? S.never_set
                                                                     : S.status + k * kRadix + d;
                uint32_t ns = 32;
                bool timed_out = false;
                while ((load_volatile(src) & ~kCountMask) == 0) {
                    if ((++spins & 15u) == 0 && global_ns() - t0 > S.timeout_ns) {
                        timed_out = true;
                        break;
                    }
                    __nanosleep(ns);
                    ns = ns < 512 ? 2 * ns : ns;
                }
                if (timed_out) {
                    set_error(S.error, CB_ERR_TIMEOUT);
                    *S.timed_out = 1;
                    atomicExch(&sh_abort, 1);
                    break;
                }
            }
        }
        store_volatile(my_status, kFlagIncl | ((excl + count) & kCountMask));
    }
    // Positions are below 2^30 and the local index below 2^12: 32 bits suffice.
    sh_goff[d] = static_cast<int32_t>(
        static_cast<int64_t>(S.digit_base[static_cast<int64_t>(t) * S.base_stride + d]) + excl - start);
    __syncthreads();

    scatter_tile<kSortThreads>(key, val, rank2, tile_count, key_base, S.shift, sh_warp, sh_keys, sh_vals);
    __syncthreads();
    if (sh_abort) return;
    write_tile<kSortThreads>(S, tile_count, key_base, sh_goff, sh_keys, sh_vals);
}

// ---------------------------------------------------------------- reduce-then-scan

// (a) Digit counts of every tile of this pass: 16 keys per thread, shared
// counters (their order does not matter here).
#ifndef CB_COUNT_MIN_BLOCKS
#define CB_COUNT_MIN_BLOCKS 8  // resident blocks per SM the count kernel is compiled for (31 registers)
#endif
__global__ void __launch_bounds__(kSortThreads, CB_COUNT_MIN_BLOCKS) radix_count_kernel(const SortPass S) {
    __shared__ uint32_t sh[kRadix];
    begin_kernel();
    const int64_t tile = blockIdx.x;
    if (tile >= *S.num_tiles) return;  // the grid is an upper bound on the tiles
    const int tid = threadIdx.x;
    sh[tid] = 0;
    const Chunk tc = S.tiles[tile];
    const int count = static_cast<int>(min64(tc.len & 0x7fffffffu, S.n - tc.k0));
    const uint32_t rb = static_cast<uint32_t>(S.tables[tc.table].key_base);
    uint32_t k[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int i = tid + j * kSortThreads;
        k[j] = i < count ? __ldg(S.keys_in + tc.k0 + i) : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j)
        if (tid + j * kSortThreads < count) atomicAdd(&sh[sort_digit(k[j], rb, S.shift)], 1u);
    __syncthreads();
    const uint32_t c = sh[tid];
    S.tile_digits[tile * kRadix + tid] = c;
    if (c) atomicAdd(S.table_digits + static_cast<int64_t>(tc.table) * kRadix + tid, c);
}

// (b) The first output slot of every (tile, digit), replacing its count: the
// table's first position, plus the table's counts of smaller digits, plus the
// counts of the digit in the table's earlier tiles. A block takes kScanDigits digits
// of a table (8 blocks per table) and a thread one digit over 1/16 of the table's
// tiles, up to kScanLoads loads in flight (6 tables of 500 tiles: sort 402 -> 373 us
// against one block per table and four threads per digit, 24 us a pass; 64 tables of
// 100 tiles, 643 us that way: 656 with 32 parts).
constexpr int kScanDigits = 32;
constexpr int kScanParts = 16;
constexpr int kScanLoads = 16;

__global__ void __launch_bounds__(kScanDigits * kScanParts) radix_slots_kernel(const SortPass S) {
    __shared__ uint32_t sh_part[kScanParts][kScanDigits];
    __shared__ uint32_t sh_start[kRadix];
    __shared__ int64_t sh_scan[33];
    begin_kernel();
    const int groups = kRadix / kScanDigits;
    const int t = blockIdx.x / groups, tid = threadIdx.x;
    const int lane = tid & (kScanDigits - 1), part = tid / kScanDigits;
    const int d = (blockIdx.x % groups) * kScanDigits + lane;
    const int64_t f = S.table_first_tile[t], e = S.table_first_tile[t + 1];
    const int64_t per = (e - f + kScanParts - 1) / kScanParts;
    const int64_t a = min64(f + part * per, e), b = min64(a + per, e);
    const uint32_t mine = tid < kRadix ? S.table_digits[static_cast<int64_t>(t) * kRadix + tid] : 0u;
    uint32_t* c = S.tile_digits + d;
    uint32_t sum = 0;
    int64_t k = a;
    for (; k + kScanLoads <= b; k += kScanLoads) {
        uint32_t v[kScanLoads];
#pragma unroll
        for (int u = 0; u < kScanLoads; ++u) v[u] = c[(k + u) * kRadix];
#pragma unroll
        for (int u = 0; u < kScanLoads; ++u) sum += v[u];
    }
    for (; k < b; ++k) sum += c[k * kRadix];
    sh_part[part][lane] = sum;
    int64_t all;
    const int64_t ex = block_excl_scan(mine, sh_scan, &all);
    // positions are below 2^30: 32 bits hold every slot
    if (tid < kRadix) sh_start[tid] = static_cast<uint32_t>(S.table_pos[t] + ex);
    __syncthreads();
    uint32_t run = sh_start[d];
    for (int q = 0; q < part; ++q) run += sh_part[q][lane];
    for (k = a; k + kScanLoads <= b; k += kScanLoads) {
        uint32_t v[kScanLoads];
#pragma unroll
        for (int u = 0; u < kScanLoads; ++u) v[u] = c[(k + u) * kRadix];
#pragma unroll
        for (int u = 0; u < kScanLoads; ++u) {
            c[(k + u) * kRadix] = run;
            run += v[u];
        }
    }
    for (; k < b; ++k) {
        const uint32_t v = c[k * kRadix];
        c[k * kRadix] = run;
        run += v;
    }
}

// (c) The scatter of tile blockIdx.x: the ranking of the single-sweep kernel,
// with the first output slot of every digit read from (b), or (FEW) summed here
// from the counts of the table's tiles. NT threads per tile
// (NT / 32 warps ranking kSortTile / NT keys per thread); threads 0..255 own one
// digit each in the prefix step.
#ifndef CB_SCATTER_THREADS
#define CB_SCATTER_THREADS 256
#endif
constexpr int kScatterThreads = CB_SCATTER_THREADS;
static_assert(kScatterThreads >= kRadix && kSortTile % kScatterThreads == 0, "scatter block shape");

template <int NT, bool FEW>
__global__ void __launch_bounds__(NT, NT == 256 ? 3 : 1024 / NT) radix_scatter_kernel(const SortPass S) {
    constexpr int NI = kSortTile / NT;
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) uint32_t sh_dyn[];
    uint32_t* sh_keys = sh_dyn;                            // tile-sorted keys
    uint32_t* sh_vals = sh_dyn + kSortTile;                // tile-sorted payloads
    __shared__ uint32_t sh_warp[NW][kRadix + 1];           // per-warp counts, then prefixes
                                                           // (slot kRadix: positions past the tile)
    __shared__ int32_t sh_goff[kRadix];                    // global destination - local index
    __shared__ int64_t sh_scan[33];

    begin_kernel();
    const int64_t tile = blockIdx.x;
    if (tile >= *S.num_tiles) return;  // the grid is an upper bound on the tiles
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int i = tid; i < NW * (kRadix + 1); i += NT) (&sh_warp[0][0])[i] = 0;
    const Chunk tc = S.tiles[tile];
    // digit tid's first output slot; FEW: the counts it follows from
    uint32_t slot = 0, digit_total = 0;
    int64_t first_tile = 0, last_tile = 0;
    if constexpr (FEW) {
        first_tile = S.table_first_tile[tc.table];
        last_tile = S.table_first_tile[tc.table + 1] - 1;
    } else {
        slot = tid < kRadix ? S.tile_digits[tile * kRadix + tid] : 0u;
    }
    const int64_t tile_base = tc.k0;
    const int tile_count = static_cast<int>(min64(tc.len & 0x7fffffffu, S.n - tile_base));
    const uint32_t key_base = static_cast<uint32_t>(S.tables[tc.table].key_base);
    uint32_t key[NI], val[NI];
#pragma unroll
    for (int j = 0; j < NI; ++j) {
        const int local = wid * (32 * NI) + j * 32 + lane;
        const bool valid = local < tile_count;
        key[j] = valid ? __ldg(S.keys_in + tile_base + local) : 0u;
        val[j] = valid ? __ldg(S.vals_in + tile_base + local) : 0u;
    }
    if constexpr (FEW) {
        if (tid < kRadix) {
            const uint32_t* c = S.tile_digits + tid;
            for (int64_t k0 = first_tile; k0 <= last_tile; k0 += 8) {
                uint32_t v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = k0 + u <= last_tile ? __ldg(c + (k0 + u) * kRadix) : 0u;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    digit_total += v[u];
                    slot += k0 + u < tile ? v[u] : 0u;
                }
            }
        }
        int64_t all;
        slot += static_cast<uint32_t>(S.table_pos[tc.table] + block_excl_scan(digit_total, sh_scan, &all));
    }
    __syncthreads();
    uint32_t rank2[NI / 2];
    rank_tile<NT>(key, tile_count, key_base, S.shift, sh_warp, rank2);
    __syncthreads();
    const int d = tid;
    uint32_t count = 0;
    if (d < kRadix) {
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const uint32_t c = sh_warp[w][d];
            sh_warp[w][d] = count;
            count += c;
        }
    }
    int64_t total;
    const int64_t start = block_excl_scan(count, sh_scan, &total);  // threads past 255 add 0
    if (d < kRadix) {
#pragma unroll
        for (int w = 0; w < NW; ++w) sh_warp[w][d] += static_cast<uint32_t>(start);
        sh_goff[d] = static_cast<int32_t>(static_cast<int64_t>(slot) - start);
    }
    __syncthreads();
    scatter_tile<NT>(key, val, rank2, tile_count, key_base, S.shift, sh_warp, sh_keys, sh_vals);
    __syncthreads();
    if (FEW && S.next_digits)
        write_tile<NT, true>(S, tile_count, key_base, sh_goff, sh_keys, sh_vals,
                             static_cast<int32_t>(S.table_pos[tc.table]), static_cast<int32_t>(first_tile),
                             static_cast<int32_t>(last_tile));
    else
        write_tile<NT>(S, tile_count, key_base, sh_goff, sh_keys, sh_vals);
}

// ---------------------------------------------------------------- single sweep

// Digit histograms of every pass, per table. Each block streams a contiguous
// range of tiles, so its shared histogram changes table only a few times.
__global__ void __launch_bounds__(256) sort_hist_kernel(const uint32_t* keys, const Chunk* tiles,
                                                        const int64_t* num_tiles,
                                                        const TableDev* tables, int passes,
                                                        uint32_t* hist) {
    __shared__ uint32_t sh[4 * kRadix];
    begin_kernel();
    const int64_t nt = *num_tiles;
    const int64_t per = (nt + gridDim.x - 1) / gridDim.x;
    const int64_t lo = static_cast<int64_t>(blockIdx.x) * per, hi = min64(lo + per, nt);
    int cur = -1;
    for (int i = threadIdx.x; i < 4 * kRadix; i += blockDim.x) sh[i] = 0;
    __syncthreads();
    for (int64_t j = lo; j < hi; ++j) {
        const Chunk tc = tiles[j];
        if (tc.table != cur) {  // uniform across the block
            __syncthreads();    // every count of the previous table has landed
            if (cur >= 0) {
                for (int i = threadIdx.x; i < passes * kRadix; i += blockDim.x) {
                    if (sh[i]) atomicAdd(hist + static_cast<int64_t>(cur) * passes * kRadix + i, sh[i]);
                    sh[i] = 0;
                }
            }
            __syncthreads();    // the flush is done before new counts start
            cur = tc.table;
        }
        const uint32_t rb = static_cast<uint32_t>(tables[cur].key_base);
        const int len = static_cast<int>(tc.len & 0x7fffffffu);
        // All of the tile's loads first, then the counts.
        uint32_t r[kSortItems];
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            const int i = threadIdx.x + k * 256;
            r[k] = i < len ? __ldg(keys + tc.k0 + i) - rb : 0u;
        }
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            if (threadIdx.x + k * 256 >= len) break;
            for (int p = 0; p < passes; ++p)
                atomicAdd(&sh[p * kRadix + ((r[k] >> (8 * p)) & 255u)], 1u);
        }
    }
    __syncthreads();
    if (cur >= 0)
        for (int i = threadIdx.x; i < passes * kRadix; i += blockDim.x)
            if (sh[i]) atomicAdd(hist + static_cast<int64_t>(cur) * passes * kRadix + i, sh[i]);
}

// First output position of each digit of each pass: the table's first position
// plus the exclusive scan of that pass's digit counts (one block per table).
__global__ void sort_base_kernel(const uint32_t* hist, const int64_t* table_pos, int passes,
                                 uint32_t* base) {
    __shared__ int64_t sh[33];
    begin_kernel();
    const int t = blockIdx.x, d = threadIdx.x;
    for (int p = 0; p < passes; ++p) {
        const int64_t i = (static_cast<int64_t>(t) * passes + p) * kRadix + d;
        int64_t total;
        const int64_t ex = block_excl_scan(hist[i], sh, &total);
        base[i] = static_cast<uint32_t>(table_pos[t] + ex);
    }
}

void launch_sort_hist(const uint32_t* keys, const Chunk* tiles, const int64_t* num_tiles,
                      int64_t tile_bound, const TableDev* tables, int passes, uint32_t* hist,
                      int num_sms, cudaStream_t s) {
    const int grid = static_cast<int>(max64(1, min64(tile_bound, static_cast<int64_t>(num_sms) * 4)));
    launch(sort_hist_kernel, grid, 256, 0, s, keys, tiles, num_tiles, tables, passes, hist);
}

void launch_sort_bases(const uint32_t* hist, const int64_t* table_pos, int T, int passes,
                       uint32_t* base, cudaStream_t s) {
    launch(sort_base_kernel, T, kRadix, 0, s, hist, table_pos, passes, base);
}

constexpr int kSortDynSmem = 2 * kSortTile * sizeof(uint32_t);  // 32 KB

template <bool FEW>
void launch_scatter(const SortPass& S, unsigned grid, cudaStream_t s) {
    // static + dynamic shared memory may pass the 48 KB default
    static const bool configured = cudaFuncSetAttribute(radix_scatter_kernel<kScatterThreads, FEW>,
                                                        cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                        kSortDynSmem) == cudaSuccess;
    (void)configured;
    launch(radix_scatter_kernel<kScatterThreads, FEW>, grid, kScatterThreads, kSortDynSmem, s, S);
}

void launch_radix_pass(const SortPass& S, int64_t tile_bound, cudaStream_t s) {
    const unsigned grid = static_cast<unsigned>(max64(tile_bound, 1));
    if (tile_bound <= kFewSortTiles) {
        launch_scatter<true>(S, grid, s);
        return;
    }
    launch(radix_count_kernel, grid, kSortThreads, 0, s, S);
    launch(radix_slots_kernel, static_cast<unsigned>(S.T) * (kRadix / kScanDigits), kScanDigits * kScanParts, 0, s, S);
    launch_scatter<false>(S, grid, s);
}

int radix_pass_launches(int64_t tile_bound) { return tile_bound <= kFewSortTiles ? 1 : 3; }

void launch_onesweep(const SortPass& S, int64_t tile_bound, cudaStream_t s) {
    static bool configured = false;
    if (!configured) {
        cudaFuncSetAttribute(onesweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSortDynSmem);
        configured = true;
    }
    launch(onesweep_kernel, static_cast<unsigned>(max64(tile_bound, 1)), kSortThreads, kSortDynSmem, s, S);
}

}  // namespace cbtbe
