// tbe_launch.h -- host-callable launchers of the kernels (internal to the library).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace cbtbe {

struct Problem;
struct Plan;

// One radix pass over n (key, payload) pairs, each table's range sorted on
// its own: tiles never straddle tables, digits are taken from key - key_base_t.
struct SortPass {
    const uint32_t* keys_in;
    const uint32_t* vals_in;
    uint32_t* keys_out;
    uint32_t* vals_out;
    const struct Chunk* tiles;        // table-aligned tiles of at most 4096 positions
    const int64_t* num_tiles;         // device scalar
    const int64_t* table_first_tile;  // [T + 1]
    const struct TableDev* tables;
    int64_t n;
    int shift;                   // digit = ((key - key_base_t) >> shift) & 255
    // reduce-then-scan
    const int64_t* table_pos;    // [T + 1] first position of each table
    uint32_t* tile_digits;       // [tiles][256]: digit counts (many tiles: then first output slots)
    uint32_t* next_digits;       // few tiles: the next pass's counts, zeroed (null: last pass)
    uint32_t* table_digits;      // many tiles: [T][256] digit counts per table, zeroed
    int T;
    // single sweep with look-back
    const uint32_t* digit_base;  // [T][stride]: this pass's 256 first output slots per table
    int base_stride;             // passes * 256
    uint32_t* status;            // [tiles * 256], zeroed before the pass
    uint32_t* tile_counter;      // zeroed before the pass
    const uint32_t* never_set;   // a zero word no kernel writes (timeout test hook)
    int force_timeout;
    int* error;
    uint32_t* timed_out;         // set when a wait ran out (zeroed before the first pass)
    uint64_t timeout_ns;
};

// Lookups per chunk. A walker's warp takes a chunk at a time, so a call needs
// several chunks for each walker warp that the GPU holds (24 to 40 per SM): with
// 512 lookups per chunk a call of up to a few million lookups left most SMs
// without work, and one warp's chain of loads was the call's time. So
// n / (num_sms * kChunksPerSm) lookups, rounded up to whole 32-lookup batches,
// at least one batch and at most kMaxChunk. Measured whole calls, 512 against
// this rule: forward of 512 lookups (1 table) 74 -> 23 us, of 1.6 M lookups (20
// tables, odd dims) 277 -> 151 us; forward + backward of 106 K one-hot lookups
// (26 tables) 682 -> 415 us; forward + fused Adagrad on 1.3 M lookups (16
// tables) 1377 -> 572 us (698 at 64 chunks per SM, 945 at 32); from 10 M lookups
// on the chunks are 512 long, where the sweep of 256, 512 and 1024 had its best.
#ifndef CB_CHUNKS_PER_SM
#define CB_CHUNKS_PER_SM 128
#endif
constexpr int64_t kChunksPerSm = CB_CHUNKS_PER_SM;
constexpr int64_t kMaxChunk = 512;
constexpr int64_t kMinChunk = 32;
inline int64_t chunk_len_for(int64_t n, int num_sms) {
    const int64_t per = n / (num_sms * kChunksPerSm) + 1;
    const int64_t len = (per + 31) / 32 * 32;
    return len < kMinChunk ? kMinChunk : (len > kMaxChunk ? kMaxChunk : len);
}
// Chunks of a call of n lookups over T tables: a whole number per table.
inline int64_t chunk_count_bound(int64_t n, int64_t chunk_len, int64_t T) { return n / chunk_len + T + 1; }
// An upper bound on the chunks of every call of up to n lookups (the count is
// not monotone in n where the chunk length grows).
inline int64_t chunk_count_limit(int64_t n, int num_sms, int64_t T) {
    const int64_t most = num_sms * kChunksPerSm;
    const int64_t small = n / kMinChunk < most ? n / kMinChunk : most;
    return (small > n / kMaxChunk ? small : n / kMaxChunk) + T + 1;
}
// Chunks that one warp of a fix-up kernel scans at a time: 32 when there are
// plenty, fewer so that the split segments of a small call spread over the GPU.
inline int fixup_span(int64_t chunk_bound, int num_sms) {
    const int64_t warps = static_cast<int64_t>(num_sms) * 64;
    const int64_t span = (chunk_bound + warps - 1) / warps;
    return static_cast<int>(span < 1 ? 1 : (span > 32 ? 32 : span));
}
inline int fixup_grid(int64_t chunk_bound, int span, int num_sms) {
    const int64_t need = (chunk_bound + 8 * span - 1) / (8 * span);  // 8 warps per block
    const int64_t cap = static_cast<int64_t>(num_sms) * 8;
    return static_cast<int>(need < 1 ? 1 : (need < cap ? need : cap));
}

// The walkers' layout of a row of `vecs` 16-byte vectors: vectors per lane, and
// rows per warp step (the most whose lanes, a power of two per row, fit a warp).
inline int row_vectors_per_lane(int vecs) { return vecs <= 32 ? 1 : (vecs <= 64 ? 2 : 4); }
inline int rows_per_step(int vecs) {
    int lanes = 1;
    while (lanes < vecs && lanes < 32) lanes *= 2;
    return 32 / lanes;
}

// Payload bag of a lookup whose index is out of range: outside every table's bags (the
// reduce reads the table's last bag for it, and drops the sum).
constexpr uint32_t kDeadBag = 0xffffffffu;

struct KeyGen {
    uint32_t* keys;    // [n] key_base_t + index (key_base_t + rows_t: out of range)
    uint32_t* vals;    // [n] bag id (kDeadBag when out of range), or lookup position
                       // when `packed` is used
    uint2* packed;     // [n] (bag id or kDeadBag, bits of w_i * s_b) by lookup position, or null
    uint32_t* tile_digits;         // counts of the first sort pass, zeroed (null: counted later)
    const int64_t* table_first_tile;
};

struct BwdOut {
    // workspace
    const uint32_t* keys_sorted; // [n] key_base_t + r
    const uint32_t* vals_sorted; // [n]
    const uint2* packed;         // [n] or null
    uint32_t* heads;             // [max_chunks] runs begun per chunk cell, and the first's offset
    uint32_t* head_bits;         // [max_chunks][chunk_len / 32] a flag per position: a run begins
    int64_t* run_count;          // [T] runs of real rows per table
    int64_t* out_first;          // [T + 1] first output row of each table (runs of
                                 // out-of-range lookups are not output)
    int64_t* float_base;         // [T + 1]
    uint32_t* tables_done;       // zero between calls
    int* cap_fail;
    const uint32_t* timed_out;   // a sort pass gave up on its wait (null: no pass waits)
    // caller's buffers
    int64_t* unique_ids;
    int64_t* table_offsets;
    int64_t* grad_offsets;
    float* grads;
    int64_t cap_rows;
    int64_t cap_floats;
    int64_t* num_unique;
    int64_t* num_floats;
    // Optimizer step fused in place of the gradient output (apply != 0): no
    // gradient buffers; every touched table row is updated where its sum ends.
    int apply;             // 0: write gradients, kApplySgd, kApplyAdagrad
    float lr;
    float eps;
    float* const* state;   // device [T] -> fp32 [rows_t] (row-wise Adagrad)
};
constexpr int kApplySgd = 1;
constexpr int kApplyAdagrad = 2;

void launch_validate_offsets(const Problem& P, int num_sms, cudaStream_t s);
// The optimizer step of O.apply from the row-sparse gradient in O's caller buffers.
void launch_apply_sparse(const Problem& P, const BwdOut& O, int num_sms, cudaStream_t s);
// Table-aligned tiles of the sort, and the words to clear before it.
struct TilePlan {
    int64_t tile_len;           // 0: no tiles
    struct Chunk* tiles;        // [max_tiles]
    int64_t max_tiles;
    int64_t* table_first_tile;  // [T + 1]
    int64_t* num_tiles;         // device scalar
    uint32_t* zero;             // [zero_words]
    int64_t zero_words;
};
// The chunk plan over the lookups and, with S, the sort's tiles.
void launch_plan(const Problem& P, const Plan& Q, const TilePlan* S, int64_t chunk_bound, int num_sms,
                 cudaStream_t s);
int plan_launches(const Problem& P);  // kernels launch_plan enqueues

constexpr int kPlanTables = 1024;  // tables that a block plans in shared memory
constexpr int kAllClasses = -1, kPlanned = -2;  // `cls` of launch_fwd_gather
// Whether a forward of one storage type runs without a plan kernel.
#ifndef CB_PLANNED_BLOCKS
#define CB_PLANNED_BLOCKS 2
#endif
constexpr int kPlannedBlocks = CB_PLANNED_BLOCKS;  // resident blocks per SM of the kernel that does
inline bool fwd_plans_itself(int64_t chunk_bound, int64_t T, int num_sms) {
    return T <= kPlanTables && chunk_bound <= static_cast<int64_t>(num_sms) * 8 * kPlannedBlocks;
}
void launch_fwd_gather(const Problem& P, const Plan& Q, void* out, int cls, int dtype, int vpl,
                       int gc, int64_t chunk_bound, int num_sms, cudaStream_t s);
void launch_fwd_fixup(const Problem& P, const Plan& Q, void* out, int64_t chunk_bound,
                      int num_sms, cudaStream_t s);

constexpr int64_t kSortTileKeys = 4096;
void launch_sort_hist(const uint32_t* keys, const struct Chunk* tiles, const int64_t* num_tiles,
                      int64_t tile_bound, const struct TableDev* tables, int passes, uint32_t* hist,
                      int num_sms, cudaStream_t s);
void launch_sort_bases(const uint32_t* hist, const int64_t* table_pos, int T, int passes,
                       uint32_t* base, cudaStream_t s);
void launch_onesweep(const SortPass& S, int64_t tile_bound, cudaStream_t s);
// Up to this many tiles, a pass is one kernel: every scatter tile sums the counts
// of its table's tiles itself, and counts the next pass's digits as it writes.
// (A pass's three kernels become one, 6 fewer in a backward of three passes: sort of
// 330 K lookups in 8 tables 58 -> 31 us, of 106 K in 26 tables 52 -> 27 us, of 1.3 M
// in 16 tables 76 -> 56 us. A tile reads its table's counts, so the reads grow with
// the square of a table's tiles: 512 tiles of one table read 268 MB from L2.)
constexpr int64_t kFewSortTiles = 512;
// One reduce-then-scan pass: tile counts and slots, unless few tiles; scatter.
void launch_radix_pass(const SortPass& S, int64_t tile_bound, cudaStream_t s);
int radix_pass_launches(int64_t tile_bound);  // kernels launch_radix_pass enqueues

void launch_keygen(const Problem& P, const Plan& Q, const KeyGen& K, bool packed, int64_t chunk_bound,
                   int num_sms, cudaStream_t s);
// Runs of equal sorted keys: counts per chunk cell, the reduce's chunks (cut at
// run ends), and the sizes and first output rows of every table.
void launch_bwd_runs(const Problem& P, const Plan& Q, const BwdOut& O, int64_t chunk_bound, int num_sms,
                     cudaStream_t s);
// The output ranges again, into other caller buffers (after launch_bwd_runs).
void launch_bwd_outputs(const Problem& P, const BwdOut& O, cudaStream_t s);
// The segmented reduce (apply: with the optimizer step fused), dispatched on
// the grad_out type P.out_dtype; one translation unit per type.
void launch_bwd_reduce(const Problem& P, const Plan& Q, const BwdOut& O, const void* grad_out, int cls,
                       int vpl, int gc, bool packed, bool apply, int64_t chunk_bound, int num_sms,
                       cudaStream_t s);
void launch_bwd_reduce_f32(const Problem& P, const Plan& Q, const BwdOut& O, const void* grad_out, int cls,
                           int vpl, int gc, bool packed, int64_t chunk_bound, int num_sms, cudaStream_t s);
void launch_bwd_reduce_f32_apply(const Problem& P, const Plan& Q, const BwdOut& O, const void* grad_out,
                                 int cls, int vpl, int gc, bool packed, int64_t chunk_bound, int num_sms,
                                 cudaStream_t s);
void launch_bwd_reduce_f16(const Problem& P, const Plan& Q, const BwdOut& O, const void* grad_out, int cls,
                           int vpl, int gc, bool packed, bool apply, int64_t chunk_bound, int num_sms,
                           cudaStream_t s);
void launch_bwd_reduce_bf16(const Problem& P, const Plan& Q, const BwdOut& O, const void* grad_out, int cls,
                            int vpl, int gc, bool packed, bool apply, int64_t chunk_bound, int num_sms,
                            cudaStream_t s);
void launch_weight_grad(const Problem& P, const Plan& Q, const void* grad_out, float* grad_w, int cls,
                        int dtype, int vpl, int gc, int64_t chunk_bound, int num_sms, cudaStream_t s);
void launch_bwd_fixup(const Problem& P, const Plan& Q, const BwdOut& O, int64_t chunk_bound,
                      int num_sms, cudaStream_t s);
}  // namespace cbtbe
