// tbe_forward.cu -- forward fix-up (bags split across chunks) and the launch
// switch over storage types; the gather-pool kernel is in tbe_forward.cuh.
#include "tbe_internal.cuh"
#include "tbe_fixup.cuh"
#include "tbe_launch.h"

namespace cbtbe {

// Bags split over chunks (only those longer than the cap of the plan's moved
// boundaries): tail and head pieces, added in fp64, then scaled.
struct BagSplit {
    static constexpr bool kNarrow = false;
    const Problem& P;
    const Plan& Q;
    void* out;
    int total;

    __device__ __forceinline__ int64_t offset(int64_t bag) const { return load_index(P.offsets, bag, P.is32); }
    // Chunks of a table are contiguous and chunk_len long while a split bag goes on, so
    // the number of chunks that a bag reaches into follows from where it ends.
    __device__ __forceinline__ int pieces(int j, uint32_t bag, int) const {
        const Chunk ch = Q.chunks[j];
        const int64_t k1 = ch.k0 + static_cast<int64_t>(ch.len & 0x7fffffffu), e = offset(static_cast<int64_t>(bag) + 1);
        if (e <= k1) return 0;
        return static_cast<int>(min64((e - k1 + Q.chunk_len - 1) / Q.chunk_len, total - j - 1));
    }
    // ... and the chunk where it begins, from where that is (checked: malformed offsets).
    // Both positions count from the table's first, in whole chunks.
    __device__ __forceinline__ bool origin(int i, int lane, int& j, int& m) const {
        const Chunk ch = Q.chunks[i];
        const int64_t p0 = min64(max64(offset(static_cast<int64_t>(ch.table) * P.B), 0), P.n), s = offset(ch.first);
        if (s < p0 || s >= ch.k0) return false;
        // (k0 - p0 is a whole number of chunks: from s's chunk on, the bag moves no boundary)
        const int64_t before = (ch.k0 - s + Q.chunk_len - 1) / Q.chunk_len;
        if (before > i) return false;
        j = i - static_cast<int>(before);
        const unsigned long long word = Q.split[j];
        if (!(word & kSplitBegins) || static_cast<uint32_t>(word) != static_cast<uint32_t>(ch.first)) return false;
        m = pieces(j, static_cast<uint32_t>(ch.first), lane);
        return j + m >= i;
    }
    struct Dest {
        int64_t col;
        double length;  // mean pooling, else 0
    };
    __device__ __forceinline__ Dest dest(int, uint32_t bag, int t) const {
        const int64_t L = P.mean ? offset(static_cast<int64_t>(bag) + 1) - offset(bag) : 0;
        return Dest{(static_cast<int64_t>(bag) - static_cast<int64_t>(t) * P.B) * P.sum_d + P.tables[t].doff,
                    static_cast<double>(L)};
    }
    __device__ __forceinline__ void store(const Dest& d, int x0, double (&acc)[4]) const {
        if (d.length > 0.0)
#pragma unroll
            for (int x = 0; x < 4; ++x) acc[x] /= d.length;
        store_out4(out, d.col + x0, static_cast<float>(acc[0]), static_cast<float>(acc[1]),
                   static_cast<float>(acc[2]), static_cast<float>(acc[3]), P.out_dtype);
    }
    __device__ __forceinline__ void stored(int, int, int) const {}
};

// BLOCKS per SM: 2 for grids of up to 3 blocks per SM, else 3 (80 registers, the heavy part
// spills). Whole forward, us, at 2, 3 and 4: 106 K one-hot lookups (446 blocks) 35.4, 41.7 and
// (another box) 34 against 32 at 2; 139 K in tables of two types (579 blocks) 34.6, 34.0,
// 38.0; 330 K (736 blocks) 33.2, 33.3, 32.7; 270 K in bags of 300 45.5, 42.2, 41.0; 1.3 M 68.1,
// 67.7, 69.0; 1.6 M on odd dims 80.2, 79.3, 79.4.
template <int BLOCKS>
__global__ void __launch_bounds__(kWarpThreads, BLOCKS) fwd_fixup_kernel(const __grid_constant__ Problem P,
                                                                         const __grid_constant__ Plan Q, void* out,
                                                                         int span, int group_blocks) {
    begin_kernel();
    const int total = static_cast<int>(min64(Q.class_chunk_base[Q.num_classes], Q.max_chunks));
    fix_split(P, Q, BagSplit{P, Q, out, total}, total, span, group_blocks);
}

void launch_fwd_gather_f32(const Problem&, const Plan&, void*, int, int, int, int64_t, int,
                           cudaStream_t);
void launch_fwd_gather_f16(const Problem&, const Plan&, void*, int, int, int, int64_t, int,
                           cudaStream_t);
void launch_fwd_gather_bf16(const Problem&, const Plan&, void*, int, int, int, int64_t, int,
                            cudaStream_t);

void launch_fwd_gather(const Problem& P, const Plan& Q, void* out, int cls, int dtype, int vpl,
                       int gc, int64_t chunk_bound, int num_sms, cudaStream_t s) {
    if (dtype == CB_F32) launch_fwd_gather_f32(P, Q, out, cls, vpl, gc, chunk_bound, num_sms, s);
    else if (dtype == CB_F16) launch_fwd_gather_f16(P, Q, out, cls, vpl, gc, chunk_bound, num_sms, s);
    else launch_fwd_gather_bf16(P, Q, out, cls, vpl, gc, chunk_bound, num_sms, s);
}

void launch_fwd_fixup(const Problem& P, const Plan& Q, void* out, int64_t chunk_bound,
                      int num_sms, cudaStream_t s) {
    const FixupGrid g(chunk_bound, num_sms);
    auto* kernel = g.blocks <= 3 * num_sms ? fwd_fixup_kernel<2> : fwd_fixup_kernel<3>;
    launch(kernel, g.blocks, kWarpThreads, 0, s, P, Q, out, g.span, g.group_blocks);
}

}  // namespace cbtbe
