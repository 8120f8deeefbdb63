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
    int64_t total;

    __device__ __forceinline__ int64_t offset(int64_t bag) const { return load_index(P.offsets, bag, P.is32); }
    // Chunks of a table are contiguous and chunk_len long while a split bag goes on, so
    // the number of chunks that a bag reaches into follows from where it ends.
    __device__ __forceinline__ int64_t pieces(int64_t j, uint32_t bag, int) const {
        const Chunk ch = Q.chunks[j];
        const int64_t k1 = ch.k0 + static_cast<int64_t>(ch.len & 0x7fffffffu), e = offset(bag + 1);
        if (e <= k1) return 0;
        return min64((e - k1 + Q.chunk_len - 1) / Q.chunk_len, total - j - 1);
    }
    // ... and the chunk where it begins, from where that is (checked: malformed offsets).
    __device__ __forceinline__ bool origin(int64_t i, int lane, int64_t& j, int64_t& m) const {
        const Chunk ch = Q.chunks[i];
        const int64_t p0 = min64(max64(offset(static_cast<int64_t>(ch.table) * P.B), 0), P.n);
        j = i - ((ch.k0 - p0) / Q.chunk_len - (offset(ch.first) - p0) / Q.chunk_len);
        if (j < 0 || j >= i) return false;
        const unsigned long long word = Q.split[j];
        if (!(word & kSplitBegins) || static_cast<uint32_t>(word) != static_cast<uint32_t>(ch.first)) return false;
        m = pieces(j, static_cast<uint32_t>(ch.first), lane);
        return j + m >= i;
    }
    __device__ __forceinline__ void store(int64_t, uint32_t bag, int t, int x0, double (&acc)[4]) const {
        if (P.mean) {
            const int64_t L = offset(bag + 1) - offset(bag);
            if (L > 0)
#pragma unroll
                for (int x = 0; x < 4; ++x) acc[x] /= static_cast<double>(L);
        }
        const int64_t col0 = (static_cast<int64_t>(bag) - static_cast<int64_t>(t) * P.B) * P.sum_d + P.tables[t].doff;
        store_out4(out, col0 + x0, static_cast<float>(acc[0]), static_cast<float>(acc[1]),
                   static_cast<float>(acc[2]), static_cast<float>(acc[3]), P.out_dtype);
    }
    __device__ __forceinline__ void stored(int64_t, int, int) const {}
};

// (80 registers; left to itself the compiler takes 64 and spills.)
__global__ void __launch_bounds__(kWarpThreads, 3) fwd_fixup_kernel(const __grid_constant__ Problem P,
                                                                 const __grid_constant__ Plan Q,
                                                                 void* out, int span) {
    begin_kernel();
    const int64_t total = min64(Q.class_chunk_base[Q.num_classes], Q.max_chunks);
    fix_split(P, Q, BagSplit{P, Q, out, total}, total, span);
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
    const int span = fixup_span(chunk_bound, num_sms);
    launch(fwd_fixup_kernel, fixup_grid(chunk_bound, span, num_sms), kWarpThreads, 0, s, P, Q, out, span);
}

}  // namespace cbtbe
