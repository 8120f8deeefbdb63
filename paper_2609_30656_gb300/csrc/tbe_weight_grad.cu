// tbe_weight_grad.cu -- gradient of the pooled output with respect to the
// per-sample weights. The pooled bag (Sec. IV.A.2 sparse_arch lookups) is
// linear in each weight, so for an upstream gradient grad_out
//
//   grad_w[i] = s_b * sum_j grad_out[b, Doff_t + j] * E_t[indices[i], j]
//
// (s_b = 1/L for mean pooling, 1 for sum), whatever the weights are: one dot
// product of the lookup's table row with its bag's grad_out slice.
//
// One warp per chunk of lookup positions (the forward's chunk plan and row
// layouts), in batches of 32 lookups: each of the G lane groups takes V = 32 / G
// consecutive lookups, so that it holds its bag's grad_out slice in registers and
// loads one only where its bag changes. Eight lookups' rows are loaded together, and
// their eight dot products are summed over the group's lanes at once: three rounds
// that halve the values a lane holds while they add, then plain butterfly rounds;
// every lane ends with its own lookup's sum. grad_out is fp32, or fp16 / bf16 when
// the handle's output is (mixed precision). Fixed order: deterministic.
// Bound by the rows served from L1 and L2, as the forward's gather, and by issue. On
// 11.8 M lookups (24 tables, 256-byte rows, Zipf 1.1, bags of 30): 771 us with the
// slice loaded and a butterfly run for every lookup, 396 us now (four lookups at a
// time: 447 us at 4 blocks per SM, 418 at 5, 508 at 3; eight at 3 blocks: 444).
#include "tbe_internal.cuh"
#include "tbe_launch.h"

namespace cbtbe {
namespace {

// Four grad_out values at g (fp32, or fp16 / bf16 with mixed precision), widened.
__device__ __forceinline__ float4 load_go4(const char* g, int go_dtype) {
    if (go_dtype == CB_F32) return __ldg(reinterpret_cast<const float4*>(g));
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(g));
    if (go_dtype == CB_BF16)
        return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                           __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
    __half2 a, b;
    memcpy(&a, &w.x, 4);
    memcpy(&b, &w.y, 4);
    const float2 fa = __half22float2(a), fb = __half22float2(b);
    return make_float4(fa.x, fa.y, fb.x, fb.y);
}

template <int DT, int VPL, int G>
__device__ __forceinline__ void weight_grad_chunk(const Problem& P, const Chunk& ch, const TableDev& td,
                                                  const void* grad_out, float* grad_w, int lane) {
    constexpr int E = Storage<DT>::kElems;
    constexpr int V = 32 / G;
    constexpr int U = V < 8 / VPL ? V : 8 / VPL;  // lookups per group whose rows are loaded together
    static_assert(VPL == 1 || G == 1, "several vectors per lane: one row per step");
    const int g = lane / V, v = lane - g * V;
    const int row_vecs = td.row_vecs;
    const uint32_t row_bytes = row_vecs * 16u;
    const uint32_t rows = static_cast<uint32_t>(td.rows);
    const int64_t k0 = ch.k0;
    const int32_t len = static_cast<int32_t>(ch.len & 0x7fffffffu);
    const int64_t bag_lo = static_cast<int64_t>(ch.table) * P.B, bag_hi = bag_lo + P.B;
    const int eb = dtype_bytes(P.out_dtype);
    const char* go_lane = static_cast<const char*>(grad_out) + (static_cast<int64_t>(td.doff) + v * E) * eb;
    const int64_t go_stride = static_cast<int64_t>(P.sum_d) * eb;
    const char* row_lane = static_cast<const char*>(td.data) + (v < row_vecs ? v : 0) * 16;
    BagWindow32 W = bag_window32(P, ch.first, bag_hi, k0, lane);
    float go[VPL][E];         // the group's bag's slice, this lane's columns
    int32_t held = -1;        // the bag
    int64_t r = lane < len ? load_index(P.indices, k0 + lane, P.is32) : -1;
    for (int32_t base = 0; base < len; base += 32) {
        const int32_t q = base + lane;
        const int64_t r_cur = r;
        r = q + 32 < len ? load_index(P.indices, k0 + q + 32, P.is32) : -1;  // the next batch's
        int64_t my_bag;
        int32_t my_s = 0, my_e = 0;
        if (!bags_by_mask(W, base, lane, P.mean, my_bag, my_s, my_e))
            find_bag32(P, W, bag_hi, k0, q, q < len, lane, my_bag, my_s, my_e);
        int32_t b_rel = 0;
        if (q < len) {
            if (my_bag >= bag_hi) {  // only reachable with malformed offsets
                set_error(P.error, CB_ERR_BAD_OFFSETS);
                my_bag = bag_hi - 1;
            }
            b_rel = static_cast<int32_t>(my_bag - bag_lo);
        }
        // An invalid lookup contributes nothing: it loads a valid one's row, and
        // its result is replaced by 0 below.
        const bool valid = static_cast<uint64_t>(r_cur) < rows;
        if (!valid && q < len) set_error(P.error, CB_ERR_INDEX_OOB);
        const uint32_t vm = __ballot_sync(kFull, valid);
        uint32_t my_a = static_cast<uint32_t>(r_cur);
        const uint32_t some = __shfl_sync(kFull, my_a, vm ? __ffs(vm) - 1 : 0);
        if (!valid) my_a = some;
        float mine = 0.f;
#pragma unroll 1
        for (int s0 = 0; vm != 0 && s0 < V && base + s0 < len; s0 += U) {
            uint4 x[U][VPL];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t a = __shfl_sync(kFull, my_a, g * V + s0 + u);
                const char* p = row_lane + static_cast<uint64_t>(a) * row_bytes;
#pragma unroll
                for (int k = 0; k < VPL; ++k)
                    x[u][k] = __ldg(reinterpret_cast<const uint4*>(p + (k > 0 && v + 32 * k < row_vecs ? 512 * k : 0)));
            }
            float dot[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int32_t bag = __shfl_sync(kFull, b_rel, g * V + s0 + u);
                if (bag != held) {
                    held = bag;
#pragma unroll
                    for (int k = 0; k < VPL; ++k)
                        if (v + 32 * k < row_vecs)
#pragma unroll
                            for (int c = 0; c < E; c += 4) {
                                const float4 f = load_go4(go_lane + held * go_stride + (32 * k * E + c) * eb, P.out_dtype);
                                go[k][c] = f.x;
                                go[k][c + 1] = f.y;
                                go[k][c + 2] = f.z;
                                go[k][c + 3] = f.w;
                            }
                }
                dot[u] = 0.f;
#pragma unroll
                for (int k = 0; k < VPL; ++k) {
                    float f[E];
                    unpack<DT>(x[u][k], f);
                    if (v + 32 * k < row_vecs)
#pragma unroll
                        for (int c = 0; c < E; ++c) dot[u] = fmaf(go[k][c], f[c], dot[u]);
                }
            }
            // The U sums over the group's V lanes: lane v ends with that of lookup v % U.
#pragma unroll
            for (int w = 1; w < U; w <<= 1) {
                // a lane keeps the sums whose number has its own bit w and adds its
                // partner's share of them
                const bool up = v & w;
#pragma unroll
                for (int i = 0; i < U; i += 2 * w)
                    dot[i] = (up ? dot[i + w] : dot[i]) + __shfl_xor_sync(kFull, up ? dot[i] : dot[i + w], w);
            }
            float z = dot[0];
#pragma unroll
            for (int off = U; off < V; off <<= 1) z += __shfl_xor_sync(kFull, z, off);
            if (v / U == s0 / U) mine = z;  // lookup g*V + v is this lane's own
        }
        if (q < len) {
            const float sc = (P.mean && my_e > my_s) ? 1.f / static_cast<float>(my_e - my_s) : 1.f;
            grad_w[k0 + q] = valid ? sc * mine : 0.f;
        }
    }
}

template <int DT, int VPL, int G>
__global__ void __launch_bounds__(kWarpThreads, VPL == 4 ? 2 : 4)
    weight_grad_kernel(const __grid_constant__ Problem P, const __grid_constant__ Plan Q, const void* grad_out,
                       float* grad_w, int cls) {
    begin_kernel();
    const int lane = threadIdx.x & 31;
    const int64_t cb = Q.class_chunk_base[cls];
    const int64_t ce = min64(Q.class_chunk_base[cls + 1], Q.max_chunks);
    for (int64_t j = first_chunk(Q, cls, cb, lane); j < ce;) {
        const int64_t nxt = fetch_next_chunk(Q, cls, cb, lane);
        const Chunk ch = Q.chunks[j];
        weight_grad_chunk<DT, VPL, G>(P, ch, P.tables[ch.table], grad_out, grad_w, lane);
        j = __shfl_sync(kFull, nxt, 0);
    }
}

template <auto Kernel>
void launch_one(const Problem& P, const Plan& Q, const void* go, float* gw, int cls, int64_t chunk_bound,
                int num_sms, cudaStream_t s) {
    static const int cap = resident_blocks(Kernel, kWarpThreads);
    launch(Kernel, warp_grid(chunk_bound, static_cast<int64_t>(cap) * num_sms), kWarpThreads, 0, s, P, Q, go, gw, cls);
}

template <int DT>
void launch_dtype(const Problem& P, const Plan& Q, const void* go, float* gw, int cls, int vpl, int gc,
                  int64_t chunk_bound, int num_sms, cudaStream_t s) {
#define CB_CASE(V, G)                                                                             \
    if (vpl == V && gc == G) {                                                                     \
        launch_one<weight_grad_kernel<DT, V, G>>(P, Q, go, gw, cls, chunk_bound, num_sms, s);       \
        return;                                                                                   \
    }
    CB_CASE(1, 1) CB_CASE(1, 2) CB_CASE(1, 4) CB_CASE(1, 8) CB_CASE(1, 16) CB_CASE(1, 32)
    CB_CASE(2, 1) CB_CASE(4, 1)
#undef CB_CASE
}

}  // namespace

void launch_weight_grad(const Problem& P, const Plan& Q, const void* grad_out, float* grad_w, int cls,
                        int dtype, int vpl, int gc, int64_t chunk_bound, int num_sms, cudaStream_t s) {
    if (dtype == CB_F32) launch_dtype<CB_F32>(P, Q, grad_out, grad_w, cls, vpl, gc, chunk_bound, num_sms, s);
    else if (dtype == CB_F16) launch_dtype<CB_F16>(P, Q, grad_out, grad_w, cls, vpl, gc, chunk_bound, num_sms, s);
    else launch_dtype<CB_BF16>(P, Q, grad_out, grad_w, cls, vpl, gc, chunk_bound, num_sms, s);
}

}  // namespace cbtbe
