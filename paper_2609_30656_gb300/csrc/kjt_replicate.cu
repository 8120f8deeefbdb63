// kjt_replicate.cu -- the batch-size preprocessor of Component Benchmark
// (Sec. III): a small captured batch of jagged lookups is replicated to the
// production batch size, which keeps the input distribution the lookup sees.
// For T tables and a key-major batch of B bags per table, the output has
// F * B bags per table, and bag r * B + b of table t is bag b of table t:
//
//   out_offsets[t*F*B + r*B + b] = F * off[t*B] + r * n_t + (off[t*B + b] - off[t*B])
//   out_indices[F * off[t*B] + r * n_t + i] = indices[off[t*B] + i]   (i < n_t)
//
// with n_t = off[(t+1)*B] - off[t*B]. One kernel: some blocks take bags, the others
// lookups; a thread reads its bag or lookup once and writes it F times (or, in
// a small call, the copies its block was given), neighbours to neighbouring
// places. A lookup's table is found once, by bisection over the table starts, held
// in shared memory up to kTables of them. Offsets are clamped into [0, n] and made
// monotone per table first, so any input stays in bounds. Bound by the writes:
// 553 K lookups with weights in 26 tables, 16 times (106 MB written): 83 -> 25 us
// (a bisection and a 64-bit modulo for every output lookup, before).
#include <cstdint>
#include <cuda_runtime.h>

#include "cb_tbe.h"
#include "tbe_internal.cuh"

namespace cbtbe {
namespace {

template <typename I>
__device__ __forceinline__ int64_t off_at(const I* off, int64_t k, int64_t n) {
    const int64_t v = static_cast<int64_t>(off[k]);
    return v < 0 ? 0 : (v > n ? n : v);
}

constexpr int kThreads = 256;
constexpr int kTables = 2048;  // table starts held in shared memory

template <typename I>
struct Replicate {
    const I* ind;
    const I* off;
    const float* w;
    I* out_ind;
    I* out_off;
    float* out_w;
    int64_t n;
    int32_t T, B, F;
    int32_t bag_blocks;    // blocks that take bags; the others take lookups
    int32_t parts;         // copies are split over this many blocks (blockIdx.y)
};

template <typename I>
__global__ void __launch_bounds__(kThreads) replicate_kernel(const Replicate<I> p) {
    __shared__ I starts[kTables + 1];
    begin_kernel();
    // this block's copies [r0, r1), in 64 bits: F may be as large as a 32-bit number gets
    const int64_t per_part = (static_cast<int64_t>(p.F) + p.parts - 1) / p.parts;
    const int r0 = static_cast<int>(min64(blockIdx.y * per_part, p.F));
    const int r1 = static_cast<int>(min64(r0 + per_part, p.F));
    if (static_cast<int>(blockIdx.x) < p.bag_blocks) {
        const int64_t bags = static_cast<int64_t>(p.T) * p.B;
        const int64_t k = static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x;
        if (k > bags) return;
        if (k == bags) {
            if (blockIdx.y == 0) p.out_off[bags * p.F] = static_cast<I>(p.F * off_at(p.off, bags, p.n));
            return;
        }
        const int64_t t = k / p.B, b = k - t * p.B;
        const int64_t s = off_at(p.off, t * p.B, p.n);
        const int64_t e0 = off_at(p.off, (t + 1) * p.B, p.n);
        const int64_t e = e0 < s ? s : e0;
        int64_t o = off_at(p.off, k, p.n);
        o = o < s ? s : (o > e ? e : o);
        I* out = p.out_off + t * p.F * p.B + b;
        for (int r = r0; r < r1; ++r)
            out[static_cast<int64_t>(r) * p.B] = static_cast<I>(p.F * s + r * (e - s) + (o - s));
        return;
    }
    const bool held = p.T <= kTables;
    if (held) {
        for (int t = threadIdx.x; t <= p.T; t += kThreads)
            starts[t] = static_cast<I>(off_at(p.off, static_cast<int64_t>(t) * p.B, p.n));
        __syncthreads();
    }
    auto start = [&](int t) -> int64_t {
        return held ? static_cast<int64_t>(starts[t]) : off_at(p.off, static_cast<int64_t>(t) * p.B, p.n);
    };
    const int64_t i = (static_cast<int64_t>(blockIdx.x) - p.bag_blocks) * kThreads + threadIdx.x;
    if (i >= p.n) return;
    const I value = p.ind[i];
    const float weight = p.w ? p.w[i] : 0.f;
    int lo = 0, hi = p.T;  // largest t with start(t) <= i
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (start(mid) <= i) lo = mid;
        else hi = mid;
    }
    const int64_t s = start(lo), nt = start(lo + 1) - s;
    if (i < s || i - s >= nt) return;  // past the last bag (or bad offsets)
    const int64_t first = p.F * s + (i - s);
#pragma unroll 4
    for (int r = r0; r < r1; ++r) {
        p.out_ind[first + r * nt] = value;
        if (p.w) p.out_w[first + r * nt] = weight;
    }
}

template <typename I>
void replicate(const void* ind, const void* off, const float* w, int32_t T, int32_t B, int64_t n, int32_t F,
            void* out_ind, void* out_off, float* out_w, cudaStream_t s) {
    Replicate<I> p{static_cast<const I*>(ind), static_cast<const I*>(off), w, static_cast<I*>(out_ind),
                   static_cast<I*>(out_off), out_w, n, T, B, F, 0, 1};
    const int64_t bags = static_cast<int64_t>(T) * B + 1;
    p.bag_blocks = static_cast<int32_t>((bags + kThreads - 1) / kThreads);
    const int64_t blocks = p.bag_blocks + (n + kThreads - 1) / kThreads;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // a call too small to fill the GPU splits the copies over blocks too
    const int64_t want = 8 * static_cast<int64_t>(sms > 0 ? sms : 1) / blocks;
    p.parts = static_cast<int32_t>(want < 1 ? 1 : (want < F ? want : F));
    if (p.parts > 65535) p.parts = 65535;
    cbtbe::launch(replicate_kernel<I>, dim3(static_cast<unsigned>(blocks), static_cast<unsigned>(p.parts)), kThreads, 0,
                  s, p);
}

}  // namespace
}  // namespace cbtbe

extern "C" cb_status cb_kjt_replicate(const void* indices, const void* offsets, const float* per_sample_weights,
                                      cb_index_dtype idx_dtype, int32_t num_tables, int32_t batch,
                                      int64_t num_indices, int32_t factor, void* out_indices,
                                      void* out_offsets, float* out_weights, cudaStream_t stream) {
    if (num_tables < 1 || batch < 0 || num_indices < 0 || factor < 1 || !offsets || !out_offsets)
        return CB_ERR_INVALID_ARG;
    if (idx_dtype != CB_I32 && idx_dtype != CB_I64) return CB_ERR_INVALID_ARG;
    if (num_indices > 0 && (!indices || !out_indices)) return CB_ERR_INVALID_ARG;
    if (per_sample_weights && num_indices > 0 && !out_weights) return CB_ERR_INVALID_ARG;
    const int64_t nn = static_cast<int64_t>(factor) * num_indices;
    const int64_t bags = static_cast<int64_t>(num_tables) * factor * batch;
    if (bags >= (int64_t(1) << 31) || (idx_dtype == CB_I32 && nn > INT32_MAX)) return CB_ERR_INVALID_ARG;
    cudaGetLastError();
    if (idx_dtype == CB_I64)
        cbtbe::replicate<long long>(indices, offsets, per_sample_weights, num_tables, batch, num_indices, factor,
                                 out_indices, out_offsets, out_weights, stream);
    else
        cbtbe::replicate<int>(indices, offsets, per_sample_weights, num_tables, batch, num_indices, factor,
                           out_indices, out_offsets, out_weights, stream);
    return cudaGetLastError() == cudaSuccess ? CB_OK : CB_ERR_CUDA;
}
