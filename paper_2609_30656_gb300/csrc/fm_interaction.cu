// fm_interaction.cu -- the factorization-machine cross term on the pooled
// embeddings and its gradient: the inter_arch.fm step that follows the
// lookups in the paper's DeepFM-based model (Sec. IV.A.2, where it is
// bandwidth-bound: a few element-wise and reduction passes over the pooled
// rows). With each table's pooled row as one field embedding,
// v_bt = y[b, t*D : (t+1)*D], the second-order term of the factorization
// machine (Rendle, 2010, cited by the paper) is
//
//   fm[b] = sum_{t < u} <v_bt, v_bu> = 1/2 sum_j [(sum_t v_btj)^2 - sum_t v_btj^2]
//
// and, for an upstream gradient g[b],
//
//   grad_y[b, t*D + j] = g[b] * (sum_u v_buj - v_btj).
//
// A warp takes a sample, or a block takes S of them (fm_by_warp says which; one,
// unless a sample has fewer vectors than a block has threads): R * nv threads per
// sample, thread (r, c) owning vector column c of fields r, r + R, ..., loaded together
// and held in registers; the R partial column sums meet in shared memory. So a sample is
// read once, with all its loads in flight, whatever T and D (D / 4 need not divide
// anything); only a block's samples of more than 16 fields per thread row are read in a
// loop, twice by the gradient. Sums are taken in a fixed order, so results are
// deterministic. Bound by HBM. From a flushed L2, us, forward + gradient, with a warp per
// sample that read in a loop, and now: 16384 samples x 26 fields x 128: 54 + 76, now 48 +
// 70; 60000 x 10 x 8: 21 + 203, now 21 + 17; 65536 x 100 x 128: 507 + 986, now 472 + 959
// (6.9 TB/s of compulsory bytes).
#include <cstdint>
#include <cuda_runtime.h>
#include <type_traits>

#include "cb_tbe.h"
#include "tbe_internal.cuh"

namespace cbtbe {
namespace {

constexpr int kFmThreads = 256;
constexpr int kFmFields = 16;  // fields per thread held in registers

__device__ __forceinline__ void add4(float4& a, const float4& x) {
    a.x += x.x;
    a.y += x.y;
    a.z += x.z;
    a.w += x.w;
}
__device__ __forceinline__ void fma4(float4& a, const float4& x) {
    a.x = fmaf(x.x, x.x, a.x);
    a.y = fmaf(x.y, x.y, a.y);
    a.z = fmaf(x.z, x.z, a.z);
    a.w = fmaf(x.w, x.w, a.w);
}

__device__ __forceinline__ float4 shfl_xor4(const float4& a, int off) {
    return make_float4(__shfl_xor_sync(kFull, a.x, off), __shfl_xor_sync(kFull, a.y, off),
                       __shfl_xor_sync(kFull, a.z, off), __shfl_xor_sync(kFull, a.w, off));
}

// The R partial sums of a column (part[c], part[c + nv], ...): up to kDirect of
// them are added by whoever needs the total; more meet in a tree first, in which
// `part` and `part2` (unless null) of thread (r, c) take those of (r + half, c).
constexpr int kDirect = 16;
__device__ __forceinline__ void tree_sum(float4* part, float4* part2, int r, int nv, int R) {
    int half = 1;
    while (half < R) half <<= 1;
    for (half >>= 1; half >= 1; half >>= 1) {
        if (r < half && r + half < R) {
            add4(part[0], part[half * nv]);
            if (part2) add4(part2[0], part2[half * nv]);
        }
        __syncthreads();
    }
}
__device__ __forceinline__ float4 column_total(const float4* part, int nv, int R) {
    float4 S = part[0];
#pragma unroll 1
    for (int q = 1; q < R; ++q) add4(S, part[q * nv]);
    return S;
}

struct FmShape {
    int B, T, nv;    // samples, fields, 16-byte vectors per field
    int R, per, S;   // thread rows per sample, threads per sample (R * nv), samples per block
    int64_t stride;  // floats from one sample to the next
};

// K > 0: up to K fields per thread, in registers. K = 0: any number, in a loop.
// The gradient takes the samples from the last to the first: after a forward pass
// the last ones are what L2 still holds.
template <int K, bool BACKWARD>
__global__ void __launch_bounds__(kFmThreads, K == 16 ? 2 : (K == 8 ? 4 : (K == 4 ? 6 : 8)))
    fm_kernel(const float* __restrict__ y, const float* __restrict__ grad_fm, const FmShape f,
              float* __restrict__ out) {
    __shared__ float4 sum[kFmThreads], sq[BACKWARD ? 1 : kFmThreads];
    begin_kernel();
    const int i = threadIdx.x;
    const int slot = i / f.per, w = i - slot * f.per, r = w / f.nv, c = w - r * f.nv;
    const int64_t b0 = static_cast<int64_t>(blockIdx.x) * f.S + slot;
    const bool live = slot < f.S && b0 < f.B;
    const int64_t b = !live ? 0 : (BACKWARD ? f.B - 1 - b0 : b0);
    const float4* row = reinterpret_cast<const float4*>(y + b * f.stride) + c;
    constexpr int kHeld = K > 0 ? K : 1;
    float4 x[kHeld];
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f), q = s;
    if constexpr (K > 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int t = r + k * f.R;
            x[k] = live && t < f.T ? __ldg(row + static_cast<int64_t>(t) * f.nv) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            add4(s, x[k]);
            if (!BACKWARD) fma4(q, x[k]);
        }
    } else if (live) {
#pragma unroll 8
        for (int t = r; t < f.T; t += f.R) {
            const float4 z = __ldg(row + static_cast<int64_t>(t) * f.nv);
            add4(s, z);
            if (!BACKWARD) fma4(q, z);
        }
    }
    sum[i] = s;
    if (!BACKWARD) sq[i] = q;
    __syncthreads();
    const int left = f.R > kDirect ? 1 : f.R;
    if (left == 1) tree_sum(sum + i, BACKWARD ? nullptr : sq + i, live ? r : f.R, f.nv, f.R);
    if constexpr (!BACKWARD) {
        // thread (0, c): its column's S^2 - Q; then a warp per sample adds the columns
        __shared__ float cols[kFmThreads];
        if (live && r == 0) {
            const float4 S = column_total(sum + i, f.nv, left), Q = column_total(sq + i, f.nv, left);
            cols[slot * f.nv + c] = (fmaf(S.x, S.x, -Q.x) + fmaf(S.y, S.y, -Q.y)) +
                                    (fmaf(S.z, S.z, -Q.z) + fmaf(S.w, S.w, -Q.w));
        }
        __syncthreads();
        const int lane = i & 31;
        for (int k = i >> 5; k < f.S; k += blockDim.x >> 5) {
            const int64_t bk = static_cast<int64_t>(blockIdx.x) * f.S + k;
            if (bk >= f.B) break;
            float part = 0.f;
            for (int j = lane; j < f.nv; j += 32) part += cols[k * f.nv + j];
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
            if (lane == 0) out[bk] = 0.5f * part;
        }
    } else if (live) {
        const float4 S = column_total(sum + slot * f.per + c, f.nv, left);
        const float g = __ldg(grad_fm + b);
        float4* dst = reinterpret_cast<float4*>(out + b * f.stride) + c;
        auto put = [&](int t, const float4& z) {
            __stcs(dst + static_cast<int64_t>(t) * f.nv,
                   make_float4(g * (S.x - z.x), g * (S.y - z.y), g * (S.z - z.z), g * (S.w - z.w)));
        };
        if constexpr (K > 0) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (r + k * f.R < f.T) put(r + k * f.R, x[k]);
        } else {
#pragma unroll 4
            for (int t = r; t < f.T; t += f.R) put(t, row[static_cast<int64_t>(t) * f.nv]);
        }
    }
}

// A warp per sample: V lanes per field (a power of two that holds it, at most 32),
// G = 32 / V fields at a time, K steps of one vector a lane, all loaded together. A field
// of more than 32 vectors takes M steps, of which a lane's sums keep their own. The
// gradient holds the sample; a forward of more steps takes them K at a time (LOOP). No
// shared memory and no barrier, so the warps' loads and stores overlap freely.
struct FmWarp {
    int B, T, nv, V;
    int64_t stride;
};

template <int K, int M, bool BACKWARD, bool LOOP = false>
__global__ void __launch_bounds__(kFmThreads)
    fm_warp_kernel(const float* __restrict__ y, const float* __restrict__ grad_fm, const FmWarp f,
                   float* __restrict__ out) {
    static_assert(K % M == 0 && (!LOOP || (K / M & (K / M - 1)) == 0), "whole fields; a loop adds them by halves");
    begin_kernel();
    const int lane = threadIdx.x & 31;
    const int g = lane / f.V, c = lane & (f.V - 1), G = 32 / f.V;
    const int64_t b0 = warp_id_global();
    if (b0 >= f.B) return;
    // the gradient from the last sample to the first, as the block's
    const int64_t b = BACKWARD ? f.B - 1 - b0 : b0;
    const int64_t at = b * f.stride + 4 * (static_cast<int64_t>(g) * f.nv + c);
    const float4* row = reinterpret_cast<const float4*>(y + at);
    float4 x[K], s[M], q[M];
#pragma unroll
    for (int m = 0; m < M; ++m) s[m] = q[m] = make_float4(0.f, 0.f, 0.f, 0.f);
    int t0 = g;
    do {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int t = t0 + k / M * G, col = c + 32 * (k % M);
            x[k] = t < f.T && col < f.nv ? __ldg(row + static_cast<int64_t>(k / M * G) * f.nv + 32 * (k % M))
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (!LOOP) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                add4(s[k % M], x[k]);
                if (!BACKWARD) fma4(q[k % M], x[k]);
            }
            break;
        }
        // A round's values by halves, in place (shorter chains of adds than one by one, so
        // smaller rounding errors): the even ones become sums, the odd ones of squares.
        constexpr int N = K / M;
#pragma unroll
        for (int m = 0; m < M; ++m) {
#pragma unroll
            for (int i = 0; i < N; i += 2) {
                float4 &a = x[i * M + m], &b = x[(i + 1) % N * M + m];
                float4 sq = make_float4(a.x * a.x, a.y * a.y, a.z * a.z, a.w * a.w);
                fma4(sq, b);
                add4(a, b);
                b = sq;
            }
#pragma unroll
            for (int w = 2; w < N; w *= 2)
#pragma unroll
                for (int i = 0; i < N; i += 2 * w) {
                    add4(x[i * M + m], x[(i + w) * M + m]);
                    add4(x[(i + 1) * M + m], x[(i + w + 1) * M + m]);
                }
            add4(s[m], x[m]);
            add4(q[m], x[M % K + m]);
        }
        t0 += N * G;
        row += static_cast<int64_t>(N * G) * f.nv;
    } while (t0 < f.T);
    for (int off = f.V; off < 32; off <<= 1)
#pragma unroll
        for (int m = 0; m < M; ++m) {
            add4(s[m], shfl_xor4(s[m], off));
            if (!BACKWARD) add4(q[m], shfl_xor4(q[m], off));
        }
    if constexpr (!BACKWARD) {
        float part = 0.f;
        if (g == 0)
#pragma unroll
            for (int m = 0; m < M; ++m)
                part += (fmaf(s[m].x, s[m].x, -q[m].x) + fmaf(s[m].y, s[m].y, -q[m].y)) +
                        (fmaf(s[m].z, s[m].z, -q[m].z) + fmaf(s[m].w, s[m].w, -q[m].w));
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) part += __shfl_xor_sync(kFull, part, off);
        if (lane == 0) out[b] = 0.5f * part;
    } else {
        const float w = __ldg(grad_fm + b);
        float4* dst = reinterpret_cast<float4*>(out + at);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int t = g + k / M * G, col = c + 32 * (k % M);
            if (t < f.T && col < f.nv)
                __stcs(dst + static_cast<int64_t>(k / M * G) * f.nv + 32 * (k % M),
                       make_float4(w * (s[k % M].x - x[k].x), w * (s[k % M].y - x[k].y), w * (s[k % M].z - x[k].z),
                                   w * (s[k % M].w - x[k].w)));
        }
    }
}

// The steps that a warp takes over a sample, M for each G fields.
struct FmSteps {
    int V, M;
    int64_t steps;
    FmSteps(int T, int nv) {
        V = 1;
        while (V < nv && V < 32) V *= 2;
        M = (nv + 31) / 32;
        steps = (static_cast<int64_t>(T) + 32 / V - 1) / (32 / V) * M;
    }
};

// Steps at a time in the loop. (64 MB of y, forward of 26 fields x 192, with the adds one
// by one: 10.6 us, at 4 steps 14.5, at 12 12.0; by halves 12.7.)
constexpr int kFmLoop = 8;
constexpr int64_t kL2Bytes = int64_t(128) << 20;

// Whether a warp takes a sample, or a block. The block has the samples of a few vectors,
// several at a time, and those of many steps; also of many in a batch too small to give
// every SM's warps one, and of many vectors in one larger than L2. Block and warp, us, y
// of 20 to 64 MB (read from L2), fields x dim. Forward: 10 x 4 (10 vectors) 24.9, 32.4;
// 2 x 32 (16) 23.2, 25.5; 10 x 8 (20) 36.8, 30.2; 16 x 64 (8 steps) 33.6, 10.2; 40 x 64
// (20) 17.6, 9.5; 40 x 96 (40) 12.5, 11.1; 100 x 128 (100) 11.0, 13.1. From HBM (256 MB):
// 26 x 96 (624 vectors) 56.1, 45.9; 26 x 128 (832) 44.7, 45.3; 40 x 256 (2560) 44.1, 52.4.
// Gradient from L2: 16 x 4 (16 vectors) 22.2, 26.1; 10 x 8 (20) 24.1, 24.8; 3 x 32 (24)
// 23.8, 23.1; 16 x 64 43.5, 20.1. (A warp per sample that read in a loop took 14.8 for the
// forward of 100 x 8, the block 43.4; now 12.6.)
bool fm_by_warp(int64_t vectors, int64_t steps, int batch, bool backward) {
    if (vectors < (backward ? 21 : 16)) return false;
    if (steps <= 16) return true;
    const bool from_hbm = 16 * vectors * batch > kL2Bytes;
    return !backward && steps <= 48 && batch >= 1024 && !(from_hbm && vectors >= 768);
}

template <int M, bool BACKWARD>
void launch_fm_warp(const float* y, const float* grad_fm, const FmWarp& f, int64_t steps, float* out, cudaStream_t s) {
    const unsigned grid = static_cast<unsigned>((static_cast<int64_t>(f.B) + kFmThreads / 32 - 1) / (kFmThreads / 32));
    constexpr int K = 16 / M * M;  // 16, 16, 15, 16
    if constexpr (!BACKWARD)
        if (steps > K) {
            launch(fm_warp_kernel<kFmLoop / M * M, M, false, true>, grid, kFmThreads, 0, s, y, grad_fm, f, out);
            return;
        }
    auto go = [&](auto fields) {
        constexpr int N = decltype(fields)::value;  // steps per M
        launch(fm_warp_kernel<N * M, M, BACKWARD>, grid, kFmThreads, 0, s, y, grad_fm, f, out);
    };
    if (steps <= 2 * M) go(std::integral_constant<int, 2>{});
    else if (steps <= 4 * M) go(std::integral_constant<int, K / M < 4 ? K / M : 4>{});
    else if (steps <= 8 * M) go(std::integral_constant<int, K / M < 8 ? K / M : 8>{});
    else go(std::integral_constant<int, K / M>{});
}

template <bool BACKWARD>
void launch_fm(const float* y, const float* grad_fm, const FmShape& f, float* out, cudaStream_t s) {
    const unsigned grid = static_cast<unsigned>((f.B + f.S - 1) / f.S);
    const int threads = (f.per * f.S + 31) / 32 * 32;
    const int k = (f.T + f.R - 1) / f.R;
    if (k <= 2) launch(fm_kernel<2, BACKWARD>, grid, threads, 0, s, y, grad_fm, f, out);
    else if (k <= 4) launch(fm_kernel<4, BACKWARD>, grid, threads, 0, s, y, grad_fm, f, out);
    else if (k <= 8) launch(fm_kernel<8, BACKWARD>, grid, threads, 0, s, y, grad_fm, f, out);
    else if (k <= kFmFields) launch(fm_kernel<kFmFields, BACKWARD>, grid, threads, 0, s, y, grad_fm, f, out);
    else launch(fm_kernel<0, BACKWARD>, grid, threads, 0, s, y, grad_fm, f, out);
}

cb_status fm_call(bool backward, const float* y, const float* grad_fm, int32_t batch, int32_t num_fields,
                  int32_t dim, int64_t row_stride, float* out, cudaStream_t stream) {
    if (batch < 0 || num_fields < 1 || dim < 4 || dim > 512 || (dim & 3) ||
        row_stride < static_cast<int64_t>(num_fields) * dim || (row_stride & 3))
        return CB_ERR_INVALID_ARG;
    if (batch > 0 && (!y || !out || (backward && !grad_fm))) return CB_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(y) & 15u) || (backward && (reinterpret_cast<uintptr_t>(out) & 15u)))
        return CB_ERR_INVALID_ARG;
    if (batch == 0) return CB_OK;
    cudaGetLastError();  // an earlier, unrelated failure is not this call's
    const FmSteps w(num_fields, dim / 4);
    if (fm_by_warp(static_cast<int64_t>(num_fields) * (dim / 4), w.steps, batch, backward)) {
        const FmWarp f{batch, num_fields, dim / 4, w.V, row_stride};
        auto go = [&](auto back) {
            constexpr bool kBack = decltype(back)::value;
            if (w.M == 1) launch_fm_warp<1, kBack>(y, grad_fm, f, w.steps, out, stream);
            else if (w.M == 2) launch_fm_warp<2, kBack>(y, grad_fm, f, w.steps, out, stream);
            else if (w.M == 3) launch_fm_warp<3, kBack>(y, grad_fm, f, w.steps, out, stream);
            else launch_fm_warp<4, kBack>(y, grad_fm, f, w.steps, out, stream);
        };
        if (backward) go(std::true_type{});
        else go(std::false_type{});
        return cudaGetLastError() == cudaSuccess ? CB_OK : CB_ERR_CUDA;
    }
    FmShape f;
    f.B = batch;
    f.T = num_fields;
    f.nv = dim / 4;
    f.R = kFmThreads / f.nv < num_fields ? kFmThreads / f.nv : num_fields;
    f.per = f.R * f.nv;
    f.S = kFmThreads / f.per;
    f.stride = row_stride;
    if (backward) launch_fm<true>(y, grad_fm, f, out, stream);
    else launch_fm<false>(y, grad_fm, f, out, stream);
    return cudaGetLastError() == cudaSuccess ? CB_OK : CB_ERR_CUDA;
}

}  // namespace
}  // namespace cbtbe

extern "C" cb_status cb_fm_forward(const float* y, int32_t batch, int32_t num_fields, int32_t dim,
                                   int64_t row_stride, float* out, cudaStream_t stream) {
    return cbtbe::fm_call(false, y, nullptr, batch, num_fields, dim, row_stride, out, stream);
}

extern "C" cb_status cb_fm_backward(const float* y, const float* grad_fm, int32_t batch,
                                    int32_t num_fields, int32_t dim, int64_t row_stride, float* grad_y,
                                    cudaStream_t stream) {
    return cbtbe::fm_call(true, y, grad_fm, batch, num_fields, dim, row_stride, grad_y, stream);
}
