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
// A block takes S samples (one, unless a sample has fewer vectors than a block has
// threads): R * nv threads per sample, thread (r, c) owning vector column c of
// fields r, r + R, ..., loaded together and held in registers; the R partial
// column sums meet in shared memory. So a sample is read once, with every load of
// the block in flight, whatever T and D (D / 4 need not divide anything); only
// samples of more than 16 fields per thread row are read in a loop, twice by the
// gradient. Sums are taken in a fixed order, so results are deterministic.
// Bound by HBM. Against a warp per sample (forward, and gradients whose vectors did
// not divide 256), us from a flushed L2, forward + gradient: 16384 samples x 26
// fields x 128: 54 + 76, now 48 + 70; 19881 x 23 x 96: 56 + 87, now 48 + 68;
// 60000 x 10 x 8: 21 + 203, now 21 + 17; 65536 x 100 x 128: 507 + 986, now 472 + 959
// (6.9 TB/s of compulsory bytes). One after the other, 16384 x 26 x 128: 118, now 107.
#include <cstdint>
#include <cuda_runtime.h>

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
