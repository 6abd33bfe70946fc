// Block-wide moments of a vector and what follows from them: CV^2 = population variance / mean^2 and its gradient
// 2/(m mu^2) ((v_i - mu) - Var/mu). Sums in double, in an order fixed by the block size.
#pragma once

#include "moe_internal.cuh"

namespace moe {

struct Moments { double mu, var; };

// sum over the block (whole warps) of one value per thread, returned to every thread; sh: 32 doubles
__device__ __forceinline__ double block_sum(double v, double *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __syncthreads();  // sh may still be read from an earlier call
    if (lane == 0) sh[w] = v;
    __syncthreads();
    v = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

__device__ __forceinline__ Moments block_moments(const float *v, int32_t m, double *sh) {
    double s = 0.0;
    for (int32_t i = threadIdx.x; i < m; i += blockDim.x) s += (double)__ldcg(v + i);
    const double mu = block_sum(s, sh) / m;
    double q = 0.0;
    for (int32_t i = threadIdx.x; i < m; i += blockDim.x) { double dv = (double)__ldcg(v + i) - mu; q += dv * dv; }
    Moments r;
    r.mu = mu;
    r.var = block_sum(q, sh) / m;
    return r;
}

// The two losses (Eq. 7, 11), by one block; `losses` and, if given, a second copy. One walk over both vectors and one reduction: sums of the
// distances to each vector's first element and of their squares (in double, the values are floats: var = E[(v - c)^2] - (E[v - c])^2
// loses nothing that the result holds). Mean and variance one after the other, vector by vector, were four reductions and four
// round trips to memory, 7 us of a 16 us kernel.
__device__ __forceinline__ void cv2_block(const float *importance, int32_t n_imp, const float *load, int32_t n_load, float w_imp,
                                          float w_load, float *losses, float *losses2, double *sh /* [32] */) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, warps = blockDim.x >> 5;  // at most eight warps
    const double c0 = (double)__ldcg(importance), c1 = (double)__ldcg(load);
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int32_t i = threadIdx.x; i < max(n_imp, n_load); i += blockDim.x) {
        const double a = i < n_imp ? (double)__ldcg(importance + i) - c0 : 0.0, b = i < n_load ? (double)__ldcg(load + i) - c1 : 0.0;
        s[0] += a; s[1] += a * a; s[2] += b; s[3] += b * b;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] += __shfl_xor_sync(0xffffffffu, s[q], off);
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) sh[4 * w + q] = s[q];
    __syncthreads();
    if (threadIdx.x < 2) {  // thread 0: Importance, thread 1: Load
        const int t = threadIdx.x;
        double s1 = 0.0, s2 = 0.0;
        for (int q = 0; q < warps; ++q) { s1 += sh[4 * q + 2 * t]; s2 += sh[4 * q + 2 * t + 1]; }
        const double m = t ? n_load : n_imp, mean = s1 / m, mu = (t ? c1 : c0) + mean;
        double var = s2 / m - mean * mean;
        if (var < 0.0) var = 0.0;  // rounding; a NaN (of an infinite element) stays one, as in the gradient
        const float l = (float)((double)(t ? w_load : w_imp) * var / (mu * mu));
        losses[t] = l;
        if (losses2) losses2[t] = l;
    }
}

// out[i] = scale * dCV^2/dv_i
__device__ __forceinline__ void cv2_grad_block(const Cv2Job &job, double *sh) {
    const Moments a = block_moments(job.v, job.m, sh);
    const double c = 2.0 / ((double)job.m * a.mu * a.mu);
    for (int32_t i = threadIdx.x; i < job.m; i += blockDim.x)
        job.out[i] = (float)((double)job.scale * c * (((double)job.v[i] - a.mu) - a.var / a.mu));
}

}  // namespace moe
