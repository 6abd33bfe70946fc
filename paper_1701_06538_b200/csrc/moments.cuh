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

// out[i] = scale * dCV^2/dv_i
__device__ __forceinline__ void cv2_grad_block(const Cv2Job &job, double *sh) {
    const Moments a = block_moments(job.v, job.m, sh);
    const double c = 2.0 / ((double)job.m * a.mu * a.mu);
    for (int32_t i = threadIdx.x; i < job.m; i += blockDim.x)
        job.out[i] = (float)((double)job.scale * c * (((double)job.v[i] - a.mu) - a.var / a.mu));
}

}  // namespace moe
