// Block-wide moments of a vector and what follows from them: CV^2 = population variance / mean^2 and its gradient
// 2/(m mu^2) ((v_i - mu) - Var/mu). Sums in double, in an order fixed by the block size.
#pragma once

#include "moe_internal.cuh"

namespace moe {

struct Moments { double mu, var; };

// sh: blockDim.x doubles (a power of two)
__device__ __forceinline__ Moments block_moments(const float *v, int32_t m, double *sh) {
    double s = 0.0;
    for (int32_t i = threadIdx.x; i < m; i += blockDim.x) s += (double)__ldcg(v + i);
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
        __syncthreads();
    }
    const double mu = sh[0] / m;
    __syncthreads();
    double q = 0.0;
    for (int32_t i = threadIdx.x; i < m; i += blockDim.x) { double dv = (double)__ldcg(v + i) - mu; q += dv * dv; }
    sh[threadIdx.x] = q;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
        __syncthreads();
    }
    Moments r;
    r.mu = mu;
    r.var = sh[0] / m;
    __syncthreads();
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
