// Balancing losses (Section 4 and Appendix A): Importance (Eq. 6), the smooth load estimator
// P(x, i) (Eq. 9), Load (Eq. 10), the two CV^2 losses (Eq. 7, 11) and their gradients.
// Batch sums are deterministic: per-chunk partial sums in float, then one ordered pass in double.
#include <math_constants.h>

#include "moe_internal.cuh"
#include "moments.cuh"

namespace moe {

constexpr int LCHUNKS_MAX = 148 * 4;

// a row per warp until the chip is full: the normal-CDF evaluations of a row are one long latency chain per lane. Up to 32
// columns one block adds up all chunks, and up to 16384 rows half as many are enough (8192 rows: 6 columns 12.0 us for both
// launches, with all chunks 15.2; 15000 rows of 30 columns 15.5, 17.9; but 60000 rows of 20 columns 28.4, 26.5)
static inline int32_t level_chunks(int64_t rows, int32_t n) {
    return (int32_t)imin(cdiv(rows, 8), n <= 32 && rows <= 16384 ? LCHUNKS_MAX / 2 : LCHUNKS_MAX);
}
int64_t losses_ws_floats(int64_t rows, int32_t n) { return 2 * (int64_t)level_chunks(rows, n) * n + 64; }

__device__ __forceinline__ float softplus_f(float r) { return fmaxf(r, 0.0f) + log1pf(expf(-fabsf(r))); }

// Thread (tl, cw): column lane cw in [0, CW), token lane tl in [0, 256/CW). A block owns a chunk of
// rows; for each of its columns a thread sums over its rows, the token lanes are then added in order.
__global__ void __launch_bounds__(256) level_sums_kernel(const int32_t *__restrict__ idx,
                                                         const float *__restrict__ gates,
                                                         const float *__restrict__ clean,
                                                         const float *__restrict__ raw,
                                                         const float *__restrict__ kth_vals, int64_t rows, int32_t n,
                                                         int32_t k, int32_t CW, float *__restrict__ part_imp,
                                                         float *__restrict__ part_load, int32_t *__restrict__ ticket) {
    wait_previous_kernel();
    if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0;  // of level_reduce_kernel
    __shared__ float red_i[256], red_l[256];
    const int cw = threadIdx.x % CW, tl = threadIdx.x / CW, TL = 256 / CW;
    const int64_t per = (rows + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = (int64_t)blockIdx.x * per, r1 = min(r0 + per, rows);
    for (int32_t jb = 0; jb < n; jb += CW) {
        const int32_t j = jb + cw;
        float s_imp = 0.0f, s_load = 0.0f;
        if (j < n) {
            for (int64_t t = r0 + tl; t < r1; t += TL) {
                bool sel = false;
                float g = 0.0f;
                for (int s = 0; s < k; ++s)
                    if (idx[t * k + s] == j) { sel = true; g = gates[t * k + s]; }
                const float thr = kth_vals[t * 2 + (sel ? 1 : 0)];  // kth_excluding(H, k, j)
                const float z = (clean[t * n + j] - thr) / softplus_f(raw[t * n + j]);
                s_load += 0.5f * erfcf(-z * 0.70710678118654752440f);  // Phi(z)
                s_imp += g;
            }
        }
        red_i[threadIdx.x] = s_imp;
        red_l[threadIdx.x] = s_load;
        __syncthreads();
        if (tl == 0 && j < n) {
            float a = 0.0f, b = 0.0f;
            for (int q = 0; q < TL; ++q) { a += red_i[q * CW + cw]; b += red_l[q * CW + cw]; }
            part_imp[(int64_t)blockIdx.x * n + j] = a;
            part_load[(int64_t)blockIdx.x * n + j] = b;
        }
        __syncthreads();
    }
}

// Same sums with one warp per row and the lanes across the columns (n <= 32 * NV): all loads of a row are
// issued first, a lane accumulates its columns over the rows of its warp, the block's 8 warps are then added
// in order through shared memory.
template <int NV>
__global__ void __launch_bounds__(256) level_sums_rows_kernel(const int32_t *__restrict__ idx,
                                                              const float *__restrict__ gates,
                                                              const float *__restrict__ clean,
                                                              const float *__restrict__ raw,
                                                              const float *__restrict__ kth_vals, int64_t rows,
                                                              int32_t n, int32_t k, float *__restrict__ part_imp,
                                                              float *__restrict__ part_load, int32_t *__restrict__ ticket) {
    wait_previous_kernel();
    if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0;  // of level_reduce_kernel
    __shared__ float red[2][8][32 * NV];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t per = (rows + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = (int64_t)blockIdx.x * per, r1 = min(r0 + per, rows);
    float s_imp[NV], s_load[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) s_imp[u] = s_load[u] = 0.0f;
    for (int64_t t = r0 + w; t < r1; t += 8) {
        float cv[NV], rv[NV];
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int32_t j = lane + 32 * u;
            cv[u] = j < n ? clean[t * n + j] : 0.0f;
            rv[u] = j < n ? raw[t * n + j] : 0.0f;
        }
        // the row's kept experts: bit u of `kept` = this lane's column lane + 32 u is one of them (its gate goes to
        // the Importance sum); an expert id outside [0, n) belongs to no lane
        uint32_t kept = 0u;
        for (int s = 0; s < k; ++s) {
            const int32_t e = idx[t * k + s];
            const float g = gates[t * k + s];
            if ((e & 31) == lane && (uint32_t)e < (uint32_t)n) {
#pragma unroll
                for (int u = 0; u < NV; ++u)
                    if ((e >> 5) == u) { kept |= 1u << u; s_imp[u] += g; }
            }
        }
        const float thr_unsel = kth_vals[t * 2 + 0], thr_sel = kth_vals[t * 2 + 1];
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int32_t j = lane + 32 * u;
            if (j < n) {
                // (the quotient may be off by two units in the last place: 1e-7 of z, far below what Load is held to)
                const float z = __fdividef(cv[u] - (((kept >> u) & 1u) ? thr_sel : thr_unsel), softplus_f(rv[u]));
                s_load[u] += 0.5f * erfcf(-z * 0.70710678118654752440f);  // Phi(z)
            }
        }
    }
#pragma unroll
    for (int u = 0; u < NV; ++u) { red[0][w][lane + 32 * u] = s_imp[u]; red[1][w][lane + 32 * u] = s_load[u]; }
    __syncthreads();
    for (int32_t j = threadIdx.x; j < n; j += 256) {
        float a = 0.0f, b = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) { a += red[0][q][j]; b += red[1][q][j]; }
        part_imp[(int64_t)blockIdx.x * n + j] = a;
        part_load[(int64_t)blockIdx.x * n + j] = b;
    }
}

// Importance / Load = the blocks' partial sums added in double. A block takes 32 columns; its eight warps each add an
// eighth of the chunks (in ascending order, ten loads in flight), the eight sums are then added in warp order. With
// fin.losses set, the block that finishes last (counted by `ticket`) also forms the two losses from the complete vectors,
// and the copies in fin.copy are written along the way.
__global__ void __launch_bounds__(256) level_reduce_kernel(const float *__restrict__ part_imp,
                                                           const float *__restrict__ part_load, int32_t chunks,
                                                           int32_t n, float *importance, float *load,
                                                           const LossFinal fin, int32_t *ticket) {
    wait_previous_kernel();
    __shared__ double red[2][8][32];
    __shared__ double sh[32];
    __shared__ int last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t j = blockIdx.x * 32 + lane;
    const int32_t per = (chunks + 7) / 8, c0 = w * per, c1 = min(c0 + per, chunks);
    double a = 0.0, b = 0.0;
    if (j < n) {
        for (int32_t c = c0; c < c1; c += 10) {
            float pa[10], pb[10];
#pragma unroll
            for (int q = 0; q < 10; ++q) {
                pa[q] = c + q < c1 ? part_imp[(int64_t)(c + q) * n + j] : 0.0f;
                pb[q] = c + q < c1 ? part_load[(int64_t)(c + q) * n + j] : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < 10; ++q) { a += (double)pa[q]; b += (double)pb[q]; }
        }
    }
    red[0][w][lane] = a;
    red[1][w][lane] = b;
    __syncthreads();
    if (w < 2 && j < n) {  // warp 0: Importance, warp 1: Load
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) s += red[w][q][lane];
        float *out = w ? load : importance, *copy = w ? fin.copy.load : fin.copy.importance;
        if (out) out[j] = (float)s;
        if (copy) copy[j] = (float)s;
    }
    if (w == 2 && j < n && fin.copy.counts) fin.copy.counts[j] = fin.copy.counts_src[j];
    if (!fin.losses) return;
    __threadfence();  // this block's sums, before its ticket
    __syncthreads();
    if (gridDim.x > 1) {
        if (threadIdx.x == 0) last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
    }
    cv2_block(importance, n, load, n, fin.w_imp, fin.w_load, fin.losses, fin.copy.losses, sh);
}

int32_t launch_level_sums(const int32_t *idx, const float *gates, const float *clean, const float *raw,
                          const float *kth_vals, int64_t rows, int32_t n, int32_t k, float *importance_out,
                          float *load_out, float *scratch, cudaStream_t st, const LossFinal *fin_in) {
    LossFinal fin = {};
    if (fin_in) fin = *fin_in;
    if (rows == 0) {
        if (importance_out) MOE_CUDA(cudaMemsetAsync(importance_out, 0, sizeof(float) * n, st));
        if (load_out) MOE_CUDA(cudaMemsetAsync(load_out, 0, sizeof(float) * n, st));
        return fin_in ? launch_cv2(importance_out, n, load_out, n, fin.w_imp, fin.w_load, fin.losses, st, fin.copy) : MOE_OK;
    }
    const int32_t chunks = level_chunks(rows, n);
    int32_t CW = 1;
    while (CW < n && CW < 256) CW <<= 1;
    float *part_imp = scratch, *part_load = scratch + (int64_t)chunks * n;
    int32_t *ticket = reinterpret_cast<int32_t *>(part_load + (int64_t)chunks * n);
    if (n <= 32) launch_kernel(level_sums_rows_kernel<1>, chunks, 256, 0, st, idx, gates, clean, raw, kth_vals, rows, n, k, part_imp, part_load, ticket);
    else if (n <= 64) launch_kernel(level_sums_rows_kernel<2>, chunks, 256, 0, st, idx, gates, clean, raw, kth_vals, rows, n, k, part_imp, part_load, ticket);
    else if (n <= 128) launch_kernel(level_sums_rows_kernel<4>, chunks, 256, 0, st, idx, gates, clean, raw, kth_vals, rows, n, k, part_imp, part_load, ticket);
    else if (n <= 256) launch_kernel(level_sums_rows_kernel<8>, chunks, 256, 0, st, idx, gates, clean, raw, kth_vals, rows, n, k, part_imp, part_load, ticket);
    else launch_kernel(level_sums_kernel, chunks, 256, 0, st, idx, gates, clean, raw, kth_vals, rows, n, k, CW, part_imp, part_load, ticket);
    MOE_LAUNCHED();
    launch_kernel(level_reduce_kernel, (unsigned)cdiv(n, 32), 256, 0, st, part_imp, part_load, chunks, n, importance_out,
                  load_out, fin, ticket);
    MOE_LAUNCHED();
    return MOE_OK;
}

// the losses of vectors that are complete already (block 0), and the copies of everything (the other blocks)
__global__ void __launch_bounds__(256) cv2_kernel(const float *importance, int32_t n_imp, const float *load,
                                                  int32_t n_load, float w_imp, float w_load, float *losses, const LossOut copy) {
    wait_previous_kernel();
    __shared__ double sh[32];
    if (blockIdx.x == 0) {
        cv2_block(importance, n_imp, load, n_load, w_imp, w_load, losses, copy.losses, sh);
        return;
    }
    const int32_t i = (blockIdx.x - 1) * 256 + threadIdx.x;
    if (i < copy.n) {
        if (copy.importance) copy.importance[i] = importance[i];
        if (copy.counts) copy.counts[i] = copy.counts_src[i];
    }
    if (i < copy.n_load && copy.load) copy.load[i] = load[i];
}

int32_t launch_cv2(const float *importance, int32_t n_imp, const float *load, int32_t n_load, float w_imp,
                   float w_load, float *losses, cudaStream_t st, const LossOut &copy) {
    launch_kernel(cv2_kernel, 1 + (unsigned)cdiv(copy.n > copy.n_load ? copy.n : copy.n_load, 256), 256, 0, st, importance, n_imp, load, n_load, w_imp, w_load, losses, copy);
    MOE_LAUNCHED();
    return MOE_OK;
}

struct Cv2Pair { Cv2Job job[2]; };
__global__ void __launch_bounds__(1024) cv2_grads_kernel(const Cv2Pair pair) {  // one block per vector
    wait_previous_kernel();
    __shared__ double sh[32];
    cv2_grad_block(pair.job[blockIdx.x], sh);
}

int32_t launch_cv2_grads(const Cv2Job *jobs, cudaStream_t st) {
    launch_kernel(cv2_grads_kernel, 2, 1024, 0, st, Cv2Pair{{jobs[0], jobs[1]}});
    MOE_LAUNCHED();
    return MOE_OK;
}

// dgates[p] += dimp[topk_idx[p]]; an expert id outside [0, n) adds nothing
__global__ void add_gathered_kernel(float *dgates, const int32_t *topk_idx, const float *dimp, int64_t R, int32_t n) {
    wait_previous_kernel();
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= R) return;
    const int32_t e = topk_idx[p];
    MOE_BOUNDS_NOTE((uint32_t)e < (uint32_t)n);
    if ((uint32_t)e < (uint32_t)n) dgates[p] += dimp[e];
}

int32_t launch_add_gathered(float *dgates, const int32_t *topk_idx, const float *dimp, int64_t R, int32_t n,
                            cudaStream_t st) {
    if (R == 0) return MOE_OK;
    launch_kernel(add_gathered_kernel, (unsigned)cdiv(R, 256), 256, 0, st, dgates, topk_idx, dimp, R, n);
    MOE_LAUNCHED();
    return MOE_OK;
}

MOE_BOUNDS_READER(bounds_violations_losses)

}  // namespace moe
