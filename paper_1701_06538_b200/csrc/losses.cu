// Balancing losses (Section 4 and Appendix A): Importance (Eq. 6), the smooth load estimator
// P(x, i) (Eq. 9), Load (Eq. 10), the two CV^2 losses (Eq. 7, 11) and their gradients.
// Batch sums are deterministic: per-chunk partial sums in float, then one ordered pass in double.
#include "losses.cuh"

namespace moe {

constexpr int LCHUNKS_MAX = 148 * 4;

// a row per warp until the chip is full: the normal-CDF evaluations of a row are one long latency chain per lane. Up to 32
// columns one block adds up all chunks, and up to 16384 rows half as many are enough (8192 rows: 6 columns 12.0 us for both
// launches, with all chunks 15.2; 15000 rows of 30 columns 15.5, 17.9; but 60000 rows of 20 columns 28.4, 26.5)
static inline int32_t level_chunks(int64_t rows, int32_t n) {
    return (int32_t)imin(cdiv(rows, 8), n <= 32 && rows <= 16384 ? LCHUNKS_MAX / 2 : LCHUNKS_MAX);
}
int64_t losses_ws_floats(int64_t rows, int32_t n) { return 2 * (int64_t)level_chunks(rows, n) * n + 64; }

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

template <int NV> __global__ void __launch_bounds__(256) level_sums_rows_kernel(const LevelSums sums) {
    wait_previous_kernel();
    level_sums_rows<NV>(sums, blockIdx.x);
}
__global__ void __launch_bounds__(256) level_reduce_kernel(const LevelSums sums) {
    wait_previous_kernel();
    level_reduce(sums, blockIdx.x);
}

LevelSums level_sums(const int32_t *idx, const float *gates, const float *clean, const float *raw, const float *kth_vals, int64_t rows,
                     int32_t n, int32_t k, float *importance, float *load, float *scratch, const LossFinal *fin) {
    LevelSums s = {};
    s.idx = idx; s.gates = gates; s.clean = clean; s.raw = raw; s.kth_vals = kth_vals;
    s.rows = rows; s.n = n; s.k = k;
    s.chunks = level_chunks(rows, n);
    s.part_imp = scratch; s.part_load = scratch + (int64_t)s.chunks * n;
    s.ticket = reinterpret_cast<int32_t *>(s.part_load + (int64_t)s.chunks * n);
    s.importance = importance; s.load = load;
    if (fin) s.fin = *fin;
    return s;
}

int32_t launch_level_sums(const LevelSums &s, cudaStream_t st) {
    const int32_t n = s.n;
    if (s.rows == 0) {
        if (s.importance) MOE_CUDA(cudaMemsetAsync(s.importance, 0, sizeof(float) * n, st));
        if (s.load) MOE_CUDA(cudaMemsetAsync(s.load, 0, sizeof(float) * n, st));
        return s.fin.losses ? launch_cv2(s.importance, n, s.load, n, s.fin.w_imp, s.fin.w_load, s.fin.losses, st, s.fin.copy) : MOE_OK;
    }
    if (n <= 32) launch_kernel(level_sums_rows_kernel<1>, s.chunks, 256, 0, st, s);
    else if (n <= 64) launch_kernel(level_sums_rows_kernel<2>, s.chunks, 256, 0, st, s);
    else if (n <= 128) launch_kernel(level_sums_rows_kernel<4>, s.chunks, 256, 0, st, s);
    else if (n <= 256) launch_kernel(level_sums_rows_kernel<8>, s.chunks, 256, 0, st, s);
    else launch_kernel(level_sums_kernel, s.chunks, 256, 0, st, s.idx, s.gates, s.clean, s.raw, s.kth_vals, s.rows, n, s.k, 256, s.part_imp, s.part_load, s.ticket);
    MOE_LAUNCHED();
    launch_kernel(level_reduce_kernel, (unsigned)cdiv(n, 32), 256, 0, st, s);
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
