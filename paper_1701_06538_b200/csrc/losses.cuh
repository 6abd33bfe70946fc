// The batch sums of the balancing losses as device code: blocks of 256 threads in launches of their own (losses.cu) or beside others'
// (route.cu: the per-chunk sums, bound by arithmetic, with the dispatch of the rows, bound by memory; the pass over the chunks
// with the combine).
#pragma once

#include <math_constants.h>

#include "moe_internal.cuh"
#include "moments.cuh"

namespace moe {

__device__ __forceinline__ float softplus_f(float r) { return fmaxf(r, 0.0f) + log1pf(expf(-fabsf(r))); }

// Per-chunk sums with one warp per row and the lanes across the columns (n <= 32 * NV): all loads of a row are
// issued first, a lane accumulates its columns over the rows of its warp, the block's 8 warps are then added
// in order through shared memory.
template <int NV> __device__ __forceinline__ void level_sums_rows(const LevelSums &a, int32_t block) {
    const int32_t *__restrict__ idx = a.idx;
    const float *__restrict__ gates = a.gates, *__restrict__ clean = a.clean, *__restrict__ raw = a.raw, *__restrict__ kth_vals = a.kth_vals;
    const int64_t rows = a.rows;
    const int32_t n = a.n, k = a.k;
    if (block == 0 && threadIdx.x == 0) *a.ticket = 0;  // of level_reduce
    __shared__ float red[2][8][32 * NV];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t per = (rows + a.chunks - 1) / a.chunks;
    const int64_t r0 = (int64_t)block * per, r1 = min(r0 + per, rows);
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
        float s_i = 0.0f, s_l = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) { s_i += red[0][q][j]; s_l += red[1][q][j]; }
        a.part_imp[(int64_t)block * n + j] = s_i;
        a.part_load[(int64_t)block * n + j] = s_l;
    }
}

// Importance / Load = the blocks' partial sums added in double. A block takes 32 columns; its eight warps each add an
// eighth of the chunks (in ascending order, eight loads in flight: with a condition on each of ten they wait for one another, both
// launches of 32768 x 64 36 us, this way 24), the eight sums are then added in warp order. With
// fin.losses set, the block that finishes last (counted by `ticket`) also forms the two losses from the complete vectors,
// and the copies in fin.copy are written along the way.
__device__ __forceinline__ void level_reduce(const LevelSums &s, int32_t block) {
    __shared__ double red[2][8][32];
    __shared__ double sh[32];
    __shared__ int last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t n = s.n, chunks = s.chunks, blocks = (n + 31) / 32, j = block * 32 + lane;
    const LossFinal &fin = s.fin;
    const int32_t per = (chunks + 7) / 8, c0 = w * per, c1 = min(c0 + per, chunks);
    double a = 0.0, b = 0.0;
    if (j < n) {
        int32_t c = c0;
        for (; c + 8 <= c1; c += 8) {
            float pa[8], pb[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                pa[q] = s.part_imp[(int64_t)(c + q) * n + j];
                pb[q] = s.part_load[(int64_t)(c + q) * n + j];
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) { a += (double)pa[q]; b += (double)pb[q]; }
        }
        for (; c < c1; ++c) {
            a += (double)s.part_imp[(int64_t)c * n + j];
            b += (double)s.part_load[(int64_t)c * n + j];
        }
    }
    red[0][w][lane] = a;
    red[1][w][lane] = b;
    __syncthreads();
    if (w < 2 && j < n) {  // warp 0: Importance, warp 1: Load
        double sum = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) sum += red[w][q][lane];
        float *out = w ? s.load : s.importance, *copy = w ? fin.copy.load : fin.copy.importance;
        if (out) out[j] = (float)sum;
        if (copy) copy[j] = (float)sum;
    }
    if (w == 2 && j < n && fin.copy.counts) fin.copy.counts[j] = fin.copy.counts_src[j];
    if (!fin.losses) return;
    __threadfence();  // this block's sums, before its ticket
    __syncthreads();
    if (blocks > 1) {
        if (threadIdx.x == 0) last = atomicAdd(s.ticket, 1) == blocks - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
    }
    cv2_block(s.importance, n, s.load, n, fin.w_imp, fin.w_load, fin.losses, fin.copy.losses, sh);
}

}  // namespace moe
