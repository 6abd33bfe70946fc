// Optimiser step on the expert parameters (Appendix D, "Training", the memory optimisations): Adam with beta1 = 0
// (no first-moment estimate) whose second-moment matrix is replaced by a factored approximation: for every expert
// weight matrix only the running row-wise and column-wise averages of the squared gradient are kept, and the matrix of
// estimators is taken to be their outer product divided by the mean of the row vector. Biases (vectors) keep a full
// second-moment estimate. All of it is HBM streaming: the gradient is read twice (averages, update), the parameters
// are read and written once (small matrices: the second look finds the gradient in L2). Sums are taken in fixed orders (no floating-point atomics): two runs agree bit for bit.
#include <math_constants.h>

#include "moe_internal.cuh"

namespace moe {

namespace {

constexpr int RB = 32;  // rows per block of the averaging pass

template <typename XT> struct Vec {
    static constexpr int N = 16 / sizeof(XT);
    uint4 raw;
    __device__ __forceinline__ float get(int i) const { return to_f32(reinterpret_cast<const XT *>(&raw)[i]); }
    __device__ __forceinline__ void set(int i, float v) { reinterpret_cast<XT *>(&raw)[i] = from_f32<XT>(v); }
};

// Row block rb of expert e: row_avg[e, row] <- beta2 * row_avg + (1 - beta2) * mean_j g^2 for its RB rows (complete rows),
// and colpart[e, rb, j] = sum over its rows of g[row, j]^2. grid (row blocks, experts); 32..256 threads, one 16-byte
// column vector per thread and pass (narrow matrices get narrower blocks, so that no thread idles).
template <typename XT>
__global__ void __launch_bounds__(256) adam_averages_kernel(const XT *__restrict__ g, int32_t rows, int32_t cols,
                                                            float beta2, float *__restrict__ row_avg,
                                                            float *__restrict__ colpart) {
    wait_previous_kernel();
    constexpr int VN = Vec<XT>::N;
    __shared__ float warp_rows[8][RB];
    const int32_t e = blockIdx.y, rb = blockIdx.x, nrb = gridDim.x;
    const int32_t row0 = rb * RB;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const XT *G = g + (int64_t)e * rows * cols;
    float *cp = colpart + ((int64_t)e * nrb + rb) * cols;
    float rowacc[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) rowacc[r] = 0.0f;
    const int nvec = cols / VN;
    for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
        float colacc[VN];
#pragma unroll
        for (int i = 0; i < VN; ++i) colacc[i] = 0.0f;
#pragma unroll
        for (int r0 = 0; r0 < RB; r0 += 8) {  // eight independent 16-byte loads in flight per thread
            Vec<XT> in[8];
#pragma unroll
            for (int r = 0; r < 8; ++r)
                in[r].raw = row0 + r0 + r < rows ? reinterpret_cast<const uint4 *>(G + (int64_t)(row0 + r0 + r) * cols)[v]
                                                 : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                float s = 0.0f;
#pragma unroll
                for (int i = 0; i < VN; ++i) {
                    const float x = in[r].get(i), q = x * x;
                    colacc[i] += q;
                    s += q;
                }
                rowacc[r0 + r] += s;
            }
        }
#pragma unroll
        for (int i = 0; i < VN; ++i) cp[v * VN + i] = colacc[i];
    }
    // row sums: lanes by butterfly, then the block's warps in order
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        float s = rowacc[r];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) warp_rows[wp][r] = s;
    }
    __syncthreads();
    if (threadIdx.x < RB && row0 + threadIdx.x < rows) {
        float s = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += warp_rows[w][threadIdx.x];
        float *ra = row_avg + (int64_t)e * rows + row0 + threadIdx.x;
        *ra = beta2 * *ra + (1.0f - beta2) * (s / (float)cols);
    }
}

// col_avg[e, j] <- beta2 * col_avg + (1 - beta2) * (sum of the row blocks' partial sums, in order) / rows for the 256
// columns of block (x, e); block x = 0 also forms row_mean[e], the mean over the rows of the (already updated) row averages.
__global__ void __launch_bounds__(256) adam_columns_kernel(const float *__restrict__ colpart, int32_t nrb, int32_t rows,
                                                           int32_t cols, float beta2, float *__restrict__ col_avg,
                                                           const float *__restrict__ row_avg,
                                                           float *__restrict__ row_mean) {
    wait_previous_kernel();
    __shared__ double part[256];
    const int32_t e = blockIdx.y;
    const int32_t j = blockIdx.x * 256 + threadIdx.x;
    if (j < cols) {
        const float *src = colpart + (int64_t)e * nrb * cols + j;
        double s = 0.0;
        int32_t rb = 0;
        for (; rb + 4 <= nrb; rb += 4) {  // four loads in flight, added in order
            const float a0 = src[(int64_t)rb * cols], a1 = src[(int64_t)(rb + 1) * cols];
            const float a2 = src[(int64_t)(rb + 2) * cols], a3 = src[(int64_t)(rb + 3) * cols];
            s += (double)a0; s += (double)a1; s += (double)a2; s += (double)a3;
        }
        for (; rb < nrb; ++rb) s += (double)src[(int64_t)rb * cols];
        float *ca = col_avg + (int64_t)e * cols + j;
        *ca = beta2 * *ca + (1.0f - beta2) * (float)(s / (double)rows);
    }
    if (blockIdx.x != 0) return;
    double s = 0.0;
    for (int32_t r = threadIdx.x; r < rows; r += 256) s += (double)row_avg[(int64_t)e * rows + r];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if (threadIdx.x < off) part[threadIdx.x] += part[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) row_mean[e] = (float)(part[0] / (double)rows);
}

// W[e, i, j] -= lr * g / (sqrt(row_avg_i * col_avg_j / row_mean / correction) + eps). grid (blocks of ur rows, experts); a thread
// keeps one 16-byte column vector, with its column averages in registers, and walks down the block's rows, four of them
// in flight. HBM bound: parameters read and written, gradients read (as one flat index space, the column averages came
// from L1 with twice the loads of the parameters: 169 us for 134 M parameters, 4.8 TB/s).
// The estimate is a product, so its root is the product of a row's and a column's root, each taken once per row and column: one
// multiply-add and one reciprocal per element.
__device__ __forceinline__ float adam_step(float w, float g, float lr, float row_root, float col_root, float eps) {
    return w - __fdividef(lr * g, fmaf(row_root, col_root, eps));
}
__device__ __forceinline__ float sqrt_fast(float x) { return x > 0.0f ? x * rsqrtf(x) : 0.0f; }  // ~2 ulp, no IEEE sqrt sequence
// 0 for what is no number as well: an infinite gradient makes its column's average infinite and every row's factor 0
__device__ __forceinline__ float root(float x) { return x > 0.0f && x < CUDART_INF_F ? sqrtf(x) : 0.0f; }
// v_hat = row_avg_i * lift * factor * col_avg_j. The averages of an expert that gets no rows decay to the smallest floats, where
// the quotient by their mean alone overflows; a row's average over that mean is at most the number of rows. 2^100 is exact and 1
// elsewhere.
struct RowFactor {
    float lift, factor;
    __device__ __forceinline__ RowFactor(float mean, float inv_correction) {
        lift = mean < 1e-30f ? 0x1p100f : 1.0f;
        mean *= lift;
        factor = mean > 0.0f ? inv_correction / mean : 0.0f;
    }
    __device__ __forceinline__ float operator()(float row_avg) const { return row_avg * lift * factor; }
};

template <typename XT>
__global__ void __launch_bounds__(256) adam_update_kernel(XT *__restrict__ W, const XT *__restrict__ g, int32_t rows,
                                                          int32_t cols, const float *__restrict__ row_avg,
                                                          const float *__restrict__ col_avg,
                                                          const float *__restrict__ row_mean, float lr,
                                                          float inv_correction, float eps, int32_t ur) {
    wait_previous_kernel();
    constexpr int VN = Vec<XT>::N;
    const int32_t e = blockIdx.y;
    const RowFactor scaled(row_mean[e], inv_correction);
    const int nvec = cols / VN;
    const float *ca = col_avg + (int64_t)e * cols;
    const int32_t r0 = blockIdx.x * ur, nr = min(ur, rows - r0);
    const int64_t base = ((int64_t)e * rows + r0) * cols;
    // narrow matrices: several rows side by side
    const int groups = nvec <= 256 ? 256 / nvec : 1, group = nvec <= 256 ? threadIdx.x / nvec : 0;
    if (group >= groups) return;
    for (int v = nvec <= 256 ? threadIdx.x % nvec : threadIdx.x; v < nvec; v += nvec <= 256 ? nvec : 256) {
        float c[VN];
#pragma unroll
        for (int q = 0; q < VN / 4; ++q) {
            const float4 f = reinterpret_cast<const float4 *>(ca + v * VN)[q];
            c[4 * q] = root(f.x); c[4 * q + 1] = root(f.y); c[4 * q + 2] = root(f.z); c[4 * q + 3] = root(f.w);
        }
        for (int r = group; r < nr; r += 4 * groups) {
            Vec<XT> w[4], gr[4];
            float rs[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int row = r + u * groups;
                if (row < nr) {
                    w[u].raw = reinterpret_cast<const uint4 *>(W + base + (int64_t)row * cols)[v];
                    gr[u].raw = reinterpret_cast<const uint4 *>(g + base + (int64_t)row * cols)[v];
                    rs[u] = sqrt_fast(scaled(row_avg[(int64_t)e * rows + r0 + row]));
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int row = r + u * groups;
                if (row >= nr) break;
#pragma unroll
                for (int i = 0; i < VN; ++i)
                    w[u].set(i, adam_step(w[u].get(i), gr[u].get(i), lr, rs[u], c[i], eps));
                reinterpret_cast<uint4 *>(W + base + (int64_t)row * cols)[v] = w[u].raw;
            }
        }
    }
}

// The same with the rows' vectors as one flat index space, four independent ones per thread in flight: no thread idles, whatever the
// width.
constexpr int FLAT_ROWS = 16;
template <typename XT>
__global__ void __launch_bounds__(256) adam_update_flat_kernel(XT *__restrict__ W, const XT *__restrict__ g, int32_t rows,
                                                          int32_t cols, const float *__restrict__ row_avg,
                                                          const float *__restrict__ col_avg,
                                                          const float *__restrict__ row_mean, float lr,
                                                          float inv_correction, float eps) {
    wait_previous_kernel();
    constexpr int VN = Vec<XT>::N;
    const int32_t e = blockIdx.y;
    const RowFactor scaled(row_mean[e], inv_correction);
    const int nvec = cols / VN;
    const float *ca = col_avg + (int64_t)e * cols;
    const int32_t r0 = blockIdx.x * FLAT_ROWS, nr = min(FLAT_ROWS, rows - r0);
    const int64_t base = ((int64_t)e * rows + r0) * cols;
    const int total = nr * nvec;
    for (int i0 = threadIdx.x; i0 < total; i0 += 4 * 256) {
        Vec<XT> w[4], gr[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = i0 + u * 256;
            if (idx < total) {
                w[u].raw = reinterpret_cast<const uint4 *>(W + base)[idx];
                gr[u].raw = reinterpret_cast<const uint4 *>(g + base)[idx];
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = i0 + u * 256;
            if (idx >= total) break;
            const int r = idx / nvec, v = idx - r * nvec;
            const float rs = scaled(row_avg[(int64_t)e * rows + r0 + r]);
#pragma unroll
            for (int i = 0; i < VN; ++i)
                w[u].set(i, w[u].get(i) - __fdividef(lr * gr[u].get(i), sqrt_fast(rs * ca[v * VN + i]) + eps));
            reinterpret_cast<uint4 *>(W + base)[idx] = w[u].raw;
        }
    }
}

// ------------------------------------------------------------------------------------------
// The whole step in one launch, for matrices that stay in L2 between the two looks at their gradient. A cluster of CTAs takes an
// expert's matrix, each CTA a slab of its rows: squared row and column sums of the slab, the column sums of the cluster's
// CTAs added through distributed shared memory, then the update of the slab, whose gradients are read from L2 the second time.
// Two blocks per SM, of different clusters: one streams while the other one is at the cluster's barrier. HBM bound: gradients read
// once, parameters read and written. The last clusters step the biases.
// A warp takes a strip of 32 column vectors (a narrow matrix: several rows side by side) and walks down its share of the
// slab's rows; strips and row shares are dealt to the 16 warps.
// ------------------------------------------------------------------------------------------
constexpr int FUSED_THREADS = 512, FUSED_WARPS = FUSED_THREADS / 32;
constexpr int64_t FUSED_MATRIX_BYTES = 4 << 20, FUSED_SLAB_BYTES = 256 << 10, FUSED_EXPERT_BYTES = 112 << 10;
struct FusedMatrix {
    void *W;
    const void *g;
    float *row_avg, *col_avg;
    int32_t rows, cols, per;            // per: rows of a CTA's slab
    int32_t lanes, strips, groups;      // lanes of a row, strips of `lanes` vectors, row shares (1 where strips exceed the warps)
};
struct FusedVector {
    void *b;
    const void *g;
    float *v;
    int64_t count;
};
struct FusedAdam {
    FusedMatrix m[2];
    FusedVector v[2];
    int32_t n, cluster;
    float lr, beta2, inv_correction, eps;
};
// floats of shared memory: column sums of the CTA, updated column and row averages, sums of the row shares / strips
static int64_t fused_smem_floats(const FusedMatrix &m) {
    return 2 * (int64_t)m.cols + m.per + (int64_t)m.groups * m.cols + (int64_t)m.strips * m.per + 4;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_address(const void *p, uint32_t cta) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(cta));
    return r;
}
__device__ __forceinline__ float ld_cluster(uint32_t at) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ double ld_cluster_double(uint32_t at) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(at) : "memory");
    return v;
}

template <typename XT>
__device__ __forceinline__ void adam_vector_step(XT *b, const XT *g, float *v, int64_t i, float lr, float beta2, float inv_correction, float eps) {
    const float gi = to_f32(g[i]);
    const float vi = beta2 * v[i] + (1.0f - beta2) * gi * gi;
    v[i] = vi;
    b[i] = from_f32<XT>(to_f32(b[i]) - lr * gi / (sqrtf(vi * inv_correction) + eps));  // tiny tensor: exact operations
}

template <typename XT>
__global__ void __launch_bounds__(FUSED_THREADS, 2) adam_fused_kernel(const __grid_constant__ FusedAdam a) {
    wait_previous_kernel();
    constexpr int VN = Vec<XT>::N, UR = 4;
    extern __shared__ __align__(16) double fused_sh[];
    double *row_total = fused_sh;  // this CTA's sum of updated row averages; [2..] its warps' shares
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t C = a.cluster, item = blockIdx.x / C, rank = blockIdx.x % C;
    if (item >= 2 * a.n) {
        const int64_t first = ((int64_t)blockIdx.x - 2 * (int64_t)a.n * C) * FUSED_THREADS + tid;
        const int64_t step = ((int64_t)gridDim.x - 2 * (int64_t)a.n * C) * FUSED_THREADS;
#pragma unroll
        for (int q = 0; q < 2; ++q)
            for (int64_t i = first; i < a.v[q].count; i += step)
                adam_vector_step((XT *)a.v[q].b, (const XT *)a.v[q].g, a.v[q].v, i, a.lr, a.beta2, a.inv_correction, a.eps);
        return;
    }
    const FusedMatrix &m = a.m[item >= a.n];
    const int32_t e = item >= a.n ? item - a.n : item;
    const int32_t rows = m.rows, cols = m.cols, L = m.lanes, strips = m.strips, groups = m.groups, nvec = cols / VN;
    const int32_t r0 = min(rank * m.per, rows), nr = min(m.per, rows - r0);
    float *col_part = reinterpret_cast<float *>(fused_sh + 2 + FUSED_WARPS), *col_now = col_part + cols;
    float *group_cols = col_now + cols, *row_now = group_cols + groups * cols, *strip_rows = row_now + m.per;
    const int64_t base = ((int64_t)e * rows + r0) * nvec;  // in vectors
    const uint4 *G = reinterpret_cast<const uint4 *>(m.g) + base;
    uint4 *W = reinterpret_cast<uint4 *>(m.W) + base;
    float *row_avg = m.row_avg + (int64_t)e * rows + r0, *col_avg = m.col_avg + (int64_t)e * cols;

    // the old averages are fetched beside the first rows; every CTA reads them before its arrival at the barrier behind which they are written
    for (int j = tid; j < cols; j += FUSED_THREADS) col_now[j] = a.beta2 * col_avg[j];
    for (int r = tid; r < nr; r += FUSED_THREADS) row_now[r] = a.beta2 * row_avg[r];
    const int side = 32 / L, sub = lane / L, vl = lane % L;             // rows side by side in a warp
    const int grp = warp / min(strips, FUSED_WARPS), row_step = groups * side;
    const bool warp_on = grp < groups;
    if (warp_on) {
        for (int strip = warp % min(strips, FUSED_WARPS); strip < strips; strip += FUSED_WARPS) {
            const int v = strip * L + vl;
            const bool live = v < nvec;
            float colacc[VN];
#pragma unroll
            for (int i = 0; i < VN; ++i) colacc[i] = 0.0f;
            for (int rb = grp * side; rb < nr; rb += UR * row_step) {
                Vec<XT> in[UR];
#pragma unroll
                for (int u = 0; u < UR; ++u) {
                    const int r = rb + sub + u * row_step;
                    in[u].raw = live && r < nr ? G[(int64_t)r * nvec + v] : make_uint4(0, 0, 0, 0);
                }
                float c4[VN], s[UR];
#pragma unroll
                for (int u = 0; u < UR; ++u) {
                    s[u] = 0.0f;
#pragma unroll
                    for (int i = 0; i < VN; ++i) {
                        const float x = in[u].get(i), q = x * x;
                        c4[i] = u ? c4[i] + q : q;
                        s[u] += q;
                    }
                }
#pragma unroll
                for (int i = 0; i < VN; ++i) colacc[i] += c4[i];
                if (L >= 4) {  // two halving steps over four rows, then one value per lane
                    const bool up = vl & (L >> 1), up2 = vl & (L >> 2);
                    const float k0 = up ? s[2] : s[0], k1 = up ? s[3] : s[1];
                    float t0 = k0 + __shfl_xor_sync(0xffffffffu, up ? s[0] : s[2], L >> 1);
                    float t1 = k1 + __shfl_xor_sync(0xffffffffu, up ? s[1] : s[3], L >> 1);
                    float t = (up2 ? t1 : t0) + __shfl_xor_sync(0xffffffffu, up2 ? t0 : t1, L >> 2);
                    for (int off = L >> 3; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
                    const int r = rb + sub + (2 * up + up2) * row_step;
                    if ((vl & ((L >> 2) - 1)) == 0 && r < nr) strip_rows[strip * m.per + r] = t;
                } else {
#pragma unroll
                    for (int u = 0; u < UR; ++u) {
                        for (int off = L >> 1; off > 0; off >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], off);
                        const int r = rb + sub + u * row_step;
                        if (vl == 0 && r < nr) strip_rows[strip * m.per + r] = s[u];
                    }
                }
            }
            for (int off = L; off < 32; off <<= 1) {
#pragma unroll
                for (int i = 0; i < VN; ++i) colacc[i] += __shfl_xor_sync(0xffffffffu, colacc[i], off);
            }
            if (live && sub == 0) {
#pragma unroll
                for (int i = 0; i < VN; ++i) group_cols[grp * cols + v * VN + i] = colacc[i];
            }
        }
    }
    __syncthreads();
    double mine = 0.0;
    for (int r = tid; r < nr; r += FUSED_THREADS) {
        float s = 0.0f;
        for (int q = 0; q < strips; ++q) s += strip_rows[q * m.per + r];
        const float ra = row_now[r] + (1.0f - a.beta2) * (s / (float)cols);
        row_avg[r] = ra;
        row_now[r] = ra;
        mine += (double)ra;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, off);
    if (lane == 0) row_total[2 + warp] = mine;
    for (int j = tid; j < cols; j += FUSED_THREADS) {
        double s = 0.0;
        for (int q = 0; q < groups; ++q) s += (double)group_cols[q * cols + j];
        col_part[j] = (float)s;
    }
    __syncthreads();
    if (warp == 0) {
        double s = lane < FUSED_WARPS ? row_total[2 + lane] : 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) row_total[0] = s;
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    double shares[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) shares[c] = c < C ? ld_cluster_double(cluster_address(row_total, c)) : 0.0;
    const int32_t own = (cols + C - 1) / C;
    for (int j = tid; j < cols; j += FUSED_THREADS) {
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = c < C ? ld_cluster(cluster_address(col_part + j, c)) : 0.0f;
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) s += (double)v[c];
        const float ca = col_now[j] + (1.0f - a.beta2) * (float)(s / (double)rows);
        col_now[j] = root(ca);
        if (j / own == rank) col_avg[j] = ca;
    }
    double total = 0.0;
#pragma unroll
    for (int c = 0; c < 8; ++c) total += shares[c];
    const RowFactor scaled((float)(total / (double)rows), a.inv_correction);
    for (int r = tid; r < nr; r += FUSED_THREADS) row_now[r] = root(scaled(row_now[r]));
    __syncthreads();
    cluster_arrive();  // no more reads of the other CTAs' shared memory
    if (warp_on) {
        for (int strip = warp % min(strips, FUSED_WARPS); strip < strips; strip += FUSED_WARPS) {
            const int v = strip * L + vl;
            if (v >= nvec) continue;
            float c[VN];
#pragma unroll
            for (int i = 0; i < VN; ++i) c[i] = col_now[v * VN + i];
            constexpr int UW = 4;
            for (int rb = grp * side + sub; rb < nr; rb += UW * row_step) {
                Vec<XT> w[UW], gr[UW];
#pragma unroll
                for (int u = 0; u < UW; ++u) {
                    const int r = rb + u * row_step;
                    if (r < nr) {
                        w[u].raw = __ldcs(W + (int64_t)r * nvec + v);
                        gr[u].raw = __ldcs(G + (int64_t)r * nvec + v);
                    }
                }
#pragma unroll
                for (int u = 0; u < UW; ++u) {
                    const int r = rb + u * row_step;
                    if (r >= nr) break;
                    const float rs = row_now[r];
#pragma unroll
                    for (int i = 0; i < VN; ++i) w[u].set(i, adam_step(w[u].get(i), gr[u].get(i), a.lr, rs, c[i], a.eps));
                    __stcs(W + (int64_t)r * nvec + v, w[u].raw);
                }
            }
        }
    }
    __syncwarp();
    cluster_wait();  // this CTA's shared memory is not read any more
}

// vectors (biases): full second-moment estimate
template <typename XT>
__global__ void __launch_bounds__(256) adam_vector_kernel(XT *__restrict__ b, const XT *__restrict__ g, int64_t count,
                                                          float *__restrict__ v, float lr, float beta2,
                                                          float inv_correction, float eps) {
    wait_previous_kernel();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    adam_vector_step(b, g, v, i, lr, beta2, inv_correction, eps);
}

template <typename XT>
int32_t adam_matrix(XT *W, const XT *g, int32_t n, int32_t rows, int32_t cols, float *row_avg, float *col_avg, float lr,
                    float beta2, float inv_correction, float eps, float *colpart, float *row_mean, cudaStream_t st) {
    const int32_t nrb = (int32_t)cdiv(rows, RB);
    const int nvec = cols / (int)(16 / sizeof(XT));
    const unsigned threads = (unsigned)imin(256, cdiv(nvec, 32) * 32);
    launch_kernel(adam_averages_kernel<XT>, dim3((unsigned)nrb, (unsigned)n), threads, 0, st, g, rows, cols, beta2, row_avg, colpart);
    MOE_LAUNCHED();
    launch_kernel(adam_columns_kernel, dim3((unsigned)cdiv(cols, 256), (unsigned)n), 256, 0, st, colpart, nrb, rows, cols, beta2, col_avg, row_avg,
                                                                                     row_mean);
    MOE_LAUNCHED();
    // A thread per column vector pays where at least 7 in 8 threads have one (256 experts, bf16, 512 x 1024: 436 us for the whole step,
    // flat 470; 64 experts, 1088 x 1088, 136 vectors on 256 threads: 384 against 293).
    const int groups = nvec <= 256 ? 256 / nvec : 1;
    const int64_t lanes = 256 * cdiv(nvec, 256), busy = nvec <= 256 ? groups * nvec : nvec;
    if (8 * busy < 7 * lanes) {
        launch_kernel(adam_update_flat_kernel<XT>, dim3((unsigned)cdiv(rows, FLAT_ROWS), (unsigned)n), 256, 0, st, W, g, rows, cols, row_avg,
                      col_avg, row_mean, lr, inv_correction, eps);
        MOE_LAUNCHED();
        return MOE_OK;
    }
    // 64 rows a block where that still leaves four blocks per SM: each thread's column averages and the block's start serve
    // more rows (256 experts, 512 x 1024: 152 us, with 16 rows 164). With float's four averages per thread 16 rows each are
    // enough, and shorter blocks spread better (the same sizes in float: 976 us for the whole step, with 64 rows 1006).
    int32_t ur = n * cdiv(rows, 64) >= 4 * 148 ? 64 : 16;
    if (sizeof(XT) == 4) ur = (int32_t)imin(ur, 16 * groups);
    launch_kernel(adam_update_kernel<XT>, dim3((unsigned)cdiv(rows, ur), (unsigned)n), 256, 0, st, W, g, rows, cols, row_avg, col_avg,
                  row_mean, lr, inv_correction, eps, ur);
    MOE_LAUNCHED();
    return MOE_OK;
}

// false: this step is not one for the fused kernel
template <typename XT>
bool plan_fused(FusedAdam &a, int32_t n, int32_t d, int32_t h, size_t *smem) {
    constexpr int VN = 16 / sizeof(XT);
    const int64_t bytes = (int64_t)d * h * sizeof(XT);
    if (bytes > FUSED_MATRIX_BYTES) return false;
    int32_t C = 1;  // slabs as large as that, smaller ones where there are few matrices
    while (C < 8 && (bytes > C * FUSED_SLAB_BYTES || (2 * (int64_t)n * C < 2 * 148 && bytes > C * (int64_t)32768))) C <<= 1;
    // Few large matrices: a slab's time is its CTA's, and the kernels of their own spread over more of the chip. A step, us, in one launch /
    // apart (bf16): 4 MiB matrices of 1 expert 46 / 34, 2 47 / 37, 4 50 / 48; 2.25 MiB 1 33 / 29, 2 34 / 32, 3 and more faster in one
    if (bytes > C * FUSED_SLAB_BYTES && bytes > C * n * FUSED_EXPERT_BYTES) return false;
    a.n = n; a.cluster = C;
    const int32_t shape[2][2] = {{d, h}, {h, d}};
    int64_t floats = 0;
    for (int q = 0; q < 2; ++q) {
        FusedMatrix &m = a.m[q];
        m.rows = shape[q][0]; m.cols = shape[q][1];
        const int32_t nvec = m.cols / VN;
        m.lanes = 1;
        while (m.lanes < 32 && m.lanes < nvec) m.lanes <<= 1;
        m.strips = (int32_t)cdiv(nvec, m.lanes);
        m.groups = m.strips < FUSED_WARPS ? FUSED_WARPS / m.strips : 1;
        m.per = (int32_t)cdiv(m.rows, C);
        if (fused_smem_floats(m) > floats) floats = fused_smem_floats(m);
    }
    *smem = (2 + FUSED_WARPS) * sizeof(double) + floats * sizeof(float);
    return *smem <= 100 * 1024 && (2 * (int64_t)n + 64) * C < (int64_t)1 << 31;
}

template <typename XT>
int32_t launch_fused(const FusedAdam &a, size_t smem, cudaStream_t st) {
    static PerDevice configured;
    if (!allow_shared(configured, adam_fused_kernel<XT>, 100 * 1024)) return MOE_ERR_CUDA;
    const int64_t count = a.v[0].count > a.v[1].count ? a.v[0].count : a.v[1].count;
    const int64_t vector_clusters = imin(cdiv(count, 2 * FUSED_THREADS * a.cluster), cdiv(2 * 148, a.cluster));
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeClusterDimension;
    attrs[0].val.clusterDim.x = (unsigned)a.cluster; attrs[0].val.clusterDim.y = 1; attrs[0].val.clusterDim.z = 1;
    attrs[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_kernel
    attrs[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((2 * (int64_t)a.n + vector_clusters) * a.cluster)); cfg.blockDim = dim3(FUSED_THREADS);
    cfg.dynamicSmemBytes = smem; cfg.stream = st; cfg.attrs = attrs; cfg.numAttrs = 2;
    MOE_CUDA(cudaLaunchKernelEx(&cfg, adam_fused_kernel<XT>, a));
    MOE_LAUNCHED();
    return MOE_OK;
}

template <typename XT>
int32_t expert_adam(int32_t n, int32_t d, int32_t h, XT *W1, XT *b1, XT *W2, XT *b2, const XT *dW1, const XT *db1, const XT *dW2,
                    const XT *db2, float *state, float lr, float beta2, float inv_correction, float eps, float *ws, cudaStream_t st) {
    // state: r1 [n,d], c1 [n,h], r2 [n,h], c2 [n,d], vb1 [n,h], vb2 [n,d]
    float *r1 = state, *c1 = r1 + (int64_t)n * d, *r2 = c1 + (int64_t)n * h, *c2 = r2 + (int64_t)n * h;
    float *vb1 = c2 + (int64_t)n * d, *vb2 = vb1 + (int64_t)n * h;
    FusedAdam a = {};
    size_t smem = 0;
    if (plan_fused<XT>(a, n, d, h, &smem)) {
        a.m[0].W = W1; a.m[0].g = dW1; a.m[0].row_avg = r1; a.m[0].col_avg = c1;
        a.m[1].W = W2; a.m[1].g = dW2; a.m[1].row_avg = r2; a.m[1].col_avg = c2;
        a.v[0] = {b1, db1, vb1, (int64_t)n * h};
        a.v[1] = {b2, db2, vb2, (int64_t)n * d};
        a.lr = lr; a.beta2 = beta2; a.inv_correction = inv_correction; a.eps = eps;
        return launch_fused<XT>(a, smem, st);
    }
    float *row_mean = ws, *colpart = ws + ((n + 63) & ~63);
    const unsigned gb1 = (unsigned)cdiv((int64_t)n * h, 256), gb2 = (unsigned)cdiv((int64_t)n * d, 256);
    MOE_TRY(adam_matrix<XT>(W1, dW1, n, d, h, r1, c1, lr, beta2, inv_correction, eps, colpart, row_mean, st));
    MOE_TRY(adam_matrix<XT>(W2, dW2, n, h, d, r2, c2, lr, beta2, inv_correction, eps, colpart, row_mean, st));
    launch_kernel(adam_vector_kernel<XT>, gb1, 256, 0, st, b1, db1, (int64_t)n * h, vb1, lr, beta2, inv_correction, eps);
    MOE_LAUNCHED();
    launch_kernel(adam_vector_kernel<XT>, gb2, 256, 0, st, b2, db2, (int64_t)n * d, vb2, lr, beta2, inv_correction, eps);
    MOE_LAUNCHED();
    return MOE_OK;
}

}  // namespace

int64_t adam_ws_floats(int32_t n, int32_t d, int32_t h) {
    const int64_t a = (int64_t)n * cdiv(d, RB) * h, b = (int64_t)n * cdiv(h, RB) * d;
    return (a > b ? a : b) + n + 64;
}

int32_t launch_expert_adam(int32_t act, int32_t n, int32_t d, int32_t h, void *W1, void *b1, void *W2, void *b2,
                           const void *dW1, const void *db1, const void *dW2, const void *db2, float *state, float lr,
                           float beta2, float eps, int32_t step, float *ws, cudaStream_t st) {
    const float inv_correction = (float)(1.0 / (1.0 - pow((double)beta2, (double)step)));
    if (act == MOE_BF16)
        return expert_adam<bf16>(n, d, h, (bf16 *)W1, (bf16 *)b1, (bf16 *)W2, (bf16 *)b2, (const bf16 *)dW1, (const bf16 *)db1,
                                 (const bf16 *)dW2, (const bf16 *)db2, state, lr, beta2, inv_correction, eps, ws, st);
    return expert_adam<float>(n, d, h, (float *)W1, (float *)b1, (float *)W2, (float *)b2, (const float *)dW1, (const float *)db1,
                              (const float *)dW2, (const float *)db2, state, lr, beta2, inv_correction, eps, ws, st);
}

}  // namespace moe
