// Strictly balanced gating (Appendix F, Eq. 15-20): dense softmax gate, batchwise mask (the m = k T / n largest values
// of every expert's column over the batch, so that every expert receives exactly m examples), gates renormalised over
// the kept experts, threshold mask and L_batchwise. An example is kept by a variable number of experts, so the routing
// tables are by sorted row (expert-major, m rows per expert, token order inside an expert) plus a per-token list
// (CSR: tok_ptr, tok_rows) for the combine and its adjoint. Integer results (mask, tables) are unique: ties go to the
// lower token. Sums are taken in fixed orders; integer atomics only.
#include <math_constants.h>

#include "moe_internal.cuh"

namespace moe {

namespace {

// p = softmax(c) per row: exponentials and their sum in double (largest logit subtracted), one rounding to float. The double
// exponential is what bounds it: rows of up to 256 columns keep theirs in registers (below), this kernel evaluates each twice.
__global__ void __launch_bounds__(256) bal_softmax_kernel(const float *__restrict__ c, int64_t T, int32_t n,
                                                          float *__restrict__ p) {
    wait_previous_kernel();
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= T) return;
    const float *row = c + t * n;
    float mx = -CUDART_INF_F;
    for (int32_t j = lane; j < n; j += 32) mx = fmaxf(mx, row[j]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    double s = 0.0;
    for (int32_t j = lane; j < n; j += 32) s += exp((double)row[j] - (double)mx);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    for (int32_t j = lane; j < n; j += 32) p[t * n + j] = (float)(exp((double)row[j] - (double)mx) / s);
}

// out [cols, rows] = in [rows, cols]^T, 32 x 32 tiles
__global__ void __launch_bounds__(256) bal_transpose_kernel(const float *__restrict__ in, int64_t rows, int32_t cols,
                                                            float *__restrict__ out) {
    wait_previous_kernel();
    __shared__ float tile[32][33];
    const int64_t r0 = (int64_t)blockIdx.x * 32;
    const int32_t c0 = blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int i = ty; i < 32; i += 8)
        if (r0 + i < rows && c0 + tx < cols) tile[i][tx] = in[(r0 + i) * cols + c0 + tx];
    __syncthreads();
    for (int i = ty; i < 32; i += 8)
        if (c0 + i < cols && r0 + tx < rows) out[(int64_t)(c0 + i) * rows + r0 + tx] = tile[tx][i];
}

// Softmax of rows of at most 32 * NV columns, and p^T [n, T] with it: a block takes 32 tokens, two per warp, and writes the
// transposed values from shared memory, 128 bytes of a column at a time (a transposing pass of its own read and wrote p again:
// 18 us of 48 for both, 32768 x 256).
template <int NV>
__global__ void __launch_bounds__(512) bal_softmax_both_kernel(const float *__restrict__ c, int64_t T, int32_t n,
                                                               float *__restrict__ p, float *__restrict__ pT) {
    wait_previous_kernel();
    __shared__ float tile[32][32 * NV + 1];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * 32;
    float v[2][NV];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int64_t t = t0 + 2 * wp + q;
            v[q][u] = t < T && lane + 32 * u < n ? c[t * n + lane + 32 * u] : -CUDART_INF_F;
        }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int64_t t = t0 + 2 * wp + q;
        if (t >= T) break;
        float mx = -CUDART_INF_F;
#pragma unroll
        for (int u = 0; u < NV; ++u) mx = fmaxf(mx, v[q][u]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        double s = 0.0, e[NV];
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            e[u] = lane + 32 * u < n ? exp((double)v[q][u] - (double)mx) : 0.0;
            s += e[u];
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
#pragma unroll
        for (int u = 0; u < NV; ++u)
            if (lane + 32 * u < n) {
                const float f = (float)(e[u] / s);
                p[t * n + lane + 32 * u] = f;
                tile[2 * wp + q][lane + 32 * u] = f;
            }
    }
    __syncthreads();
    if (t0 + lane < T)
        for (int32_t j = wp; j < n; j += 16) pT[(int64_t)j * T + t0 + lane] = tile[lane][j];
}

// Batchwise mask of one expert (block = column i of p, given transposed: col [T]): the m largest values, equal values to
// the lower token. Radix select of the m-th largest key (the bit patterns of non-negative floats order like the
// values), then an order-preserving compaction: tok_of_row[i * m + q] = q-th kept token, and the expert's bit is set
// in the token's mask words. A warp owns a contiguous run of tokens, so that its place in the list needs one scan over the
// warps. NK > 0: up to 1024 * NK keys stay in registers and the column is read once; NK = 0: any length, one sweep per digit
// and two for the compaction, eight loads per thread in flight. Three digits of 11, 11 and 10 bits: the first one holds the exponent
// and two bits of the mantissa, so that the lanes' additions to its few counters collide less (four digits of 8 bits and a sweep
// each: 62 us at 32768 x 256).
constexpr int SEL_BATCH = 8, SEL_BINS = 2048;
template <int NK>
__global__ void __launch_bounds__(1024, NK > 8 ? 1 : 2) bal_select_kernel(const float *__restrict__ pT, int64_t T, int32_t n, int32_t m,
                                                          int32_t words, int32_t *__restrict__ tok_of_row,
                                                          uint32_t *__restrict__ mask_bits) {
    wait_previous_kernel();
    __shared__ int32_t hist[SEL_BINS];
    __shared__ int32_t warp_gt[32], warp_eq[32];
    __shared__ uint32_t s_prefix;
    __shared__ int32_t s_need;
    constexpr int NB = NK > 0 ? NK : SEL_BATCH;
    const int32_t i = blockIdx.x;
    const uint32_t *col = reinterpret_cast<const uint32_t *>(pT + (int64_t)i * T);
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int64_t run = ((T + 31) / 32 + 31) / 32 * 32, t_first = wp * run, t_last = min(T, t_first + run);
    uint32_t key[NB];
    // f(token of this lane, key, inside the run) for the warp's run in ascending order; all lanes take part
    auto load = [&](int64_t t00) {
#pragma unroll
        for (int u = 0; u < NB; ++u) key[u] = t00 + 32 * u + lane < t_last ? col[t00 + 32 * u + lane] : 0u;
    };
    auto sweep = [&](auto f) {
        for (int64_t t00 = t_first; t00 < t_last; t00 += 32 * NB) {
            if (NK == 0) load(t00);
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int64_t t = t00 + 32 * u + lane;
                f(t, key[u], t < t_last);
            }
        }
    };
    if (NK > 0) load(t_first);
    if (tid == 0) { s_prefix = 0u; s_need = m; }
    uint32_t known = 0u;  // mask of the key bits fixed so far
#pragma unroll
    for (int digit = 0; digit < 3; ++digit) {
        const int shift = digit == 0 ? 21 : digit == 1 ? 10 : 0;
        const uint32_t bins = digit == 2 ? 1024u : 2048u;
        hist[tid] = 0; hist[tid + 1024] = 0;
        __syncthreads();
        const uint32_t prefix = s_prefix;
        sweep([&](int64_t, uint32_t k, bool in) {
            if (in && (k & known) == prefix) atomicAdd(&hist[(k >> shift) & (bins - 1u)], 1);
        });
        __syncthreads();
        // the digit that holds the need-th largest key: thread tid holds the digits 2047 - 2 tid and the one below
        const int32_t need = s_need, h0 = hist[SEL_BINS - 1 - 2 * tid], h1 = hist[SEL_BINS - 2 - 2 * tid];
        int32_t inc = h0 + h1;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t o = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += o;
        }
        if (lane == 31) warp_gt[wp] = inc;
        __syncthreads();
        const int32_t before = __reduce_add_sync(0xffffffffu, lane < wp ? warp_gt[lane] : 0) + inc - h0 - h1;  // keys with a larger digit
        if (before < need && need <= before + h0) {
            s_need = need - before;
            s_prefix = prefix | ((uint32_t)(SEL_BINS - 1 - 2 * tid) << shift);
        } else if (before + h0 < need && need <= before + h0 + h1) {
            s_need = need - before - h0;
            s_prefix = prefix | ((uint32_t)(SEL_BINS - 2 - 2 * tid) << shift);
        }
        known |= (bins - 1u) << shift;
        __syncthreads();
    }
    const uint32_t kth = s_prefix;    // the m-th largest key
    const int32_t take_eq = s_need;   // how many of the keys equal to it are kept (the first ones in token order)
    int32_t gt = 0, eq = 0;
    sweep([&](int64_t, uint32_t k, bool in) {
        if (in) { gt += k > kth; eq += k == kth; }
    });
    gt = __reduce_add_sync(0xffffffffu, gt);
    eq = __reduce_add_sync(0xffffffffu, eq);
    if (lane == 0) { warp_gt[wp] = gt; warp_eq[wp] = eq; }
    __syncthreads();
    int32_t eq_base = __reduce_add_sync(0xffffffffu, lane < wp ? warp_eq[lane] : 0);  // in the warps before
    int32_t pos = __reduce_add_sync(0xffffffffu, lane < wp ? warp_gt[lane] : 0) + min(eq_base, take_eq);
    sweep([&](int64_t t, uint32_t k, bool in) {
        const bool is_eq = in && k == kth;
        const uint32_t below = (1u << lane) - 1u, b_eq = __ballot_sync(0xffffffffu, is_eq);
        const bool keep = (in && k > kth) || (is_eq && eq_base + __popc(b_eq & below) < take_eq);
        const uint32_t b_keep = __ballot_sync(0xffffffffu, keep);
        const int32_t at = pos + __popc(b_keep & below);
        if (keep && at < m) {  // at < m always: exactly m keys are kept
            tok_of_row[(int64_t)i * m + at] = (int32_t)t;
            atomicOr(&mask_bits[t * words + (i >> 5)], 1u << (i & 31));
        }
        eq_base += __popc(b_eq);
        pos += __popc(b_keep);
    });
}

// Per token (one warp): den = sum of p over the kept experts, cnt = how many keep it, the token's part of L_batchwise
// (Eq. 20), and the per-expert counts of the threshold mask. Block partials of the loss go to loss_part. A warp takes up to
// eight tokens, so that a block clears and adds up its n counts once per 64 tokens, but no more than leave four blocks per SM:
// the sweeps over a token's row are its time (whole gate, 4096 tokens x 2048 experts: 279 us, with eight tokens each 375;
// 8192 x 8192: 1633, 2066; 32768 x 256 with eight: 184, with one: 234).
constexpr int TOK_PER_WARP = 8;
int32_t tokens_per_warp(int64_t T) {
    const int64_t fit = T / (8 * 4 * 148);
    return (int32_t)(fit < 1 ? 1 : imin(fit, TOK_PER_WARP));
}
__global__ void __launch_bounds__(256) bal_token_kernel(const float *__restrict__ p, const uint32_t *__restrict__ mask_bits,
                                                        const float *__restrict__ thr, int64_t T, int32_t n, int32_t words,
                                                        float *__restrict__ den, int32_t *__restrict__ cnt,
                                                        int32_t *__restrict__ thr_counts, double *__restrict__ loss_part,
                                                        int32_t per_warp) {
    wait_previous_kernel();
    extern __shared__ int32_t s_cnt[];  // [n] threshold-mask counts of this block
    __shared__ double s_loss[8];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    for (int32_t j = threadIdx.x; j < n; j += blockDim.x) s_cnt[j] = 0;
    __syncthreads();
    double loss = 0.0;
    for (int q = 0; q < per_warp; ++q) {
        const int64_t t = ((int64_t)blockIdx.x * 8 + wp) * per_warp + q;
        if (t >= T) break;
        double d = 0.0, l = 0.0;
        int32_t c = 0;
#pragma unroll 4
        for (int32_t j = lane; j < n; j += 32) {
            const float pj = p[t * n + j];
            const bool mb = (mask_bits[t * words + (j >> 5)] >> (j & 31)) & 1u;
            const bool mt = pj > thr[j];
            if (mb) { d += (double)pj; ++c; }
            if (mt) atomicAdd(&s_cnt[j], 1);
            if (mt != mb) l += (mt ? 1.0 : -1.0) * ((double)pj - (double)thr[j]);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            d += __shfl_xor_sync(0xffffffffu, d, off);
            l += __shfl_xor_sync(0xffffffffu, l, off);
            c += __shfl_xor_sync(0xffffffffu, c, off);
        }
        if (lane == 0) { den[t] = (float)d; cnt[t] = c; }
        loss += l;
    }
    if (lane == 0) s_loss[wp] = loss;
    __syncthreads();
    for (int32_t j = threadIdx.x; j < n; j += blockDim.x)
        if (s_cnt[j]) atomicAdd(&thr_counts[j], s_cnt[j]);
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += s_loss[w];
        loss_part[blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(256) bal_loss_final_kernel(const double *__restrict__ part, int64_t nparts,
                                                             float *__restrict__ loss) {
    wait_previous_kernel();
    __shared__ double sh[256];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < nparts; i += 256) s += part[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if (threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) loss[0] = (float)sh[0];
}

// rank of expert e among the experts that keep token t
__device__ __forceinline__ int32_t rank_in_token(const uint32_t *bits, int32_t e) {
    int32_t r = 0;
    for (int32_t w = 0; w < (e >> 5); ++w) r += __popc(bits[w]);
    return r + __popc(bits[e >> 5] & ((1u << (e & 31)) - 1u));
}

// Per sorted row: its place in its token's list (ascending expert); offsets[e] = e * m.
__global__ void __launch_bounds__(256) bal_fill_kernel(const int32_t *__restrict__ tok_of_row,
                                                       const uint32_t *__restrict__ mask_bits,
                                                       const int32_t *__restrict__ tok_ptr, int64_t R, int32_t n, int32_t m,
                                                       int32_t words, int32_t *__restrict__ tok_rows,
                                                       int32_t *__restrict__ offsets) {
    wait_previous_kernel();
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r <= n) offsets[r] = (int32_t)(r * m);
    if (r >= R) return;
    const int32_t t = tok_of_row[r], e = (int32_t)(r / m);
    tok_rows[tok_ptr[t] + rank_in_token(mask_bits + (int64_t)t * words, e)] = (int32_t)r;
}

template <typename XT> struct V16 {
    static constexpr int N = 16 / sizeof(XT);
    uint4 raw;
    __device__ __forceinline__ float get(int i) const { return to_f32(reinterpret_cast<const XT *>(&raw)[i]); }
    __device__ __forceinline__ void set(int i, float v) { reinterpret_cast<XT *>(&raw)[i] = from_f32<XT>(v); }
};

// xs[r] = x[tok_of_row[r]], one warp per row
template <typename XT>
__global__ void __launch_bounds__(256) bal_gather_kernel(const XT *__restrict__ x, const int32_t *__restrict__ tok_of_row,
                                                         int64_t R, int64_t T, int32_t d, XT *__restrict__ xs) {
    wait_previous_kernel();
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= R) return;
    const int32_t t = tok_of_row[r];
    if ((uint32_t)t >= (uint32_t)T) return;
    const int nvec = d / V16<XT>::N;
    const uint4 *src = reinterpret_cast<const uint4 *>(x + (int64_t)t * d);
    uint4 *dst = reinterpret_cast<uint4 *>(xs + r * d);
    for (int v0 = lane; v0 < nvec; v0 += 128) {
        uint4 val[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (v0 + 32 * u < nvec) val[u] = src[v0 + 32 * u];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (v0 + 32 * u < nvec) dst[v0 + 32 * u] = val[u];
    }
}

// Rows of token t that a lane holds for its warp: entry j of the list in lane j (the first 32 entries; `first` moves on). A row
// outside [0, R) is -1 and contributes nothing.
__device__ __forceinline__ int32_t token_row(const int32_t *tok_rows, int32_t first, int32_t j1, int64_t R, int lane) {
    const int32_t r = first + lane < j1 ? tok_rows[first + lane] : -1;
    return (uint32_t)r < (uint32_t)R ? r : -1;
}

// A warp's walk over tokens t, t + step, ...: the next token's list is fetched while the rows of this one move, and the bounds of the
// list after it (the numbers of a token's rows, their gates and the rows are three loads one behind the other).
struct TokenWalk {
    const int32_t *tok_ptr, *tok_rows;
    int64_t T, R, t, step;
    int32_t j0, j1, n0, n1, row;  // this token's list, the next one's, this lane's entry of this one's
    int lane;
    __device__ __forceinline__ TokenWalk(const int32_t *tok_ptr_, const int32_t *tok_rows_, int64_t T_, int64_t R_, int lane_)
        : tok_ptr(tok_ptr_), tok_rows(tok_rows_), T(T_), R(R_), t((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)),
          step((int64_t)gridDim.x * 8), j0(0), j1(0), n0(0), n1(0), row(-1), lane(lane_) {
        if (t < T) { j0 = tok_ptr[t]; j1 = tok_ptr[t + 1]; }
        bounds();
        row = token_row(tok_rows, j0, j1, R, lane);
    }
    __device__ __forceinline__ void bounds() {
        n0 = n1 = 0;
        if (t + step < T) { n0 = tok_ptr[t + step]; n1 = tok_ptr[t + step + 1]; }
    }
    __device__ __forceinline__ int32_t next_row() const { return token_row(tok_rows, n0, n1, R, lane); }
    __device__ __forceinline__ void advance(int32_t row_) {
        t += step;
        j0 = n0; j1 = n1; row = row_;
        bounds();
    }
};

// y[t] = sum over the rows of token t (ascending expert) of p[t, e] / den[t] * ys[row]   (Eq. 1 with the gates of Eq. 16).
// One warp per token, a vector of four rows in flight per lane (one row after the other, each behind the load of its number: 74 us
// at 32768 tokens x 512 with four rows each, this way 58; the adjoints below, with the same walk, lost what it took in registers).
template <typename XT>
__global__ void __launch_bounds__(256) bal_combine_kernel(const XT *__restrict__ ys, const float *__restrict__ p,
                                                          const float *__restrict__ den, const int32_t *__restrict__ tok_ptr,
                                                          const int32_t *__restrict__ tok_rows, int64_t T, int64_t R,
                                                          int32_t n, int32_t m, int32_t d, XT *__restrict__ y) {
    wait_previous_kernel();
    constexpr int VN = V16<XT>::N;
    const int lane = threadIdx.x & 31;
    const int nvec = d / VN;
    for (TokenWalk w(tok_ptr, tok_rows, T, R, lane); w.t < T;) {
        const int32_t next = w.next_row();
        const float dn = den[w.t];
        const float gate0 = w.row >= 0 ? p[w.t * n + w.row / m] / dn : 0.0f;
        for (int v = lane; v - lane < nvec; v += 32) {
            float acc[VN];
#pragma unroll
            for (int i = 0; i < VN; ++i) acc[i] = 0.0f;
            int32_t row = w.row;
            float gate = gate0;
            for (int32_t first = w.j0; first < w.j1; first += 32) {
                if (first > w.j0) {  // lists of more than 32 rows
                    row = token_row(tok_rows, first, w.j1, R, lane);
                    gate = row >= 0 ? p[w.t * n + row / m] / dn : 0.0f;
                }
                const int count = min(32, w.j1 - first);
                for (int q0 = 0; q0 < count; q0 += 4) {
                    V16<XT> in[4];
                    int32_t r[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        r[q] = __shfl_sync(0xffffffffu, row, (q0 + q) & 31);
                        if (q0 + q >= count) r[q] = -1;
                        if (r[q] >= 0 && v < nvec) in[q].raw = reinterpret_cast<const uint4 *>(ys + (int64_t)r[q] * d)[v];
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float g = __shfl_sync(0xffffffffu, gate, (q0 + q) & 31);
                        if (r[q] >= 0) {
#pragma unroll
                            for (int i = 0; i < VN; ++i) acc[i] = fmaf(g, in[q].get(i), acc[i]);
                        }
                    }
                }
            }
            if (v < nvec) {
                V16<XT> out;
#pragma unroll
                for (int i = 0; i < VN; ++i) out.set(i, acc[i]);
                reinterpret_cast<uint4 *>(y + w.t * d)[v] = out.raw;
            }
        }
        w.advance(next);
    }
}

// per row: dG_row[r] = <dY[t], ys[r]>, dys[r] = g * dY[t]
template <typename XT>
__global__ void __launch_bounds__(256) bal_combine_bwd_kernel(const XT *__restrict__ dY, const XT *__restrict__ ys,
                                                              const float *__restrict__ p, const float *__restrict__ den,
                                                              const int32_t *__restrict__ tok_of_row, int64_t R, int64_t T,
                                                              int32_t n, int32_t m, int32_t d, float *__restrict__ dG_row,
                                                              XT *__restrict__ dys) {
    wait_previous_kernel();
    constexpr int VN = V16<XT>::N;
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= R) return;
    const int32_t t = tok_of_row[r];
    if ((uint32_t)t >= (uint32_t)T) return;
    const float g = p[(int64_t)t * n + r / m] / den[t];
    const int nvec = d / VN;
    float dot = 0.0f;
    for (int v = lane; v < nvec; v += 32) {
        V16<XT> a, b, o;
        a.raw = reinterpret_cast<const uint4 *>(dY + (int64_t)t * d)[v];
        b.raw = reinterpret_cast<const uint4 *>(ys + r * d)[v];
#pragma unroll
        for (int i = 0; i < VN; ++i) {
            dot = fmaf(a.get(i), b.get(i), dot);
            o.set(i, g * a.get(i));
        }
        reinterpret_cast<uint4 *>(dys + r * d)[v] = o.raw;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    if (lane == 0) dG_row[r] = dot;
}

// Logit gradients of one token (one warp): through Eq. 16 (mask constant), Eq. 20 scaled by w, and the softmax.
__global__ void __launch_bounds__(256) bal_gate_bwd_kernel(const float *__restrict__ p, const uint32_t *__restrict__ mask_bits,
                                                           const float *__restrict__ den, const float *__restrict__ thr,
                                                           const int32_t *__restrict__ tok_ptr,
                                                           const int32_t *__restrict__ tok_rows,
                                                           const float *__restrict__ dG_row, float w, int64_t T, int32_t n,
                                                           int32_t m, int32_t words, float *__restrict__ dc,
                                                           bf16 *__restrict__ dsplit) {
    wait_previous_kernel();
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (t >= T) return;
    const int32_t j0 = tok_ptr[t], j1 = tok_ptr[t + 1];
    const double dn = (double)den[t];
    double inner = 0.0;  // sum over the kept experts of G * dG
    for (int32_t j = j0 + lane; j < j1; j += 32) {
        const int32_t r = tok_rows[j];
        inner += (double)p[t * n + r / m] / dn * (double)dG_row[r];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) inner += __shfl_xor_sync(0xffffffffu, inner, off);
    const uint32_t *bits = mask_bits + t * words;
    double s2 = 0.0;
    for (int32_t j = lane; j < n; j += 32) {
        const double pj = (double)p[t * n + j];
        const bool mb = (bits[j >> 5] >> (j & 31)) & 1u;
        const bool mt = (float)pj > thr[j];
        double dp = (double)w * ((mt ? 1.0 : 0.0) - (mb ? 1.0 : 0.0));
        if (mb) dp += ((double)dG_row[tok_rows[j0 + rank_in_token(bits, j)]] - inner) / dn;
        s2 += dp * pj;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, off);
    for (int32_t j = lane; j < n; j += 32) {
        const double pj = (double)p[t * n + j];
        const bool mb = (bits[j >> 5] >> (j & 31)) & 1u;
        const bool mt = (float)pj > thr[j];
        double dp = (double)w * ((mt ? 1.0 : 0.0) - (mb ? 1.0 : 0.0));
        if (mb) dp += ((double)dG_row[tok_rows[j0 + rank_in_token(bits, j)]] - inner) / dn;
        const float v = (float)(pj * (dp - s2));
        if (dsplit) {  // three bf16 terms carry the 24 mantissa bits: [T, 3n] = (hi | mid | lo)
            const bf16 hi = __float2bfloat16_rn(v);
            const float r1 = v - __bfloat162float(hi);
            const bf16 mid = __float2bfloat16_rn(r1);
            bf16 *row = dsplit + t * 3 * n;
            row[j] = hi; row[n + j] = mid; row[2 * n + j] = __float2bfloat16_rn(r1 - __bfloat162float(mid));
        } else {
            dc[t * n + j] = v;
        }
    }
}

// The same for the tensor-core path and at most 64 * NP columns (n even): a lane owns pairs of adjacent columns, reads the row once
// and keeps it, with the gradients of the kept ones, in registers, and the three bf16 terms of a pair leave as 4-byte stores
// (three walks over the row, each behind its own loads: 85 us at 32768 x 256).
template <int NP>
__global__ void __launch_bounds__(256) bal_gate_bwd_pairs_kernel(const float *__restrict__ p, const uint32_t *__restrict__ mask_bits,
                                                                 const float *__restrict__ den, const float *__restrict__ thr,
                                                                 const int32_t *__restrict__ tok_ptr,
                                                                 const int32_t *__restrict__ tok_rows,
                                                                 const float *__restrict__ dG_row, float w, int64_t T, int32_t n,
                                                                 int32_t words, bf16 *__restrict__ dsplit) {
    wait_previous_kernel();
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (t >= T) return;
    const int32_t j0 = tok_ptr[t];
    const double dn = (double)den[t];
    const uint32_t mine = lane < words ? mask_bits[t * words + lane] : 0u;  // word `lane` of the token's mask
    float2 pv[NP], tv[NP];
#pragma unroll
    for (int u = 0; u < NP; ++u) {
        const int32_t j = 2 * lane + 64 * u;
        pv[u] = j < n ? *reinterpret_cast<const float2 *>(p + t * n + j) : make_float2(0.0f, 0.0f);
        tv[u] = j < n ? *reinterpret_cast<const float2 *>(thr + j) : make_float2(0.0f, 0.0f);
    }
    float dg[2 * NP];
    bool kept[2 * NP];
    int32_t rank0 = 0;  // kept experts in the words before
#pragma unroll
    for (int u = 0; u < NP; ++u) {
        const uint32_t w0 = __shfl_sync(0xffffffffu, mine, 2 * u), w1 = __shfl_sync(0xffffffffu, mine, 2 * u + 1);
        const uint32_t word = lane < 16 ? w0 : w1;
        const int bit = (2 * lane) & 31;
        int32_t rank = rank0 + (lane < 16 ? 0 : __popc(w0)) + __popc(word & ((1u << bit) - 1u));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            kept[2 * u + h] = (word >> (bit + h)) & 1u;
            dg[2 * u + h] = kept[2 * u + h] ? dG_row[tok_rows[j0 + rank]] : 0.0f;
            rank += kept[2 * u + h];
        }
        rank0 += __popc(w0) + __popc(w1);
    }
    auto value = [](const float2 &v, int h) { return h ? v.y : v.x; };
    double inner = 0.0;  // sum over the kept experts of G * dG
#pragma unroll
    for (int q = 0; q < 2 * NP; ++q)
        if (kept[q]) inner += (double)value(pv[q >> 1], q & 1) / dn * (double)dg[q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) inner += __shfl_xor_sync(0xffffffffu, inner, off);
    double dp[2 * NP], s2 = 0.0;
#pragma unroll
    for (int q = 0; q < 2 * NP; ++q) {
        const float pj = value(pv[q >> 1], q & 1);
        dp[q] = (double)w * ((pj > value(tv[q >> 1], q & 1) ? 1.0 : 0.0) - (kept[q] ? 1.0 : 0.0));
        if (kept[q]) dp[q] += ((double)dg[q] - inner) / dn;
        s2 += dp[q] * (double)pj;  // columns behind the row: p = 0
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, off);
    bf16 *row = dsplit + t * 3 * n;  // three bf16 terms carry the 24 mantissa bits: [T, 3n] = (hi | mid | lo)
#pragma unroll
    for (int u = 0; u < NP; ++u) {
        const int32_t j = 2 * lane + 64 * u;
        if (j >= n) continue;
        float v0 = (float)((double)pv[u].x * (dp[2 * u] - s2)), v1 = (float)((double)pv[u].y * (dp[2 * u + 1] - s2));
#pragma unroll
        for (int term = 0; term < 3; ++term) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
            *reinterpret_cast<__nv_bfloat162 *>(row + term * n + j) = h;
            v0 -= __bfloat162float(h.x); v1 -= __bfloat162float(h.y);
        }
    }
}

__global__ void bal_dthr_kernel(const int32_t *__restrict__ thr_counts, int32_t n, int32_t m, float w,
                                float *__restrict__ dthr) {
    wait_previous_kernel();
    const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n) dthr[j] = -w * (float)(thr_counts[j] - m);
}

// dX[t] = sum over the rows of token t of dxs[row] + dX_gate[t], rounded to the act type
template <typename XT>
__global__ void __launch_bounds__(256) bal_dispatch_bwd_kernel(const XT *__restrict__ dxs, const int32_t *__restrict__ tok_ptr,
                                                               const int32_t *__restrict__ tok_rows,
                                                               const float *__restrict__ dX_gate, int64_t T, int64_t R,
                                                               int32_t d, XT *__restrict__ dX) {
    wait_previous_kernel();
    constexpr int VN = V16<XT>::N;
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (t >= T) return;
    const int32_t j0 = tok_ptr[t], j1 = tok_ptr[t + 1];
    const int nvec = d / VN;
    for (int v = lane; v < nvec; v += 32) {
        float acc[VN];
#pragma unroll
        for (int i = 0; i < VN; ++i) acc[i] = 0.0f;
        for (int32_t j = j0; j < j1; ++j) {
            const int32_t r = tok_rows[j];
            if ((uint32_t)r >= (uint32_t)R) continue;
            V16<XT> in;
            in.raw = reinterpret_cast<const uint4 *>(dxs + (int64_t)r * d)[v];
#pragma unroll
            for (int i = 0; i < VN; ++i) acc[i] += in.get(i);
        }
        V16<XT> out;
#pragma unroll
        for (int i = 0; i < VN; ++i) out.set(i, acc[i] + dX_gate[t * d + v * VN + i]);
        reinterpret_cast<uint4 *>(dX + t * d)[v] = out.raw;
    }
}

}  // namespace

int64_t balanced_ws_bytes(int64_t T, int32_t n) {
    // p^T, per-token counts, loss partials, tile sums of the scan over the tokens
    const int64_t a = (T * n * 4 + 255) & ~255ll, c = (T * 4 + 255) & ~255ll, e = (cdiv(T, 8) * 8 + 255) & ~255ll;
    const int64_t f = (cdiv(T + 1, 4096) * 4 + 255) & ~255ll;
    return a + c + e + f + 256;
}

int32_t launch_balanced_gate(const void *x, int32_t act, int64_t T, int32_t d, int32_t n, int32_t k, const float *Wg,
                             const float *thr, float *logits, float *probs, uint32_t *mask_bits, int32_t *tok_of_row,
                             int32_t *offsets, float *den, int32_t *tok_ptr, int32_t *tok_rows, float *loss,
                             int32_t *thr_counts, void *ws, cudaStream_t st) {
    const int64_t R = T * k;
    const int32_t m = (int32_t)(R / n), words = (n + 31) / 32;
    Carver cv(ws);
    float *pT = cv.take<float>(T * n);
    int32_t *cnt = cv.take<int32_t>(T);
    double *loss_part = cv.take<double>(cdiv(T, 8));  // one per block of the token kernel, at most
    int32_t *tile_sums = cv.take<int32_t>(cdiv(T + 1, 4096));
    MOE_CUDA(cudaMemsetAsync(mask_bits, 0, sizeof(uint32_t) * T * words, st));
    MOE_CUDA(cudaMemsetAsync(thr_counts, 0, sizeof(int32_t) * n, st));
    if (T == 0) {
        MOE_CUDA(cudaMemsetAsync(offsets, 0, sizeof(int32_t) * (n + 1), st));
        MOE_CUDA(cudaMemsetAsync(tok_ptr, 0, sizeof(int32_t), st));
        MOE_CUDA(cudaMemsetAsync(loss, 0, sizeof(float), st));
        return MOE_OK;
    }
    // logits by the fixed fma chain (one matrix: the projection kernel's second one is absent)
    MOE_TRY(launch_projection(x, act, T, d, n, Wg, nullptr, logits, nullptr, nullptr, 0, nullptr, 1, nullptr, st));
    const unsigned both = (unsigned)cdiv(T, 32);
    if (n <= 64) launch_kernel(bal_softmax_both_kernel<2>, both, 512, 0, st, logits, T, n, probs, pT);
    else if (n <= 128) launch_kernel(bal_softmax_both_kernel<4>, both, 512, 0, st, logits, T, n, probs, pT);
    else if (n <= 256) launch_kernel(bal_softmax_both_kernel<8>, both, 512, 0, st, logits, T, n, probs, pT);
    else {
        launch_kernel(bal_softmax_kernel, (unsigned)cdiv(T, 8), 256, 0, st, logits, T, n, probs);
        MOE_LAUNCHED();
        launch_kernel(bal_transpose_kernel, dim3((unsigned)cdiv(T, 32), (unsigned)cdiv(n, 32)), 256, 0, st, probs, T, n, pT);
    }
    MOE_LAUNCHED();
    if (T <= 8 * 1024) launch_kernel(bal_select_kernel<8>, (unsigned)n, 1024, 0, st, pT, T, n, m, words, tok_of_row, mask_bits);
    else if (T <= 32 * 1024) launch_kernel(bal_select_kernel<32>, (unsigned)n, 1024, 0, st, pT, T, n, m, words, tok_of_row, mask_bits);
    else launch_kernel(bal_select_kernel<0>, (unsigned)n, 1024, 0, st, pT, T, n, m, words, tok_of_row, mask_bits);
    MOE_LAUNCHED();
    const int32_t per_warp = tokens_per_warp(T);
    const int64_t tok_blocks = cdiv(T, 8 * per_warp);
    launch_kernel(bal_token_kernel, (unsigned)tok_blocks, 256, n * sizeof(int32_t), st, probs, mask_bits, thr, T, n, words, den, cnt,
                  thr_counts, loss_part, per_warp);
    MOE_LAUNCHED();
    launch_kernel(bal_loss_final_kernel, 1, 256, 0, st, loss_part, tok_blocks, loss);
    MOE_LAUNCHED();
    MOE_TRY(launch_exclusive_scan(cnt, (int32_t)T, tok_ptr, st, tile_sums));
    launch_kernel(bal_fill_kernel, (unsigned)cdiv(R > n ? R : n + 1, 256) + 1, 256, 0, st, tok_of_row, mask_bits, tok_ptr, R, n, m, words,
                                                                                tok_rows, offsets);
    MOE_LAUNCHED();
    return MOE_OK;
}

int32_t launch_balanced_gather(const void *x, int32_t act, const int32_t *tok_of_row, int64_t R, int64_t T, int32_t d,
                               void *xs, cudaStream_t st) {
    if (R == 0) return MOE_OK;
    if (act == MOE_BF16) launch_kernel(bal_gather_kernel<bf16>, (unsigned)cdiv(R, 8), 256, 0, st, (const bf16 *)x, tok_of_row, R, T, d, (bf16 *)xs);
    else launch_kernel(bal_gather_kernel<float>, (unsigned)cdiv(R, 8), 256, 0, st, (const float *)x, tok_of_row, R, T, d, (float *)xs);
    MOE_LAUNCHED();
    return MOE_OK;
}

int32_t launch_balanced_combine(const void *ys, int32_t act, const float *p, const float *den, const int32_t *tok_ptr,
                                const int32_t *tok_rows, int64_t T, int64_t R, int32_t n, int32_t m, int32_t d, void *y,
                                cudaStream_t st) {
    if (T == 0) return MOE_OK;
    if (act == MOE_BF16)
        launch_kernel(bal_combine_kernel<bf16>, (unsigned)imin(cdiv(T, 8), 148 * 8), 256, 0, st, (const bf16 *)ys, p, den, tok_ptr, tok_rows, T, R, n, m, d, (bf16 *)y);
    else
        launch_kernel(bal_combine_kernel<float>, (unsigned)imin(cdiv(T, 8), 148 * 8), 256, 0, st, (const float *)ys, p, den, tok_ptr, tok_rows, T, R, n, m, d, (float *)y);
    MOE_LAUNCHED();
    return MOE_OK;
}

int32_t launch_balanced_combine_bwd(const void *dY, const void *ys, int32_t act, const float *p, const float *den,
                                    const int32_t *tok_of_row, int64_t R, int64_t T, int32_t n, int32_t m, int32_t d,
                                    float *dG_row, void *dys, cudaStream_t st) {
    if (R == 0) return MOE_OK;
    if (act == MOE_BF16)
        launch_kernel(bal_combine_bwd_kernel<bf16>, (unsigned)cdiv(R, 8), 256, 0, st, (const bf16 *)dY, (const bf16 *)ys, p, den, tok_of_row, R, T, n, m, d, dG_row, (bf16 *)dys);
    else
        launch_kernel(bal_combine_bwd_kernel<float>, (unsigned)cdiv(R, 8), 256, 0, st, (const float *)dY, (const float *)ys, p, den, tok_of_row, R, T, n, m, d, dG_row, (float *)dys);
    MOE_LAUNCHED();
    return MOE_OK;
}

int32_t launch_balanced_gate_bwd(const float *p, const uint32_t *mask_bits, const float *den, const float *thr,
                                 const int32_t *tok_ptr, const int32_t *tok_rows, const float *dG_row,
                                 const int32_t *thr_counts, float w, int64_t T, int32_t n, int32_t m, float *dc,
                                 void *dsplit, float *dthr, cudaStream_t st) {
    const int32_t words = (n + 31) / 32;
    if (T > 0 && dsplit && n % 2 == 0 && n <= 256) {
        if (n <= 64)
            launch_kernel(bal_gate_bwd_pairs_kernel<1>, (unsigned)cdiv(T, 8), 256, 0, st, p, mask_bits, den, thr, tok_ptr, tok_rows, dG_row, w, T, n,
                          words, (bf16 *)dsplit);
        else
            launch_kernel(bal_gate_bwd_pairs_kernel<4>, (unsigned)cdiv(T, 8), 256, 0, st, p, mask_bits, den, thr, tok_ptr, tok_rows, dG_row, w, T, n,
                          words, (bf16 *)dsplit);
        MOE_LAUNCHED();
    } else if (T > 0) {
        launch_kernel(bal_gate_bwd_kernel, (unsigned)cdiv(T, 8), 256, 0, st, p, mask_bits, den, thr, tok_ptr, tok_rows, dG_row, w, T, n, m, words, dc,
                                                                  (bf16 *)dsplit);
        MOE_LAUNCHED();
    }
    launch_kernel(bal_dthr_kernel, (unsigned)cdiv(n, 256), 256, 0, st, thr_counts, n, T > 0 ? m : 0, w, dthr);
    MOE_LAUNCHED();
    return MOE_OK;
}

int32_t launch_balanced_dispatch_bwd(const void *dxs, int32_t act, const int32_t *tok_ptr, const int32_t *tok_rows,
                                     const float *dX_gate, int64_t T, int64_t R, int32_t d, void *dX, cudaStream_t st) {
    if (T == 0) return MOE_OK;
    if (act == MOE_BF16)
        launch_kernel(bal_dispatch_bwd_kernel<bf16>, (unsigned)cdiv(T, 8), 256, 0, st, (const bf16 *)dxs, tok_ptr, tok_rows, dX_gate, T, R, d, (bf16 *)dX);
    else
        launch_kernel(bal_dispatch_bwd_kernel<float>, (unsigned)cdiv(T, 8), 256, 0, st, (const float *)dxs, tok_ptr, tok_rows, dX_gate, T, R, d, (float *)dX);
    MOE_LAUNCHED();
    return MOE_OK;
}

}  // namespace moe
