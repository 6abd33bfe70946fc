// Noisy top-k gating (Section 2.1, Eq. 3-5): projection, noisy logits, KeepTopK, masked softmax.
#include <math_constants.h>
#include <string.h>

#include "moe_internal.cuh"

namespace moe {

// rows that a block of 256 threads takes: a thread per column as far as that goes
__host__ __device__ __forceinline__ int select_rows_per_block(int32_t n) { return n <= 64 ? 4 : n <= 128 ? 2 : 1; }

// ------------------------------------------------------------------------------------------
// Noisy logits H = clean + noise * softplus(raw) (Eq. 4), KeepTopK (Eq. 5) and the softmax over
// the kept entries (Eq. 3). A row is selected by one warp: each lane keeps the k+1 best of its columns in a
// sorted register list (value descending, then index ascending); k+1 rounds of a warp arg-max
// over the list heads then produce the global order. Lowest index wins ties everywhere.
// softplus is evaluated in double and rounded once, H by one fused multiply-add.
// ------------------------------------------------------------------------------------------
// STAGED (n > 32, few rows): the noisy logits of the block's rows are formed first, one column per thread and step, and parked
// in shared memory for the row's warp. The softplus in double is a chain of 3000 cycles, and a warp that walks a wide row
// alone goes through it n / 32 times (1019 rows of 256 columns: 14 us). Where the rows alone fill the chip with warps, the
// chains of different rows overlap and the unstaged form wins, which leaves no warp of a block idle (see launch_gate_select).
template <int KL, bool STAGED>  // KL: length of the per-lane sorted lists, >= k + 1
__global__ void __launch_bounds__(256) gate_select_kernel(const float *__restrict__ clean,
                                                          const float *__restrict__ raw,
                                                          const float *__restrict__ noise, int64_t rows, int32_t n,
                                                          int32_t k, int32_t *__restrict__ idx,
                                                          float *__restrict__ gates, float *__restrict__ kth_vals,
                                                          int32_t *__restrict__ kth_idx,
                                                          const int32_t *__restrict__ row_list,
                                                          const int32_t *__restrict__ row_count,
                                                          const int2 *__restrict__ row_span,
                                                          const int2 *__restrict__ chain_list, const HierMerge merge) {
    wait_previous_kernel();
    extern __shared__ float staged[];  // [rows of the block][n]
    const int lane = threadIdx.x & 31, rpb = STAGED ? select_rows_per_block(n) : blockDim.x >> 5;
    int64_t row = (int64_t)blockIdx.x * rpb + (threadIdx.x >> 5);
    auto noisy = [](float c, float r, float e) {
        const double rd = (double)r;
        const float sigma = (float)(fmax(rd, 0.0) + log1p(exp(-fabs(rd))));
        const float v = fmaf(e, sigma, c);
        return v == v ? v : -CUDART_INF_F;  // a NaN logit ranks last: the selection stays total, indices stay in [0, n)
    };
    if (STAGED) {
        const int64_t first = (int64_t)blockIdx.x * rpb * n, total = min((int64_t)rpb * n, rows * n - first);
        for (int i = threadIdx.x; i < total; i += 256) staged[i] = noisy(clean[first + i], raw[first + i], noise[first + i]);
        __syncthreads();
        if ((int)(threadIdx.x >> 5) >= rpb) return;
    }
    // row_span (with a row list): {first chain entry, number of candidate columns} of a listed row whose other
    // columns are known to rank below k + 1, so only the candidates are looked at; {., -1}: every column
    int32_t cand_base = 0, cand_total = -1;
    if (row_list) {  // only the listed rows (their number is read on the device)
        if (row >= *row_count) return;
        if (row_span) { const int2 sp = row_span[row]; cand_base = sp.x; cand_total = sp.y; }
        row = row_list[row];
    } else if (row >= rows) {
        return;
    }
    float lv[KL];
    int32_t li[KL];
#pragma unroll
    for (int s = 0; s < KL; ++s) { lv[s] = -CUDART_INF_F; li[s] = INT32_MAX; }
    const float *c = clean + row * n, *r = raw + row * n, *e = noise + row * n;
    const int32_t visits = cand_total >= 0 ? cand_total : n;
    for (int32_t q = lane; q < visits; q += 32) {
        // a candidate's column is the code of its first chain entry (the clean one), modulo the group's block of 2n
        const int32_t j = cand_total >= 0 ? chain_list[cand_base + 2 * q].y % (2 * n) : q;
        float v = STAGED ? staged[(threadIdx.x >> 5) * n + j] : noisy(c[j], r[j], e[j]);
        int32_t id = j;
        bool shifting = false;
#pragma unroll
        for (int s = 0; s < KL; ++s) {
            if (shifting || v > lv[s] || li[s] == INT32_MAX) {  // an empty slot takes anything, -inf included
                float tv = lv[s]; int32_t ti = li[s];
                lv[s] = v; li[s] = id; v = tv; id = ti;
                shifting = true;
            }
        }
    }
    const int rounds = (k < n) ? k + 1 : k;
    float myv = -CUDART_INF_F;
    int32_t myi = -1;
    float v_k = -CUDART_INF_F, v_k1 = -CUDART_INF_F;
    int32_t i_k = -1, i_k1 = -1;
    for (int s = 0; s < rounds; ++s) {
        float hv = lv[0];
        int32_t hi = li[0];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            float ov = __shfl_xor_sync(0xffffffffu, hv, off);
            int32_t oi = __shfl_xor_sync(0xffffffffu, hi, off);
            if (ov > hv || (ov == hv && oi < hi)) { hv = ov; hi = oi; }
        }
        if (li[0] == hi) {  // this lane held the winner: pop it
#pragma unroll
            for (int q = 0; q < KL - 1; ++q) { lv[q] = lv[q + 1]; li[q] = li[q + 1]; }
            lv[KL - 1] = -CUDART_INF_F;
            li[KL - 1] = INT32_MAX;
        }
        if (s < k && lane == s) { myv = hv; myi = hi; }
        if (s == k - 1) { v_k = hv; i_k = hi; }
        if (s == k) { v_k1 = hv; i_k1 = hi; }
    }
    // softmax over the k kept logits, denominator summed in slot order
    const float m = __shfl_sync(0xffffffffu, myv, 0);
    const float ex = lane < k ? expf(myv - m) : 0.0f;
    float den = 0.0f;
    for (int s = 0; s < k; ++s) den += __shfl_sync(0xffffffffu, ex, s);
    if (lane < k) {
        const float g = ex / den;
        idx[row * k + lane] = myi;
        gates[row * k + lane] = g;
        if (merge.idx) merge.put(row, k, lane, myi, g);
    }
    if (lane == 0) {
        kth_vals[row * 2 + 0] = v_k;
        kth_vals[row * 2 + 1] = v_k1;
        kth_idx[row * 2 + 0] = i_k;
        kth_idx[row * 2 + 1] = i_k1;
    }
}

int32_t launch_gate_select(const float *clean, const float *raw, const float *noise, int64_t rows, int32_t n,
                           int32_t k, int32_t *idx, float *gates, float *kth_vals, int32_t *kth_idx,
                           cudaStream_t st, const int32_t *row_list, const int32_t *row_count, const void *row_span,
                           const void *chain_list, const HierMerge &merge) {
    if (rows == 0) return MOE_OK;
    // Staged up to eight rows per SM, wider rows up to n / 32 of them. A whole moe_gate with 16 features, staged / unstaged us:
    // n = 129 (half of a step's threads idle): 1019 rows 12.3 / 11.8, 2048 rows 15.8 / 13.2, 65536 rows 239 / 170; n = 256: 12.1 / 13.6,
    // 16.5 / 15.7, 290 / 236; n = 512: 1019 rows 16.6 / 21.0, 2048 rows 22.0 / 23.5, 3000 rows 31.5 / 30.8, 32768 rows 260 / 224; n = 4096:
    // 2048 rows 129 / 156, 4096 rows 246 / 259.
    const bool stage = n > 32 && !row_list && rows <= 148 * (int64_t)(n >= 256 ? n / 32 : 8);
    const int rpb = stage ? select_rows_per_block(n) : 8;
    const unsigned grid = (unsigned)cdiv(rows, rpb);
    const size_t sh = stage ? sizeof(float) * rpb * n : 0;  // at most 32 KiB
#define MOE_SELECT_AS(KL, STAGED)                                                                                        \
    launch_kernel((gate_select_kernel<KL, STAGED>), grid, 256, sh, st, clean, raw, noise, rows, n, k, idx, gates, kth_vals, \
                  kth_idx, row_list, row_count, (const int2 *)row_span, (const int2 *)chain_list, merge)
#define MOE_SELECT(KL)                        \
    do {                                      \
        if (stage) MOE_SELECT_AS(KL, true);   \
        else MOE_SELECT_AS(KL, false);        \
    } while (0)
    if (k <= 2) MOE_SELECT(3);
    else if (k <= 4) MOE_SELECT(5);
    else MOE_SELECT(MOE_MAX_K + 1);
#undef MOE_SELECT_AS
#undef MOE_SELECT
    MOE_LAUNCHED();
    return MOE_OK;
}

// ------------------------------------------------------------------------------------------
// Tensor-core screening of the routing (bf16 activations). The projection x.[W_g|W_noise] is first
// done on the tensor cores with W split into three bf16 terms (~1e-7 of the fma-chain value). From
// those approximate logits each token's top-(k+2) is found together with a bound U on how far any
// approximate noisy logit can be from the value the fixed fma chain would give:
//     |H~_j - H_j| <= theta * |x|_2 * (|W_g[:,j]|_2 + |noise_j| * |W_noise[:,j]|_2) + rounding slack,
// theta covering the worst-case rounding of the chain (d * 2^-24) and of the tensor-core accumulation
// (modelled as one truncation of an fp32 accumulator per MMA step, doubled). If every gap between
// consecutive ranks 1..k+2 exceeds 2U, the order of the top k+1 under the chain values is provably the
// same, so the routing taken from the approximate logits IS the bit-exact routing. The other tokens
// (a few per cent) are listed and redone with the fma chain by the kernels above.
// ------------------------------------------------------------------------------------------
// What the screen needs beside its product, in one launch. The first blocks take 32 columns of [W_g | W_noise] each (of one group
// where matrices are stacked [groups, d, n]) and walk down the features, four 32 x 32 tiles in flight: the three-term bf16 split
// wsplit [3][groups * d][2n], the transposed weights wt [groups][2n][d] for single chains, and the columns' norms (slightly rounded
// up) wnorm [groups][2n]. The other blocks: |x_t|_2 (slightly rounded up), one warp per row, 16 bytes per lane, four loads in flight.
__global__ void __launch_bounds__(256) gate_prepare_kernel(const bf16 *__restrict__ x, int64_t T, int32_t d, int32_t n,
                                                           const float *__restrict__ Wg, const float *__restrict__ Wn,
                                                           int32_t groups, bf16 *__restrict__ wsplit, float *__restrict__ wt,
                                                           float *__restrict__ wnorm, float *__restrict__ xnorm,
                                                           int32_t *__restrict__ counters, int32_t *__restrict__ clear) {
    wait_previous_kernel();
    const int32_t n2 = 2 * n, column_blocks = groups * (n2 / 32);
    if ((int32_t)blockIdx.x >= column_blocks) {
        const int lane = threadIdx.x & 31;
        const int64_t t = (int64_t)(blockIdx.x - column_blocks) * 8 + (threadIdx.x >> 5);
        if (t >= T) return;
        float s = 0.0f;
        const uint4 *row = reinterpret_cast<const uint4 *>(x + t * d);
        const int32_t pieces = d / 8;
        for (int32_t q0 = lane; q0 < pieces; q0 += 128) {
            uint4 v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = q0 + 32 * i < pieces ? row[q0 + 32 * i] : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const bf16 *h = reinterpret_cast<const bf16 *>(&v[i]);
#pragma unroll
                for (int e = 0; e < 8; ++e) { const float f = __bfloat162float(h[e]); s = fmaf(f, f, s); }
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) xnorm[t] = sqrtf(s) * (1.0f + 1e-5f);
        return;
    }
    if (blockIdx.x == 0) {  // rows to re-select, chains, full-chain rows; the status word
        if (threadIdx.x < 4) counters[threadIdx.x] = 0;
        if (threadIdx.x == 4 && clear) *clear = 0;
    }
    __shared__ float tile[4][32][33];
    __shared__ double sums[8][32];
    const int32_t group = blockIdx.x / (n2 / 32), c0 = (blockIdx.x % (n2 / 32)) * 32;  // 2n and d are multiples of 64 on this path
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int32_t c = c0 + tx;
    const float *W = (c < n ? Wg + c : Wn + (c - n)) + (int64_t)group * d * n;
    wt += ((int64_t)group * n2 + c0) * d;
    double sum = 0.0;
    for (int32_t q0 = 0; q0 < d; q0 += 128) {
        const int tiles = min(4, (d - q0) / 32);
        float v[4][4];
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int i = 0; i < 4; ++i) v[b][i] = b < tiles ? W[(int64_t)(q0 + 32 * b + ty + 8 * i) * n] : 0.0f;
        __syncthreads();  // the tiles before have been read
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (b >= tiles) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float f = v[b][i];
                sum += (double)f * (double)f;
                tile[b][ty + 8 * i][tx] = f;
                const int64_t q = (int64_t)group * d + q0 + 32 * b + ty + 8 * i;
#pragma unroll
                for (int term = 0; term < 3; ++term) {  // hi, mid, lo
                    const bf16 h = __float2bfloat16_rn(f);
                    wsplit[((int64_t)term * groups * d + q) * n2 + c] = h;
                    f -= __bfloat162float(h);
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (b >= tiles) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) wt[(int64_t)(ty + 8 * i) * d + q0 + 32 * b + tx] = tile[b][tx][ty + 8 * i];
        }
    }
    sums[ty][tx] = sum;
    __syncthreads();
    if (ty == 0) {
        double s = sums[0][tx];
#pragma unroll
        for (int q = 1; q < 8; ++q) s += sums[q][tx];
        wnorm[group * n2 + c] = (float)(sqrt(s) * (1.0 + 1e-6));
    }
}

// Approximate noisy logit v of one column and a bound u on its distance from the fma chain's value; c, r = the
// tensor-core products, e = the noise, xn = theta |x|, wg / wn = the column norms of W_g / W_noise. Both screening
// kernels call this one function, written with the non-contracting intrinsics so that they get the same bits.
// The hardware exponential and logarithm are enough here: their error is an absolute 7.2e-7 at most on sigma (2.4e-7
// from __expf on [-inf, 0], 1.2e-7 from rounding 1 + y, 2^-21.41 from __logf on [1, 2]) and goes into u with a margin
// (2e-6 |noise|).
__device__ __forceinline__ void screen_eval(float c, float r, float e, float xn, float wg, float wn, float &v, float &u) {
    const float sigma = __fadd_rn(fmaxf(r, 0.0f), __logf(__fadd_rn(1.0f, __expf(-fabsf(r)))));
    v = __fmaf_rn(e, sigma, c);
    // |H~_j - H_j|: projection errors through c and through softplus(r) (slope <= 1) times |noise|, plus the error of
    // softplus (here approximate, there double rounded once) and of the final fma on both sides
    const float ae = fabsf(e);
    const float rounding = __fmul_rn(1.1920929e-7f, __fmaf_rn(16.0f * ae, sigma, 8.0f * fabsf(v)));
    u = __fmaf_rn(2.0e-6f, ae, __fmaf_rn(xn, __fmaf_rn(ae, wn, wg), rounding));
}

// The screen. P adjacent lanes take a row (sorted row): each walks every P-th quad of its columns, one quad ahead in registers,
// and keeps a sorted list of the KL >= k + 2 largest approximate logits with their
// bounds and the largest possible value of everything else; the P lists are then merged by exchanging them. Bound by the
// arithmetic of the list where the rows fill the chip, by the latency of one lane's walk where they do not, hence P by the
// number of rows (see launch_gate_screen). Certified rows get their routing here; the others are listed with `low`, the
// bound that decides which of their columns need an exact chain (gate_candidates_kernel).
// Grouped use (secondary gates of the hierarchical layer): neighbours in a warp are of one group; perm maps a sorted row to its
// row (the slot t * k1 + s1), the token is output row / kdiv, group_of gives the slot's group, whose column
// norms are used. Flat use: perm = group_of = nullptr, kdiv = 1.
// four floats at p: one 16-byte access where the tensor allows it (V16), else four 4-byte ones (the secondary gates'
// part of noise / clean / raw starts T * a floats into the tensor, not always a multiple of four)
template <bool V16>
__device__ __forceinline__ float4 load4(const float *p) {
    if constexpr (V16) return *reinterpret_cast<const float4 *>(p);
    else return make_float4(p[0], p[1], p[2], p[3]);
}
template <int KL, int P, bool V16>
__global__ void __launch_bounds__(128) gate_screen_rows_kernel(const float *__restrict__ noise,
                                                               const float *__restrict__ xnorm,
                                                               const float *__restrict__ wnorm, float theta, int64_t T,
                                                               int32_t n, int32_t k, int32_t *__restrict__ idx,
                                                               float *__restrict__ gates, const float *__restrict__ clean,
                                                               const float *__restrict__ raw, float *__restrict__ kth_vals,
                                                               int32_t *__restrict__ kth_idx,
                                                               int32_t *__restrict__ unsafe_list,
                                                               float *__restrict__ unsafe_low,
                                                               int32_t *__restrict__ unsafe_count,
                                                               const int32_t *__restrict__ perm, int32_t kdiv,
                                                               const int32_t *__restrict__ group_of, const HierMerge merge) {
    wait_previous_kernel();
    const int lane = threadIdx.x & 31, sub = lane % P;
    const int64_t s0 = ((int64_t)blockIdx.x * 4 + (threadIdx.x >> 5)) * (32 / P);  // first sorted row of this warp
    if (s0 >= T) return;
    const int64_t srow = s0 + lane / P;
    const bool live = srow < T;
    const int64_t row = live ? (perm ? (int64_t)perm[srow] : srow) : 0;
    const float *wn = wnorm + (int64_t)(group_of && live ? group_of[row] : 0) * 2 * n;
    const float xn = live ? theta * xnorm[row / kdiv] : 0.0f;
    float lv[KL], lu[KL];
    int32_t li[KL];
#pragma unroll
    for (int s = 0; s < KL; ++s) { lv[s] = -CUDART_INF_F; li[s] = INT32_MAX; lu[s] = 0.0f; }
    float rest_hi = -CUDART_INF_F;  // largest possible chain value of anything that is not in the list
    auto insert = [&](int32_t j, float v, float u) {
        if (v > lv[KL - 1]) {
            // enters the list behind every entry that is at least as large, the last entry falls off (equal values are
            // never certified: their order does not matter here)
            rest_hi = fmaxf(rest_hi, lv[KL - 1] + lu[KL - 1]);
#pragma unroll
            for (int s = KL - 1; s >= 1; --s) {
                const bool stays = lv[s] >= v && s != KL - 1, here = lv[s - 1] >= v;
                if (!stays) {
                    lv[s] = here ? v : lv[s - 1];
                    lu[s] = here ? u : lu[s - 1];
                    li[s] = here ? j : li[s - 1];
                }
            }
            if (!(lv[0] >= v)) { lv[0] = v; lu[0] = u; li[0] = j; }
        } else {
            rest_hi = fmaxf(rest_hi, v + u);
        }
    };
    // four columns at a time: their values and bounds first (independent of each other, so the exponentials and
    // logarithms overlap), then the four list updates, which depend on one another
    auto consider4 = [&](int32_t j, const float4 &c4, const float4 &r4, const float4 &e4) {
        const float4 wg4 = *reinterpret_cast<const float4 *>(wn + j), wn4 = *reinterpret_cast<const float4 *>(wn + n + j);
        float v0, v1, v2, v3, u0, u1, u2, u3;
        screen_eval(c4.x, r4.x, e4.x, xn, wg4.x, wn4.x, v0, u0);
        screen_eval(c4.y, r4.y, e4.y, xn, wg4.y, wn4.y, v1, u1);
        screen_eval(c4.z, r4.z, e4.z, xn, wg4.z, wn4.z, v2, u2);
        screen_eval(c4.w, r4.w, e4.w, xn, wg4.w, wn4.w, v3, u3);
        insert(j, v0, u0);
        insert(j + 1, v1, u1);
        insert(j + 2, v2, u2);
        insert(j + 3, v3, u3);
    };
    const float *cp = clean + row * n + 4 * sub, *rp = raw + row * n + 4 * sub, *ep = noise + row * n + 4 * sub;  // a dead lane walks row 0
    float4 c4 = load4<V16>(cp), r4 = load4<V16>(rp), e4 = load4<V16>(ep);  // n is a multiple of 4 P
    for (int32_t j0 = 0; j0 < n; j0 += 4 * P) {
        const int32_t next = j0 + 4 * P;
        float4 cn = c4, rn = r4, en = e4;
        if (next < n) { cn = load4<V16>(cp + next); rn = load4<V16>(rp + next); en = load4<V16>(ep + next); }
        consider4(j0 + 4 * sub, c4, r4, e4);
        c4 = cn; r4 = rn; e4 = en;
    }
#pragma unroll
    for (int off = 1; off < P; off <<= 1) {  // afterwards every lane of the row holds the list of all columns
        float ov[KL], ou[KL];
        int32_t oi[KL];
#pragma unroll
        for (int s = 0; s < KL; ++s) {
            ov[s] = __shfl_xor_sync(0xffffffffu, lv[s], off);
            ou[s] = __shfl_xor_sync(0xffffffffu, lu[s], off);
            oi[s] = __shfl_xor_sync(0xffffffffu, li[s], off);
        }
        rest_hi = fmaxf(rest_hi, __shfl_xor_sync(0xffffffffu, rest_hi, off));
#pragma unroll
        for (int s = 0; s < KL; ++s) insert(oi[s], ov[s], ou[s]);
    }
    // the first `rounds` entries are the ranked ones, whatever else is in the list is "rest" as well
    const int rounds = min(k + 2, n);
#pragma unroll
    for (int s = 0; s < KL; ++s)
        if (s >= rounds && li[s] != INT32_MAX) rest_hi = fmaxf(rest_hi, lv[s] + lu[s]);
    // ranks 1..k+1 are certain iff each one's lowest possible value beats the highest possible value of everything
    // ranked after it
    bool safe = true;
    float suffix = rest_hi;
#pragma unroll
    for (int s = KL - 1; s >= 0; --s) {
        if (s < rounds) {
            if (s <= k && !(lv[s] - lu[s] > suffix)) safe = false;
            suffix = fmaxf(suffix, lv[s] + lu[s]);
        }
    }
    // Not provably the chain's routing: only the columns that can still reach rank k+1 matter, those whose highest
    // possible value is at least `low`, a lower bound of the (k+1)-th largest chain value (the (k+1)-th largest lower end
    // among the ranked columns).
    float low = -CUDART_INF_F;
    if (!safe && k < rounds) {
#pragma unroll
        for (int s = 0; s < KL; ++s) {
            if (s < rounds) {
                const float ls = lv[s] - lu[s];
                int above = 0;
#pragma unroll
                for (int s2 = 0; s2 < KL; ++s2)
                    if (s2 < rounds && s2 != s) {
                        const float l2 = lv[s2] - lu[s2];
                        above += (l2 > ls || (l2 == ls && s2 < s)) ? 1 : 0;
                    }
                if (above == k) low = ls;
            }
        }
    }
    const bool listed = live && !safe && sub == 0;  // one lane of a row reports it
    const uint32_t lb = __ballot_sync(0xffffffffu, listed);
    if (lb) {
        int32_t base = 0;
        if (lane == 0) base = atomicAdd(unsafe_count, __popc(lb));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (listed) {
            const int32_t at = base + __popc(lb & ((1u << lane) - 1u));
            unsafe_list[at] = (int32_t)row;
            unsafe_low[at] = low;
        }
    }
    if (!live || !safe || sub != 0) return;
    float ex[KL], den = 0.0f;
#pragma unroll
    for (int s = 0; s < KL; ++s) {
        ex[s] = 0.0f;
        if (s < k) { ex[s] = expf(lv[s] - lv[0]); den += ex[s]; }
    }
#pragma unroll
    for (int s = 0; s < KL; ++s)
        if (s < k) {
            const float g = ex[s] / den;
            idx[row * k + s] = li[s];
            gates[row * k + s] = g;
            if (merge.idx) merge.put(row, k, s, li[s], g);
        }
    float v_k = -CUDART_INF_F, v_k1 = -CUDART_INF_F;
    int32_t i_k = -1, i_k1 = -1;
#pragma unroll
    for (int s = 0; s < KL; ++s) {
        if (s == k - 1) { v_k = lv[s]; i_k = li[s]; }
        if (s == k && k < n) { v_k1 = lv[s]; i_k1 = li[s]; }
    }
    kth_vals[row * 2 + 0] = v_k;
    kth_vals[row * 2 + 1] = v_k1;
    kth_idx[row * 2 + 0] = i_k;
    kth_idx[row * 2 + 1] = i_k1;
}

// The rows the screen listed, one warp per row: the columns whose highest possible value reaches the row's `low` get
// their two fma chains redone (chain_list), the selection is then repeated on the patched row. Rows with more than
// SCREEN_MAX_CAND candidates (ties) take the full chain (full_list), or, where there is no whole-row fallback
// (full_list == nullptr), the chains of all their columns.
__global__ void __launch_bounds__(256) gate_candidates_kernel(const float *__restrict__ clean, const float *__restrict__ raw,
                                                              const float *__restrict__ noise,
                                                              const float *__restrict__ xnorm,
                                                              const float *__restrict__ wnorm, float theta, int32_t n,
                                                              const int32_t *__restrict__ unsafe_list,
                                                              const float *__restrict__ unsafe_low,
                                                              int32_t *__restrict__ unsafe_count,
                                                              int2 *__restrict__ chain_list,
                                                              int32_t *__restrict__ full_list, int32_t kdiv,
                                                              const int32_t *__restrict__ group_of, int32_t k,
                                                              int2 *__restrict__ unsafe_span) {
    wait_previous_kernel();
    // unsafe_span[i] = {first entry of the row's chains in chain_list, number of candidate columns}, or {0, -1}
    // where the repeated selection has to look at every column
    const int lane = threadIdx.x & 31;
    const int32_t total_rows = *unsafe_count;  // complete: the screen ran before this kernel
    const int32_t nwarps = gridDim.x * (blockDim.x >> 5);
    for (int32_t it = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < total_rows; it += nwarps) {
        const int64_t row = unsafe_list[it];
        const float low = unsafe_low[it];
        const int32_t group = group_of ? group_of[row] : 0;
        const float *wn = wnorm + (int64_t)group * 2 * n;
        const float xn = theta * xnorm[row / kdiv];
        const float *c = clean + row * n, *r = raw + row * n, *e = noise + row * n;
        auto candidate = [&](int32_t j) {
            if (j >= n) return false;
            float v, u;
            screen_eval(c[j], r[j], e[j], xn, wn[j], wn[n + j], v, u);
            return v + u >= low;
        };
        // one pass over the row: lane g keeps the ballot of the g-th group of 32 columns (rows wider than 1024
        // columns are evaluated again when their entries are written)
        int total = 0;
        uint32_t kept_word = 0u;
        for (int32_t j0 = 0; j0 < n; j0 += 32) {
            const uint32_t b = __ballot_sync(0xffffffffu, candidate(j0 + lane));
            if ((j0 >> 5) == lane) kept_word = b;
            total += __popc(b);
        }
        // (fewer than k + 1 candidates happens only with NaN logits, which are nobody's candidate)
        const bool few = total <= SCREEN_MAX_CAND && total >= min(k + 1, n);
        const int32_t wbase = group * 2 * n;  // this group's rows of the transposed weights
        int32_t base = 0;
        if (lane == 0) {
            if (few) base = atomicAdd(unsafe_count + 1, 2 * total);
            else if (full_list) full_list[atomicAdd(unsafe_count + 2, 1)] = (int32_t)row;
            else base = atomicAdd(unsafe_count + 1, 2 * n);
        }
        base = __shfl_sync(0xffffffffu, base, 0);
        if (lane == 0) unsafe_span[it] = few ? make_int2(base, total) : make_int2(0, -1);
        if (!few) {
            if (!full_list)
                for (int32_t j = lane; j < n; j += 32) {
                    chain_list[base + 2 * j] = make_int2((int32_t)row, wbase + j);
                    chain_list[base + 2 * j + 1] = make_int2((int32_t)row, wbase + n + j);
                }
            continue;
        }
        int pos = 0;
        for (int32_t j0 = 0; j0 < n; j0 += 32) {
            const int32_t j = j0 + lane;
            const uint32_t b = n <= 1024 ? __shfl_sync(0xffffffffu, kept_word, j0 >> 5)
                                         : __ballot_sync(0xffffffffu, candidate(j));
            const bool cand = (b >> lane) & 1u;
            if (cand) {
                const int at = base + 2 * (pos + __popc(b & ((1u << lane) - 1u)));
                chain_list[at] = make_int2((int32_t)row, wbase + j);
                chain_list[at + 1] = make_int2((int32_t)row, wbase + n + j);
            }
            pos += __popc(b);
        }
    }
}

// One fma chain per thread: entry (row, c) of chain_list recomputes clean[row, c] (c < n) or raw[row, c - n] exactly
// as the projection kernel does: fp32, from +0, ascending input feature. Wt [2n, d] holds the columns of
// [W_g | W_noise] as rows. The 32 chains of a warp read 32 different weight rows; a load instruction that touches 32
// lines costs the load/store unit 32 tag look-ups, which is what bounds this kernel, so the warp fetches the next 32
// features of its 32 rows cooperatively (eight lanes per 128-byte line, four lines per instruction), parks them in
// shared memory and every lane then reads its own row back. Loads for step s + 1 are in flight during the 32
// dependent fused multiply-adds of step s.
constexpr int CHAIN_PITCH = 144;  // bytes per staged row: 128 + 16, conflict-free both ways
__global__ void __launch_bounds__(128) gate_chain_kernel(const bf16 *__restrict__ x, int32_t d, int32_t n,
                                                         const float *__restrict__ Wt,
                                                         const int2 *__restrict__ chain_list,
                                                         const int32_t *__restrict__ chain_count,
                                                         float *__restrict__ clean, float *__restrict__ raw,
                                                         int32_t kdiv) {
    wait_previous_kernel();
    // entry {output row, row of Wt}: the token is output row / kdiv, the column code is Wt row mod 2n (grouped gates
    // keep one [2n, d] block of Wt per group)
    __shared__ __align__(16) uint8_t stage[4][2][32 * CHAIN_PITCH];
    const int32_t total = *chain_count;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int32_t steps = d / 32;  // d is a multiple of 64 on this path
    for (int32_t i0 = (blockIdx.x * 4 + wp) * 32; i0 < total; i0 += gridDim.x * 128) {  // warp-uniform
        const int32_t i = i0 + lane;
        const int2 en = chain_list[i < total ? i : total - 1];  // idle lanes shadow the last chain
        const bf16 *xr = x + (int64_t)(en.x / kdiv) * d;
        const float *wrow = Wt + (int64_t)en.y * d;
        // instruction u of a step loads 16 bytes of the row of lane 4 u + lane / 8, at byte (lane % 8) * 16
        const float *src[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const unsigned long long ptr = __shfl_sync(0xffffffffu, (unsigned long long)wrow, 4 * u + (lane >> 3));
            src[u] = reinterpret_cast<const float *>(ptr) + (lane & 7) * 4;
        }
        float4 wreg[8];
        uint4 xreg[4];
        auto fetch = [&](int32_t st) {
#pragma unroll
            for (int u = 0; u < 8; ++u) wreg[u] = *reinterpret_cast<const float4 *>(src[u] + st * 32);
#pragma unroll
            for (int g = 0; g < 4; ++g) xreg[g] = *reinterpret_cast<const uint4 *>(xr + st * 32 + 8 * g);
        };
        auto park = [&](int b) {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                *reinterpret_cast<float4 *>(&stage[wp][b][(4 * u + (lane >> 3)) * CHAIN_PITCH + (lane & 7) * 16]) = wreg[u];
        };
        float acc = 0.0f;
        fetch(0);
        __syncwarp();  // the previous chains' last reads of the staging rows are done
        park(0);
        uint4 xcur[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) xcur[g] = xreg[g];
        __syncwarp();
        for (int32_t st = 0; st < steps; ++st) {
            if (st + 1 < steps) fetch(st + 1);
            const uint8_t *mine = &stage[wp][st & 1][lane * CHAIN_PITCH];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float4 wv = *reinterpret_cast<const float4 *>(mine + 16 * u);
                const bf16 *hx = reinterpret_cast<const bf16 *>(&xcur[u >> 1]) + 4 * (u & 1);
                acc = fmaf(__bfloat162float(hx[0]), wv.x, acc); acc = fmaf(__bfloat162float(hx[1]), wv.y, acc);
                acc = fmaf(__bfloat162float(hx[2]), wv.z, acc); acc = fmaf(__bfloat162float(hx[3]), wv.w, acc);
            }
            if (st + 1 < steps) {
                park((st + 1) & 1);  // the other buffer: its readers finished a step ago (syncwarp below)
#pragma unroll
                for (int g = 0; g < 4; ++g) xcur[g] = xreg[g];
            }
            __syncwarp();
        }
        if (i < total) {
            const int32_t code = en.y % (2 * n);
            if (code >= n) raw[(int64_t)en.x * n + (code - n)] = acc;
            else clean[(int64_t)en.x * n + code] = acc;
        }
    }
}

int32_t launch_gate_chains(const void *x, int32_t d, int32_t n, const float *Wt, const void *chain_list,
                           const int32_t *chain_count, float *clean, float *raw, cudaStream_t st, int32_t kdiv) {
    launch_kernel(gate_chain_kernel, 148 * 16, 128, 0, st, (const bf16 *)x, d, n, Wt, (const int2 *)chain_list, chain_count, clean, raw, kdiv);
    MOE_LAUNCHED();
    return MOE_OK;
}

// Lanes a row: one lane's walk while the rows do not fill the chip, the arithmetic of the lists and their merging when they do. A whole
// moe_gate of 128 features, two kept of 256 columns, us with 8 / 4 / 2 lanes: 2048 rows 35.6 / 38.5 / 47.7, 16384 48.5 / 47.9 / 55.1,
// 32768 81.2 / 76.2 / 81.0, 65536 135.0 / 125.7 / 123.1, 131072 227 / 215 / 212. (Narrower or with more kept the lines lie a little
// lower: 64 columns, four kept, 24576 rows 49.7 / 44.0 / 41.9.)
static int screen_lanes(int64_t rows) { return rows >= 65536 ? 2 : rows >= 16384 ? 4 : 8; }

int32_t launch_gate_screen_prepare(const void *x, int64_t T, int32_t d, int32_t n, const float *Wg, const float *Wn, void *wsplit,
                                   float *wnorm, float *xnorm, int32_t *unsafe_count, float *wt, cudaStream_t st, int32_t groups,
                                   bool with_xnorm, int32_t *clear) {
    // groups > 1: Wg, Wn are stacks [groups, d, n]; wsplit [3][groups * d][2n], wnorm [groups][2n], wt [groups][2n][d]
    const int64_t blocks = (int64_t)groups * (2 * n / 32) + (with_xnorm ? cdiv(T, 8) : 0);
    launch_kernel(gate_prepare_kernel, (unsigned)blocks, 256, 0, st, (const bf16 *)x, T, d, n, Wg, Wn, groups, (bf16 *)wsplit, wt, wnorm,
                  xnorm, unsafe_count, clear);
    MOE_LAUNCHED();
    return MOE_OK;
}

int32_t launch_gate_screen(const float *noise, const float *xnorm, const float *wnorm,
                           int32_t d, int64_t T, int32_t n, int32_t k, int32_t *idx, float *gates, float *clean, float *raw,
                           float *kth_vals, int32_t *kth_idx, int32_t *unsafe_list, float *unsafe_low, int32_t *unsafe_count,
                           void *chain_list, int32_t *full_list, void *unsafe_span, cudaStream_t st, const int32_t *perm, int32_t kdiv,
                           const int32_t *group_of, const HierMerge &merge) {
    // worst-case rounding of the fma chain, plus two truncations of an fp32 accumulator per MMA step of the
    // three-term tensor-core product (3d/16 steps and the additions inside a step), plus the split residual
    const double u = ldexp(1.0, -24);
    const double chain = d * u / (1.0 - d * u);
    const double tc = 2.0 * (3.0 * d / 16.0 + 8.0) * ldexp(1.0, -23) + ldexp(1.0, -22);
    const float theta = (float)((chain + tc) * 1.01);
    if (T == 0) return MOE_OK;
    if (n % 32 != 0) return MOE_ERR_INVALID_ARG;  // the screened path has 2n a multiple of 64
    const bool v16 = (((uintptr_t)noise | (uintptr_t)clean | (uintptr_t)raw) & 15) == 0;
    const int p = screen_lanes(T);
#define MOE_SCREEN(KL, P, V16)                                                                                                     \
    launch_kernel((gate_screen_rows_kernel<KL, P, V16>), (unsigned)cdiv(T, 4 * (32 / P)), 128, 0, st, noise, xnorm, wnorm, theta, T, n, \
                  k, idx, gates, clean, raw, kth_vals, kth_idx, unsafe_list, unsafe_low, unsafe_count, perm, kdiv, group_of, merge)
#define MOE_SCREEN_P(KL, P)                    \
    do {                                       \
        if (v16) MOE_SCREEN(KL, P, true);      \
        else MOE_SCREEN(KL, P, false);         \
    } while (0)
#define MOE_SCREEN_KL(KL)                      \
    do {                                       \
        if (p == 2) MOE_SCREEN_P(KL, 2);       \
        else if (p == 4) MOE_SCREEN_P(KL, 4);  \
        else MOE_SCREEN_P(KL, 8);              \
    } while (0)
    if (k <= 2) MOE_SCREEN_KL(4);
    else if (k <= 4) MOE_SCREEN_KL(6);
    else MOE_SCREEN_KL(MOE_MAX_K + 2);
#undef MOE_SCREEN_KL
#undef MOE_SCREEN_P
#undef MOE_SCREEN
    MOE_LAUNCHED();
    launch_kernel(gate_candidates_kernel, 148 * 4, 256, 0, st, clean, raw, noise, xnorm, wnorm, theta, n, unsafe_list, unsafe_low,
                  unsafe_count, (int2 *)chain_list, full_list, kdiv, group_of, k, (int2 *)unsafe_span);
    MOE_LAUNCHED();
    return MOE_OK;
}

MOE_BOUNDS_READER(bounds_violations_gate)

}  // namespace moe
