// Strided SIMT grouped GEMM in float accumulation. It serves the largest float projections and those of short single-float rows (the others:
// projection.cu), the first product of float layers and of bf16 layers of odd widths and, with many rows an expert, the other ones of widths that are no multiples of 64 or of little
// work (else: products_f32.cu, few_rows.cu), and the contractions of the gate backward where neither the tensor cores (ffn_tc.cu) nor
// gate_products.cu take them.
//
// Every output is one chain of fused multiply-adds over the contraction index in ascending order, starting from +0
// (contractions cut into slices: one such chain per slice, the slices added in double). That is bound by the FP32
// pipes where the grid fills the chip and by the length of the chain where it does not, so the tile is chosen by the
// number of blocks it leaves (see pick_tile). Operand tiles go through registers into one of two shared-memory buffers
// while the other one is used: one barrier per K block, the loads of a block are in flight during the arithmetic of
// the one before, and the shared-memory reads of step k + 1 during the arithmetic of step k.
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "sums.cuh"

namespace moe {

namespace {

template <typename T> __device__ __forceinline__ float ld_as_f32(const void *p, int64_t i) {
    return to_f32(reinterpret_cast<const T *>(p)[i]);
}
// two fused multiply-adds with one instruction (each rounded as fmaf rounds it): c += a * b
__device__ __forceinline__ void fma_pair(float &c0, float &c1, float a, float b0, float b1) {
    asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%2, %2};\n mov.b64 b, {%3, %4};\n mov.b64 c, {%0, %1};\n"
        " fma.rn.f32x2 c, a, b, c;\n mov.b64 {%0, %1}, c;\n}"
        : "+f"(c0), "+f"(c1) : "f"(a), "f"(b0), "f"(b1));
}
// four consecutive elements as they lie in memory (aligned to their size), converted where they are stored: a conversion
// next to the load would wait for it
template <typename T> struct Quad;
template <> struct Quad<float> {
    float4 raw;
    __device__ __forceinline__ void load(const float *p) { raw = *reinterpret_cast<const float4 *>(p); }
    __device__ __forceinline__ void clear() { raw = make_float4(0.0f, 0.0f, 0.0f, 0.0f); }
    __device__ __forceinline__ void set(int i, float v) { reinterpret_cast<float *>(&raw)[i] = v; }
    __device__ __forceinline__ float4 get() const { return raw; }
};
template <> struct Quad<bf16> {
    uint2 raw;
    __device__ __forceinline__ void load(const bf16 *p) { raw = *reinterpret_cast<const uint2 *>(p); }
    __device__ __forceinline__ void clear() { raw = make_uint2(0u, 0u); }
    __device__ __forceinline__ void set(int i, bf16 v) { reinterpret_cast<bf16 *>(&raw)[i] = v; }
    __device__ __forceinline__ float4 get() const {
        return make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u), __uint_as_float(raw.y << 16),
                           __uint_as_float(raw.y & 0xffff0000u));
    }
};

struct SimtRun {
    SimtGemm g;
    const int32_t *tile_prefix;
    int32_t vec_c;       // four elements along a row of C can be stored at once
    int32_t splits;      // mode 1: the contraction range of a segment is cut into this many slices
    const SegmentPlan *plan;  // host side: tile prefixes made already, or nullptr
    float *part;         // splits > 1: [splits][nseg][M][N] partial results instead of C
    GateParts *parts_left;  // host side: where a product over one segment leaves its partial results to be added later, or nullptr
};

// AK: A(i, k) is contiguous along k (else along i); BJ: B(k, j) is contiguous along j (else along k). QA4, QB4: quads of A / B can
// be loaded at once (extents, strides, addresses and the border between two concatenated matrices are multiples of four
// elements). Their loads are not guarded by branches: a quad outside the operand reads the operand's first elements
// instead and counts as zero.
template <typename TA, typename TB, typename TC, bool QA4, bool QB4, bool AK, bool BJ, int BM, int BN, int TM, int TN, int BK>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), TM * TN >= 64 ? 3 : TM * TN >= 32 ? 4 : 8) simt_gemm_kernel(const __grid_constant__ SimtRun run) {
    wait_previous_kernel();
    constexpr int NTX = BN / TN, NTY = BM / TM, NT = NTX * NTY;
    // An operand whose contraction index is the contiguous one is stored transposed, four elements of a quad in four rows of the
    // tile: the lanes of a warp hold BK / 4 quads of 128 / BK tile rows, and without a swizzle those stores met in a few banks (four
    // to a bank at 32 x 32 x 32). Tile row i of step k stands at i ^ swizzle(k). The reads of every step pay for it, so only where both
    // operands are stored that way, or one of two bytes an element in 32 x 32 tiles, and not in the larger tiles, where two stores meet
    // (the backward products of 256 experts x 16 rows of 256 x 256 floats 229 us, without 240; a whole forward call with a gate of
    // 1019 x 512 x 512 145.0, without 146.9; but a gate of 24 x 512 x 64 12.1, without 11.3, of 4000 x 256 x 64 floats
    // 14.1, 13.4, and 4170 x 512 x 256 in larger tiles 41, 38).
    constexpr int LDA = BM + 4, LDB = BN + 4;
    constexpr bool SWZ = AK && (BJ ? BM * BN == 32 * 32 && sizeof(TA) == 2 : BM * BN <= 32 * 32);
    constexpr int SWZ_UNIT = BK <= 32 ? 128 / BK : 4, SWZ_K = BK <= 32 ? 4 : 8;
    auto swizzle_a = [](int k) { return SWZ && AK ? (k / SWZ_K % ((BM < 32 ? BM : 32) / SWZ_UNIT)) * SWZ_UNIT : 0; };
    auto swizzle_b = [](int k) { return SWZ && !BJ ? (k / SWZ_K % ((BN < 32 ? BN : 32) / SWZ_UNIT)) * SWZ_UNIT : 0; };
    constexpr int QA = BM * BK / 4 / NT, QB = BN * BK / 4 / NT;  // quads a thread stages per K block
    constexpr int VA = TM < 4 ? TM : 4, VB = TN < 4 ? TN : 4;    // rows / columns per shared-memory read
    static_assert(QA * NT * 4 == BM * BK && QB * NT * 4 == BN * BK, "whole quads per thread");
    // A projection onto weights of any width: a thread loads one column of B element by element, so that a warp's loads are
    // adjacent and the choice between the two matrices is made once. (As guarded quads, four elements apart between the
    // lanes, 32768 tokens x 512 features x 500 columns took 950 us, this way 400.)
    constexpr bool COL_B = !QB4 && AK && BJ;
    static_assert(!COL_B || NT % BN == 0, "a thread's column");
    static_assert(NT % (BK / 4) == 0 && NT % (BM / 4) == 0 && NT % (BN / 4) == 0, "a thread's quads are a fixed step apart");
    __shared__ __align__(16) float As[2][BK * LDA];
    __shared__ __align__(16) float Bs[2][BK * LDB];
    __shared__ int4 tile_at;
    const SimtGemm &g = run.g;
    if (g.clear && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) *g.clear = 0;
    const int tid = threadIdx.x, tx = tid % NTX, ty = tid / NTX;

    int64_t m0, m_end, kbeg, kend;
    int32_t e = 0, slice = 0;
    if (g.mode == 0) {
        if (g.offsets) {
            const int4 at = segment_of_tile(run.tile_prefix, g.offsets, g.nseg, blockIdx.x, &tile_at);
            if (at.x < 0) return;
            e = at.x;
            m0 = at.y + (int64_t)at.w * BM;
            m_end = at.z;
        } else {
            m0 = (int64_t)blockIdx.x * BM;
            m_end = g.row_count ? (int64_t)*g.row_count : g.M;
            if (m0 >= m_end) return;
        }
        kbeg = 0;
        kend = g.K;
    } else {
        e = blockIdx.z / run.splits;
        slice = blockIdx.z - e * run.splits;
        m0 = (int64_t)blockIdx.x * BM;
        m_end = g.M;
        kbeg = g.offsets ? g.offsets[e] : 0;
        kend = g.offsets ? g.offsets[e + 1] : g.K;
        if (run.splits > 1) {
            const int64_t len = ((kend - kbeg + run.splits - 1) / run.splits + BK - 1) / BK * BK;
            kbeg += slice * len;
            kend = min(kend, kbeg + len);
        }
    }
    const int64_t n0 = (int64_t)blockIdx.y * BN;
    const TA *A = reinterpret_cast<const TA *>(g.A);
    const TB *B = reinterpret_cast<const TB *>(g.B) + (g.mode == 0 ? (int64_t)e * g.b_e : 0);
    const TB *B2 = g.B2 ? reinterpret_cast<const TB *>(g.B2) + (g.mode == 0 ? (int64_t)e * g.b_e : 0) : nullptr;
    const int rows_valid = (int)min((int64_t)BM, m_end - m0), cols_valid = (int)min((int64_t)BN, g.N - n0);
    const int klen = (int)max((int64_t)0, kend - kbeg);

    // Quad q of this thread: contraction index ka(q) of the K block (AK: its first one) and tile row ia(q) (else its first
    // one). pa[q] points at the quad of the current K block; where rows are gathered along the contraction
    // index (mode 1) it points at the column instead.
    auto ka = [&](int q) { return AK ? 4 * (tid % (BK / 4)) : (tid + q * NT) / (BM / 4); };
    auto ia = [&](int q) { return AK ? (tid + q * NT) / (BK / 4) : 4 * (tid % (BM / 4)); };
    auto kb = [&](int q) { return BJ ? (tid + q * NT) / (BN / 4) : 4 * (tid % (BK / 4)); };
    auto jb = [&](int q) { return BJ ? 4 * (tid % (BN / 4)) : (tid + q * NT) / (BK / 4); };
    const bool gather_a = !AK && g.a_row_index, gather_b = BJ && g.mode == 1 && g.b_row_index;
    const TA *pa[QA];
    const TB *pb[QB];
#pragma unroll
    for (int q = 0; q < QA; ++q) {
        if (AK) {
            int64_t r = m0 + ia(q);
            if (g.a_row_index && ia(q) < rows_valid) r = g.a_row_index[r] / g.a_row_div;
            pa[q] = A + r * g.sa_i + kbeg + ka(q);
        } else {
            pa[q] = A + m0 + ia(q) + (gather_a ? 0 : (kbeg + ka(q)) * g.sa_k);
        }
    }
#pragma unroll
    for (int q = 0; q < QB; ++q) {
        const int64_t j = n0 + jb(q);
        if (BJ) pb[q] = (B2 && j >= g.b_split ? B2 + (j - g.b_split) : B + j) + (gather_b ? 0 : (kbeg + kb(q)) * g.sb_k);
        else pb[q] = B + j * g.sb_j + kbeg + kb(q);
    }
    // !BJ: distance from B to the place where the second matrix stands for the contraction indices from b_split on
    const int64_t to_b2 = B2 ? ((int64_t)reinterpret_cast<uintptr_t>(B2) - (int64_t)reinterpret_cast<uintptr_t>(B)) /
                                       (int64_t)sizeof(TB) - g.b_split : 0;
    const int b_switch = !BJ && B2 ? (int)(g.b_split - kbeg) : INT32_MAX;

    Quad<TA> ra[QA];
    Quad<TB> rb[QB];
    constexpr int COL_STEP = NT / BN, COL_N = COL_B ? 4 * QB : 1;  // COL_B: rows kcol, kcol + COL_STEP, ... of column jcol
    const int jcol = tid % BN, kcol = tid / BN;
    const TB *pcol = nullptr;
    if (COL_B) pcol = (B2 && n0 + jcol >= g.b_split ? B2 + (n0 + jcol - g.b_split) : B + n0 + jcol) + (kbeg + kcol) * g.sb_k;
    TB ecol[COL_N];
    uint32_t live_a = 0u, live_b = 0u;  // QA4 / QB4: which quads lie inside the operand
    // rows gathered along the contraction index: the row numbers of the next K block, fetched one block ahead
    int32_t ga[QA], gb[QB];
    auto fetch_rows = [&](int k0) {
        if (gather_a) {
#pragma unroll
            for (int q = 0; q < QA; ++q) ga[q] = k0 + ka(q) < klen ? g.a_row_index[kbeg + k0 + ka(q)] : 0;
        }
        if (gather_b) {
#pragma unroll
            for (int q = 0; q < QB; ++q) gb[q] = k0 + kb(q) < klen ? g.b_row_index[kbeg + k0 + kb(q)] : 0;
        }
    };
    auto load_tiles = [&](int k0) {  // k0: first contraction index of the block, counted from kbeg
        live_a = live_b = 0u;
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            const int k = k0 + ka(q);
            const bool live = ia(q) < rows_valid && k < klen;
            const TA *src = gather_a ? pa[q] + (int64_t)(ga[q] / g.a_row_div) * g.sa_k : pa[q];
            if constexpr (QA4) {
                ra[q].load(live ? src : A);
                live_a |= (uint32_t)live << q;
            } else {
                ra[q].clear();
                const int left = AK ? klen - k : rows_valid - ia(q);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (live && u < left) ra[q].set(u, src[u]);
            }
            if (AK) pa[q] += BK;
            else if (!gather_a) pa[q] += BK * g.sa_k;
        }
        if constexpr (COL_B) {  // (mode 0: no rows to fetch)
#pragma unroll
            for (int q = 0; q < COL_N; ++q)
                ecol[q] = jcol < cols_valid && k0 + kcol + q * COL_STEP < klen ? pcol[q * COL_STEP * g.sb_k] : from_f32<TB>(0.0f);
            pcol += BK * g.sb_k;
            return;
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int k = k0 + kb(q);
            const bool live = jb(q) < cols_valid && k < klen;
            const TB *src = gather_b ? pb[q] + (int64_t)gb[q] * g.sb_k : pb[q];
            if constexpr (QB4) {
                if (!BJ && k >= b_switch) src += to_b2;
                rb[q].load(live ? src : B);
                live_b |= (uint32_t)live << q;
            } else {
                rb[q].clear();
                const int left = BJ ? cols_valid - jb(q) : klen - k;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (!live || u >= left) continue;
                    if (BJ) {  // the quad may straddle the border between the two matrices
                        const int64_t row = (gather_b ? (int64_t)gb[q] : kbeg + k) * g.sb_k, j = n0 + jb(q) + u;
                        rb[q].set(u, B2 && j >= g.b_split ? B2[row + j - g.b_split] : B[row + j]);
                    } else {
                        rb[q].set(u, src[u + (k + u >= b_switch ? to_b2 : 0)]);
                    }
                }
            }
            if (!BJ) pb[q] += BK;
            else if (!gather_b) pb[q] += BK * g.sb_k;
        }
        fetch_rows(k0 + BK);
    };
    auto store_tiles = [&](int buf) {
        const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            const float4 v = !QA4 || ((live_a >> q) & 1u) ? ra[q].get() : zero;
            float *dst = &As[buf][ka(q) * LDA + (ia(q) ^ swizzle_a(ka(q)))];
            if (AK) { dst[0] = v.x; dst[LDA] = v.y; dst[2 * LDA] = v.z; dst[3 * LDA] = v.w; }
            else *reinterpret_cast<float4 *>(dst) = v;
        }
        if constexpr (COL_B) {
#pragma unroll
            for (int q = 0; q < COL_N; ++q) Bs[buf][(kcol + q * COL_STEP) * LDB + jcol] = to_f32(ecol[q]);
            return;
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const float4 v = !QB4 || ((live_b >> q) & 1u) ? rb[q].get() : zero;
            float *dst = &Bs[buf][kb(q) * LDB + (jb(q) ^ swizzle_b(kb(q)))];
            if (!BJ) { dst[0] = v.x; dst[LDB] = v.y; dst[2 * LDB] = v.z; dst[3 * LDB] = v.w; }
            else *reinterpret_cast<float4 *>(dst) = v;
        }
    };
    // tile row of accumulator row i / tile column of accumulator column j
    auto row_at = [&](int i) { return (i / VA) * (VA * NTY) + ty * VA + i % VA; };
    auto col_at = [&](int j) { return (j / VB) * (VB * NTX) + tx * VB + j % VB; };

    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0f;
    float fa[2][TM], fb[2][TN];
    auto load_frag = [&](int buf, int k, int f) {
#pragma unroll
        for (int i = 0; i < TM; i += VA) {
            const float *src = &As[buf][k * LDA + (row_at(i) ^ swizzle_a(k))];
            if constexpr (VA == 4) {
                const float4 w = *reinterpret_cast<const float4 *>(src);
                fa[f][i] = w.x; fa[f][i + 1] = w.y; fa[f][i + 2] = w.z; fa[f][i + 3] = w.w;
            } else {
                const float2 w = *reinterpret_cast<const float2 *>(src);
                fa[f][i] = w.x; fa[f][i + 1] = w.y;
            }
        }
#pragma unroll
        for (int j = 0; j < TN; j += VB) {
            const float *src = &Bs[buf][k * LDB + (col_at(j) ^ swizzle_b(k))];
            if constexpr (VB == 4) {
                const float4 w = *reinterpret_cast<const float4 *>(src);
                fb[f][j] = w.x; fb[f][j + 1] = w.y; fb[f][j + 2] = w.z; fb[f][j + 3] = w.w;
            } else {
                const float2 w = *reinterpret_cast<const float2 *>(src);
                fb[f][j] = w.x; fb[f][j + 1] = w.y;
            }
        }
    };
    auto multiply = [&](int buf, auto rows_) {  // one K block for the first rows_ accumulator rows
        constexpr int ROWS = decltype(rows_)::value;
        load_frag(buf, 0, 0);
#pragma unroll 4
        for (int k = 0; k < BK; ++k) {  // the operands of step k + 1 are read during step k (after the last one: unused)
            load_frag(buf, k + 1 < BK ? k + 1 : 0, (k + 1) & 1);
#pragma unroll
            for (int i = 0; i < ROWS; ++i)
#pragma unroll
                for (int j = 0; j < TN; j += 2) fma_pair(acc[i][j], acc[i][j + 1], fa[k & 1][i], fb[k & 1][j], fb[k & 1][j + 1]);
        }
    };
    // Rows behind the segment's end are not computed: whole warps of them (a warp's lanes own VA * 32 / NTX adjacent rows of
    // every group of VA * NTY) and, in a tile less than half full, the accumulators' upper half.
    const bool busy = __any_sync(0xffffffffu, row_at(0) < rows_valid);
    const bool upper = rows_valid > VA * NTY;  // then every warp is busy
    if (klen > 0) {
        fetch_rows(0);
        load_tiles(0);
        store_tiles(0);
        __syncthreads();
    }
    int buf = 0;
    for (int k0 = 0; k0 < klen; k0 += BK) {
        const bool more = k0 + BK < klen;
        if (more) load_tiles(k0 + BK);
        if (upper) multiply(buf, std::integral_constant<int, TM>());
        else if (busy) multiply(buf, std::integral_constant<int, VA>());
        if (more) store_tiles(buf ^ 1);  // everybody left that buffer at the last barrier
        __syncthreads();
        buf ^= 1;
    }

    const bool partial = g.mode == 1 && run.splits > 1;
    float *part = partial ? run.part + ((int64_t)slice * g.nseg + e) * g.M * g.N : nullptr;
    const int64_t c_off = g.mode == 1 ? (int64_t)e * g.c_e : 0;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int64_t r = m0 + row_at(i);
        if (r >= m_end) continue;
        if (partial) {
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (n0 + col_at(j) < g.N) part[r * g.N + n0 + col_at(j)] = acc[i][j];
            continue;
        }
        const int64_t cr = (g.mode == 0 && g.c_row_index) ? g.c_row_index[r] : r;
#pragma unroll
        for (int j0 = 0; j0 < TN; j0 += VB) {
            TC out[VB];
#pragma unroll
            for (int z = 0; z < VB; ++z) {
                const int64_t col = n0 + col_at(j0 + z);
                float v = acc[i][j0 + z];
                if (col < g.N) {
                    if (g.bias) v += ld_as_f32<TC>(g.bias, (int64_t)e * g.N + col);
                    if (g.relu) v = fmaxf(v, 0.0f);
                    if (g.mask && !(ld_as_f32<TC>(g.mask, c_off + cr * g.sc_i + col) > 0.0f)) v = 0.0f;
                }
                out[z] = from_f32<TC>(v);
            }
            // C2 takes the columns from c_split on (same row stride)
            auto at = [&](int64_t col) {
                return g.C2 && col >= g.c_split ? reinterpret_cast<TC *>(g.C2) + c_off + cr * g.sc_i + (col - g.c_split)
                                                : reinterpret_cast<TC *>(g.C) + c_off + cr * g.sc_i + col;
            };
            if (BJ && VB == 4 && run.vec_c) {
                const int64_t col = n0 + col_at(j0);
                if (col < g.N) {
                    if constexpr (sizeof(TC) == 4) *reinterpret_cast<uint4 *>(at(col)) = *reinterpret_cast<const uint4 *>(out);
                    else *reinterpret_cast<uint2 *>(at(col)) = *reinterpret_cast<const uint2 *>(out);
                }
            } else {
#pragma unroll
                for (int z = 0; z < VB; ++z)
                    if (n0 + col_at(j0 + z) < g.N) *at(n0 + col_at(j0 + z)) = out[z];
            }
        }
    }
}

// C (and C2) = the slices' partial results added in double, in slice order
__global__ void __launch_bounds__(256) simt_reduce_kernel(const __grid_constant__ SimtRun run) {
    wait_previous_kernel();
    const SimtGemm &g = run.g;
    const int64_t per = g.M * g.N, total = per * g.nseg;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    double s = 0.0;
    int32_t c = 0;
    for (; c + 8 <= run.splits; c += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = run.part[(int64_t)(c + u) * total + i];
#pragma unroll
        for (int u = 0; u < 8; ++u) s += (double)v[u];
    }
    for (; c < run.splits; ++c) s += (double)run.part[(int64_t)c * total + i];
    const int64_t e = i / per, r = i % per / g.N, col = i % g.N;
    float *out = reinterpret_cast<float *>(g.C2 && col >= g.c_split ? g.C2 : g.C);
    out[e * g.c_e + r * g.sc_i + (g.C2 && col >= g.c_split ? col - g.c_split : col)] = (float)s;
}

constexpr int SLICE_ROWS = 64;  // shortest slice worth a block

}  // namespace

// Slices the contraction of a mode-1 product [M, N] over K rows in nseg segments is cut into: enough blocks for four per
// SM. A gate has a few hundred features and a few dozen columns, so its weight gradient is a handful of tiles, each one
// chain over the whole batch (2085 tokens x 256 features x 32 columns: 260 us on 4 blocks).
int32_t simt_wgrad_splits(int64_t M, int64_t N, int32_t nseg, int64_t K) {
    const int64_t tiles = cdiv(M, N <= 32 ? 32 : 64) * cdiv(N, N <= 32 ? 32 : 64) * nseg;
    const int64_t want = cdiv(4 * 148, tiles), most = cdiv(cdiv(K, nseg), SLICE_ROWS);
    return (int32_t)std::max<int64_t>(1, std::min(std::min(want, most), (int64_t)65535 / nseg));
}

static bool quad_aligned(const void *p, int32_t t) { return (reinterpret_cast<uintptr_t>(p) & (t == G_F32 ? 15 : 7)) == 0; }

template <typename TA, typename TB, typename TC, bool QA4, bool QB4, bool AK, bool BJ, int BM, int BN, int TM, int TN, int BK>
static int32_t simt_launch(SimtRun &run, int32_t *tile_prefix, cudaStream_t st) {
    const SimtGemm &g = run.g;
    const int32_t *ready = g.mode == 0 && g.offsets && run.plan ? run.plan->prefix_of(BM) : nullptr;
    dim3 grid;
    if (g.mode == 0) {
        int64_t tiles = cdiv(g.M, BM);
        if (g.offsets) {
            if (!ready) {
                if (!tile_prefix) return MOE_ERR_WORKSPACE;
                MOE_TRY(launch_tile_prefix(g.offsets, g.nseg, BM, tile_prefix, st));
            }
            tiles += g.nseg;
        }
        grid = dim3((unsigned)tiles, (unsigned)cdiv(g.N, BN), 1);
    } else {
        grid = dim3((unsigned)cdiv(g.M, BM), (unsigned)cdiv(g.N, BN), (unsigned)(g.nseg * run.splits));
    }
    if (grid.y > 65535 || grid.z > 65535) return MOE_ERR_UNSUPPORTED;
    run.tile_prefix = ready ? ready : tile_prefix;
    launch_kernel((simt_gemm_kernel<TA, TB, TC, QA4, QB4, AK, BJ, BM, BN, TM, TN, BK>), grid, (BM / TM) * (BN / TN), 0, st, run);
    MOE_LAUNCHED();
    if (run.part && run.parts_left) {  // left for a later launch
        *run.parts_left = {run.part, run.splits, (int32_t)g.M, (int32_t)g.N, (int32_t)(g.C2 ? g.c_split : g.N), (int32_t)g.sc_i, (float *)g.C, (float *)g.C2};
    } else if (run.part) {
        launch_kernel(simt_reduce_kernel, (unsigned)cdiv(g.M * g.N * g.nseg, 256), 256, 0, st, run);
        MOE_LAUNCHED();
    }
    return MOE_OK;
}

// The tile. What bounds a block is the issue of its instructions and the shared-memory reads that feed them, so the more
// outputs per thread the better, as long as the blocks spread over the chip: 64 x 128 tiles (8 x 8 outputs per thread)
// from six blocks per SM on (32768 tokens x 512 features x 256 columns: 186 us = 46 TFLOP/s, with 64 x 64 tiles 213);
// 64 x 64 tiles (8 x 4) from two per SM on (the 16-expert float layer with 4170 rows: 46 us per product, with 64 x 128
// tiles 58); else 32 x 32 tiles (4 x 4), and where even those leave SMs idle 16 x 16 (2 x 2, K blocks of 64): there a
// block's time is the latency of one chain and its loads (24 tokens x 512 features x 64 columns: 9 us; one 128 x 64
// tile: 40).
// Gate widths that are no multiple of four: the projections that come here (projection.cu keeps the smaller ones) have six 128 x 64 tiles and more
// per SM; the gradient of x takes 32 x 32 element-wise tiles.
template <typename TA, typename TB, typename TC, bool AK, bool BJ>
static int32_t simt_pick_tile(SimtRun &run, bool vec_a, bool vec_b, int32_t *tile_prefix, cudaStream_t st) {
    const SimtGemm &g = run.g;
    const int64_t segs = g.offsets || g.mode == 1 ? g.nseg : 0;
    auto blocks = [&](int64_t bm, int64_t bn) {
        return (g.mode == 0 ? cdiv(g.M, bm) + segs : cdiv(g.M, bm) * segs * run.splits) * cdiv(g.N, bn);
    };
    const bool short_rows = g.mode == 0 && g.offsets && g.M <= 32 * (int64_t)g.nseg;  // segments of few rows: less padding
    if (!(vec_a && vec_b)) {
        if constexpr (std::is_same<TC, bf16>::value) {  // an expert product: widths are whole 16-byte vectors
            return MOE_ERR_UNSUPPORTED;
        } else if constexpr (AK && BJ) {
            if (!vec_a) return MOE_ERR_UNSUPPORTED;  // activations have rows of whole 16-byte vectors
            return simt_launch<TA, TB, TC, true, false, AK, BJ, 128, 64, 8, 8, 16>(run, tile_prefix, st);
        } else if constexpr (AK) {
            return simt_launch<TA, TB, TC, false, false, AK, BJ, 32, 32, 4, 4, 32>(run, tile_prefix, st);
        } else {
            return MOE_ERR_UNSUPPORTED;  // gate_products.cu
        }
    }
    if constexpr (AK && BJ && std::is_same<TA, bf16>::value && std::is_same<TB, float>::value) {
        return MOE_ERR_UNSUPPORTED;  // projections of whole quads: projection.cu
    } else {
        if (blocks(64, 128) >= 6 * 148 && !short_rows && g.N > 64)
            return simt_launch<TA, TB, TC, true, true, AK, BJ, 64, 128, 8, 8, 16>(run, tile_prefix, st);
        if (blocks(64, 64) >= 2 * 148 && !short_rows && !(run.part && g.N <= 32))
            return simt_launch<TA, TB, TC, true, true, AK, BJ, 64, 64, 8, 4, 16>(run, tile_prefix, st);
        if (blocks(32, 32) >= 148) return simt_launch<TA, TB, TC, true, true, AK, BJ, 32, 32, 4, 4, 32>(run, tile_prefix, st);
        return simt_launch<TA, TB, TC, true, true, AK, BJ, 16, 16, 2, 2, 64>(run, tile_prefix, st);
    }
}

int32_t launch_slices_sum(float *part, int32_t splits, int32_t groups, int32_t d, int32_t cols, int32_t n, float *dW, float *dW2, cudaStream_t st) {
    SimtRun run;
    memset(&run, 0, sizeof(run));
    run.g.M = d; run.g.N = cols; run.g.nseg = groups; run.g.C = dW; run.g.C2 = dW2; run.g.c_split = n; run.g.sc_i = n; run.g.c_e = (int64_t)d * n;
    run.splits = splits; run.part = part;
    launch_kernel(simt_reduce_kernel, (unsigned)cdiv((int64_t)d * cols * groups, 256), 256, 0, st, run);
    MOE_LAUNCHED();
    return MOE_OK;
}

// part: simt_wgrad_splits(M, N, nseg, rows) * nseg * M * N floats (mode 1, float results), or nullptr: no slices
int32_t launch_simt_gemm(const SimtGemm &g_in, int32_t *tile_prefix, cudaStream_t st, float *part, const SegmentPlan *plan,
                         GateParts *parts_left) {
    SimtRun run;
    run.plan = plan;
    run.parts_left = parts_left;
    run.g = g_in;
    SimtGemm &g = run.g;
    if (!g.offsets) g.nseg = 1;
    if (g.mode == 0 && g.M == 0) return MOE_OK;
    const bool ak = g.sa_k == 1, bj = g.sb_j == 1 && !g.b_k_contiguous;
    const int64_t sa = ak ? g.sa_i : g.sa_k, sb = bj ? g.sb_k : g.sb_j;
    const int64_t ext_a = ak ? g.K : g.M, ext_b = bj ? g.N : g.K;
    const bool vec_a = ext_a % 4 == 0 && sa % 4 == 0 && quad_aligned(g.A, g.ta);
    const bool vec_b = ext_b % 4 == 0 && sb % 4 == 0 && g.b_e % 4 == 0 && quad_aligned(g.B, g.tb) &&
                (!g.B2 || (g.b_split % 4 == 0 && quad_aligned(g.B2, g.tb)));
    run.vec_c = g.N % 4 == 0 && g.sc_i % 4 == 0 && g.c_e % 4 == 0 && quad_aligned(g.C, g.tc) &&
                (!g.C2 || (g.c_split % 4 == 0 && quad_aligned(g.C2, g.tc)));
    run.splits = 1;
    run.part = nullptr;
    if (g.mode == 1 && part) {
        run.splits = simt_wgrad_splits(g.M, g.N, g.nseg, g.K);
        if (run.splits > 1) run.part = part;
    }
    const bool fff = g.ta == G_F32 && g.tb == G_F32 && g.tc == G_F32;
    const bool bff = g.ta == G_BF16 && g.tb == G_F32 && g.tc == G_F32;
    if (ak && bj) {  // rows x weight [K, N]
        if (fff) return simt_pick_tile<float, float, float, true, true>(run, vec_a, vec_b, tile_prefix, st);
        if (bff) return simt_pick_tile<bf16, float, float, true, true>(run, vec_a, vec_b, tile_prefix, st);
        if (g.ta == G_BF16 && g.tb == G_BF16 && g.tc == G_BF16) return simt_pick_tile<bf16, bf16, bf16, true, true>(run, vec_a, vec_b, tile_prefix, st);
    } else if (ak) {  // rows x weight [N, K] read transposed
        if (fff) return simt_pick_tile<float, float, float, true, false>(run, vec_a, vec_b, tile_prefix, st);
    } else if (bj) {  // contraction over rows
        if (fff) return simt_pick_tile<float, float, float, false, true>(run, vec_a, vec_b, tile_prefix, st);
        if (bff) return simt_pick_tile<bf16, float, float, false, true>(run, vec_a, vec_b, tile_prefix, st);
    }
    return MOE_ERR_UNSUPPORTED;
}

// ------------------------------------------------------------------------------------------
// Column sums per segment (bias gradients): partial sums over tiles of 128 rows, then an ordered
// pass over each segment's tiles. Deterministic.
// ------------------------------------------------------------------------------------------
int64_t colsum_ws_floats(int64_t R, int32_t n, int32_t N) { return (cdiv(R, COLSUM_ROWS) + n) * (int64_t)N + 64; }

template <typename XT> __global__ void __launch_bounds__(256) colsum_partial_kernel(const ColumnSums a) {
    wait_previous_kernel();
    column_sums_partial<XT>(a, blockIdx.x, blockIdx.y);
}
template <int COLS> __global__ void __launch_bounds__(256) colsum_final_kernel(const ColumnSums a) {
    wait_previous_kernel();
    __shared__ float sh[8][32];
    column_sums_final<COLS>(a, blockIdx.x, blockIdx.y, sh);
}

int32_t launch_segment_colsum(const ColumnSums &a, cudaStream_t st) {
    const dim3 tiles((unsigned)column_tiles(a), (unsigned)column_slabs(a));
    if (a.act == MOE_BF16) launch_kernel(colsum_partial_kernel<bf16>, tiles, 256, 0, st, a);
    else launch_kernel(colsum_partial_kernel<float>, tiles, 256, 0, st, a);
    MOE_LAUNCHED();
    return MOE_OK;
}
int32_t launch_segment_colsum_final(const ColumnSums &a, cudaStream_t st) {
    if (a.nseg >= COLSUM_MANY) launch_kernel(colsum_final_kernel<256>, dim3((unsigned)a.nseg, (unsigned)cdiv(a.N, 256)), 256, 0, st, a);
    else launch_kernel(colsum_final_kernel<32>, dim3((unsigned)a.nseg, (unsigned)cdiv(a.N, 32)), 256, 0, st, a);
    MOE_LAUNCHED();
    return MOE_OK;
}

}  // namespace moe
