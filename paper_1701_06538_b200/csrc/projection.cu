// Projection onto the gating matrices  clean = x.W_g,  raw = x.W_noise   (the two products of Eq. 4)
//
// The routing must be reproducible bit for bit, so every output is ONE chain of fused multiply-adds over the input features in
// ascending order, starting from +0: each accumulator sees feature 0, 1, 2, ... A tensor-core MMA would not keep that order.
// It is bound by the FP32 pipes where the outputs fill the chip, by the chain and the way to memory where they do not. The operands come in by
// asynchronous copies several K blocks ahead, rows of x as they lie: a thread reads its rows sixteen bytes along the features at a time (eight
// features of a bf16 row, where a transposed float tile takes eight reads), so that the shared-memory reads, which with float tiles of both
// operands took as long as the multiply-adds, leave these the pipes. `fma.rn.f32x2` does two columns with one instruction.
#include <math.h>
#include <string.h>

#include <type_traits>

#include "async_copy.cuh"
#include "moe_internal.cuh"

namespace moe {

namespace {

struct ProjectionArgs {
    const void *x;
    const float *W0, *W1;  // [d, n0] each (per group); columns from n0 on are W1's
    float *out0, *out1;
    int64_t rows, group_stride;  // elements of a group's matrix
    int32_t d, n0, N;            // N = n0 or 2 n0
    const int32_t *offsets, *tile_prefix;  // rows sorted by group, or nullptr: one group
    int32_t groups;
    const int32_t *row_index;    // row r: x row row_index[r] / row_div, output row row_index[r]; or nullptr
    int32_t row_div, vec_out, quads;
    const int32_t *row_count;    // number of rows, read on the device (at most `rows`), or nullptr
    int32_t *clear;              // status word, cleared if given
};

// element v of sixteen bytes
template <typename T> __device__ __forceinline__ float element(const uint4 &q, int v) {
    const uint32_t *w = reinterpret_cast<const uint32_t *>(&q);
    if constexpr (sizeof(T) == 4) return __uint_as_float(w[v]);
    else return __uint_as_float(v & 1 ? w[v >> 1] & 0xffff0000u : w[v >> 1] << 16);
}

// BM x BN outputs a block, TM x TN a thread; a warp's lanes are 4 (rows) x 8 (columns). K blocks of BK features, S of them in shared memory.
template <typename T, int BM, int BN, int TM, int TN, int BK, int S> struct ProjectionTile {
    static constexpr int WARPS_M = BM / (4 * TM), WARPS_N = BN / (8 * TN), NT = 32 * WARPS_M * WARPS_N;
    static constexpr int ROW_BYTES = BK * (int)sizeof(T) + 16;  // 16 more: the four rows that a warp reads together stand in different banks
    static constexpr int A_STAGE = BM * ROW_BYTES, B_STAGE = BK * BN * 4, STAGE = A_STAGE + B_STAGE, SHARED = S * STAGE;
};
// QUADS: rows of the weights come in sixteen bytes at a time; otherwise (widths that are no multiple of four) four
template <typename T, int BM, int BN, int TM, int TN, int BK, int S, int BLOCKS, bool QUADS>
__global__ void __launch_bounds__(ProjectionTile<T, BM, BN, TM, TN, BK, S>::NT, BLOCKS) projection_kernel(const __grid_constant__ ProjectionArgs p) {
    using Tile = ProjectionTile<T, BM, BN, TM, TN, BK, S>;
    constexpr int NT = Tile::NT, VK = 16 / sizeof(T), A_ROW = BK / VK, A_COPIES = BM * A_ROW, VB = QUADS ? 4 : 1, B_ROW = BN / VB, B_COPIES = BK * B_ROW;
    constexpr int QA = A_COPIES / NT, QB = B_COPIES / NT, COLS = QUADS ? QB : (BN > NT ? BN / NT : 1), VN = TN < 4 ? TN : 4;
    static_assert(QUADS || NT % BN == 0 || BN % NT == 0, "a thread's single floats are of COLS columns");
    static_assert(QA * NT == A_COPIES && QB * NT == B_COPIES, "whole copies a thread");
    wait_previous_kernel();
    extern __shared__ __align__(16) uint8_t stages[];
    __shared__ int4 tile_at;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (p.clear && tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) *p.clear = 0;
    int64_t m0 = (int64_t)blockIdx.x * BM, m_end = p.row_count ? (int64_t)*p.row_count : p.rows;
    int32_t group = 0;
    if (p.offsets) {
        const int4 at = segment_of_tile(p.tile_prefix, p.offsets, p.groups, blockIdx.x, &tile_at);
        if (at.x < 0) return;
        group = at.x;
        m0 = at.y + (int64_t)at.w * BM;
        m_end = at.z;
    }
    if (m0 >= m_end) return;
    const int32_t n_at = blockIdx.y * BN;
    const float *W0 = p.W0 + group * p.group_stride, *W1 = p.W1 + group * p.group_stride;

    // the copies of this thread: the same rows of x and columns of W in every K block
    const T *from_a[QA];
    const float *from_b[COLS];
#pragma unroll
    for (int q = 0; q < QA; ++q) {
        const int id = tid + q * NT;
        int64_t r = m0 + id / A_ROW;
        if (r >= m_end) r = m0;  // (not copied)
        if (p.row_index) r = p.row_index[r] / p.row_div;
        from_a[q] = static_cast<const T *>(p.x) + r * p.d + id % A_ROW * VK;
    }
#pragma unroll
    for (int q = 0; q < COLS; ++q) {
        const int id = tid + q * NT;
        int32_t col = n_at + id % B_ROW * VB;
        // columns behind the last one are computed and dropped; not all from one column: copies from one address go one by one (6000 x 512 x 174 in
        // 64 x 128 tiles 92 us, 58; 20000 x 1024 x 40 100, 79)
        if (col >= p.N) col = min(col - p.N, p.N - VB);
        from_b[q] = (col < p.n0 ? W0 + col : W1 + (col - p.n0)) + (int64_t)(id / B_ROW) * p.n0;
    }
    const int64_t step = (int64_t)(NT > BN ? NT / BN : 1) * p.n0;  // single floats: a thread's copies of a column stand this far apart
    const int blocks = (p.d + BK - 1) / BK;
    // Features behind the last one are not used, rows behind the last one are whatever is there, computed and dropped. (Neither is copied: copies from one address, of zeros
    // too, go one by one: 29 rows of 56 features onto 1448 columns 7.3 us, this way 3.0; 3 of 128 onto 4000 9.1, 4.6; 24 bf16 rows of 512 onto 2048 11.0, 9.2.)
    const bool all_rows = m0 + BM <= m_end;
    auto load = [&](int kb) {
        uint8_t *to = stages + kb % S * Tile::STAGE;
        const int k0 = kb * BK;
        auto copies = [&](auto whole_) {
            constexpr bool WHOLE = decltype(whole_)::value;  // all rows and features are there
#pragma unroll
            for (int q = 0; q < QA; ++q) {
                const int id = tid + q * NT;
                uint8_t *at = to + id / A_ROW * Tile::ROW_BYTES + id % A_ROW * 16;
                if (WHOLE || (k0 + id % A_ROW * VK < p.d && m0 + id / A_ROW < m_end)) copy16(at, from_a[q] + k0);
            }
            if constexpr (QUADS) {
#pragma unroll
                for (int q = 0; q < QB; ++q) {
                    const int id = tid + q * NT;
                    uint8_t *at = to + Tile::A_STAGE + id * 16;
                    if (WHOLE || k0 + id / B_ROW < p.d) copy16(at, from_b[q] + (int64_t)k0 * p.n0);
                }
            } else {
#pragma unroll
                for (int c = 0; c < COLS; ++c) {
                    const float *from = from_b[c] + (int64_t)k0 * p.n0;
#pragma unroll
                    for (int q = c; q < QB; q += COLS, from += step) {
                        const int id = tid + q * NT;
                        uint8_t *at = to + Tile::A_STAGE + id * 4;
                        if (WHOLE || k0 + id / B_ROW < p.d) copy4(at, from);
                    }
                }
            }
        };
        if (all_rows && k0 + BK <= p.d) copies(std::true_type());
        else copies(std::false_type());
    };
#pragma unroll
    for (int s = 0; s < S - 1; ++s) {
        if (s < blocks) load(s);
        copies_commit();
    }
    const int tx = lane & 7, ty = lane >> 3;
    const int row0 = warp % Tile::WARPS_M * 4 * TM + ty, col0 = warp / Tile::WARPS_M * 8 * TN + tx * VN;  // rows row0 + 4 i, columns col0 + 32 (j / 4) + j % 4
    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0f;
    for (int kb = 0; kb < blocks; ++kb) {
        copies_wait<S - 2>();
        __syncthreads();  // block kb is there for all, block kb - 1 is read by all
        if (kb + S - 1 < blocks) load(kb + S - 1);
        copies_commit();
        const uint8_t *a = stages + kb % S * Tile::STAGE + row0 * Tile::ROW_BYTES;
        const float *b = reinterpret_cast<const float *>(stages + kb % S * Tile::STAGE + Tile::A_STAGE) + col0;
        auto multiply = [&](int steps) {
#pragma unroll 2
            for (int kk = 0; kk < steps; kk += VK) {
                uint4 av[TM];
#pragma unroll
                for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const uint4 *>(a + 4 * i * Tile::ROW_BYTES + kk * sizeof(T));
#pragma unroll
                for (int v = 0; v < VK; ++v) {
                    float bv[TN];
#pragma unroll
                    for (int j = 0; j < TN; j += VN) {
                        if constexpr (VN == 4) *reinterpret_cast<float4 *>(bv + j) = *reinterpret_cast<const float4 *>(b + (kk + v) * BN + 8 * j);
                        else *reinterpret_cast<float2 *>(bv + j) = *reinterpret_cast<const float2 *>(b + (kk + v) * BN + 8 * j);
                    }
#pragma unroll
                    for (int i = 0; i < TM; ++i) {
                        const float x = element<T>(av[i], v);
#pragma unroll
                        for (int j = 0; j < TN; j += 2) fma_two(acc[i][j], acc[i][j + 1], x, bv[j], bv[j + 1]);
                    }
                }
            }
        };
        if (kb * BK + BK <= p.d) multiply(BK);
        else multiply(p.d - kb * BK);  // (features are whole vectors)
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        int64_t r = m0 + row0 + 4 * i;
        if (r >= m_end) continue;
        if (p.row_index) r = p.row_index[r];
#pragma unroll
        for (int j = 0; j < TN; j += VN) {
            const int32_t col = n_at + col0 + 8 * j;
            if constexpr (QUADS) {
                if (col >= p.N) continue;  // N and n0 are multiples of four
                float *to = (col < p.n0 ? p.out0 + col : p.out1 + (col - p.n0)) + r * p.n0;
                if (VN == 4 && p.vec_out) {
                    *reinterpret_cast<float4 *>(to) = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + VN - 2], acc[i][j + VN - 1]);
                } else {
#pragma unroll
                    for (int z = 0; z < VN; ++z) to[z] = acc[i][j + z];
                }
            } else {
#pragma unroll
                for (int z = 0; z < VN; ++z)
                    if (col + z < p.N) (col + z < p.n0 ? p.out0 + (col + z) : p.out1 + (col + z - p.n0))[r * p.n0] = acc[i][j + z];
            }
        }
    }
}

template <typename T, int BM, int BN, int TM, int TN, int BK, int S, int BLOCKS, bool QUADS>
int32_t launch_tile_as(ProjectionArgs p, int32_t *tile_prefix, cudaStream_t st) {
    using Tile = ProjectionTile<T, BM, BN, TM, TN, BK, S>;
    int64_t tiles = cdiv(p.rows, BM);
    if (p.offsets) {
        if (!tile_prefix) return MOE_ERR_WORKSPACE;
        MOE_TRY(launch_tile_prefix(p.offsets, p.groups, BM, tile_prefix, st));
        tiles += p.groups;
        p.tile_prefix = tile_prefix;
    }
    if (cdiv(p.N, BN) > 65535) return MOE_ERR_UNSUPPORTED;
    static PerDevice configured;
    const auto kernel = projection_kernel<T, BM, BN, TM, TN, BK, S, BLOCKS, QUADS>;
    if (!allow_shared(configured, kernel, Tile::SHARED)) return MOE_ERR_CUDA;
    launch_kernel(kernel, dim3((unsigned)tiles, (unsigned)cdiv(p.N, BN)), Tile::NT, Tile::SHARED, st, p);
    MOE_LAUNCHED();
    return MOE_OK;
}

template <typename T, int BM, int BN, int TM, int TN, int BK, int S, int BLOCKS>
int32_t launch_tile(const ProjectionArgs &p, int32_t *tile_prefix, cudaStream_t st) {
    return p.quads ? launch_tile_as<T, BM, BN, TM, TN, BK, S, BLOCKS, true>(p, tile_prefix, st)
                   : launch_tile_as<T, BM, BN, TM, TN, BK, S, BLOCKS, false>(p, tile_prefix, st);
}

// The tile that takes the least time by an estimate: an SM's first block takes `chain` ns a feature, each further one `share`, and each `more` us besides.
// Read off kernels of all sizes; us, by the 64 x 128 tile and the others in order:
//   32768 x 512 x 510 363 406 460 - 507 550;  6000 x 512 x 168 54 35 38 81 42 39;  1019 x 512 x 222 33 22 14 25 15 14;  24 x 512 x 64 30 21 12 6.4 15 10;
//   20000 x 1024 x 44 157 95 89 159 80 75;  15000 x 256 x 648 125 132 138 - 159 164;  60000 x 256 x 10 (float) 90 53 38 50 26 25.
// Against one chain per output of float tiles in shared memory (gemm_simt.cu): 24 x 512 x 64 10.5 6.1, 1019 x 512 x 512 25 21, 3001 x 320 x 40 13 7.8,
// 8192 x 512 x 64 25 21, 15000 x 128 x 72 21 16, 32768 x 512 x 256 185 179. Widths that are no multiple of four cost next to nothing more (single floats
// of the weights are a tenth of a thread's instructions), and that way twice: 24 x 512 x 66 18.4 7.0, 300 x 256 x 50 11.2 4.3, 60000 x 256 x 10 61 26.
constexpr int32_t PROJECTION_ELSEWHERE = -1;  // (no status)
struct ProjectionCost { int32_t bm, bn; double chain, share[2], more; };  // [bf16, float]
template <typename T> int32_t pick_tile(const ProjectionArgs &p, int32_t *tile_prefix, cudaStream_t st) {
    constexpr int F = sizeof(T) == 4 ? 1 : 0;
    static const ProjectionCost costs[6] = {{64, 128, 53, {44, 45}, 2.5}, {64, 64, 33, {24, 24}, 2.3}, {32, 32, 19.5, {6.5, 8}, 0.75},
                                            {16, 16, 10, {5.2, 6.5}, 0.5}, {128, 16, 27, {16, 22}, 0.9}, {64, 16, 18, {9, 14}, 0.6}};
    int best = 0;
    double least = 0.0;
    for (int i = 0; i < 6; ++i) {
        const ProjectionCost &c = costs[i];
        // (tiles of groups: half a tile more each, and as much again as their number may exceed that: 1244 rows in 32 groups, 1648 x 234, 143 tiles by the halves alone,
        // one wave, was two: 64 x 64 tiles, 143 us a call of moe_gate, 32 x 32 110)
        const int64_t blocks = (cdiv(p.rows, c.bm) + (p.offsets ? p.groups / 2 + (int64_t)(0.5 * sqrt((double)p.groups)) : 0)) * cdiv(p.N, c.bn);
        const double cost = 1e-3 * c.chain * p.d + c.more + (double)(cdiv(blocks, 148) - 1) * (1e-3 * c.share[F] * p.d + c.more);
        if (i == 0 || cost < least) { best = i; least = cost; }
    }
    // Single floats of the weights that the float product takes in 128 x 64 tiles, whose number may fall better onto the SMs (its kernels of 3554 x 1200 x 1970, 868
    // tiles, 355 us, 896 of 64 x 128 here or 1736 of 64 x 64 398; 7117 x 1632 x 262, 280 tiles, 175 and 187)
    if (!p.quads && !p.offsets) {
        const int64_t blocks = cdiv(p.rows, 128) * cdiv(p.N, 64);
        const double more = costs[0].more, there = 1e-3 * costs[0].chain * p.d + more + (double)(cdiv(blocks, 148) - 1) * (1e-3 * costs[0].share[F] * p.d + more);
        // (float rows in 64 x 128 tiles take 2 % longer than there with as many waves: 6040 x 896 x 986 274 us, 268)
        if (2 * blocks >= 3 * 148 && (F && best == 0 ? 1.0 : 1.02) * there <= least) return PROJECTION_ELSEWHERE;
    }
    // float rows have as many shared-memory reads in the largest tiles as the float product has (32768 x 512 x 512: 362, that way 349)
    if (F && best == 0 && p.d >= 256 && !p.offsets && cdiv(p.rows, 64) * cdiv(p.N, 128) >= 6 * 148) return PROJECTION_ELSEWHERE;
    // and short chains of single floats fill the pipeline of the copies too often (15000 x 256 x 650: 136, that way 130; 32768 x 512 x 510: 363, 367)
    if (!p.quads && best == 0 && p.d < 512 && !p.offsets && cdiv(p.rows, 64) * cdiv(p.N, 128) >= 6 * 148) return PROJECTION_ELSEWHERE;
    switch (best) {
        case 0: return launch_tile<T, 64, 128, 8, 8, 32, 3, 3>(p, tile_prefix, st);
        case 1: return launch_tile<T, 64, 64, 8, 4, 32, 4, 3>(p, tile_prefix, st);
        case 2: return launch_tile<T, 32, 32, 4, 4, 32, 4, 6>(p, tile_prefix, st);
        case 3: return launch_tile<T, 16, 16, 1, 2, 64, 8, 3>(p, tile_prefix, st);
        case 4: return launch_tile<T, 128, 16, 8, 2, 32, 4, 4>(p, tile_prefix, st);
        default: return launch_tile<T, 64, 16, 4, 2, 32, 4, 4>(p, tile_prefix, st);
    }
}

}  // namespace

int32_t launch_projection(const void *x, int32_t act, int64_t M, int32_t d, int32_t n0, const float *W0,
                          const float *W1, float *out0, float *out1, const int32_t *offsets, int32_t nseg,
                          const int32_t *perm, int32_t kdiv, int32_t *tile_prefix, cudaStream_t st,
                          const int32_t *row_count, int32_t *clear) {
    if (M == 0) return MOE_OK;
    {
        ProjectionArgs p;
        memset(&p, 0, sizeof(p));
        p.x = x; p.W0 = W0; p.W1 = W1 ? W1 : W0; p.out0 = out0; p.out1 = out1; p.rows = M; p.group_stride = (int64_t)d * n0;
        p.d = d; p.n0 = n0; p.N = W1 ? 2 * n0 : n0; p.offsets = offsets; p.groups = nseg; p.row_index = perm; p.row_div = kdiv > 0 ? kdiv : 1;
        p.quads = n0 % 4 == 0 && aligned16(W0) && (!W1 || aligned16(W1));
        p.vec_out = aligned16(out0) && (!W1 || aligned16(out1));
        p.row_count = row_count; p.clear = clear;
        const int32_t rc = act == MOE_BF16 ? pick_tile<bf16>(p, tile_prefix, st) : pick_tile<float>(p, tile_prefix, st);
        if (rc != PROJECTION_ELSEWHERE) return rc;
    }
    SimtGemm g;  // rows x [W0 | W1] (W1 == nullptr: one matrix only)
    memset(&g, 0, sizeof(g));
    g.ta = act == MOE_BF16 ? G_BF16 : G_F32; g.tb = g.tc = G_F32;
    g.A = x; g.B = W0; g.B2 = W1; g.C = out0; g.C2 = W1 ? out1 : nullptr; g.b_split = g.c_split = n0;
    g.sa_i = d; g.sa_k = 1; g.sb_k = n0; g.sb_j = 1; g.sc_i = n0;
    g.mode = 0; g.offsets = offsets; g.nseg = nseg; g.M = M; g.N = W1 ? 2 * n0 : n0; g.K = d; g.b_e = (int64_t)d * n0;
    g.a_row_index = perm; g.a_row_div = kdiv; g.c_row_index = perm; g.row_count = row_count; g.clear = clear;
    return launch_simt_gemm(g, tile_prefix, st);
}

}  // namespace moe
