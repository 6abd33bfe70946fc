// The two products of a gate's backward pass by FP32 multiply-adds (gates that the tensor-core contractions do not take: float tokens, widths that
// are no multiple of 32, most levels of a hierarchy):
//   dX[r] = dlogit[r] . [W_g | W_noise]^T      contraction over the logits, a few dozen
//   dW    = x^T . dlogit                       contraction over the tokens, cut into slices
// Narrow gates are small next to the latency of their loads: 5000 tokens x 512 features x 32 logits are 2 us of multiply-adds each. So the K blocks come
// in by asynchronous copies, all in flight together or several ahead, sixteen bytes of a row at a time and as the rows lie in memory. Wider ones stay
// with the float product of gemm_simt.cu (see gate_rows_supported). Every output of dX is one chain of multiply-adds in ascending order,
// every slice of dW likewise.
#include <string.h>

#include <type_traits>

#include "async_copy.cuh"
#include "moe_internal.cuh"

namespace moe {

namespace {

// lanes of a warp: 4 (rows) x 8 (columns)
template <int BM, int BN, int TM, int TN, int BK, int S> struct RowsTile {
    static constexpr int WARPS_M = BM / (4 * TM), WARPS_N = BN / (8 * TN), NT = 32 * WARPS_M * WARPS_N;
    static constexpr int ROW_BYTES = BK * 4 + 16;  // the rows that a warp reads together stand in different banks
    static constexpr int A_STAGE = BM * ROW_BYTES, STAGE = A_STAGE + BN * ROW_BYTES, SHARED = S * STAGE;
};
// QUADS: rows of logits come in sixteen bytes at a time; otherwise (widths that are no multiple of four) four
template <int BM, int BN, int TM, int TN, int BK, int S, int BLOCKS, bool QUADS>
__global__ void __launch_bounds__(RowsTile<BM, BN, TM, TN, BK, S>::NT, BLOCKS) gate_rows_kernel(const __grid_constant__ GateProduct p, const int32_t *__restrict__ tile_prefix) {
    using Tile = RowsTile<BM, BN, TM, TN, BK, S>;
    constexpr int NT = Tile::NT, V = QUADS ? 4 : 1, ROW = BK / V, QA = BM * ROW / NT, QB = BN * ROW / NT;
    static_assert(QA * NT == BM * ROW && QB * NT == BN * ROW && TN % 2 == 0, "whole copies a thread, pairs of columns");
    wait_previous_kernel();
    extern __shared__ __align__(16) uint8_t stages[];
    __shared__ int4 tile_at;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t m0 = (int64_t)blockIdx.x * BM, m_end = p.rows;
    int32_t group = 0;
    if (p.offsets) {
        const int4 at = segment_of_tile(tile_prefix, p.offsets, p.groups, blockIdx.x, &tile_at);
        if (at.x < 0) return;
        group = at.x;
        m0 = at.y + (int64_t)at.w * BM;
        m_end = at.z;
    }
    if (m0 >= m_end) return;
    const int32_t n_at = blockIdx.y * BN, cols = p.W2 ? 2 * p.n : p.n;
    const int64_t matrix = (int64_t)group * p.d * p.n;
    int32_t from_a[QA], from_b[QB];  // rows of dlogit and W that this thread copies from
#pragma unroll
    for (int q = 0; q < QA; ++q) {
        int64_t r = m0 + (tid + q * NT) / ROW;
        if (r >= m_end) r = m0;  // (a row that is computed and dropped)
        from_a[q] = p.perm ? p.perm[r] : (int32_t)r;
    }
#pragma unroll
    for (int q = 0; q < QB; ++q) {
        const int32_t j = n_at + (tid + q * NT) / ROW;
        from_b[q] = j < p.d ? j : 0;  // (a column that is computed and dropped)
    }
    const int blocks = (cols + BK - 1) / BK;
    auto load = [&](int kb) {  // logits behind the last one are zero in both operands
        uint8_t *to = stages + kb % S * Tile::STAGE;
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            const int id = tid + q * NT, k = kb * BK + id % ROW * V;
            uint8_t *at = to + id / ROW * Tile::ROW_BYTES + id % ROW * (4 * V);
            const float *from = k < cols ? p.dlogit + (int64_t)from_a[q] * cols + k : p.dlogit;
            if (QUADS) copy16(at, from, k < cols);
            else copy4(at, from, k < cols);
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int id = tid + q * NT, k = kb * BK + id % ROW * V;
            uint8_t *at = to + Tile::A_STAGE + id / ROW * Tile::ROW_BYTES + id % ROW * (4 * V);
            const float *from = k >= cols ? p.W : (k < p.n ? p.W + k : p.W2 + (k - p.n)) + matrix + (int64_t)from_b[q] * p.n;
            if (QUADS) copy16(at, from, k < cols);
            else copy4(at, from, k < cols);
        }
    };
#pragma unroll
    for (int s = 0; s < S - 1; ++s) {
        if (s < blocks) load(s);
        copies_commit();
    }
    const int tx = lane & 7, ty = lane >> 3;
    const int row0 = warp % Tile::WARPS_M * 4 * TM + ty, col0 = warp / Tile::WARPS_M * 8 * TN + tx;  // rows row0 + 4 i, columns col0 + 8 j
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
        const uint8_t *a = stages + kb % S * Tile::STAGE + row0 * Tile::ROW_BYTES, *b = stages + kb % S * Tile::STAGE + Tile::A_STAGE + col0 * Tile::ROW_BYTES;
        const int steps = min(BK, (cols - kb * BK + 3) & ~3);
        for (int kk = 0; kk < steps; kk += 4) {
            float4 av[TM], bv[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4 *>(a + 4 * i * Tile::ROW_BYTES + kk * 4);
#pragma unroll
            for (int j = 0; j < TN; ++j) bv[j] = *reinterpret_cast<const float4 *>(b + 8 * j * Tile::ROW_BYTES + kk * 4);
#pragma unroll
            for (int v = 0; v < 4; ++v)
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; j += 2)
                        fma_two(acc[i][j], acc[i][j + 1], reinterpret_cast<const float *>(&av[i])[v], reinterpret_cast<const float *>(&bv[j])[v],
                                reinterpret_cast<const float *>(&bv[j + 1])[v]);
        }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        int64_t r = m0 + row0 + 4 * i;
        if (r >= m_end) continue;
        if (p.perm) r = p.perm[r];
        float *to = p.dX + r * p.d + n_at + col0;
#pragma unroll
        for (int j = 0; j < TN; ++j)
            if (n_at + col0 + 8 * j < p.d) to[8 * j] = acc[i][j];
    }
}

// dW: a thread has four features, or eight (two quads 16 apart), and TN logits
template <typename T, int BM, int BN, int TM, int TN, int BK, int S> struct WgradTile {
    static constexpr int WARPS_M = BM / (4 * TM), WARPS_N = BN / (8 * TN), NT = 32 * WARPS_M * WARPS_N;
    static constexpr int A_STAGE = BK * BM * (int)sizeof(T), STAGE = A_STAGE + BK * BN * 4, SHARED = S * STAGE;
};
template <typename T, int BM, int BN, int TM, int TN, int BK, int S, int BLOCKS, bool QUADS>
__global__ void __launch_bounds__(WgradTile<T, BM, BN, TM, TN, BK, S>::NT, BLOCKS) gate_wgrad_kernel(const __grid_constant__ GateProduct p, int32_t splits, float *__restrict__ part) {
    using Tile = WgradTile<T, BM, BN, TM, TN, BK, S>;
    constexpr int NT = Tile::NT, VK = 16 / sizeof(T), A_ROW = BM / VK, VB = QUADS ? 4 : 1, B_ROW = BN / VB, QA = BK * A_ROW / NT, QB = BK * B_ROW / NT;
    static_assert(QA * NT == BK * A_ROW && QB * NT == BK * B_ROW, "whole copies a thread");
    wait_previous_kernel();
    extern __shared__ __align__(16) uint8_t stages[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t group = blockIdx.z / splits, slice = blockIdx.z % splits, cols = p.W2 ? 2 * p.n : p.n, m_at = blockIdx.x * BM, n_at = blockIdx.y * BN;
    int64_t begin = p.offsets ? p.offsets[group] : 0, end = p.offsets ? p.offsets[group + 1] : p.rows;
    const int64_t len = ((end - begin + splits - 1) / splits + BK - 1) / BK * BK;
    begin += slice * len;
    if (begin + len < end) end = begin + len;
    const int count = (int)(end > begin ? end - begin : 0), blocks = (count + BK - 1) / BK;
    // rows of a K block that this thread copies, fetched one block ahead where they are gathered
    int32_t ra[QA], rb[QB];
    auto fetch = [&](int kb) {
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            const int k = kb * BK + (tid + q * NT) / A_ROW;
            ra[q] = k < count ? (p.perm ? p.perm[begin + k] : (int32_t)(begin + k)) : -1;
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int k = kb * BK + (tid + q * NT) / B_ROW;
            rb[q] = k < count ? (p.perm ? p.perm[begin + k] : (int32_t)(begin + k)) : -1;
        }
    };
    // rows behind the last one are zero in both operands; features and logits behind the last ones are whatever is there, computed and dropped
    const bool whole_tile = m_at + BM <= p.d && n_at + BN <= cols;
    auto load = [&](int kb) {
        uint8_t *to = stages + kb % S * Tile::STAGE;
        auto copies = [&](auto whole_) {
            constexpr bool WHOLE = decltype(whole_)::value;
#pragma unroll
            for (int q = 0; q < QA; ++q) {
                const int id = tid + q * NT, m = m_at + id % A_ROW * VK;
                if (!WHOLE && m >= p.d) continue;
                if (WHOLE || ra[q] >= 0) copy16(to + id * 16, static_cast<const T *>(p.x) + (int64_t)(ra[q] / p.row_div) * p.d + m);
                else zero16(to + id * 16);
            }
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int id = tid + q * NT, c = n_at + id % B_ROW * VB;
                if (!WHOLE && c >= cols) continue;
                uint8_t *at = to + Tile::A_STAGE + id * 4 * VB;
                const float *from = p.dlogit + (int64_t)rb[q] * cols + c;
                if (WHOLE || rb[q] >= 0) {
                    if (QUADS) copy16(at, from);
                    else copy4(at, from);
                } else if (QUADS) zero16(at);
                else zero4(at);
            }
        };
        if (whole_tile && (kb + 1) * BK <= count) copies(std::true_type());
        else copies(std::false_type());
        fetch(kb + 1);
    };
    fetch(0);
#pragma unroll
    for (int s = 0; s < S - 1; ++s) {
        if (s < blocks) load(s);
        copies_commit();
    }
    const int tx = lane & 7, ty = lane >> 3, m0 = warp % Tile::WARPS_M * 4 * TM + ty * 4, c0 = warp / Tile::WARPS_M * 8 * TN + tx * TN;  // features m0 + i % 4 + 16 (i / 4)
    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0f;
    for (int kb = 0; kb < blocks; ++kb) {
        copies_wait<S - 2>();
        __syncthreads();
        if (kb + S - 1 < blocks) load(kb + S - 1);
        copies_commit();
        const T *a = reinterpret_cast<const T *>(stages + kb % S * Tile::STAGE) + m0;
        const float *b = reinterpret_cast<const float *>(stages + kb % S * Tile::STAGE + Tile::A_STAGE) + c0;
#pragma unroll 4
        for (int k = 0; k < BK; ++k) {
            float av[TM], bv[TN];
#pragma unroll
            for (int h = 0; h < TM / 4; ++h) {
                if constexpr (sizeof(T) == 4) {
                    *reinterpret_cast<float4 *>(av + 4 * h) = *reinterpret_cast<const float4 *>(a + k * BM + 16 * h);
                } else {
                    const uint2 w = *reinterpret_cast<const uint2 *>(a + k * BM + 16 * h);
                    av[4 * h] = __uint_as_float(w.x << 16); av[4 * h + 1] = __uint_as_float(w.x & 0xffff0000u);
                    av[4 * h + 2] = __uint_as_float(w.y << 16); av[4 * h + 3] = __uint_as_float(w.y & 0xffff0000u);
                }
            }
            if constexpr (TN == 4) *reinterpret_cast<float4 *>(bv) = *reinterpret_cast<const float4 *>(b + k * BN);
            else *reinterpret_cast<float2 *>(bv) = *reinterpret_cast<const float2 *>(b + k * BN);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; j += 2) fma_two(acc[i][j], acc[i][j + 1], av[i], bv[j], bv[j + 1]);
        }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int32_t m = m_at + m0 + i % 4 + 16 * (i / 4), c = n_at + c0;
        if (m >= p.d) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            if (c + j >= cols) break;
            if (splits > 1) part[(((int64_t)slice * p.groups + group) * p.d + m) * cols + c + j] = acc[i][j];
            else ((c + j < p.n ? p.dW + c : p.dW2 + (c - p.n)) + ((int64_t)group * p.d + m) * p.n)[j] = acc[i][j];
        }
    }
}

// whether rows come in sixteen bytes at a time: of logits, and of the weights as well
bool quads_of_logits(const GateProduct &p) { return (p.W2 ? 2 * (int64_t)p.n : p.n) % 4 == 0 && aligned16(p.dlogit); }
bool quads_of_rows(const GateProduct &p) { return p.n % 4 == 0 && aligned16(p.W) && (!p.W2 || aligned16(p.W2)) && quads_of_logits(p); }

template <int BM, int BN, int TM, int TN, int BK, int S, int BLOCKS> int32_t launch_rows(const GateProduct &p, int32_t *tile_prefix, cudaStream_t st) {
    using Tile = RowsTile<BM, BN, TM, TN, BK, S>;
    int64_t tiles = cdiv(p.rows, BM);
    if (p.offsets) {
        MOE_TRY(launch_tile_prefix(p.offsets, p.groups, BM, tile_prefix, st));
        tiles += p.groups;
    }
    if (cdiv(p.d, BN) > 65535) return MOE_ERR_UNSUPPORTED;
    auto run = [&](auto quads) -> int32_t {
        static PerDevice configured;
        const auto kernel = gate_rows_kernel<BM, BN, TM, TN, BK, S, BLOCKS, decltype(quads)::value>;
        if (!allow_shared(configured, kernel, Tile::SHARED)) return MOE_ERR_CUDA;
        launch_kernel(kernel, dim3((unsigned)tiles, (unsigned)cdiv(p.d, BN)), Tile::NT, Tile::SHARED, st, p, (const int32_t *)tile_prefix);
        MOE_LAUNCHED();
        return MOE_OK;
    };
    return quads_of_rows(p) ? run(std::true_type()) : run(std::false_type());
}
template <typename T, int BM, int BN, int TM, int TN, int BK, int S, int BLOCKS> int32_t launch_wgrad(const GateProduct &p, int32_t splits, float *part, cudaStream_t st) {
    using Tile = WgradTile<T, BM, BN, TM, TN, BK, S>;
    const int64_t cols = p.W2 ? 2 * (int64_t)p.n : p.n;
    if (cdiv(cols, BN) > 65535 || (int64_t)p.groups * splits > 65535) return MOE_ERR_UNSUPPORTED;
    auto run = [&](auto quads) -> int32_t {
        static PerDevice configured;
        const auto kernel = gate_wgrad_kernel<T, BM, BN, TM, TN, BK, S, BLOCKS, decltype(quads)::value>;
        if (!allow_shared(configured, kernel, Tile::SHARED)) return MOE_ERR_CUDA;
        launch_kernel(kernel, dim3((unsigned)cdiv(p.d, BM), (unsigned)cdiv(cols, BN), (unsigned)(p.groups * splits)), Tile::NT, Tile::SHARED, st, p, splits, part);
        MOE_LAUNCHED();
        return MOE_OK;
    };
    return quads_of_logits(p) ? run(std::true_type()) : run(std::false_type());
}
}  // namespace

// Where the products below are faster than the float product of gemm_simt.cu; us, that way and this way, tokens x features x logits:
//   dX: 256 x 64 x 16 4.1 2.4; 81 x 128 x 128 5.4 4.1 (16 x 16 tiles); 2085 x 256 x 32 5.7 5.0; 3001 x 320 x 40 9.7 7.9; 5000 x 512 x 32 14.8 12.1;
//       15000 x 512 x 16 34.8 19.1; but 15000 x 128 x 72 16.3 20.8, 12000 x 256 x 128 30 44: with a wider contraction the multiply-adds count, of which
//       eight rows and columns a thread from transposed tiles need fewer moves
//       single floats (n no multiple of four): 24 x 512 x 66 7.0 4.4; 3000 x 128 x 14 5.3 5.0; 5000 x 320 x 26 11.5 9.0; 60000 x 256 x 10 63 40;
//       20000 x 1024 x 44 131 120; but 2000 x 1024 x 78 22 26, 8192 x 512 x 94 41 48, 1019 x 512 x 222 15 25: the same line
//   dW: 256 x 64 x 16 4.4 4.1, 15000 x 512 x 16 22.9 15.8 (64 x 16 tiles); 1000 x 512 x 24 6.2 4.4, 2085 x 256 x 32 6.3 4.6 (32 x 32, two warps);
//       3001 x 320 x 40 9.2 7.3, 5000 x 512 x 32 11.5 9.2, 15000 x 128 x 72 17.7 15.5 (64 x 32); but 12000 x 256 x 128 26.8 28.6, 20000 x 1024 x 40 70 75
//       single floats (rows of logits that are no multiple of sixteen bytes): that way twice at all sizes, 3000 x 128 x 14 11.1 4.2, 8192 x 512 x 94
//       64 29, 60000 x 256 x 10 69 35, 15000 x 256 x 650 276 153, 5000 x 512 x 1970 582 309
bool gate_rows_supported(const GateProduct &p) {
    const int32_t cols = p.W2 ? 2 * p.n : p.n;
    if (cdiv(p.d, 16) > 65535) return false;
    return p.rows < 512 ? cols <= 256 : cols <= 40 && 4 * cdiv(p.d, 64) * 64 <= 5 * (int64_t)p.d;
}
int32_t launch_gate_rows(const GateProduct &p, int32_t *tile_prefix, cudaStream_t st) {
    if (p.rows == 0) return MOE_OK;
    if (p.rows < 512) return launch_rows<16, 16, 2, 2, 32, 4, 8>(p, tile_prefix, st);
    if (2 * (cdiv(p.rows, 64) + p.groups / 2) * cdiv(p.d, 64) >= 148) return launch_rows<64, 64, 8, 4, 32, 2, 4>(p, tile_prefix, st);
    return launch_rows<32, 32, 4, 4, 32, 2, 8>(p, tile_prefix, st);
}

static bool few_blocks(const GateProduct &p, int32_t cols, int32_t splits) { return cdiv(p.d, 32) * cdiv(cols, 32) * p.groups * splits <= 2 * 148; }
bool gate_wgrad_supported(const GateProduct &p) {
    const int32_t cols = p.W2 ? 2 * p.n : p.n, splits = simt_wgrad_splits(p.d, cols, p.groups, p.rows);
    if (cdiv(cols, 16) > 65535 || (int64_t)p.groups * splits > 65535) return false;
    return !quads_of_logits(p) || cols <= 16 || few_blocks(p, cols, splits) || (cols <= 72 && p.d <= 512);
}
// part: simt_wgrad_splits(d, logits, groups, rows) * groups * d * logits floats
int32_t launch_gate_wgrad(const GateProduct &p, float *part, cudaStream_t st, GateParts *parts_left) {
    const int32_t cols = p.W2 ? 2 * p.n : p.n, splits = simt_wgrad_splits(p.d, cols, p.groups, p.rows);
    auto run = [&](auto x) {
        using T = decltype(x);
        // few features, of which a wider tile would mostly be empty; with few slices its warps are worth more. 32000 tokens x 8 x 72 logits 18.7 us, this way
        // 9.5, 26346 x 16 x 40 12.0, 6.0; but 3000 x 16 x 80 3.8, 5.2
        if (p.d <= 16 && !few_blocks(p, cols, splits))
            return cols <= 16 ? launch_wgrad<T, 16, 16, 4, 2, 32, 4, 8>(p, splits, part, st) : launch_wgrad<T, 16, 32, 4, 4, 32, 4, 8>(p, splits, part, st);
        if (cols <= 16) return launch_wgrad<T, 64, 16, 4, 2, 32, 4, 4>(p, splits, part, st);
        if (few_blocks(p, cols, splits) || p.d <= 32) return launch_wgrad<T, 32, 32, 4, 2, 32, 4, 4>(p, splits, part, st);
        return launch_wgrad<T, 64, 32, 4, 4, 32, 4, 4>(p, splits, part, st);
    };
    MOE_TRY(p.act == MOE_BF16 ? run(bf16()) : run(float()));
    if (splits == 1) return MOE_OK;
    if (parts_left) {
        *parts_left = {part, splits, p.d, cols, p.n, p.n, p.dW, p.dW2};
        return MOE_OK;
    }
    return launch_slices_sum(part, splits, p.groups, p.d, cols, p.n, p.dW, p.dW2, st);
}

}  // namespace moe
