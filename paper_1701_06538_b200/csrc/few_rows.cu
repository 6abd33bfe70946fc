// Products of float experts with few rows each:
//   rows        C[r] = A[r] . W[e]        W[e] as [K, N], or [N, K] read transposed
//   gradients   C[e] = A_e^T . B_e        over the rows of segment e
// These read, or write, an expert's whole matrix for a handful of rows: bound by memory (5.9 floats a cycle and SM come in, sixteen multiply-adds each
// are what the FP32 pipes do meanwhile). So the weights go from memory to registers without a stop, every
// load sixteen bytes a lane along their rows and many in flight; the rows of A wait in shared memory or the first-level cache. Sixteen rows a tile; a tile
// with fewer runs with eight or four, so that the arithmetic follows the rows that are there. The float product of gemm_simt.cu, whose tiles of 32
// rows and more stage both operands in shared memory, and this way, us:
//   416 experts x 1 row of 832 x 512 (709 MB of weights): rows 312 -> 138; transposed 334, 333 -> 133, 128; gradients 402, 374 -> 122, 119
//   (5.5 TB/s in, 5.9 TB/s out); 32 x 9 of 512 x 3712 (243 MB): rows 190 -> 100; transposed 139, 208 -> 89, 88; gradients 142, 138 -> 53, 53
// The product that makes hid is not among them: its signs are the ReLU mask, and it keeps one chain of multiply-adds per output (api.cu).
#include "async_copy.cuh"
#include "moe_internal.cuh"

#include <type_traits>

namespace moe {

namespace {

constexpr int FEW_ROWS = 16, FEW_THREADS = 128, FEW_WARPS = FEW_THREADS / 32;

struct FewRows {
    const float *A, *W;
    float *C;
    const float *bias, *mask;  // of rows; of transposed products
    int32_t N, K, nseg;
    int64_t w_e;
    const int32_t *offsets, *prefix;
};

// A tile: the rows of a segment from row0 on, by the least of 4, 8 and 16 that holds them
struct FewTile { int32_t e, row0, rows; };
__device__ __forceinline__ bool few_tile(const FewRows &p, int4 *sh, FewTile &t) {
    const int4 at = segment_of_tile(p.prefix, p.offsets, p.nseg, blockIdx.x, sh);
    t.e = at.x;
    t.row0 = at.y + at.w * FEW_ROWS;
    t.rows = min(FEW_ROWS, at.z - t.row0);
    return at.x >= 0;
}
template <typename Run> __device__ __forceinline__ void with_rows(int rows, Run run) {
    if (rows <= 4) run(std::integral_constant<int, 4>());
    else if (rows <= 8) run(std::integral_constant<int, 8>());
    else run(std::integral_constant<int, 16>());
}

// W[e] [K, N]: LC lanes take 4 LC columns of a row of W, the 32 / LC groups of lanes and the warps share the contraction, 32 features at a time
template <int LC, int WARPS> __global__ void __launch_bounds__(32 * WARPS, WARPS > 4 ? 1 : 3) few_rows_kernel(const FewRows p) {
    constexpr int CW = 4 * LC, NT = 32 * WARPS;
    wait_previous_kernel();
    __shared__ int4 tile_at;
    __shared__ __align__(16) float buf[WARPS * FEW_ROWS * CW];  // x: [warp][row][32], then the warps' sums [warp][row][CW]
    FewTile t;
    if (!few_tile(p, &tile_at, t)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, group = lane / LC, n_at = blockIdx.y * CW, col = n_at + lane % LC * 4;
    const float *__restrict__ w = p.W + t.e * p.w_e + (col < p.N ? col : 0);  // (columns that are computed and dropped)
    const float *__restrict__ a = p.A + (int64_t)t.row0 * p.K;
    with_rows(t.rows, [&](auto rows_) {
        constexpr int RB = decltype(rows_)::value;
        float acc[RB][4], next[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[r][j] = 0.0f;
        float *x = buf + warp * FEW_ROWS * 32;
        const int chunks = (p.K + 31) / 32;
        auto fetch = [&](int c) {
            const int k = c * 32 + lane;
            const float *__restrict__ from = a + k;
#pragma unroll
            for (int r = 0; r < RB; ++r, from += p.K) next[r] = r < t.rows && k < p.K ? *from : 0.0f;  // (one address: sixteen of them were spilled)
        };
        if (warp < chunks) fetch(warp);
        for (int c = warp; c < chunks; c += WARPS) {
            __syncwarp();
#pragma unroll
            for (int r = 0; r < RB; ++r) x[r * 32 + lane] = next[r];
            __syncwarp();
            if (c + WARPS < chunks) fetch(c + WARPS);
            const int k0 = c * 32 + group * LC;
#pragma unroll(WARPS > 4 ? 1 : 2)
            for (int j = 0; j < LC; j += 4) {
                float4 wv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    wv[u] = k0 + j + u < p.K ? __ldg(reinterpret_cast<const float4 *>(w + (int64_t)(k0 + j + u) * p.N)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    const float4 xv = *reinterpret_cast<const float4 *>(x + r * 32 + group * LC + j);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float s = reinterpret_cast<const float *>(&xv)[u];
                        fma_two(acc[r][0], acc[r][1], s, wv[u].x, wv[u].y);
                        fma_two(acc[r][2], acc[r][3], s, wv[u].z, wv[u].w);
                    }
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < RB; ++r) {
#pragma unroll
            for (int off = LC; off < 32; off <<= 1)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[r][j] += __shfl_xor_sync(0xffffffffu, acc[r][j], off);
            if (group == 0) *reinterpret_cast<float4 *>(buf + (warp * FEW_ROWS + r) * CW + lane * 4) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
        }
        __syncthreads();
        for (int id = tid; id < t.rows * LC; id += NT) {
            const int r = id / LC, c = n_at + id % LC * 4;
            if (c >= p.N) continue;
            float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
            for (int q = 0; q < WARPS; ++q) {
                const float4 v = *reinterpret_cast<const float4 *>(buf + (q * FEW_ROWS + r) * CW + id % LC * 4);
                s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
            }
            const int64_t at = (int64_t)(t.row0 + r) * p.N + c;
            const float4 b = p.bias ? *reinterpret_cast<const float4 *>(p.bias + (int64_t)t.e * p.N + c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            *reinterpret_cast<float4 *>(p.C + at) = make_float4(s.x + b.x, s.y + b.y, s.z + b.z, s.w + b.w);
        }
    });
}

// W[e] [N, K]: a warp takes the dot products of all rows with a few columns at a time, LK lanes along the contraction; KS: so do the warps
constexpr int transposed_columns(int lk, int ks) { return 8 * (32 / lk) * FEW_WARPS / ks; }  // of a block, eight a group of lanes
template <int LK, int KS> __global__ void __launch_bounds__(FEW_THREADS, 4) few_rows_transposed_kernel(const FewRows p) {
    constexpr int GROUPS = 32 / LK, PER_GROUP = 8, COLS = transposed_columns(LK, KS);
    wait_previous_kernel();
    __shared__ int4 tile_at;
    __shared__ float sums[KS > 1 ? FEW_WARPS : 1][KS > 1 ? 64 * GROUPS : 1];
    FewTile t;
    if (!few_tile(p, &tile_at, t)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = warp % KS, in = lane % LK, group = lane / LK;
    const float *__restrict__ w = p.W + t.e * p.w_e;
    const float *__restrict__ a = p.A + (int64_t)t.row0 * p.K;
    with_rows(t.rows, [&](auto rows_) {
        constexpr int RB = decltype(rows_)::value, NB = RB == 16 ? 4 : 8, V = RB * NB;
#pragma unroll 1
        for (int pass = 0; pass < PER_GROUP / NB; ++pass) {
            const int n0 = blockIdx.y * COLS + (warp / KS * GROUPS + group) * PER_GROUP + pass * NB;
            float acc[V];
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q] = 0.0f;
            for (int k = (part * LK + in) * 4; k < p.K; k += 4 * LK * KS) {
                float4 wv[NB];
#pragma unroll
                for (int i = 0; i < NB; ++i) wv[i] = __ldg(reinterpret_cast<const float4 *>(w + (int64_t)min(n0 + i, p.N - 1) * p.K + k));  // (computed and dropped)
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    const float4 x = __ldg(reinterpret_cast<const float4 *>(a + (int64_t)min(r, t.rows - 1) * p.K + k));
#pragma unroll
                    for (int i = 0; i < NB; ++i) {
                        float &s = acc[r * NB + i];
                        s = fmaf(x.x, wv[i].x, s); s = fmaf(x.y, wv[i].y, s); s = fmaf(x.z, wv[i].z, s); s = fmaf(x.w, wv[i].w, s);
                    }
                }
            }
            // sums over the group's lanes; lane l of it keeps values l V / LK and up
#pragma unroll
            for (int off = LK / 2, half = V / 2; off > 0; off >>= 1, half >>= 1) {
                const bool up = lane & off;
#pragma unroll
                for (int q = 0; q < half; ++q) {
                    const float keep = up ? acc[q + half] : acc[q], give = up ? acc[q] : acc[q + half];
                    acc[q] = keep + __shfl_xor_sync(0xffffffffu, give, off);
                }
            }
            auto store = [&](int first, int f, float v) {
                const int r = f / NB, n = first + f % NB;
                if (r >= t.rows || n >= p.N) return;
                const int64_t at = (int64_t)(t.row0 + r) * p.N + n;
                p.C[at] = !p.mask || p.mask[at] > 0.0f ? v : 0.0f;
            };
            if constexpr (KS == 1) {
#pragma unroll
                for (int q = 0; q < V / LK; ++q) store(n0, in * (V / LK) + q, acc[q]);
            } else {
                static_assert(KS == 1 || KS == FEW_WARPS, "the warps of a block have the same columns");
#pragma unroll
                for (int q = 0; q < V / LK; ++q) sums[warp][group * V + in * (V / LK) + q] = acc[q];
                __syncthreads();
                for (int id = threadIdx.x; id < GROUPS * V; id += FEW_THREADS) {
                    float s = 0.0f;
#pragma unroll
                    for (int q = 0; q < KS; ++q) s += sums[q][id];
                    store(blockIdx.y * COLS + id / V * PER_GROUP + pass * NB, id % V, s);
                }
                __syncthreads();
            }
        }
    });
}

// C[e] [M, N]: 8 TM x 64 outputs a block, TM rows and four columns a thread; sixteen rows of the segment in shared memory and the next ones on their way. A
// block goes through its whole segment, so that where loads are uneven the longest one is the launch's time: a row of it takes 32 ns with TM = 4, 51 with 8 and 94 with 16
// and nothing on the way meanwhile, and 31 in gemm_simt.cu. With blocks enough for all SMs all along TM = 8 reads less of shared memory (see launch_float_expert_product).
// A backward call, us, by the float product and this way: 126 experts, 4410 rows, the longest segment 1399, of 64 x 64 112, 83; 416, 6656, 684, 64 x 128 127,
// 103 (TM = 16: 175); 377, 25259, 2655, 704 x 448 2317, 1413; 416 x 1 row of 832 x 512 1456, 520
struct FewGradients {
    const float *A, *B;
    float *C;
    int32_t M, N, nseg, tiles_n;
    const int32_t *offsets;
};
constexpr int GRAD_N = 64;
constexpr int grad_rows(int tm) { return FEW_WARPS * 2 * tm; }  // of a block
template <int TM> __global__ void __launch_bounds__(FEW_THREADS, TM == 4 ? 8 : 6) few_gradients_kernel(const FewGradients p) {
    constexpr int LC = GRAD_N / 4, G = 32 / LC, S = 2, GRAD_M = grad_rows(TM);
    wait_previous_kernel();
    __shared__ __align__(16) float as[S][FEW_ROWS][GRAD_M], bs[S][FEW_ROWS][GRAD_N];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, e = blockIdx.y, m_at = blockIdx.x / p.tiles_n * GRAD_M, n_at = blockIdx.x % p.tiles_n * GRAD_N;
    const int begin = p.offsets[e], end = p.offsets[e + 1], blocks = (end - begin + FEW_ROWS - 1) / FEW_ROWS;
    const int row = (warp * G + lane / LC) * TM, col = lane % LC * 4;
    auto load = [&](int block, int s) {
        const int r0 = begin + block * FEW_ROWS, rows = min(FEW_ROWS, end - r0);
        for (int id = tid; id < rows * (GRAD_M / 4); id += FEW_THREADS) {
            const int r = id / (GRAD_M / 4), m = id % (GRAD_M / 4) * 4;
            if (m_at + m < p.M) copy16(&as[s][r][m], p.A + (int64_t)(r0 + r) * p.M + m_at + m);  // (what lies behind is computed from whatever is there and dropped)
        }
        for (int id = tid; id < rows * LC; id += FEW_THREADS) {
            const int r = id / LC, n = id % LC * 4;
            if (n_at + n < p.N) copy16(&bs[s][r][n], p.B + (int64_t)(r0 + r) * p.N + n_at + n);
        }
    };
    float acc[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
#pragma unroll
    for (int s = 0; s < S - 1; ++s) {
        if (s < blocks) load(s, s);
        copies_commit();
    }
    int s = 0;
    for (int block = 0; block < blocks; ++block) {
        copies_wait<S - 2>();
        __syncthreads();  // this block is there for all, the one before is read by all
        if (block + S - 1 < blocks) load(block + S - 1, s == 0 ? S - 1 : s - 1);
        copies_commit();
        const int rows = min(FEW_ROWS, end - begin - block * FEW_ROWS);
#pragma unroll 4
        for (int r = 0; r < rows; ++r) {
            const float4 b = *reinterpret_cast<const float4 *>(&bs[s][r][col]);
#pragma unroll
            for (int i = 0; i < TM; i += 4) {
                const float4 a = *reinterpret_cast<const float4 *>(&as[s][r][row + i]);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float v = reinterpret_cast<const float *>(&a)[u];
                    fma_two(acc[i + u][0], acc[i + u][1], v, b.x, b.y);
                    fma_two(acc[i + u][2], acc[i + u][3], v, b.z, b.w);
                }
            }
        }
        if (++s == S) s = 0;
    }
    if (n_at + col >= p.N) return;
    float *c = p.C + ((int64_t)e * p.M + m_at + row) * p.N + n_at + col;
#pragma unroll
    for (int i = 0; i < TM; ++i)
        if (m_at + row + i < p.M) *reinterpret_cast<float4 *>(c + (int64_t)i * p.N) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
}

int64_t grad_blocks(const SimtGemm &g) { return cdiv(g.M, grad_rows(4)) * cdiv(g.N, GRAD_N); }  // of an expert

// Where this way is the faster one, by the rows an expert has on average: read off both ways' times of 780 products each (1 to 10000 rows an expert, widths of 8 to 4096,
// equal and Zipf loads). Of the times that the rule takes, geometric means and the worst against the float product's: rows 0.62 and 1.21, transposed
// 0.56 and 1.35, gradients 0.53 and 1.27. us, by the float product and this way:
//   rows         64 experts of 200 x 520, 16 rows 34.6, 24.4;  48 54.4, 38.0;  but 120 x 60 of 1728 x 960 580, 818;  47 x 61 of 3136 x 1344 612, 792;
//                narrow results of many experts: 209 x 16 of 384 x 64 19.6, 22.4;  432 x 51 of 64 x 64 14.6, 27.7;  short contractions: 134 x 31 of 64 x 1408 105, 119 (a forward call)
//   transposed   64 of 200 x 520, 16 31.3 + 35.5, 22.5 + 22.5;  32 37.7 + 37.0, 36.0 + 31.4;  48 37.0 + 53.0, 49.4 + 43.1
//   gradients    more than 32 rows an expert want four blocks and more an expert, or eight a SM in all: 126 x 35, the longest 1399, of 64 x 64 43, 53;
//                one block an expert 16: 59 x 26 of 28 x 24, the longest 257, 34.8, 40.8 (a backward call)
bool few_rows_take(const SimtGemm &g, const SegmentPlan &plan, int64_t R) {
    const bool grad = g.mode == 1;
    if (g.N % 4 != 0 || g.K % 4 != 0 || g.M % (grad ? 4 : 1) != 0 || !aligned16(g.A) || !aligned16(g.B) || !aligned16(g.C)) return false;
    if ((g.bias && !aligned16(g.bias)) || (g.mask && !aligned16(g.mask)) || g.nseg > 65535 || cdiv(g.N, 8) > 65535) return false;
    if (g.relu || (!grad && (!plan.prefix_of(FEW_ROWS) || (g.sb_j == 1 ? g.mask : g.bias)))) return false;
    const int64_t n = g.nseg;
    if (grad) {
        const int64_t blocks = grad_blocks(g);
        return R <= (blocks > 1 ? 32 : 16) * n || (R <= 64 * n && blocks > 4) || (R <= 128 * n && n * blocks >= 8 * 148);
    }
    if (g.sb_j != 1) return R <= 32 * n;
    const bool wide = g.N > 64 || n < 100;
    return R <= (wide ? 16 : 8) * n || (wide && g.K > 64 && R <= (n * g.K * g.N < 5000000 ? 64 : 32) * n);
}

template <int LC, int WARPS> int32_t launch_rows(const FewRows &p, int64_t tiles, cudaStream_t st) {
    launch_kernel(few_rows_kernel<LC, WARPS>, dim3((unsigned)tiles, (unsigned)cdiv(p.N, 4 * LC)), 32 * WARPS, 0, st, p);
    MOE_LAUNCHED();
    return MOE_OK;
}
template <int LK, int KS> int32_t launch_transposed(const FewRows &p, int64_t tiles, cudaStream_t st) {
    launch_kernel(few_rows_transposed_kernel<LK, KS>, dim3((unsigned)tiles, (unsigned)cdiv(p.N, transposed_columns(LK, KS))), FEW_THREADS, 0, st, p);
    MOE_LAUNCHED();
    return MOE_OK;
}
template <int TM> int32_t launch_gradients(FewGradients p, cudaStream_t st) {
    p.tiles_n = (int32_t)cdiv(p.N, GRAD_N);
    launch_kernel(few_gradients_kernel<TM>, dim3((unsigned)(cdiv(p.M, grad_rows(TM)) * p.tiles_n), (unsigned)p.nseg), FEW_THREADS, 0, st, p);
    MOE_LAUNCHED();
    return MOE_OK;
}
}  // namespace

int32_t launch_float_expert_product(const SimtGemm &g, const SegmentPlan &plan, int64_t R, cudaStream_t st) {
    if (R == 0 || !few_rows_take(g, plan, R)) return launch_simt_gemm(g, nullptr, st, nullptr, &plan);
    if (g.mode == 1) {
        FewGradients p = {(const float *)g.A, (const float *)g.B, (float *)g.C, (int32_t)g.M, (int32_t)g.N, g.nseg, 0, g.offsets};
        // (416 x 1 row of 832 x 512, 86528 blocks of TM = 4: a backward call 576, with TM = 8 520; 128 x 24 of 512 x 1024, 32768, 573, 535; 416 x 16 of
        // 64 x 128, the longest 684, 3328 blocks: 103, 135)
        return g.nseg * grad_blocks(g) >= 64 * 148 ? launch_gradients<8>(p, st) : launch_gradients<4>(p, st);
    }
    const FewRows p = {(const float *)g.A, (const float *)g.B, (float *)g.C, (const float *)g.bias, (const float *)g.mask, (int32_t)g.N, (int32_t)g.K, g.nseg, g.b_e,
                       g.offsets, plan.prefix_of(FEW_ROWS)};
    const int64_t tiles = imin(cdiv(R, FEW_ROWS) + g.nseg, R), live = imin(R, cdiv(R, FEW_ROWS) + g.nseg / 2);  // launched, and about how many have rows
    // Blocks enough for every SM first, then the widest rows; warps that share a long contraction where there are few blocks. us:
    //   transposed, 8 lanes a row (128 columns a block), 32 lanes (32 columns), 32 lanes and four warps a contraction (8 columns):
    //     96 experts x 1 row, 64 -> 2880 14.9 26.9 82;  13 x 15, 128 -> 3840 17.0 21.6 54;  179 x 2, 128 -> 128 9.2 6.7 12;
    //     32 x 9, 512 -> 3712 110 89 135, 3712 -> 512 426 122 88;  192 x 2, 2728 -> 72 305 94 40;  16 x 5, 256 -> 128 19 8.0 4.6
    //   rows, 128, 64, 32 columns a block, and 32 with 16 warps a contraction:
    //     32 x 9, 512 -> 3712 74 85 94 154, 3712 -> 512 181 127 107 100;  88 x 0.4, 1088 -> 896 36 25 27 45;  13 x 15, 3840 -> 128 170 111 64 30;
    //     192 x 2, 72 -> 2728 52 70 97 351, 2728 -> 72 84 70 51 60;  73 x 10, 704 -> 128 39 28 19 21
    if (g.sb_j != 1) {
        if (g.K <= 128 && live * cdiv(g.N, 128) >= 2 * 148) return launch_transposed<8, 1>(p, tiles, st);
        if (live * cdiv(g.N, 32) < (g.K >= 1024 ? 4 : 1) * 148 && g.K >= 256) return launch_transposed<32, 4>(p, tiles, st);
        return launch_transposed<32, 1>(p, tiles, st);
    }
    if (live * cdiv(g.N, 128) >= 2 * 148) return launch_rows<32, 4>(p, tiles, st);
    if (live * cdiv(g.N, 64) >= 2 * 148) return launch_rows<16, 4>(p, tiles, st);
    if (live * cdiv(g.N, 32) > 148 || g.K < 512) return launch_rows<8, 4>(p, tiles, st);
    return launch_rows<8, 16>(p, tiles, st);
}

}  // namespace moe
