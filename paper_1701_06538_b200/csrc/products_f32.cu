// The float experts' products on the tensor cores: every operand as three bf16 terms (hi + mid + lo hold a float's 24 bits, see three_terms), a product as the
// six terms of at most 2^-16 of the leading one and more: hi.hi, and hi.mid, mid.hi, mid.mid, hi.lo, lo.hi. Float products by FP32
// multiply-adds (gemm_simt.cu) run at 20 to 29 of the chip's 74 TFLOP/s; this way five of the six products of a step with 16 experts x 260 rows
// of 256 x 512 take 14 to 16 us each instead of 38 to 52, most of it the way of the operands from L2. (The first, whose signs are the ReLU mask, stays
// with one chain of multiply-adds per output.)
//
// Precision. A tensor core's accumulator drops low bits at every step of 16: over a long contraction more than the one rounding per term of a
// chain of multiply-adds. So the leading products are summed in tensor memory over 128 terms of the contraction only and these sums added,
// rounding to nearest, in registers; the five small ones, 2^-8 of them, have an accumulator of their own for the whole contraction.
// Relative error against 64 bits (2-norms) of y, dX, dW1 by multiply-adds and this way: 16 experts, 4170 rows, 256 x 512: 4.8e-7, 4.8e-7, 4.3e-7
// and 3.1e-7, 3.2e-7, 3.2e-7; 12 experts, 3000 rows, 128 x 4096: 8.5e-7, 8.5e-7, 3.3e-7 and 2.7e-7, 2.8e-7, 2.5e-7.
//
// Values that are no numbers. An infinite operand meets terms of either sign and zeros, and becomes NaN where the float chain has an infinity. Every
// element that does not come out finite is therefore computed again as the float chain that gemm_simt.cu computes, with its result: by the CTA that has
// the tile, when its tensor-core work is done and nothing waits for it any more, as a tile of multiply-adds. (Sums whose
// parts leave float's range on the way depend on the order of the parts, as ever.)
//
// One CTA, 128 x 128 tiles, K blocks of 64: a stage holds the three terms of both operands (96 KiB, two stages), of which the six products
// read what otherwise would be loaded twice: L2 delivers a stage in about the time of its 1536 cycles of tensor work. Warp 0 copies, warp 1
// issues, warps 2-9 add, finish and store: float results, and where a later product reads them their three terms.
#include <string.h>

#include <type_traits>

#include "async_copy.cuh"
#include "tc.cuh"

namespace moe {

namespace {

constexpr int F_TILE = 128, F_STAGES = 2, F_OPERAND = F_TILE * BK * 2 /* 16 KiB */, F_STAGE = 6 * F_OPERAND;
constexpr int F_SUB = 2;  // K blocks of a sum of leading products
constexpr int F_SHARED = F_STAGES * F_STAGE + 1024 /*alignment*/ + 8 * 4096 /*a slab per epilogue warp*/ + 256 /*barriers*/;

struct FloatProduct {
    const int32_t *offsets, *row_tiles;  // [nseg + 1] bounds of the segments (rows); &number of row tiles
    const int4 *info;                    // per row tile {segment, first row, segment end, number}
    int32_t N, M, K;                     // ROW_*: K is the contraction, M unused; WGRAD: [M, N] per segment
    int32_t tiles_n, per_e, total;       // tiles beside each other; WGRAD: of a segment, of all segments; ROW_*: at most
    Divisor by_tiles_n, by_per_e;
    float *out;
    bf16 *terms;                         // [rows][3 N], or nullptr
    const float *bias, *mask, *A, *B;    // [nseg, N]; [R, N]; the operands themselves
    int32_t *status;
};
enum FloatEpilogue { FE_PLAIN = 0, FE_BIAS, FE_MASK };

// Three bf16 terms of a float times 2^16: hi + mid + lo == 2^16 v exactly, down to float's smallest bit 2^-149, since bf16's is 2^-133 (without the factor
// values of 1e-36 had 15 bits, and ys of such activations errors of 1e-4 of its size). Values from 2^112 on, and sums of products from 2^96, leave float's range: these
// outputs are not finite and computed again. (Rounding to nearest; values that would round to infinity are cut instead. Infinities and NaN are
// their own leading term.)
constexpr float F_SCALE = 0x1p16f, F_UNSCALE = 0x1p-32f;  // of an operand; of a product of two
__device__ __forceinline__ void three_terms(float unscaled, bf16 &hi, bf16 &mid, bf16 &lo) {
    const float v = unscaled * F_SCALE;
    const uint32_t size = __float_as_uint(v) & 0x7fffffffu;
    hi = __float2bfloat16_rn(v);
    if (size >= 0x7f7f8000u && size < 0x7f800000u) hi = __ushort_as_bfloat16((unsigned short)(__float_as_uint(v) >> 16));
    const float r = size < 0x7f800000u ? v - __bfloat162float(hi) : 0.0f;
    mid = __float2bfloat16_rn(r);
    lo = __float2bfloat16_rn(r - __bfloat162float(mid));
}
// of four neighbours, to places `apart` elements apart
__device__ __forceinline__ void store_terms(const float4 &v, bf16 *to, int64_t apart) {
    const float in[4] = {v.x, v.y, v.z, v.w};
    __align__(8) bf16 t[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) three_terms(in[i], t[0][i], t[1][i], t[2][i]);
#pragma unroll
    for (int q = 0; q < 3; ++q) *reinterpret_cast<uint2 *>(to + q * apart) = *reinterpret_cast<const uint2 *>(t[q]);
}

// What one launch computes: a weight gradient, a row product, or a weight gradient and then a row product that does not need it (they fill each
// other's last wave: a step with 16 experts x 260 rows of 256 x 512, 128 and up to 196 tiles, 174 us, this way 161). Tiles are dealt.
template <int ROW, int EPI, bool WITH_WGRAD> struct FloatLaunch {
    CUtensorMap row_a, row_b, wgrad_a, wgrad_b;
    FloatProduct row, wgrad;
};
struct FloatTile { int32_t e, row0, row_end, m0, n0, blocks; bool wgrad; };
template <int ROW, int EPI, bool WITH_WGRAD> __device__ __forceinline__ bool float_tile(const FloatLaunch<ROW, EPI, WITH_WGRAD> &L, int32_t id, FloatTile &t) {
    int32_t rest, tn;
    t.wgrad = WITH_WGRAD && id < L.wgrad.total;
    if (t.wgrad) {
        const FloatProduct &p = L.wgrad;
        t.e = p.by_per_e(id, rest);
        t.m0 = p.by_tiles_n(rest, tn) * F_TILE;
        t.row0 = p.offsets[t.e];
        t.row_end = p.offsets[t.e + 1];
        t.blocks = (t.row_end - t.row0 + BK - 1) / BK;
    } else {
        const FloatProduct &p = L.row;
        if (WITH_WGRAD) id -= L.wgrad.total;
        if (id >= p.total) return false;
        const int4 at = p.info[p.by_tiles_n(id, tn)];
        if (id >= *p.row_tiles * p.tiles_n) return false;
        t.e = at.x; t.row0 = at.y; t.row_end = at.z; t.m0 = 0;
        t.blocks = p.K / BK;
    }
    t.n0 = tn * F_TILE;
    return true;
}
// f(product, kind, epilogue) for a tile's product
template <int ROW, int EPI, bool WITH_WGRAD, typename F> __device__ __forceinline__ void with_product(const FloatLaunch<ROW, EPI, WITH_WGRAD> &L, const FloatTile &t, F f) {
    if constexpr (WITH_WGRAD) {
        if (t.wgrad) return f(L.wgrad, std::integral_constant<int, WGRAD>(), std::integral_constant<int, FE_PLAIN>());
    }
    f(L.row, std::integral_constant<int, ROW>(), std::integral_constant<int, EPI>());
}

// The elements of a stored tile that are not finite once more, each as one chain of multiply-adds in ascending order, through shared memory: 8 x 8 outputs a
// thread of the first 256, bound by the reads of shared memory (16 cycles a warp and row of 180 in all). A backward call, and with a NaN in dys, which makes whole
// matrices of gradients NaN: 4 experts x 2000 rows of 128 x 256 105 us, 535; 20000 rows of 64 x 128, one tile, 0.80 ms, 4.6. Every element by itself,
// straight from memory and while the MMA warp waited with its limit of 2 s, 3.8 ms and 37.
constexpr int R_BK = 32, R_PITCH = F_TILE + 4;
template <int KIND, int EPI> __device__ __forceinline__ void repair_tile(const FloatProduct &p, const FloatTile &t) {
    const int tid = threadIdx.x;
    const int64_t row0 = KIND == WGRAD ? t.m0 : t.row0;
    float *out = p.out + ((KIND == WGRAD ? (int64_t)t.e * p.M : 0) + row0) * p.N + t.n0;
    const int rows = (int)min((int64_t)F_TILE, (KIND == WGRAD ? p.M : t.row_end) - row0), cols = min(F_TILE, p.N - t.n0);
    bool odd = false;
    for (int i = tid; i < rows * (cols / 4); i += NTHREADS) {
        const float4 v = *reinterpret_cast<const float4 *>(out + (int64_t)(i / (cols / 4)) * p.N + i % (cols / 4) * 4);
        odd = odd || !isfinite(v.x) || !isfinite(v.y) || !isfinite(v.z) || !isfinite(v.w);
    }
    if (!__syncthreads_or(odd)) return;
    extern __shared__ uint8_t smem_raw[];  // the stages are free
    constexpr int OPERAND = R_BK * R_PITCH, LOADS = R_BK * F_TILE / 4 / 256;  // [R_BK][R_PITCH] floats: the contraction's index first
    float *stage = reinterpret_cast<float *>(smem_raw);
    const int depth = KIND == WGRAD ? t.row_end - t.row0 : p.K, tx = tid & 15, ty = tid >> 4;
    float acc[8][8];  // rows 4 ty + i % 4 + 64 (i / 4), columns 4 tx + j % 4 + 64 (j / 4)
#pragma unroll
    for (int i = 0; i < 64; ++i) acc[i >> 3][i & 7] = 0.0f;
    // Four neighbours at a time, into one stage while the other one is used: as they lie, by asynchronous copies; or, where they are neighbours along the
    // contraction, through registers, turned on the way
    constexpr bool TURN_A = KIND != WGRAD, TURN_B = KIND == ROW_BK;
    auto place = [&](bool turn, int q, int &across, int &along) {
        const int i = tid + 256 * q;
        across = turn ? i / (R_BK / 4) : i % (F_TILE / 4) * 4;
        along = turn ? i % (R_BK / 4) * 4 : i / (F_TILE / 4);
    };
    float4 turned[TURN_A + TURN_B + 1][LOADS];
    auto fetch = [&](int k0, float *as) {
        float *bs = as + OPERAND;
#pragma unroll
        for (int q = 0; q < LOADS; ++q) {
            int c, k;
            place(TURN_A, q, c, k);
            const bool live_a = c < rows && k0 + k < depth;
            const float *a = !live_a ? p.A : TURN_A ? p.A + (t.row0 + c) * (int64_t)p.K + k0 + k : p.A + (int64_t)(t.row0 + k0 + k) * p.M + t.m0 + c;
            if (TURN_A) turned[0][q] = live_a ? *reinterpret_cast<const float4 *>(a) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            else if (live_a) copy16(as + k * R_PITCH + c, a);
            else zero16(as + k * R_PITCH + c);
            place(TURN_B, q, c, k);
            const bool live_b = c < cols && k0 + k < depth;
            const float *b = !live_b         ? p.B
                             : KIND == WGRAD ? p.B + (int64_t)(t.row0 + k0 + k) * p.N + t.n0 + c
                             : TURN_B        ? p.B + ((int64_t)t.e * p.N + t.n0 + c) * p.K + k0 + k
                                             : p.B + ((int64_t)t.e * p.K + k0 + k) * p.N + t.n0 + c;
            if (TURN_B) turned[1][q] = live_b ? *reinterpret_cast<const float4 *>(b) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            else if (live_b) copy16(bs + k * R_PITCH + c, b);
            else zero16(bs + k * R_PITCH + c);
        }
        copies_commit();
    };
    auto put = [&](float *to, bool turn, const float4 (&v)[LOADS]) {
        if (!turn) return;
#pragma unroll
        for (int q = 0; q < LOADS; ++q) {
            int c, k;
            place(true, q, c, k);
            float *at = to + k * R_PITCH + c;
            at[0] = v[q].x; at[R_PITCH] = v[q].y; at[2 * R_PITCH] = v[q].z; at[3 * R_PITCH] = v[q].w;
        }
    };
    const int last_row = rows > 64, last_col = cols > 64;  // whether the tile's second halves have elements
    __syncthreads();
    if (tid < 256) fetch(0, stage);
    int at = 0;
    for (int k0 = 0; k0 < depth; k0 += R_BK, at ^= 1) {
        float *as = stage + at * 2 * OPERAND, *bs = as + OPERAND;
        if (tid < 256) {
            put(as, TURN_A, turned[0]);
            put(bs, TURN_B, turned[TURN_B]);
            copies_wait<0>();
        }
        __syncthreads();  // this stage is there for all, the other one is read by all
        if (tid >= 256) continue;
        if (k0 + R_BK < depth) fetch(k0 + R_BK, stage + (at ^ 1) * 2 * OPERAND);
#pragma unroll 4
        for (int k = 0; k < R_BK; ++k) {  // (zeros behind the end: a sum that began with +0 is never -0, so they do not change it)
            float a[8], b[8];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                *reinterpret_cast<float4 *>(a + 4 * u) = *reinterpret_cast<const float4 *>(as + k * R_PITCH + 4 * ty + 64 * u);
                *reinterpret_cast<float4 *>(b + 4 * u) = *reinterpret_cast<const float4 *>(bs + k * R_PITCH + 4 * tx + 64 * u);
            }
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                if ((h >> 1) > last_row || (h & 1) > last_col) continue;
#pragma unroll
                for (int i = 4 * (h >> 1); i < 4 * (h >> 1) + 4; ++i)
#pragma unroll
                    for (int j = 4 * (h & 1); j < 4 * (h & 1) + 4; j += 2) fma_two(acc[i][j], acc[i][j + 1], a[i], b[j], b[j + 1]);
            }
        }
    }
    if (tid < 256) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = 4 * ty + i % 4 + 64 * (i / 4);
            if (r >= rows) break;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = 4 * tx + j % 4 + 64 * (j / 4);
                if (c >= cols) continue;
                float *to = out + (int64_t)r * p.N + c;
                if (isfinite(*to)) continue;  // (zeros of the mask among them)
                float v = acc[i][j];
                if (EPI == FE_BIAS) v += p.bias[(int64_t)t.e * p.N + t.n0 + c];
                *to = v;
                if (EPI == FE_MASK && p.terms) {
                    bf16 *terms = p.terms + (row0 + r) * 3 * p.N + t.n0 + c;
                    three_terms(v, terms[0], terms[p.N], terms[2 * (int64_t)p.N]);
                }
            }
        }
    }
}
template <int ROW, int EPI_ROW, bool WITH_WGRAD> __device__ __noinline__ void repair_tiles(const FloatLaunch<ROW, EPI_ROW, WITH_WGRAD> &L) {
    FloatTile t;
    for (int32_t id = blockIdx.x; float_tile(L, id, t); id += gridDim.x)
        with_product(L, t, [&](const FloatProduct &p, auto KIND_, auto EPI_) { repair_tile<decltype(KIND_)::value, decltype(EPI_)::value>(p, t); });
}

template <int ROW, int EPI_ROW, bool WITH_WGRAD>
__global__ void __launch_bounds__(NTHREADS, 1) float_products_kernel(const __grid_constant__ FloatLaunch<ROW, EPI_ROW, WITH_WGRAD> L) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bars = base + F_STAGES * F_STAGE + 8 * 4096;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 16u + 8u * s; };
    auto tfull_bar = [&](int a) { return bars + 32u + 8u * a; };    // sums of leading products: two accumulators in turn
    auto tempty_bar = [&](int a) { return bars + 48u + 8u * a; };
    auto sfull_bar = [&](int a) { return bars + 64u + 8u * a; };    // small products: an accumulator per tile, two in turn
    auto sempty_bar = [&](int a) { return bars + 80u + 8u * a; };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + F_STAGES * F_STAGE + 8 * 4096 + 96);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + F_STAGES * F_STAGE + 8 * 4096 + 104);
    volatile int *odd_tiles = reinterpret_cast<volatile int *>(smem + F_STAGES * F_STAGE + 8 * 4096 + 108);  // a stored element is not finite
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1);
            mbar_init(tfull_bar(s), 1); mbar_init(tempty_bar(s), 8);
            mbar_init(sfull_bar(s), 1); mbar_init(sempty_bar(s), 8);
        }
        *abort_flag = 0;
        *odd_tiles = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(WITH_WGRAD ? &L.wgrad_a : &L.row_a) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(WITH_WGRAD ? &L.wgrad_b : &L.row_b) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void *)tmem_slot)),
                     "r"((uint32_t)TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    wait_previous_kernel();
    FloatTile t;

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int32_t id = blockIdx.x; ok && float_tile(L, id, t); id += gridDim.x) {
                with_product(L, t, [&](const FloatProduct &p, auto KIND_, auto) {
                    constexpr int KIND = decltype(KIND_)::value;
                    const CUtensorMap *tm_a = KIND == WGRAD ? &L.wgrad_a : &L.row_a, *tm_b = KIND == WGRAD ? &L.wgrad_b : &L.row_b;
                    for (int kb = 0; kb < t.blocks; ++kb) {
                        ok = mbar_wait(empty_bar(s), ph ^ 1u, abort_flag, L.row.status);
                        if (!ok) break;
                        const uint32_t at = base + s * F_STAGE;
                        mbar_expect_tx(full_bar(s), F_STAGE);
#pragma unroll
                        for (int q = 0; q < 3; ++q) {  // term q of A and of B
                            const uint32_t a = at + q * F_OPERAND, b = at + (3 + q) * F_OPERAND;
                            if (KIND == WGRAD) {
                                tma_load_3d(a, tm_a, full_bar(s), 0, t.row0 + kb * BK, (q * p.M + t.m0) / 64);
                                tma_load_3d(b, tm_b, full_bar(s), 0, t.row0 + kb * BK, (q * p.N + t.n0) / 64);
                            } else {
                                tma_load_2d(a, tm_a, full_bar(s), q * p.K + kb * BK, t.row0);
                                if (KIND == ROW_BMN) tma_load_4d(b, tm_b, full_bar(s), 0, kb * BK, (q * p.N + t.n0) / 64, t.e);
                                else tma_load_3d(b, tm_b, full_bar(s), q * p.K + kb * BK, t.n0, t.e);
                            }
                        }
                        if (++s == F_STAGES) { s = 0; ph ^= 1u; }
                    }
                });
            }
            // drain: every copy this thread started must have landed before the CTA may exit
            if (!ok)
                for (int q = 0; q < F_STAGES; ++q) {
                    const unsigned long long t0 = global_ns();
                    while (!mbar_try_wait(full_bar(q), 0) && !mbar_try_wait(full_bar(q), 1) && global_ns() - t0 < WAIT_LIMIT_NS) {}
                }
        }
    } else if (warp == 1) {
        int s = 0, acc = 0, small = 0;
        uint32_t ph = 0, acc_ph = 0, small_ph = 0;
        bool ok = true;
        for (int32_t id = blockIdx.x; ok && float_tile(L, id, t); id += gridDim.x) {
            if (t.blocks == 0) continue;  // empty segment: the epilogue writes zeros
            with_product(L, t, [&](const FloatProduct &p, auto KIND_, auto) {
            constexpr int KIND = decltype(KIND_)::value;
            const int n = min(F_TILE, p.N - t.n0);  // columns behind the output's are not computed
            const uint32_t idesc = make_idesc(KIND == WGRAD ? 1 : 0, KIND == ROW_BK ? 0 : 1, n);
            constexpr uint64_t a_step = KIND == WGRAD ? (16 * 128) >> 4 : 32 >> 4, b_step = KIND == ROW_BK ? 32 >> 4 : (16 * 128) >> 4;
            ok = mbar_wait(sempty_bar(small), small_ph ^ 1u, abort_flag, L.row.status);
            if (!ok) return;
            const uint32_t d_small = tmem_base + 256 + small * F_TILE;
            for (int kb = 0; kb < t.blocks; ++kb) {
                const bool begins = kb % F_SUB == 0;
                if (begins) {
                    ok = mbar_wait(tempty_bar(acc), acc_ph ^ 1u, abort_flag, L.row.status);
                    if (!ok) break;
                }
                ok = mbar_wait(full_bar(s), ph, abort_flag, L.row.status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_main = tmem_base + acc * F_TILE;
                int ksteps = BK / 16;
                if (KIND == WGRAD && kb == t.blocks - 1) {
                    // rows behind the segment's end, up to the end of the step that holds it, are the next segment's: zeroed in all terms
                    const int valid = t.row_end - (t.row0 + kb * BK);
                    ksteps = (valid + 15) / 16;
                    if (ksteps * 16 > valid) {
                        uint8_t *z = smem + s * F_STAGE + (valid + (lane >> 3)) * 128 + (lane & 7) * 16;
                        for (int r = lane >> 3; r < ksteps * 16 - valid; r += 4, z += 4 * 128)
#pragma unroll
                            for (int chunk = 0; chunk < F_STAGE / (BK * 128); ++chunk)
                                *reinterpret_cast<uint4 *>(z + chunk * (BK * 128)) = make_uint4(0, 0, 0, 0);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                    }
                }
                if (lane == 0) {
                    uint64_t ad[3], bd[3];
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const uint32_t a = base + s * F_STAGE + q * F_OPERAND, b = a + 3 * F_OPERAND;
                        ad[q] = KIND == WGRAD ? desc_mnmajor(a) : desc_kmajor(a);
                        bd[q] = KIND == ROW_BK ? desc_kmajor(b) : desc_mnmajor(b);
                    }
                    constexpr int at[5] = {2, 0, 1, 0, 1}, bt[5] = {0, 2, 1, 1, 0};  // the small products, smallest first
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        if (k >= ksteps) break;
#pragma unroll
                        for (int q = 0; q < 5; ++q)
                            tc_mma_bf16(d_small, ad[at[q]] + k * a_step, bd[bt[q]] + k * b_step, idesc, (kb > 0 || k > 0 || q > 0) ? 1u : 0u);
                        tc_mma_bf16(d_main, ad[0] + k * a_step, bd[0] + k * b_step, idesc, (!begins || k > 0) ? 1u : 0u);
                    }
                    tc_commit(empty_bar(s));
                }
                __syncwarp();
                if (++s == F_STAGES) { s = 0; ph ^= 1u; }
                if (kb % F_SUB == F_SUB - 1 || kb == t.blocks - 1) {
                    if (lane == 0) {
                        tc_commit(tfull_bar(acc));
                        if (kb == t.blocks - 1) tc_commit(sfull_bar(small));
                    }
                    __syncwarp();
                    if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
                }
            }
            if (++small == 2) { small = 0; small_ph ^= 1u; }
            });
        }
    } else {
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        uint8_t *slab = smem + F_STAGES * F_STAGE + (warp - 2) * 4096;
        int acc = 0, small = 0;
        uint32_t acc_ph = 0, small_ph = 0;
        bool ok = true;
        for (int32_t id = blockIdx.x; ok && float_tile(L, id, t); id += gridDim.x) {
            float sums[2][32];  // a lane's row of the warp's 64 columns
#pragma unroll
            for (int i = 0; i < 64; ++i) sums[i >> 5][i & 31] = 0.0f;
            auto add = [&](uint32_t column, uint32_t empty) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    uint32_t v[32];
                    tc_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + column + half * 64 + 32 * u, v);
                    tc_ld_wait();
                    if (u == 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(empty);
                    }
#pragma unroll
                    for (int j = 0; j < 32; ++j) sums[u][j] += __uint_as_float(v[j]);
                }
            };
            for (int kb = 0; kb < t.blocks && ok; kb += F_SUB) {
                ok = mbar_wait(tfull_bar(acc), acc_ph, abort_flag, L.row.status);
                if (!ok) break;
                tc_fence_after();
                add(acc * F_TILE, tempty_bar(acc));
                if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
            }
            if (!ok) break;
            if (t.blocks > 0) {
                ok = mbar_wait(sfull_bar(small), small_ph, abort_flag, L.row.status);
                if (!ok) break;
                tc_fence_after();
                add(256 + small * F_TILE, sempty_bar(small));
                if (++small == 2) { small = 0; small_ph ^= 1u; }
            }
#pragma unroll
            for (int i = 0; i < 64; ++i) sums[i >> 5][i & 31] *= F_UNSCALE;
            with_product(L, t, [&](const FloatProduct &p, auto KIND_, auto EPI_) {
            constexpr int KIND = decltype(KIND_)::value, EPI = decltype(EPI_)::value;
            const int64_t row0 = (KIND == WGRAD ? t.m0 : t.row0) + quarter * 32, out0 = KIND == WGRAD ? (int64_t)t.e * p.M : 0;
            const int rows_valid = (int)((KIND == WGRAD ? p.M : t.row_end) - row0);
            const int32_t col0 = t.n0 + half * 64;
            if (col0 >= p.N) return;  // N is a multiple of 64
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int32_t col = col0 + 32 * u;
                if (EPI == FE_BIAS) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 b = reinterpret_cast<const float4 *>(p.bias + (int64_t)t.e * p.N + col)[q];
                        sums[u][4 * q] += b.x; sums[u][4 * q + 1] += b.y; sums[u][4 * q + 2] += b.z; sums[u][4 * q + 3] += b.w;
                    }
                }
                if (EPI == FE_MASK && lane < rows_valid) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 m = reinterpret_cast<const float4 *>(p.mask + (row0 + lane) * p.N + col)[q];
                        if (!(m.x > 0.0f)) sums[u][4 * q] = 0.0f;
                        if (!(m.y > 0.0f)) sums[u][4 * q + 1] = 0.0f;
                        if (!(m.z > 0.0f)) sums[u][4 * q + 2] = 0.0f;
                        if (!(m.w > 0.0f)) sums[u][4 * q + 3] = 0.0f;
                    }
                }
                float odd = 0.0f;  // x - x is 0, or NaN where x is not finite
#pragma unroll
                for (int j = 0; j < 32; ++j) odd += sums[u][j] - sums[u][j];
                if (odd != 0.0f && lane < rows_valid) *odd_tiles = 1;
                // through the warp's slab: lane l moves piece l % 8 of row 4 * i + l / 8
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    *reinterpret_cast<float4 *>(slab + lane * 128 + ((q ^ (lane & 7)) << 4)) =
                        make_float4(sums[u][4 * q], sums[u][4 * q + 1], sums[u][4 * q + 2], sums[u][4 * q + 3]);
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int row = 4 * i + (lane >> 3);
                    if (row >= rows_valid) continue;
                    const float4 v = *reinterpret_cast<const float4 *>(slab + row * 128 + (((lane & 7) ^ (row & 7)) << 4));
                    const int64_t r = out0 + row0 + row;
                    const int32_t c = col + (lane & 7) * 4;
                    *reinterpret_cast<float4 *>(p.out + r * p.N + c) = v;
                    if (EPI == FE_MASK && p.terms) store_terms(v, p.terms + r * 3 * p.N + c, p.N);
                }
                __syncwarp();
            }
            });
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
    }
    if (*odd_tiles && !*abort_flag) repair_tiles(L);
}

// The three terms of several tensors [rows, cols] in one launch, to [rows][3 cols]: four neighbours a thread, four times
struct TermsJob { const float *from; bf16 *to; int64_t quads; Divisor by_quads; int32_t block0; };
struct TermsJobs { TermsJob job[5]; int32_t count; };
constexpr int TERMS_QUADS = 4 * 256;
__global__ void __launch_bounds__(256) split_terms_kernel(const __grid_constant__ TermsJobs jobs) {
    wait_previous_kernel();
    int which = 0;
    while (which + 1 < jobs.count && (int32_t)blockIdx.x >= jobs.job[which + 1].block0) ++which;
    const TermsJob &j = jobs.job[which];
    const int64_t first = (int64_t)((int32_t)blockIdx.x - j.block0) * TERMS_QUADS + threadIdx.x;
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (first + 256 * u < j.quads) v[u] = reinterpret_cast<const float4 *>(j.from)[first + 256 * u];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t q = first + 256 * u;
        if (q >= j.quads) break;
        int32_t col;
        const int64_t row = j.by_quads((int32_t)q, col);
        store_terms(v[u], j.to + row * 12 * (int64_t)j.by_quads.d + 4 * col, 4 * (int64_t)j.by_quads.d);
    }
}

class TermsList {
    TermsJobs jobs;
    int32_t blocks = 0;

  public:
    TermsList() { memset(&jobs, 0, sizeof(jobs)); }
    void add(const void *from, void *to, int64_t rows, int64_t cols) {
        TermsJob &j = jobs.job[jobs.count++];
        j.from = (const float *)from; j.to = (bf16 *)to; j.quads = rows * cols / 4; j.by_quads = Divisor::of(cols / 4); j.block0 = blocks;
        blocks += (int32_t)cdiv(j.quads, TERMS_QUADS);
    }
    int32_t launch(cudaStream_t st) {
        launch_kernel(split_terms_kernel, (unsigned)blocks, 256, 0, st, jobs);
        MOE_LAUNCHED();
        return MOE_OK;
    }
};

struct FloatCall {
    const moe_config &c;
    const SegmentPlan &plan;
    const int32_t *offsets;
    int32_t *status;
    cudaStream_t st;
    int64_t R;
    FloatProduct product(const void *A, const void *B, int32_t N, void *out) const {
        FloatProduct p;
        memset(&p, 0, sizeof(p));
        p.offsets = offsets; p.row_tiles = plan.by_rank + c.n; p.info = plan.info; p.N = N;
        p.tiles_n = (int32_t)cdiv(N, F_TILE); p.by_tiles_n = Divisor::of(p.tiles_n);
        p.out = (float *)out; p.A = (const float *)A; p.B = (const float *)B; p.status = status;
        return p;
    }
    // out [R, N] = epilogue(A [R, K] . W[e]) from the terms a [R, 3 K] and w [n][.][3 .]
    template <int ROW, int EPI, bool W>
    int32_t row(FloatLaunch<ROW, EPI, W> *L, const void *A, const void *a, const void *B, const void *b, int32_t N, int32_t K, void *out, const void *bias,
                const void *mask, void *terms) const {
        FloatProduct &p = L->row = product(A, B, N, out);
        p.K = K; p.bias = (const float *)bias; p.mask = (const float *)mask; p.terms = (bf16 *)terms;
        const int64_t tiles = (cdiv(R, F_TILE) + c.n) * p.tiles_n;
        if (tiles >= (int64_t)1 << 30) return MOE_ERR_UNSUPPORTED;
        p.total = (int32_t)tiles;
        MOE_TRY(tc_map_rows_kmajor(&L->row_a, a, R, 3 * (int64_t)K, F_TILE));
        if (ROW == ROW_BMN) return tc_map_weight_mnmajor(&L->row_b, b, c.n, K, 3 * (int64_t)N, F_TILE);
        return tc_map_weight_kmajor(&L->row_b, b, c.n, N, 3 * (int64_t)K, F_TILE);
    }
    // out[e] [M, N] = A_e^T . B_e from the terms a [R, 3 M], b [R, 3 N]
    template <typename Launch> int32_t wgrad(Launch *L, const void *A, const void *a, const void *B, const void *b, int32_t M, int32_t N, void *out) const {
        FloatProduct &p = L->wgrad = product(A, B, N, out);
        p.M = M;
        p.per_e = (int32_t)cdiv(M, F_TILE) * p.tiles_n; p.by_per_e = Divisor::of(p.per_e);
        const int64_t tiles = (int64_t)c.n * p.per_e;
        if (tiles >= (int64_t)1 << 30) return MOE_ERR_UNSUPPORTED;
        p.total = (int32_t)tiles;
        MOE_TRY(tc_map_rows_mnmajor(&L->wgrad_a, a, R, 3 * (int64_t)M, 2));
        return tc_map_rows_mnmajor(&L->wgrad_b, b, R, 3 * (int64_t)N, 2);
    }
    template <int ROW, int EPI, bool W> int32_t launch(const FloatLaunch<ROW, EPI, W> &L) const {
        static PerDevice configured;
        if (!allow_shared(configured, float_products_kernel<ROW, EPI, W>, F_SHARED)) return MOE_ERR_CUDA;
        const int64_t tiles = (int64_t)L.row.total + (W ? L.wgrad.total : 0);
        launch_kernel((float_products_kernel<ROW, EPI, W>), (unsigned)imin(tiles, tc_sm_count()), NTHREADS, F_SHARED, st, L);
        MOE_LAUNCHED();
        return MOE_OK;
    }
};

}  // namespace

// A call has to make the terms (4 bytes of a float read, 6 written). Where they pay, us, by FP32 multiply-adds (few_rows.cu among them) and this way:
// A forward call, one product: from 65 rows an expert, 1e8 multiply-adds and 16 tiles on. 256 experts x 64 rows of 256 x 512 216, 225, x 72 329, 284;
// 32 x 40 of 256 x 512 47.1, 51.9; 16 x 50 34.3, 37.7, x 100 56.6, 48.9; 64 x 72 of 512 x 512 195, 157; 120 x 60 of 960 x 1728 1134, 1168, x 70 1674, 1420;
// 8 x 1500 of 64 x 128 (9.8e7) 25.6, 23.8; 2 x 136 of 192 x 3072, 8 tiles, 82.7, 86.3; 6 x 144 of 64 x 2496, 10 tiles, 68.3, 72.6; 2 x 500 of 256 x 512, 18, 34.4, 33.6.
// A backward call, four products: from 33 rows and 4e6 on. 64 x 32 of 256 x 512 105, 95, x 40 146, 100; 300 x 30 434, 390, x 40 497, 417; 8 x 30 of 512 x 4096 182,
// 222, x 40 294, 216; 200 x 30 of 64 x 128 40.9, 45.9; 72 x 31 27.3, 29.3, x 40 39.7, 29.9; 400 x 40 of 64 x 64 57.5, 63.6. Small ones, by multiply-adds in
// 1e6: 2.1 (4 x 64 of 64 x 128) 25.9, 26.9; 4.2 (16 x 64 of 64 x 64, 8 x 128 of 64 x 64) 25.8, 25.3 and 28.5, 27.5; 4.7 (8 x 36 of 64 x 256) 26.0, 28.8;
// 6.3 (16 x 48 of 64 x 128) 30.3, 27.7; 8.4 (8 x 64 of 128 x 128) 27.9, 28.5, (16 x 64 of 64 x 128) 30.2, 27.6. A few tiles that are chains of many rows are the
// exception: 1 x 20000 of 128 x 128 673, 820; 2 x 5000 205, 222; 4 x 5000 of 64 x 64 193, 228; 1 x 981 55.9, 60.9; 27 experts, 34799 rows, the longest segment
// 12894, of 64 x 64 444, 547; but 1 x 512 40.4, 38.9; equal loads of 19 x 2000 of 64 x 64 144, 131; 1 x 3000 of 512 x 128 160, 143.
// The terms take 6 bytes of workspace a float: as much again as all other buffers of a backward call. At most 8 GiB of them, a twentieth of the memory, and 1 GiB
// for callers that recompute hid to save memory. Larger layers keep the FP32 products, which take three and a half times as long (a backward call, ms: 8 experts x
// 20000 rows of 1024 x 2048, 5.9 GB, by terms 15.1, by multiply-adds 53.3; 16 x 10000 of 1024 x 1024, 4.1 GB, 8.0 and 26.9).
bool tc_float_supported(const moe_config &c, bool backward) {
    const int64_t R = (int64_t)c.T * c.k, weights = (int64_t)c.n * c.d * c.h, most = c.flags & MOE_FLAG_RECOMPUTE_HID ? (int64_t)1 << 30 : (int64_t)8 << 30;
    if (c.act != MOE_F32 || c.d % 64 != 0 || c.h % 64 != 0) return false;
    if (6 * (backward ? 2 * (R * ((int64_t)c.d + c.h) + weights) : R * c.h + weights) > most) return false;  // (quads are numbered with 31 bits: far below)
    const double work = (double)R * c.d * c.h;
    if (!backward) return R > 64 * (int64_t)c.n && work >= 1.0e8 && (cdiv(R, F_TILE) + c.n / 2) * cdiv(c.d, F_TILE) >= 16;
    if (weights < 32 * 64 * 64 && R >= 700 * (int64_t)c.n) return false;
    return R > 32 * (int64_t)c.n && work >= 4.0e6;
}

int32_t launch_float_ys(const moe_config &c, const int32_t *offsets, const void *hid, const void *W2, const void *b2, void *ys, const SegmentPlan &plan,
                        const FloatTerms &t, int32_t *status, cudaStream_t st) {
    const FloatCall call = {c, plan, offsets, status, st, (int64_t)c.T * c.k};
    TermsList list;
    list.add(hid, t.hid, call.R, c.h);
    list.add(W2, t.W2, (int64_t)c.n * c.h, c.d);
    MOE_TRY(list.launch(st));
    FloatLaunch<ROW_BMN, FE_BIAS, false> L;
    MOE_TRY(call.row(&L, hid, t.hid, W2, t.W2, c.d, c.h, ys, b2, nullptr, nullptr));
    return call.launch(L);
}

int32_t launch_float_ffn_bwd(const moe_config &c, const void *xs, const void *hid, const void *dys, const int32_t *offsets, const void *W1,
                             const void *W2, void *dxs, void *dW1, void *dW2, void *dz, const SegmentPlan &plan, const FloatTerms &t,
                             int32_t *status, cudaStream_t st) {
    const FloatCall call = {c, plan, offsets, status, st, (int64_t)c.T * c.k};
    TermsList list;
    list.add(xs, t.xs, call.R, c.d);
    list.add(dys, t.dys, call.R, c.d);
    list.add(hid, t.hid, call.R, c.h);
    list.add(W1, t.W1, (int64_t)c.n * c.d, c.h);
    list.add(W2, t.W2, (int64_t)c.n * c.h, c.d);
    MOE_TRY(list.launch(st));
    FloatLaunch<ROW_BK, FE_MASK, true> by_w2;
    MOE_TRY(call.wgrad(&by_w2, hid, t.hid, dys, t.dys, c.h, c.d, dW2));
    MOE_TRY(call.row(&by_w2, dys, t.dys, W2, t.W2, c.h, c.d, dz, nullptr, hid, t.dz));
    MOE_TRY(call.launch(by_w2));
    FloatLaunch<ROW_BK, FE_PLAIN, true> by_w1;
    MOE_TRY(call.wgrad(&by_w1, xs, t.xs, dz, t.dz, c.d, c.h, dW1));
    MOE_TRY(call.row(&by_w1, dz, t.dz, W1, t.W1, c.d, c.h, dxs, nullptr, nullptr, nullptr));
    const int64_t xs_bytes = call.R * c.d * (int64_t)sizeof(float);
    if (overlap(xs, xs_bytes, dxs, xs_bytes)) {  // the caller has no use for xs any more: dxs waits until dW1 has read it (elements that are not finite do)
        const int32_t rows = by_w1.row.total;
        by_w1.row.total = 0;
        MOE_TRY(call.launch(by_w1));
        by_w1.row.total = rows;
        by_w1.wgrad.total = 0;
    }
    return call.launch(by_w1);
}

}  // namespace moe
