// Expert feed-forward networks on the 5th-generation tensor cores (Section 3.2, Appendix C):
// variable-size grouped GEMMs, bf16 operands, fp32 accumulation in tensor memory.
//
// One persistent kernel template, one CTA per SM, 128 x 256 output tiles, K blocks of 64:
//   warp 0      TMA producer: one bulk tensor copy per operand per stage into 128-byte-swizzled
//               shared memory, completion counted on an mbarrier (4 stages)
//   warp 1      MMA issuer: tcgen05.mma (cta_group::1, kind::f16, M 128, N 256, K 16), accumulator
//               in TMEM, double buffered (2 x 256 columns) so the epilogue of one tile overlaps
//               the main loop of the next; tcgen05.commit releases the stage / publishes the tile
//   warps 2-9   epilogue: tcgen05.ld (32 lanes x 32 columns per instruction), bias / ReLU / ReLU
//               mask, round to bf16; whole [32][64] boxes leave as bulk tensor stores, boxes cut by a
//               segment end as guarded row stores
//
// Three operand arrangements (KIND):
//   ROW_BMN  rows x K activations (K-major A) times a per-expert [K, N] weight (N contiguous,
//            "MN-major" B): forward GEMMs  hid = relu(xs.W1 + b1),  ys = hid.W2 + b2
//   ROW_BK   same A, per-expert weight read transposed ([N, K], K contiguous, K-major B):
//            dz = (dys.W2^T) * [hid > 0],  dxs = dz.W1^T
//   WGRAD    contraction over the rows of a segment, both operands MN-major:
//            dW2 = hid^T.dys,  dW1 = xs^T.dz.
// The last rows of a segment are loaded through a tensor map that ends with the segment: what lies behind them (the next
// segment's rows) reads as zero, in both operands of a weight gradient (short segments: see tc_wgrad_gemm). Zeros also cost the
// tensor cores less power than the next segment's rows, which bounds the large products.
// Weights are addressed through one tensor map with the expert as a coordinate, segment bounds
// are read on the device: no per-expert descriptors and no host synchronisation.
//
// Every wait on an mbarrier is bounded (2 s of %globaltimer); on expiry the CTA records
// MOE_ERR_TIMEOUT in the workspace status word, stops issuing work, drains and frees its TMEM.
#include <cuda.h>
#include <stdlib.h>
#include <string.h>

#include <type_traits>

#include "sums.cuh"

namespace moe {

namespace {

constexpr int BM = 128, BN = 256, BK = 64, STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;  // 16 KiB
constexpr int B_BYTES = BN * BK * 2;  // 32 KiB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int EPI_STAGE_BYTES = 8 * 4096;  // per epilogue warp: a 32 x 128 B slab for float output
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*alignment slack*/ + 1024 /*barriers; the boxes behind them are 1024-byte aligned*/ + EPI_STAGE_BYTES;
constexpr int TMEM_COLS = 512;
constexpr int NTHREADS = 320;   // TMA warp, MMA warp, 8 epilogue warps
constexpr int NTHREADS2 = 352;  // two-CTA kernel: + the tile scheduler warp
constexpr unsigned long long WAIT_LIMIT_NS = 2000000000ull;

enum Kind { ROW_BMN = 0, ROW_BK = 1, WGRAD = 2 };
// What the epilogue does with an accumulator, fixed at compile time (a run-time choice kept every variant's registers and
// code in one kernel: 950 cycles for the 32 conversions of a box without any option)
enum Epilogue { EPI_PLAIN = 0, EPI_BIAS = 1, EPI_RELU = 2, EPI_MASK = 4, EPI_BITS = 8, EPI_F32 = 16, EPI_TWO_BOXES = 32 };

constexpr int MAX_TERMS = 8;

// Division by a launch's constant as a multiplication (Granlund and Montgomery, 1994): q = (high word of x * m + x) >> s for
// 0 <= x < 2^31. A tile's place is three divisions, which every warp role makes between two tiles: as integer divisions they and the
// look-up behind them were 700 of a 3700-cycle tile of 64 rows.
struct Divisor {
    uint32_t d, m, s;
    static Divisor of(int64_t by) {
        Divisor v = {(uint32_t)(by > 0 ? by : 1), 0, 0};
        while ((1ull << v.s) < v.d) ++v.s;
        v.m = (uint32_t)((((1ull << v.s) - v.d) << 32) / v.d + 1);
        return v;
    }
    __device__ __forceinline__ int32_t operator()(int32_t x, int32_t &rest) const {
        const int32_t q = (int32_t)((__umulhi((uint32_t)x, m) + (uint32_t)x) >> s);
        rest = x - q * (int32_t)d;
        return q;
    }
};
struct GemmParams {
    const int32_t *offsets;      // [nseg + 1] segment bounds (rows); nullptr = uniform segments
    const int32_t *tile_prefix;  // ROW_* with offsets: [nseg + 1] prefix of the M tiles
    const int4 *tile_info;       // ROW_* with offsets: per M tile {segment or -1, first row, segment end, 0}
    // set by the launchers: N tiles per row of tiles, WGRAD tiles per segment, number of tile ids, K blocks of a ROW tile
    int32_t tiles_n, per_e, total_tiles, kblocks_row;
    Divisor by_tiles_n, by_per_e, by_mod, by_terms, by_interleave, by_group;  // tiles_n, per_e, off_mod, segs_per_term, interleave, sched_group
    int32_t tile_n;  // columns of a tile: BN, or 128 in row products of the one-CTA kernel (see tc_row_gemm)
    int32_t nseg;
    int32_t M;  // WGRAD: rows of the per-segment output; ROW_*: unused
    int32_t N;  // output columns
    int32_t K;  // ROW_*: contraction length of one term; WGRAD: unused (segment rows)
    bf16 *out;  // ROW_*: [R, N]; WGRAD: [nseg, M, N]
    float *out_f32;    // if set, results are written here as float instead of `out`
    // float results of two matrices side by side: columns from split_n on go to out2, both with rows of split_n (a multiple of 32);
    // out_rows: where an output row goes (rows sorted by group); out_words: rows that do not start on 16 bytes
    float *out2;
    const int32_t *out_rows;
    int32_t split_n, out_words;
    const bf16 *bias;  // [nseg, N] or nullptr
    const bf16 *mask;  // [R, N] or nullptr: result kept where mask > 0
    // the same mask as one bit per element, [R, N / 32] words (bit j of word c: column 32 c + j): bits_out is written by
    // the GEMM whose output the mask is taken of (bit = stored value > 0), bits_in is applied like `mask`
    uint32_t *bits_out;
    const uint32_t *bits_in;
    // ROW_* with bf16 output: if set, column sums of the stored values over each epilogue warp's 32 rows,
    // [32-row block][N] floats; block = (global M tile * CTAs per tile + CTA rank) * 4 + row quarter
    float *colsum_part;
    int32_t tma_out;  // two-CTA ROW_*: full 32-row pieces leave through shared memory and bulk tensor stores
    int32_t relu;
    int32_t *status;
    // uniform segments (offsets == nullptr): ROW_*: one segment of R rows. WGRAD: segment s covers
    // rows [c * rows_per_seg, min(R, (c+1) * rows_per_seg)) with c = s % segs_per_term, and reads the
    // B columns shifted by (s / segs_per_term) * b_term_chunks chunks of 64 (split-precision terms).
    int64_t R;
    int32_t rows_per_seg, segs_per_term, b_term_chunks;
    int32_t segs_term0, rows_per_seg0;  // if segs_term0 > 0: term 0 is cut into that many ranges of rows_per_seg0
    int32_t interleave;                 // uniform WGRAD: number of terms whose tiles alternate in the id order (0: none)
    int32_t sub_kb0, sub_kb;            // ACC kernel: K blocks per separately accumulated sub-block, term 0 / other terms
    int32_t off_mod;                    // WGRAD with offsets: see tile_fetch
    // one map per segment that ends with the segment: for the box of A (WGRAD: of A and of B) that reaches beyond it. Row
    // products may do without (their rows behind the end are computed and dropped)
    const CUtensorMap *seg_a, *seg_b;
    // ROW_*: the contraction is the concatenation of nterms pieces of length K; piece i reads A
    // columns a_term_col[i] + [0, K) and B columns b_term_col[i] + [0, K)
    int32_t nterms;
    int32_t a_term_col[MAX_TERMS], b_term_col[MAX_TERMS];
    // two-CTA kernels over ragged segments: tiles are handed out at run time (see PairTiles). sched_counter = next tile
    // id; sched_table[id / sched_group] = {segment, first row, end row, 0} (segment -1: no more tiles). WGRAD: the
    // segments in descending size, sched_group = tiles per segment; ROW_*: tile_info, sched_group = N tiles per M tile
    const int4 *sched_table;
    int32_t *sched_counter;
    int32_t sched_group;
    int32_t trace;  // diagnostics build only: this launch records the tile trace
};

// Diagnostics build (-DMOE_TILE_TRACE): the first CTA records, per tile, when each warp role started, finished and how
// long it waited; read back with moe_debug_tile_trace. Compiled out otherwise.
#ifdef MOE_TILE_TRACE
__device__ long long g_tile_trace[3][256][6];
#define TILE_TRACE_SET(role, tile, field, val) do { if (p.trace && blockIdx.x == 0 && (tile) < 256) g_tile_trace[role][tile][field] = (val); } while (0)

#define TILE_CLOCK() clock64()
static int g_trace_launch_no = 0;
#else
#define TILE_TRACE_SET(role, tile, field, val) do {} while (0)
#define TILE_CLOCK() 0ll
#endif

// ------------------------------------------------------------------------------------------ PTX
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// same, with cluster-scope acquire (the arrival comes from the other CTA of the pair)
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait. Returns false (and raises the CTA's abort flag + the status word) on expiry.
__device__ __forceinline__ bool mbar_wait_limit(uint32_t bar, uint32_t parity, volatile int *abort_flag, int32_t *status,
                                                unsigned long long limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (global_ns() - t0 > limit_ns) {
            *abort_flag = 1;
            atomicExch(status, (int32_t)MOE_ERR_TIMEOUT);
            return false;
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int32_t *status) {
    return mbar_wait_limit(bar, parity, abort_flag, status, WAIT_LIMIT_NS);
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1,
                                            int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1,
                                            int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

// bulk tensor store of a [32 rows][64 columns] box from 128-byte-swizzled shared memory
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *tm, uint32_t src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(tm), "r"(src), "r"(c0),
                 "r"(c1)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read_but_one() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// A map in global memory that an earlier kernel has written: made visible to the copies of this thread, and fetched ahead
__device__ __forceinline__ void acquire_map(const CUtensorMap *tm) {
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(tm) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
}

// 256-bit store (sm_100): a whole 32-byte sector per instruction
__device__ __forceinline__ void st_global_32B(uint4 *dst, const uint4 &a, const uint4 &b) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(a.x), "r"(a.y), "r"(a.z),
                 "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_ld_32x32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tc_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptors (128-byte swizzle, descriptor version 1 at bit 46).
// K-major: rows of 64 bf16 (128 B); 8-row groups 1024 B apart (stride byte offset).
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// MN-major: 64 contiguous MN elements (128 B) per K row; 8 K rows per 1024-B atom (stride byte
// offset); the next 64 MN elements start BK * 128 B further (leading byte offset).
__device__ __forceinline__ uint64_t desc_mnmajor(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)((BK * 128) >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Instruction descriptor: D fp32, A/B bf16, majors, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t make_idesc(int a_mn, int b_mn, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

// Column sums over the 32 rows a warp holds (one row per lane, 32 columns per lane): returns in lane l
// the sum of column l. Butterfly: each step a lane keeps one half of its columns and sends the other.
__device__ __forceinline__ float warp_column_sums(float (&a)[32], int lane) {
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int i = 0; i < s; ++i) {
            const float keep = up ? a[i + s] : a[i];
            const float send = up ? a[i] : a[i + s];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
    return a[0];
}

// Epilogue arithmetic of one thread's 32 accumulator columns: bias, ReLU, ReLU mask, rounding to bf16. The three
// options are template parameters so that the loop body has no branches (with run-time flags every element pair became
// its own basic block and the chain add -> max -> convert ran serially, 16 times).
template <int EPI>
__device__ __forceinline__ void pack32(const uint32_t (&v)[32], const uint4 (&bias_raw)[4], const uint4 (&mask_raw)[4],
                                            uint4 (&packed)[4], uint32_t keep_word) {
    constexpr bool BIAS = EPI & EPI_BIAS, RELU = EPI & EPI_RELU, MASK = EPI & EPI_MASK, BITS = EPI & EPI_BITS;
    const uint32_t *bw = reinterpret_cast<const uint32_t *>(bias_raw);
    const uint32_t *mw = reinterpret_cast<const uint32_t *>(mask_raw);
    uint32_t *out = reinterpret_cast<uint32_t *>(packed);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        float x0 = __uint_as_float(v[2 * j]), x1 = __uint_as_float(v[2 * j + 1]);
        if (BIAS) { x0 += __uint_as_float(bw[j] << 16); x1 += __uint_as_float(bw[j] & 0xffff0000u); }
        if (MASK) {
            if (!(__uint_as_float(mw[j] << 16) > 0.0f)) x0 = 0.0f;
            if (!(__uint_as_float(mw[j] & 0xffff0000u) > 0.0f)) x1 = 0.0f;
        }
        if (BITS) {
            if (!((keep_word >> (2 * j)) & 1u)) x0 = 0.0f;
            if (!((keep_word >> (2 * j + 1)) & 1u)) x1 = 0.0f;
        }
        __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
        if (RELU) h = __hmax2(h, __float2bfloat162_rn(0.0f));  // rounding keeps the sign: the same value as max before rounding
        out[j] = *reinterpret_cast<const uint32_t *>(&h);
    }
}
// one bit per packed value: set where the stored bf16 value is greater than zero. The pairs' comparison masks are collected
// as bit j (element 2j) and bit 16 + j (element 2j + 1), two instructions a pair, and interleaved once at the end.
__device__ __forceinline__ uint32_t spread_bits(uint32_t x) {  // bit i of the low half -> bit 2 i
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}
__device__ __forceinline__ uint32_t positive_bits(const uint4 (&packed)[4]) {
    const __nv_bfloat162 *pw = reinterpret_cast<const __nv_bfloat162 *>(packed);
    const __nv_bfloat162 zero = __float2bfloat162_rn(0.0f);
    uint32_t even = 0u, odd = 0u;  // two chains
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
        even |= __hgt2_mask(pw[j], zero) & (0x00010001u << j);
        odd |= __hgt2_mask(pw[j + 1], zero) & (0x00010001u << (j + 1));
    }
    const uint32_t all = even | odd;
    return spread_bits(all & 0xffffu) | (spread_bits(all >> 16) << 1);
}
// The bias values of a 64-column box, the same for every lane (broadcast loads). They are fetched one box ahead: the
// first box's before the warp waits for its accumulator.
__device__ __forceinline__ void bias_load(const bf16 *bias, uint4 (&out)[2][4]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) out[q >> 2][q & 3] = reinterpret_cast<const uint4 *>(bias)[q];
}

// One [32 rows][64 columns] box of an output tile, by one warp (a lane owns a row): tensor memory -> bias / ReLU / mask ->
// bf16 -> global memory. With eight epilogue warps an SM sub-partition has two to hide the latencies of this chain, so a
// box is taken whole: both 32-column loads are in flight together and everything behind them has twice the independent
// work (with 32-column steps the epilogue of a 256 x 256 tile took 8500 cycles, against 4900 of tensor work at K = 512).
// Whole boxes leave as bulk tensor stores through the warp's 4 KiB of shared memory (rows of 128 bytes, 16-byte pieces
// swizzled by row); boxes cut by a segment end as guarded row stores. MASKT: the box holds the mask values on entry.
// release() hands the accumulator back; it is called once the box is in registers.
struct BoxArgs {
    const CUtensorMap *tm_out;
    uint8_t *box;
    uint32_t taddr;             // tensor-memory address of the box
    int64_t out_off, row0;      // output row of lane 0 is row0 of the matrix that starts at element out_off
    int32_t rows_valid, col0;
    int32_t map_row;            // the same row in the output's tensor map
    int64_t colsum_row;
    const bf16 *next_bias;      // of the warp's next box, or nullptr
    uint2 keep;                 // mask bits
    bool have_acc;
};
template <int EPI, bool MASKT, typename Release>
__device__ __forceinline__ void epilogue_box(const GemmParams &p, int lane, const BoxArgs &b, uint4 (&bias)[2][4],
                                             Release release) {
    uint32_t v[2][32];
    if (b.have_acc) {
        tc_ld_32x32(b.taddr, v[0]);
        tc_ld_32x32(b.taddr + 32, v[1]);
        tc_ld_wait();
        release();
    } else {
#pragma unroll
        for (int j = 0; j < 64; ++j) v[j >> 5][j & 31] = 0u;
    }
    if constexpr (EPI & EPI_F32) {  // 128-byte row segments: lane l moves piece l % 8 of row 4 * i + l / 8
        const int my_piece = lane & 7, my_sub = lane >> 3;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                *reinterpret_cast<uint4 *>(b.box + lane * 128 + ((q ^ (lane & 7)) << 4)) =
                    make_uint4(v[u][4 * q], v[u][4 * q + 1], v[u][4 * q + 2], v[u][4 * q + 3]);
            __syncwarp();
            const int32_t col = b.col0 + 32 * u;
            float *dst = p.out_f32 + b.out_off + col + my_piece * 4;
            int64_t pitch = p.N;
            if (p.out2) {
                dst = (col < p.split_n ? p.out_f32 + col : p.out2 + (col - p.split_n)) + my_piece * 4;
                pitch = p.split_n;
            }
            auto piece = [&](int row) { return *reinterpret_cast<const uint4 *>(b.box + row * 128 + ((my_piece ^ (row & 7)) << 4)); };
            if (!p.out_rows && !p.out_words) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int row = 4 * i + my_sub;
                    if (row < b.rows_valid) *reinterpret_cast<uint4 *>(dst + (b.row0 + row) * pitch) = piece(row);
                }
            } else {
                int32_t to[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int64_t row = b.row0 + 4 * i + my_sub;
                    to[i] = 4 * i + my_sub >= b.rows_valid ? -1 : p.out_rows ? p.out_rows[row] : (int32_t)row;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (to[i] < 0) continue;
                    const uint4 v = piece(4 * i + my_sub);
                    float *at = dst + (int64_t)to[i] * pitch;
                    if (!p.out_words) {
                        *reinterpret_cast<uint4 *>(at) = v;
                    } else {
                        at[0] = __uint_as_float(v.x); at[1] = __uint_as_float(v.y);
                        at[2] = __uint_as_float(v.z); at[3] = __uint_as_float(v.w);
                    }
                }
            }
            __syncwarp();
        }
        return;
    } else {
    const bool row_ok = lane < b.rows_valid, staged = p.tma_out && b.rows_valid >= 32;
    const int64_t out_row = b.row0 + lane;
    uint8_t *mine = b.box + lane * 128;
    uint4 packed[2][4];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        uint4 mask_raw[4];
        if (MASKT) {
#pragma unroll
            for (int q = 0; q < 4; ++q) mask_raw[q] = *reinterpret_cast<const uint4 *>(mine + (((u * 4 + q) ^ (lane & 7)) << 4));
        } else if ((EPI & EPI_MASK) && row_ok) {
#pragma unroll
            for (int q = 0; q < 4; ++q) mask_raw[q] = reinterpret_cast<const uint4 *>(p.mask + out_row * p.N + b.col0 + 32 * u)[q];
        }
        pack32<EPI>(v[u], bias[u], mask_raw, packed[u], u ? b.keep.y : b.keep.x);
    }
    if ((EPI & EPI_BIAS) && b.next_bias) bias_load(b.next_bias, bias);
    if ((EPI & EPI_RELU) && p.bits_out && row_ok)
        *reinterpret_cast<uint2 *>(p.bits_out + out_row * (p.N >> 5) + (b.col0 >> 5)) =
            make_uint2(positive_bits(packed[0]), positive_bits(packed[1]));
    if (staged) {
        if (!MASKT) {  // an earlier store may still be reading the box
            if (lane == 0) {
                if (EPI & EPI_TWO_BOXES) tma_store_wait_read_but_one();
                else tma_store_wait_read();
            }
            __syncwarp();
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) *reinterpret_cast<uint4 *>(mine + ((q ^ (lane & 7)) << 4)) = packed[q >> 2][q & 3];
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
            tma_store_2d(b.tm_out, smem_u32(b.box), b.col0, b.map_row);
            tma_store_commit();
        }
        if ((EPI & (EPI_MASK | EPI_BITS)) && p.colsum_part) {
            // sums of the box's columns over its 32 rows: a lane reads its two columns down the rows (one 4-byte word a
            // row, conflict free), half the instructions of a butterfly over registers
            float s0 = 0.0f, s1 = 0.0f, u0 = 0.0f, u1 = 0.0f;
            const uint8_t *word = b.box + (lane & 3) * 4;
#pragma unroll 8
            for (int r = 0; r < 32; r += 2) {
                const uint32_t w0 = *reinterpret_cast<const uint32_t *>(word + r * 128 + (((lane >> 2) ^ (r & 7)) << 4));
                const uint32_t w1 = *reinterpret_cast<const uint32_t *>(word + (r + 1) * 128 + (((lane >> 2) ^ ((r + 1) & 7)) << 4));
                s0 += __uint_as_float(w0 << 16); s1 += __uint_as_float(w0 & 0xffff0000u);
                u0 += __uint_as_float(w1 << 16); u1 += __uint_as_float(w1 & 0xffff0000u);
            }
            *reinterpret_cast<float2 *>(p.colsum_part + b.colsum_row * p.N + b.col0 + 2 * lane) = make_float2(s0 + u0, s1 + u1);
            __syncwarp();  // read before the next box overwrites this one
        }
        return;
    }
    if (row_ok) {
        uint4 *dst = reinterpret_cast<uint4 *>(p.out + b.out_off + out_row * p.N + b.col0);
#pragma unroll
        for (int q = 0; q < 4; ++q) st_global_32B(dst + 2 * q, packed[q >> 1][2 * (q & 1)], packed[q >> 1][2 * (q & 1) + 1]);
    }
    if ((EPI & (EPI_MASK | EPI_BITS)) && p.colsum_part) {  // sums of the rounded values, rows past the segment end count as 0; the whole warp: shuffles
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float a[32];
            const uint32_t *pw = reinterpret_cast<const uint32_t *>(packed[u]);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                a[2 * j] = row_ok ? __uint_as_float(pw[j] << 16) : 0.0f;
                a[2 * j + 1] = row_ok ? __uint_as_float(pw[j] & 0xffff0000u) : 0.0f;
            }
            p.colsum_part[b.colsum_row * p.N + b.col0 + 32 * u + lane] = warp_column_sums(a, lane);
        }
    }
    }
}
// mask bits of a row's 128 columns from col0 on (two boxes), as far as the row has them
__device__ __forceinline__ void keep_load(const GemmParams &p, int64_t row, int32_t col0, uint2 (&keep)[2]) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        keep[u] = make_uint2(0u, 0u);
        if (col0 + 64 * u < p.N) keep[u] = *reinterpret_cast<const uint2 *>(p.bits_in + row * (p.N >> 5) + ((col0 + 64 * u) >> 5));
    }
}

struct Tile {
    int32_t e;        // expert / segment
    int32_t row0;     // ROW_*: first sorted row; WGRAD: first row of the segment
    int32_t row_end;  // end of the segment
    int32_t m0;       // WGRAD: first output row of the tile
    int32_t n0;       // first output column
    int32_t kblocks;  // number of K blocks
    int32_t b_chunk;  // WGRAD: first 64-column chunk of B
    int32_t mt;       // ROW_*: index of the M tile over all segments
};

// Tile ids are handed out round-robin. What a tile needs from global memory (its segment's bounds) is
// fetched one tile ahead (tile_fetch) and only turned into a Tile (tile_decode) when the tile starts, so
// the load latency never sits between two tiles. ROW_* with ragged segments read one 16-byte record per
// M tile (the experts' from the call's segment plan, the grouped gates' from tile_table_kernel); WGRAD reads the two
// segment bounds.
template <int KIND>
__device__ __forceinline__ int4 tile_fetch(const GemmParams &p, int32_t id) {
    if (!p.offsets || id >= p.total_tiles) return make_int4(-1, 0, 0, 0);
    if (KIND == WGRAD) {
        int32_t rest, seg;
        const int32_t e = p.by_per_e(id, rest);
        if (p.off_mod > 0) p.by_mod(e, seg);  // segment s reads the rows of group s % off_mod
        else seg = e;
        return make_int4(e, p.offsets[seg], p.offsets[seg + 1], 0);
    }
    int32_t rest;
    return p.tile_info[p.by_tiles_n(id, rest)];
}

template <int KIND, int TM>
__device__ __forceinline__ bool tile_decode(const GemmParams &p, int32_t id, const int4 &raw, Tile &t) {
    if (id >= p.total_tiles) return false;
    if (KIND == WGRAD) {
        int32_t rem, tn;
        int32_t e = p.by_per_e(id, rem);
        // uniform ranges, interleaved terms: consecutive ids walk the terms of one row range (its rows stay in L2 for all
        // of them) while the segment index stays term-major
        if (p.interleave > 1) {
            int32_t term;
            const int32_t range = p.by_interleave(e, term);
            e = term * p.segs_per_term + range;
        }
        const int32_t tm = p.by_tiles_n(rem, tn);
        t.e = e;
        t.mt = 0;
        t.m0 = tm * TM;
        t.n0 = tn * p.tile_n;
        t.b_chunk = t.n0 / 64;
        if (p.offsets) {
            t.row0 = raw.y;
            t.row_end = raw.z;
            if (p.off_mod > 0) {
                int32_t group;
                t.b_chunk += p.by_mod(e, group) * p.b_term_chunks;  // B term s / off_mod
            }
        } else {
            int64_t rps;
            int32_t c, term;
            if (e < p.segs_term0) {  // term 0 may use its own (shorter) row ranges
                c = e; rps = p.rows_per_seg0; term = 0;
            } else {
                term = p.by_terms(e - p.segs_term0, c) + (p.segs_term0 > 0 ? 1 : 0);
                rps = p.rows_per_seg;
            }
            t.row0 = (int32_t)(c * rps);
            t.row_end = (int32_t)(((c + 1) * rps < p.R) ? (c + 1) * rps : p.R);
            if (t.row_end < t.row0) t.row_end = t.row0;
            t.b_chunk += term * p.b_term_chunks;
        }
        t.kblocks = (t.row_end - t.row0 + BK - 1) / BK;
        return true;
    } else {
        int32_t tn;
        const int32_t mt = p.by_tiles_n(id, tn);
        t.mt = mt;
        t.m0 = 0;
        t.b_chunk = 0;
        t.kblocks = p.kblocks_row;
        t.n0 = tn * p.tile_n;
        if (!p.offsets) {  // one segment of R rows; total_tiles is exact
            t.e = 0;
            t.row0 = mt * TM;
            t.row_end = (int32_t)p.R;
            return true;
        }
        if (raw.x < 0) return false;  // past the last M tile
        MOE_BOUNDS_NOTE(raw.x < p.nseg && raw.y >= 0 && raw.y <= raw.z && (int64_t)raw.z <= p.R);
        t.e = raw.x;
        t.row0 = raw.y;
        t.row_end = raw.z;
        return true;
    }
}

template <int KIND, int TM> struct TileIter {
    const GemmParams &p;
    int32_t id, stride;
    int4 raw;
    __device__ __forceinline__ TileIter(const GemmParams &p_, int32_t first, int32_t stride_)
        : p(p_), id(first), stride(stride_) { raw = tile_fetch<KIND>(p, id); }
    // the current tile; starts the fetch for the following one
    __device__ __forceinline__ bool next(Tile &t) {
        if (!tile_decode<KIND, TM>(p, id, raw, t)) return false;
        id += stride;
        raw = tile_fetch<KIND>(p, id);
        return true;
    }
};

// The maps of a tile whose last box of rows reaches beyond its segment (first row `row0` of a box of `height` rows; WGRAD: the
// segment's last K block)
template <int KIND> struct SegmentEnd {
    const CUtensorMap *a, *b;
    bool ragged;
    __device__ __forceinline__ SegmentEnd(const GemmParams &p, const Tile &t, int32_t row0, int height) : a(nullptr), b(nullptr) {
        if (KIND == WGRAD) ragged = p.seg_a && (t.row_end - t.row0) % BK != 0;  // (never with off_mod)
        else ragged = p.seg_a && row0 + height > t.row_end;
        if (!ragged) return;
        a = p.seg_a + t.e;
        acquire_map(a);
        if (KIND == WGRAD) {
            b = p.seg_b + t.e;
            acquire_map(b);
        }
    }
};

// The epilogue of an ACC tile (see grouped_gemm_kernel) by one warp: a lane's row of the warp's 128 columns, the running sums in registers.
// row0: the warp's first output row; tfull0: the barriers of the two accumulators; release() hands the current one back.
template <typename Release>
__device__ __forceinline__ bool acc_tile(const GemmParams &p, const Tile &t, int lane, int quarter, int half, int64_t row0, uint8_t *slab,
                                         uint32_t tmem_base, uint32_t tfull0, volatile int *abort_flag, int &acc, uint32_t &acc_ph,
                                         Release release) {
    float sums[4][32];
#pragma unroll
    for (int i = 0; i < 128; ++i) sums[i >> 5][i & 31] = 0.0f;
    const int sub = t.e < p.segs_term0 ? p.sub_kb0 : p.sub_kb;
    const int nsub = (t.kblocks + sub - 1) / sub;
    const int columns = p.N - (t.n0 + half * 128);  // the warp's that exist (a multiple of 64); the others were not computed
    for (int sb = 0; sb < nsub; ++sb) {
        if (!mbar_wait(tfull0 + 8u * acc, acc_ph, abort_flag, p.status)) return false;
        tc_fence_after();
        // the accumulator goes back when it is read, before the last additions
        auto drain = [&](auto count_) {
            constexpr int COUNT = decltype(count_)::value;
            if (COUNT == 0) release();
#pragma unroll
            for (int cl = 0; cl < COUNT; ++cl) {
                uint32_t v[32];
                tc_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + (half * 4 + cl) * 32, v);
                tc_ld_wait();
                if (cl == COUNT - 1) release();
#pragma unroll
                for (int j = 0; j < 32; ++j) sums[cl][j] += __uint_as_float(v[j]);
            }
        };
        if (columns >= 128) drain(std::integral_constant<int, 4>());
        else if (columns > 0) drain(std::integral_constant<int, 2>());
        else drain(std::integral_constant<int, 0>());
        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
    }
    // to global memory by way of the warp's 4 KiB: lane l moves piece l % 8 of row 4 * i + l / 8
    float *dst = p.out_f32 + (int64_t)t.e * p.M * p.N + row0 * p.N + t.n0 + half * 128 + (lane & 7) * 4;
#pragma unroll
    for (int cl = 0; cl < 4; ++cl) {
        if (t.n0 + half * 128 + cl * 32 >= p.N) break;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            *reinterpret_cast<float4 *>(slab + lane * 128 + ((q ^ (lane & 7)) << 4)) =
                make_float4(sums[cl][4 * q], sums[cl][4 * q + 1], sums[cl][4 * q + 2], sums[cl][4 * q + 3]);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = 4 * i + (lane >> 3);
            if (row0 + row < p.M)
                *reinterpret_cast<float4 *>(dst + (int64_t)row * p.N + cl * 32) =
                    *reinterpret_cast<const float4 *>(slab + row * 128 + (((lane & 7) ^ (row & 7)) << 4));
        }
        __syncwarp();
    }
    return true;
}

// EPI_TWO_BOXES (WGRAD over short segments): a warp's boxes take turns in two 4 KiB pieces, for one operand stage less. With one or two K
// blocks a tile the epilogue is what a tile lasts, 1100 cycles a box, 420 of them waiting until the store before had read the box
// out: 4096 experts x 64 rows 1056 and 1087 us -> 981 to 1012 and 1056 to 1076, 256 x 78 rows 61 -> 58; with three K blocks a tile the stage is worth
// more (256 x 188 rows 83 -> 86). Sixteen epilogue warps, eight an accumulator, were no faster than the second box.
// ACC (WGRAD with float output over long uniform row ranges, the gate backward): the contraction of a tile is cut
// into sub-blocks of p.sub_kb0 / p.sub_kb K blocks (first term / other terms). Each sub-block is accumulated in TMEM on
// its own (an fp32 tensor-core accumulator truncates, and a long run of same-sign terms loses low bits: 128 rows keep
// that below 1e-5), handed to the epilogue like a tile, and added there, with rounding to nearest, to running sums in
// registers (a lane's row of the warp's 128 columns; the cap of 168 registers makes the compiler spill 96 bytes of other
// values, 132 on SM pairs); the sums go to global memory once per tile. (With the sums in shared memory, which left room for two operand
// stages, a K block took 1850 cycles: the latency of its loads.)
template <int KIND, int EPI, bool ACC = false>
__global__ void __launch_bounds__(NTHREADS, 1)
grouped_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmO, const GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;  // 1024-B aligned for the 128-B swizzle
    uint8_t *smem = smem_raw + (base - smem_u32(smem_raw));
    constexpr bool TWO_BOXES = (EPI & EPI_TWO_BOXES) != 0;
    constexpr int NST = TWO_BOXES ? STAGES - 1 : STAGES;
    const uint32_t bars = base + NST * STAGE_BYTES;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (NST + s); };
    auto tfull_bar = [&](int a) { return bars + 8u * (2 * NST + a); };
    auto tempty_bar = [&](int a) { return bars + 8u * (2 * NST + 2 + a); };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + NST * STAGE_BYTES + 8 * (2 * NST + 4));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + NST * STAGE_BYTES + 8 * (2 * NST + 4) + 8);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 8); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void *)tmem_slot)),
                     "r"((uint32_t)TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    wait_previous_kernel();  // barriers and tensor memory are set up while the previous kernel drains

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            TileIter<KIND, BM> it(p, (int32_t)blockIdx.x, (int32_t)gridDim.x);
            Tile t;
            while (ok && it.next(t)) {
                int term = 0, kk = 0;  // ROW_*: piece of the contraction and column inside it
                const SegmentEnd<KIND> end(p, t, t.row0, BM);
                const CUtensorMap *row_a = KIND != WGRAD && end.ragged ? end.a : &tmA;
                for (int kb = 0; kb < t.kblocks && ok; ++kb) {
                    ok = mbar_wait(empty_bar(s), ph ^ 1u, abort_flag, p.status);
                    if (!ok) break;
                    const uint32_t a_dst = base + s * STAGE_BYTES, b_dst = a_dst + A_BYTES;
                    mbar_expect_tx(full_bar(s), A_BYTES + p.tile_n * BK * 2);
                    if (KIND == WGRAD) {
                        const int r = t.row0 + kb * BK;
                        const bool tail = end.ragged && kb == t.kblocks - 1;
                        tma_load_3d(a_dst, tail ? end.a : &tmA, full_bar(s), 0, r, t.m0 / 64);
                        tma_load_3d(b_dst, tail ? end.b : &tmB, full_bar(s), 0, r, t.b_chunk);
                    } else {
                        tma_load_2d(a_dst, row_a, full_bar(s), p.a_term_col[term] + kk, t.row0);
                        if (KIND == ROW_BMN) tma_load_4d(b_dst, &tmB, full_bar(s), 0, p.b_term_col[term] + kk, t.n0 / 64, t.e);
                        else tma_load_3d(b_dst, &tmB, full_bar(s), p.b_term_col[term] + kk, t.n0, t.e);
                        kk += BK;
                        if (kk == p.K) { kk = 0; ++term; }
                    }
                    if (++s == NST) { s = 0; ph ^= 1u; }
                }
            }
            // drain: every copy this thread started must have landed before the CTA may exit
            if (!ok)
                for (int q = 0; q < NST; ++q) {
                    const unsigned long long t0 = global_ns();
                    while (!mbar_try_wait(full_bar(q), 0) && !mbar_try_wait(full_bar(q), 1) &&
                           global_ns() - t0 < WAIT_LIMIT_NS) {}
                }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        int s = 0, acc = 0;
        uint32_t ph = 0, acc_ph = 0;
        bool ok = true;
        TileIter<KIND, BM> it(p, (int32_t)blockIdx.x, (int32_t)gridDim.x);
        Tile t;
        while (ok && it.next(t)) {
            if (t.kblocks == 0) continue;  // empty segment (WGRAD): the epilogue writes zeros
            // columns behind the output's are not computed (N is a multiple of 64)
            const uint32_t idesc = make_idesc(KIND == WGRAD ? 1 : 0, KIND == ROW_BK ? 0 : 1, min(p.tile_n, p.N - t.n0));
            const int sub = ACC ? (t.e < p.segs_term0 ? p.sub_kb0 : p.sub_kb) : t.kblocks;  // K blocks per accumulator
            uint32_t d_tmem = tmem_base + acc * BN;
            int kin = 0;  // K block inside the accumulator's sub-block
            for (int kb = 0; kb < t.kblocks; ++kb, ++kin) {
                if (ACC && kin == sub) kin = 0;
                if (kin == 0) {
                    ok = mbar_wait(tempty_bar(acc), acc_ph ^ 1u, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    d_tmem = tmem_base + acc * BN;
                }
                ok = mbar_wait(full_bar(s), ph, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_src = base + s * STAGE_BYTES, b_src = a_src + A_BYTES;
                int ksteps = BK / 16;  // K steps of 16 rows to issue for this block: none that lies behind the segment's end
                if (KIND == WGRAD && kb == t.kblocks - 1) {
                    const int valid = min(BK, t.row_end - (t.row0 + kb * BK));  // rows of this block inside the segment
                    ksteps = (valid + 15) / 16;
                    const int nz = ksteps * 16 - valid;
                    // Without the segments' own maps (see tc_wgrad_gemm) the rows behind the end, up to the end of the step that holds
                    // it, are the next segment's: zeroed in A AND in B (0 x finite = 0 would do for finite data; both keep a
                    // non-finite value of the next segment out of this segment's sums): 128-B lines in all 64-column
                    // chunks, the A tile's two chunks directly followed by the B tile's four.
                    if (p.offsets && !p.seg_a && nz > 0) {
                        // eight lanes a line of one chunk, four lines at a time (as one loop over all lines, with a division for
                        // each, this was 1450 cycles a tile of 64 rows)
                        uint8_t *z = smem + s * STAGE_BYTES + (valid + (lane >> 3)) * 128 + (lane & 7) * 16;
                        for (int r = lane >> 3; r < nz; r += 4, z += 4 * 128)
#pragma unroll
                            for (int chunk = 0; chunk < (BM + BN) / 64; ++chunk)
                                *reinterpret_cast<uint4 *>(z + chunk * (BK * 128)) = make_uint4(0, 0, 0, 0);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                    }
                }
                if (lane == 0) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        if (k >= ksteps) break;
                        uint64_t ad, bd;
                        if (KIND == WGRAD) ad = desc_mnmajor(a_src + k * 16 * 128);
                        else ad = desc_kmajor(a_src + k * 32);
                        if (KIND == ROW_BK) bd = desc_kmajor(b_src + k * 32);
                        else bd = desc_mnmajor(b_src + k * 16 * 128);
                        tc_mma_bf16(d_tmem, ad, bd, idesc, (kin > 0 || k > 0) ? 1u : 0u);
                    }
                    tc_commit(empty_bar(s));  // the stage may be refilled once these MMAs have read it
                }
                __syncwarp();
                if (++s == NST) { s = 0; ph ^= 1u; }
                if (ACC && (kin == sub - 1 || kb == t.kblocks - 1)) {  // sub-block complete
                    if (lane == 0) tc_commit(tfull_bar(acc));
                    __syncwarp();
                    if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
                }
            }
            if (!ACC) {
                if (ok && lane == 0) tc_commit(tfull_bar(acc));  // accumulator complete
                __syncwarp();
                if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..9)
        const int quarter = warp & 3;  // TMEM lanes 32*quarter .. 32*quarter + 31 belong to this warp
        int acc = 0, turn = 0;
        uint32_t acc_ph = 0;
        bool ok = true;
        TileIter<KIND, BM> it(p, (int32_t)blockIdx.x, (int32_t)gridDim.x);
        Tile t;
        while (ok && it.next(t)) {
            const bool have_acc = t.kblocks > 0;
            if constexpr (ACC) {
                auto release = [&]() {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty_bar(acc));
                };
                ok = acc_tile(p, t, lane, quarter, (warp - 2) >> 2, (int64_t)t.m0 + quarter * 32, smem + NST * STAGE_BYTES + 1024 + (warp - 2) * 4096,
                              tmem_base, bars + 8u * 2 * NST, abort_flag, acc, acc_ph, release);
                if (!ok) break;
                continue;
            }
            // Two warps share each quarter of the accumulator's rows and take half of its columns each, in boxes of 64.
            const int half = (warp - 2) >> 2;
            const int32_t first = t.n0 + half * (p.tile_n / 2);
            const int boxes = min(p.tile_n / 128, max(0, (p.N - first) / 64));  // N is a multiple of 64
            BoxArgs b;
            b.tm_out = &tmO;
            b.out_off = KIND == WGRAD ? (int64_t)t.e * p.M * p.N : 0;
            b.row0 = (KIND == WGRAD ? t.m0 : t.row0) + quarter * 32;
            b.rows_valid = (KIND == WGRAD ? p.M : t.row_end) - (int32_t)b.row0;
            b.map_row = (int32_t)b.row0 + (KIND == WGRAD ? t.e * p.M : 0);
            b.colsum_row = t.mt * 4 + quarter;
            b.have_acc = have_acc;
            uint4 bias[2][4];
            const bf16 *bias_at = (EPI & EPI_BIAS) ? p.bias + (int64_t)t.e * p.N + first : nullptr;
            if ((EPI & EPI_BIAS) && boxes > 0) bias_load(bias_at, bias);
            uint2 keep[2] = {make_uint2(0u, 0u), make_uint2(0u, 0u)};
            if ((EPI & EPI_BITS) && lane < b.rows_valid) keep_load(p, b.row0 + lane, first, keep);
            if (have_acc) {  // (the loads above are in flight while the warp waits for its accumulator)
                ok = mbar_wait(tfull_bar(acc), acc_ph, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
            }
            auto release = [&]() {  // the warp's part of the accumulator is in registers: the buffer goes back
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty_bar(acc));
            };
            for (int u = 0; u < boxes; ++u) {
                b.col0 = first + 64 * u;
                b.taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + half * (p.tile_n / 2) + 64 * u;
                b.next_bias = (EPI & EPI_BIAS) && u + 1 < boxes ? bias_at + 64 : nullptr;
                b.keep = u ? keep[1] : keep[0];
                b.box = smem + NST * STAGE_BYTES + 1024 + (TWO_BOXES ? (warp - 2) * 8192 + turn * 4096 : (warp - 2) * 4096);
                if (b.rows_valid >= 32) turn ^= 1;  // (else nothing is stored from the box)
                epilogue_box<EPI, false>(p, lane, b, bias, [&]() { if (u + 1 == boxes) release(); });
            }
            if (have_acc) {
                if (boxes == 0) release();
                if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
            }
        }
        if (p.tma_out && lane == 0) tma_store_wait_all();  // no bulk store may outlive the CTA's shared memory
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS)
                     : "memory");
    }
}


// ------------------------------------------------------------------------------------------
// Two-CTA variant for the row GEMMs (ROW_BMN, ROW_BK): a cluster of two CTAs (an SM pair) works on a
// 256 x 256 tile with tcgen05.mma cta_group::2 (M 256). Each CTA stages its own 128 rows of A and its
// own 128 columns of B (32 KiB per stage instead of 48, six stages), the pair's tensor cores exchange
// the B halves, and each CTA keeps the accumulator of its 128 rows in its own TMEM. The even CTA of
// the pair issues the MMAs; the loads of both CTAs count on its "full" barrier; tcgen05.commit
// releases a stage / publishes an accumulator in both CTAs at once; the odd CTA's epilogue warps
// hand their accumulator buffer back with an arrive on the even CTA's barrier.
// ------------------------------------------------------------------------------------------
constexpr int STAGES2 = 6;
constexpr int A2_BYTES = 128 * BK * 2, B2_BYTES = 128 * BK * 2, STAGE2_BYTES = A2_BYTES + B2_BYTES;
constexpr int DATA2_BYTES = STAGES2 * STAGE2_BYTES + EPI_STAGE_BYTES;  // 224 KiB: 6 stages + float staging, or 5 stages + mask tile
constexpr int SMEM2_BYTES = DATA2_BYTES + 1024 + 512;  // + alignment slack, barriers, scheduler ring
constexpr uint32_t PEER_BIT_MASK = 0xFEFFFFFFu;  // clears the CTA-rank bit of a shared::cluster address of the pair

__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// arrive on the barrier at this shared-memory offset in the EVEN CTA of the pair
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar & PEER_BIT_MASK) : "memory");
}
// The same without release semantics, for handing an accumulator buffer back: the tensor-memory reads are
// complete (tcgen05.wait::ld) and fenced (tcgen05.fence::before_thread_sync) before the arrive, and nothing
// the other side reads was written through memory. A release at cluster scope would wait here for all of this
// thread's earlier global stores (the output rows) to reach L2, several thousand cycles per tile.
__device__ __forceinline__ void mbar_arrive_leader_relaxed(uint32_t bar) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar & PEER_BIT_MASK) : "memory");
}
__device__ __forceinline__ void tc_commit2(uint32_t bar) {  // arrives at this offset in both CTAs of the pair
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(bar), "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void tc_mma2_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p;\n}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(0u)
        : "memory");
}
// loads of the pair: both CTAs' transaction bytes are counted on the even CTA's barrier
__device__ __forceinline__ void tma2_load_2d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar & PEER_BIT_MASK), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma2_load_3d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1,
                                             int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar & PEER_BIT_MASK), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma2_load_4d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1,
                                             int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(dst), "l"(tm), "r"(bar & PEER_BIT_MASK), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__host__ __device__ constexpr uint32_t make_idesc2(int a_mn, int b_mn) {  // M 256, N 256
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
}

// Tile source of the two-CTA kernel. Static mode: ids dealt round-robin to the pairs (TileIter). Dynamic mode (ragged
// segments): a fixed deal leaves pairs idle at the end, because the tiles of a weight-gradient GEMM differ in length by
// the ratio of the largest to the smallest expert, and because SM pairs do not all run at the same speed (distance to
// the L2 slices, the two dies). The scheduler warp of the even CTA draws tile ids from a global counter (WGRAD: in
// descending order of segment size, longest first) and publishes one 16-byte record per tile {segment, first row,
// end row, tile id} in a four-slot ring in the shared memory of BOTH CTAs; every warp role of both CTAs reads the
// same sequence of records. A record with segment -1 ends the sequence. Which pair computes a tile does not change
// the tile's result, so the output stays bit-reproducible.
constexpr int SCHED_SLOTS = 4;
__device__ __forceinline__ uint32_t peer_smem_addr(uint32_t addr, uint32_t cta) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
    return r;
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, const int4 &v) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster_addr(uint32_t cluster_addr) {  // release at cluster scope
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

template <int KIND> struct PairTiles {
    const GemmParams &p;
    TileIter<KIND, 256> fixed;
    const bool dyn, warp_wide, arrives;
    const uint32_t ring, full0, empty0;
    volatile int *abort_flag;
    int i;
    // warp_wide: all 32 lanes of the warp call next() together; arrives: this thread reports the slot as read
    __device__ __forceinline__ PairTiles(const GemmParams &p_, bool dyn_, int32_t first, int32_t stride, uint32_t ring_,
                                         uint32_t full0_, uint32_t empty0_, volatile int *abort_, bool warp_wide_, bool arrives_)
        : p(p_), fixed(p_, dyn_ ? p_.total_tiles : first, stride), dyn(dyn_), warp_wide(warp_wide_), arrives(arrives_),
          ring(ring_), full0(full0_), empty0(empty0_), abort_flag(abort_), i(0) {}
    __device__ __forceinline__ bool next(Tile &t) {
        if (!dyn) return fixed.next(t);
        const int slot = i & (SCHED_SLOTS - 1);
        const uint32_t par = (uint32_t)(i / SCHED_SLOTS) & 1u;
        if (!mbar_wait(full0 + 8u * slot, par, abort_flag, p.status)) return false;
        mbar_try_wait_cluster(full0 + 8u * slot, par);  // acquire at cluster scope: the record came from the other CTA's thread
        // The slot is overwritten once every reader has reported it read, so a reader's copy has to be in its registers
        // before its report leaves. The report is a relaxed arrive (a release at cluster scope would wait for the thread's
        // earlier output stores, 3 % of a step), which by itself orders nothing: with an ordinary load the assembler was
        // free to fetch the record again later instead of keeping it in registers, and in the register-heaviest epilogue
        // (mask bits + column sums) one warp then now and again worked on the record of four tiles ahead and left its
        // piece of the output unwritten. Hence a volatile load (issued once, where it stands) and an arrive whose address
        // is computed from the loaded words of all lanes (sign bit of the tile id, always 0), which cannot issue before
        // those loads have returned.
        int4 rec;
        asm volatile("ld.volatile.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(rec.x), "=r"(rec.y), "=r"(rec.z), "=r"(rec.w)
                     : "r"(ring + 16u * slot) : "memory");
        uint32_t seen = (uint32_t)rec.w;
        if (warp_wide) seen = __reduce_or_sync(0xffffffffu, seen);
        if (arrives) mbar_arrive_leader_relaxed(empty0 + 8u * slot + ((seen >> 31) << 3));
        ++i;
        if (rec.x < 0) return false;
        MOE_BOUNDS_NOTE(rec.x < p.nseg && rec.y >= 0 && rec.y <= rec.z && (int64_t)rec.z <= p.R);
        t.e = rec.x; t.row0 = rec.y; t.row_end = rec.z;
        int32_t rem, tn;
        const int32_t grp = p.by_group(rec.w, rem);  // rec.w: the tile id
        if (KIND == WGRAD) {
            const int32_t tm = p.by_tiles_n(rem, tn);
            t.mt = 0;
            t.m0 = tm * 256;
            t.n0 = tn * BN;
            t.b_chunk = t.n0 / 64;
            t.kblocks = (t.row_end - t.row0 + BK - 1) / BK;
        } else {
            t.mt = grp;
            t.m0 = 0;
            t.b_chunk = 0;
            t.n0 = rem * BN;
            t.kblocks = p.kblocks_row;
        }
        return true;
    }
};

// MASKT: the ReLU mask of the dgrad GEMM is not read row by row from global memory by the epilogue but
// fetched as a 128 x 256 tile by TMA (one stage fewer in exchange for the 64 KiB it occupies).
template <int KIND, int EPI, bool MASKT, bool ACC>
__global__ void __launch_bounds__(NTHREADS2, 1)
grouped_gemm2_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ CUtensorMap tmM, const __grid_constant__ CUtensorMap tmO,
                     const GemmParams p) {
    // ROW_* with a mask tile: 5 stages and a 64 KiB region of four [128 rows][64 columns] blocks (128-byte swizzle) that
    // holds the ReLU-mask tile and stages the bf16 output for bulk tensor stores; every other kind: 6 stages + 32 KiB of
    // staging (row GEMMs: two such blocks, a warp's two output boxes of a tile pass through the same 4 KiB one after
    // the other; the sixth stage took a seventh off the time the MMA thread waited for operands at 16 K blocks per tile)
    constexpr int NST = (KIND == WGRAD || !MASKT) ? 6 : 5;  // the mask tile needs the 64 KiB region, everything else 32 KiB
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bars = base + DATA2_BYTES;  // [stages][float staging or mask tile] then the barriers
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (NST + s); };
    auto tfull_bar = [&](int a) { return bars + 8u * (2 * NST + a); };
    auto tempty_bar = [&](int a) { return bars + 8u * (2 * NST + 2 + a); };
    const uint32_t mfull_bar = bars + 8u * 28, mempty_bar = bars + 8u * 29;  // mask tile landed / read by all 8 epilogue warps
    // dynamic tile scheduling (WGRAD): record published / record read by every role of both CTAs (barrier in the even CTA)
    const uint32_t sched_full0 = bars + 256, sched_empty0 = bars + 256 + 8u * SCHED_SLOTS, sched_ring = bars + 384;
    const bool dyn = p.sched_counter != nullptr;
    const uint32_t mask_smem = base + NST * STAGE2_BYTES;                     // 4 blocks of [128 rows][64 columns], 128-B swizzle
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + DATA2_BYTES + 240);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + DATA2_BYTES + 248);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();  // 0: issues the MMAs, owns the full / tempty barriers
    const int64_t cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 16); }
        mbar_init(mfull_bar, 1); mbar_init(mempty_bar, 8);
        // readers of a scheduler record: producer, 8 epilogue warps in each CTA, the MMA thread in the even one
        for (int q = 0; q < SCHED_SLOTS; ++q) { mbar_init(sched_full0 + 8u * q, 1); mbar_init(sched_empty0 + 8u * q, 19); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
        if (MASKT) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmM) : "memory");
        if (p.tma_out) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmO) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void *)tmem_slot)),
                     "r"((uint32_t)TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // both CTAs' barriers exist before anything is signalled across the pair
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    wait_previous_kernel();  // barriers and tensor memory are set up while the previous kernel drains

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0, mask_ph = 0;
            bool ok = true;
            PairTiles<KIND> it(p, dyn, (int32_t)cluster_id, (int32_t)n_clusters, sched_ring, sched_full0, sched_empty0, abort_flag, false, true);
            Tile t;
            // MASKT: the mask tile of a row tile can only land after the epilogue has read the previous one, which
            // happens while the next tile's K blocks are already being loaded: the load stays "due" and is issued
            // from the K loop as soon as the region is free, so the producer never stops to wait for the epilogue.
            bool mask_due = false;
            int mask_n0 = 0, mask_row0 = 0;
            auto load_mask = [&](bool blocking) -> bool {
                if (blocking) {
                    if (!mbar_wait(mempty_bar, mask_ph ^ 1u, abort_flag, p.status)) return false;
                } else if (!mbar_try_wait(mempty_bar, mask_ph ^ 1u)) {
                    return true;
                }
                const int nblk = min(4, (p.N - mask_n0) / 64);
                mbar_expect_tx(mfull_bar, nblk * 16384);
                for (int b = 0; b < nblk; ++b)
                    tma_load_2d(mask_smem + b * 16384, &tmM, mfull_bar, mask_n0 + b * 64, mask_row0 + 128 * (int)rank);
                mask_ph ^= 1u;
                mask_due = false;
                return true;
            };
            int trace_tile = -1;
            while (ok && it.next(t)) {
                int term = 0, kk = 0;  // ROW_*: piece of the contraction and column inside it
                const SegmentEnd<KIND> end(p, t, t.row0 + 128 * (int)rank, 128);
                const CUtensorMap *row_a = KIND != WGRAD && end.ragged ? end.a : &tmA;
                ++trace_tile;
                long long tr_empty = 0;
                for (int kb = 0; kb < t.kblocks && ok; ++kb) {
                    if (MASKT && mask_due) load_mask(false);
                    const long long tw0 = TILE_CLOCK();
                    ok = mbar_wait(empty_bar(s), ph ^ 1u, abort_flag, p.status);
                    if (!ok) break;
                    tr_empty += TILE_CLOCK() - tw0;
                    if (kb == 0) TILE_TRACE_SET(0, trace_tile, 0, TILE_CLOCK());
                    if (kb == t.kblocks - 1) { TILE_TRACE_SET(0, trace_tile, 2, TILE_CLOCK()); TILE_TRACE_SET(0, trace_tile, 1, tr_empty); }
                    const uint32_t a_dst = base + s * STAGE2_BYTES, b_dst = a_dst + A2_BYTES;
                    if (KIND == WGRAD) {
                        const int r = t.row0 + kb * BK;
                        const bool tail = end.ragged && kb == t.kblocks - 1;
                        if (rank == 0) mbar_expect_tx(full_bar(s), 2 * STAGE2_BYTES);
                        tma2_load_3d(a_dst, tail ? end.a : &tmA, full_bar(s), 0, r, t.m0 / 64 + 2 * (int)rank);
                        tma2_load_3d(b_dst, tail ? end.b : &tmB, full_bar(s), 0, r, t.b_chunk + 2 * (int)rank);
                    } else {
                        if (rank == 0) mbar_expect_tx(full_bar(s), 2 * STAGE2_BYTES);
                        tma2_load_2d(a_dst, row_a, full_bar(s), p.a_term_col[term] + kk, t.row0 + 128 * (int)rank);
                        if (KIND == ROW_BMN)
                            tma2_load_4d(b_dst, &tmB, full_bar(s), 0, p.b_term_col[term] + kk, t.n0 / 64 + 2 * (int)rank, t.e);
                        else
                            tma2_load_3d(b_dst, &tmB, full_bar(s), p.b_term_col[term] + kk, t.n0 + 128 * (int)rank, t.e);
                        kk += BK;
                        if (kk == p.K) { kk = 0; ++term; }
                    }
                    if (++s == NST) { s = 0; ph ^= 1u; }
                }
                if (MASKT && ok) {  // this tile's mask rows are due once the previous tile's have been read
                    if (mask_due) ok = load_mask(true);  // the previous tile's mask is still due: now it has to go
                    mask_due = ok;
                    mask_n0 = t.n0; mask_row0 = t.row0;
                    if (ok) load_mask(false);
                }
            }
            if (MASKT && ok && mask_due) load_mask(true);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (even CTA only)
        // One thread runs the whole loop: nothing in it needs the other lanes, and a single-thread loop has no
        // divergence / reconvergence around the issue of every K block.
        if (rank == 0 && lane == 0) {
            constexpr uint32_t idesc = make_idesc2(KIND == WGRAD ? 1 : 0, KIND == ROW_BK ? 0 : 1);
            int s = 0, acc = 0;
            uint32_t ph = 0, acc_ph = 0;
            bool ok = true;
            PairTiles<KIND> it(p, dyn, (int32_t)cluster_id, (int32_t)n_clusters, sched_ring, sched_full0, sched_empty0, abort_flag, false, true);
            Tile t;
            int trace_tile = -1;
            while (ok && it.next(t)) {
                ++trace_tile;
                if (t.kblocks == 0) continue;  // empty segment (WGRAD): the epilogue writes zeros
                TILE_TRACE_SET(1, trace_tile, 0, TILE_CLOCK());
                const int sub = !ACC ? t.kblocks : t.e < p.segs_term0 ? p.sub_kb0 : p.sub_kb;  // K blocks per accumulator
                int kin = 0;                                                                  // the block's place among them
                ok = mbar_wait(tempty_bar(acc), acc_ph ^ 1u, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                TILE_TRACE_SET(1, trace_tile, 1, TILE_CLOCK());
                long long tr_wait = 0, tr_issue = 0;
                uint32_t d_tmem = tmem_base + acc * BN;
                const int tail_valid = KIND == WGRAD ? (t.row_end - t.row0) - (t.kblocks - 1) * BK : BK;  // rows of the last block
                for (int kb = 0; kb < t.kblocks; ++kb) {
                    const long long tw0 = TILE_CLOCK();
                    ok = mbar_wait(full_bar(s), ph, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    tr_wait += TILE_CLOCK() - tw0;
                    const uint32_t a_src = base + s * STAGE2_BYTES, b_src = a_src + A2_BYTES;
                    const long long ti0 = TILE_CLOCK();
                    const uint64_t ad0 = KIND == WGRAD ? desc_mnmajor(a_src) : desc_kmajor(a_src);
                    const uint64_t bd0 = KIND == ROW_BK ? desc_kmajor(b_src) : desc_mnmajor(b_src);
                    // a K step of 16 advances the start address (low descriptor bits, in 16-byte units) by 32 bytes in a
                    // K-major tile and by 16 rows of 128 bytes in an MN-major one; the sum never leaves the address field
                    constexpr uint64_t a_step = KIND == WGRAD ? (16 * 128) >> 4 : 32 >> 4;
                    constexpr uint64_t b_step = KIND == ROW_BK ? 32 >> 4 : (16 * 128) >> 4;
                    const int ksteps = (KIND == WGRAD && kb == t.kblocks - 1) ? (tail_valid + 15) / 16 : BK / 16;
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        if (k < ksteps) tc_mma2_bf16(d_tmem, ad0 + k * a_step, bd0 + k * b_step, idesc, (kin > 0 || k > 0) ? 1u : 0u);
                    tc_commit2(empty_bar(s));
                    ++kin;
                    if (ACC && kin == sub && kb + 1 < t.kblocks) {  // sub-block complete: the next one has the other accumulator
                        tc_commit2(tfull_bar(acc));
                        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
                        kin = 0;
                        ok = mbar_wait(tempty_bar(acc), acc_ph ^ 1u, abort_flag, p.status);
                        if (!ok) break;
                        tc_fence_after();
                        d_tmem = tmem_base + acc * BN;
                    }
                    tr_issue += TILE_CLOCK() - ti0;
                    if (++s == NST) { s = 0; ph ^= 1u; }
                }
                if (ok) tc_commit2(tfull_bar(acc));
                TILE_TRACE_SET(1, trace_tile, 3, TILE_CLOCK());
                TILE_TRACE_SET(1, trace_tile, 2, tr_wait); TILE_TRACE_SET(0, trace_tile, 3, tr_issue);
                if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
            }
        }
    } else if (warp == 10) {
        // ------------------------------------------------------------------ tile scheduler (even CTA, one thread)
        if (dyn && rank == 0 && lane == 0) {
            const uint32_t peer_ring = peer_smem_addr(sched_ring, 1), peer_full0 = peer_smem_addr(sched_full0, 1);
            bool ok = true;
            for (int i = 0; ok; ++i) {
                const int slot = i & (SCHED_SLOTS - 1);
                if (i >= SCHED_SLOTS) {  // every reader of the record this slot held has its copy
                    const uint32_t par = (uint32_t)(i / SCHED_SLOTS - 1) & 1u;
                    ok = mbar_wait(sched_empty0 + 8u * slot, par, abort_flag, p.status) && mbar_try_wait_cluster(sched_empty0 + 8u * slot, par);
                    if (!ok) break;
                }
                const int32_t id = atomicAdd(p.sched_counter, 1);
                int4 rec = make_int4(-1, 0, 0, 0);
                if (id < p.total_tiles) {
                    int32_t rest;
                    rec = p.sched_table[p.by_group(id, rest)];
                    rec.w = id;
                }
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(sched_ring + 16u * slot), "r"(rec.x), "r"(rec.y), "r"(rec.z), "r"(rec.w) : "memory");
                st_cluster_v4(peer_ring + 16u * slot, rec);
                mbar_arrive(sched_full0 + 8u * slot);
                mbar_arrive_cluster_addr(peer_full0 + 8u * slot);
                if (rec.x < 0) break;
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        uint32_t mask_ph = 0;
        int acc = 0;
        uint32_t acc_ph = 0;
        bool ok = true;
        PairTiles<KIND> it(p, dyn, (int32_t)cluster_id, (int32_t)n_clusters, sched_ring, sched_full0, sched_empty0, abort_flag, true, lane == 0);
        Tile t;
        int trace_tile = -1;
        while (ok && it.next(t)) {
            const bool have_acc = t.kblocks > 0;
            ++trace_tile;
            if (warp == 2 && lane == 0) TILE_TRACE_SET(2, trace_tile, 0, TILE_CLOCK());
            if constexpr (ACC) {
                auto release = [&]() {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_leader_relaxed(tempty_bar(acc));
                };
                ok = acc_tile(p, t, lane, quarter, half, (int64_t)t.m0 + 128 * (int)rank + quarter * 32, smem + NST * STAGE2_BYTES + (warp - 2) * 4096,
                              tmem_base, bars + 8u * 2 * NST, abort_flag, acc, acc_ph, release);
                if (!ok) break;
                continue;
            }
            const int32_t first = t.n0 + half * (BN / 2);
            const int boxes = min(2, max(0, (p.N - first) / 64));  // N is a multiple of 64
            BoxArgs b;
            b.tm_out = &tmO;
            b.out_off = KIND == WGRAD ? (int64_t)t.e * p.M * p.N : 0;
            b.row0 = (KIND == WGRAD ? t.m0 : t.row0) + 128 * (int)rank + quarter * 32;
            b.rows_valid = (KIND == WGRAD ? p.M : t.row_end) - (int32_t)b.row0;
            b.map_row = (int32_t)b.row0 + (KIND == WGRAD ? t.e * p.M : 0);
            b.colsum_row = (t.mt * 2 + (int)rank) * 4 + quarter;
            b.have_acc = have_acc;
            uint4 bias[2][4];
            const bf16 *bias_at = (EPI & EPI_BIAS) ? p.bias + (int64_t)t.e * p.N + first : nullptr;
            if ((EPI & EPI_BIAS) && boxes > 0) bias_load(bias_at, bias);
            uint2 keep[2] = {make_uint2(0u, 0u), make_uint2(0u, 0u)};
            if ((EPI & EPI_BITS) && lane < b.rows_valid) keep_load(p, b.row0 + lane, first, keep);
            if (have_acc) {  // (the loads above are in flight while the warp waits for its accumulator)
                ok = mbar_wait(tfull_bar(acc), acc_ph, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
            }
            if (warp == 2 && lane == 0) TILE_TRACE_SET(2, trace_tile, 1, TILE_CLOCK());
            if (MASKT) {
                ok = mbar_wait(mfull_bar, mask_ph, abort_flag, p.status);
                if (!ok) break;
                mask_ph ^= 1u;
            }
            auto release = [&]() {  // the warp's part of the accumulator is in registers: the buffer goes back
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_leader_relaxed(tempty_bar(acc));
            };
            for (int u = 0; u < boxes; ++u) {
                b.col0 = first + 64 * u;
                b.taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + half * (BN / 2) + 64 * u;
                b.box = smem + NST * STAGE2_BYTES + (MASKT ? (2 * half + u) * 16384 + quarter * 4096 : (warp - 2) * 4096);
                b.next_bias = (EPI & EPI_BIAS) && u + 1 < boxes ? bias_at + 64 : nullptr;
                b.keep = u ? keep[1] : keep[0];
                epilogue_box<EPI, MASKT>(p, lane, b, bias, [&]() { if (u + 1 == boxes) release(); });
            }
            if (have_acc) {
                if (boxes == 0) release();
                if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
            }
            if (warp == 2 && lane == 0) {
                TILE_TRACE_SET(2, trace_tile, 2, TILE_CLOCK());
            }
            if (MASKT) {  // the next mask tile may land once this warp's boxes have been read out
                __syncwarp();
                if (lane == 0) {
                    tma_store_wait_read();
                    mbar_arrive(mempty_bar);
                }
            }
        }
        if (lane == 0) tma_store_wait_all();  // no bulk store may outlive the CTA's shared memory
    }

    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // the pair's MMAs read both CTAs' shared memory: leave together
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS)
                     : "memory");
    }
}

// ------------------------------------------------------------------------------------------ host
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

// bf16 tensor map; dims innermost first, strides (bytes) for dims 1.., box per dim; 128-B swizzle
int32_t make_map(CUtensorMap *tm, const void *base, int rank, const uint64_t *dims, const uint64_t *strides,
                 const uint32_t *box) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return MOE_ERR_CUDA;
    cuuint64_t gdim[5], gstr[4];
    cuuint32_t bx[5], es[5];
    for (int i = 0; i < rank; ++i) { gdim[i] = dims[i]; bx[i] = box[i]; es[i] = 1; }
    for (int i = 0; i + 1 < rank; ++i) gstr[i] = strides[i];
    CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(base), gdim, gstr, bx,
                    es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? MOE_OK : MOE_ERR_CUDA;
}

// rows x cols activations, K-major operand: box 64 (cols) x 128 (rows)
int32_t map_rows_kmajor(CUtensorMap *tm, const void *p, int64_t rows, int64_t cols) {
    const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows}, str[1] = {(uint64_t)cols * 2};
    const uint32_t box[2] = {64, BM};
    return make_map(tm, p, 2, dims, str, box);
}
// rows x cols activations, MN-major operand (contraction over rows): dims (64, rows, cols/64)
int32_t map_rows_mnmajor(CUtensorMap *tm, const void *p, int64_t rows, int64_t cols, int chunks) {
    const uint64_t dims[3] = {64, (uint64_t)rows, (uint64_t)(cols / 64)}, str[2] = {(uint64_t)cols * 2, 128};
    const uint32_t box[3] = {64, BK, (uint32_t)chunks};
    return make_map(tm, p, 3, dims, str, box);
}
// per-expert weight [n, K, N] used as MN-major B: dims (64, K, N/64, n)
int32_t map_weight_mnmajor(CUtensorMap *tm, const void *p, int64_t n, int64_t K, int64_t N, int tile_n = BN) {
    const uint64_t dims[4] = {64, (uint64_t)K, (uint64_t)(N / 64), (uint64_t)n};
    const uint64_t str[3] = {(uint64_t)N * 2, 128, (uint64_t)K * N * 2};
    const uint32_t box[4] = {64, BK, (uint32_t)tile_n / 64, 1};
    return make_map(tm, p, 4, dims, str, box);
}
// per-expert weight [n, N, K] used as K-major B: dims (K, N, n)
int32_t map_weight_kmajor(CUtensorMap *tm, const void *p, int64_t n, int64_t N, int64_t K, int tile_n = BN) {
    const uint64_t dims[3] = {(uint64_t)K, (uint64_t)N, (uint64_t)n};
    const uint64_t str[2] = {(uint64_t)K * 2, (uint64_t)N * K * 2};
    const uint32_t box[3] = {64, (uint32_t)tile_n, 1};
    return make_map(tm, p, 3, dims, str, box);
}

// bf16 output rows as [32][64] boxes
int32_t map_out_boxes(CUtensorMap *tm, const void *p, int64_t rows, int64_t cols) {
    const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows}, str[1] = {(uint64_t)cols * 2};
    const uint32_t box[2] = {64, 32};
    return make_map(tm, p, 2, dims, str, box);
}

GemmParams default_params() {
    GemmParams p;
    memset(&p, 0, sizeof(p));
    p.nterms = 1;
    p.segs_per_term = 1;
    return p;
}

// per-expert weight as B of the two-CTA kernel: each CTA of the pair loads 128 of the 256 columns
int32_t map_weight_mnmajor_half(CUtensorMap *tm, const void *p, int64_t n, int64_t K, int64_t N) {
    const uint64_t dims[4] = {64, (uint64_t)K, (uint64_t)(N / 64), (uint64_t)n};
    const uint64_t str[3] = {(uint64_t)N * 2, 128, (uint64_t)K * N * 2};
    const uint32_t box[4] = {64, BK, 2, 1};
    return make_map(tm, p, 4, dims, str, box);
}
int32_t map_weight_kmajor_half(CUtensorMap *tm, const void *p, int64_t n, int64_t N, int64_t K) {
    const uint64_t dims[3] = {(uint64_t)K, (uint64_t)N, (uint64_t)n};
    const uint64_t str[2] = {(uint64_t)K * 2, (uint64_t)N * K * 2};
    const uint32_t box[3] = {64, 128, 1};
    return make_map(tm, p, 3, dims, str, box);
}

int sm_count() {
    static PerDevice count;
    const int n = count.get([]() {
        int dev = 0, v = 0;
        return cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? v : 0;
    });
    return n > 0 ? n : 148;
}

// Derived tile counts the device code divides by; ids are 32-bit.
template <int KIND, int TM> int32_t complete_params(GemmParams &q, int64_t max_tiles) {
    if (max_tiles >= ((int64_t)1 << 31) - ((int64_t)1 << 22)) return MOE_ERR_UNSUPPORTED;
    if (!q.tile_n) q.tile_n = BN;
    q.tiles_n = (int32_t)cdiv(q.N, q.tile_n);
    q.per_e = KIND == WGRAD ? (int32_t)cdiv(q.M, TM) * q.tiles_n : 1;
    q.total_tiles = (int32_t)max_tiles;
    q.by_tiles_n = Divisor::of(q.tiles_n); q.by_per_e = Divisor::of(q.per_e); q.by_mod = Divisor::of(q.off_mod);
    q.by_terms = Divisor::of(q.segs_per_term); q.by_interleave = Divisor::of(q.interleave); q.by_group = Divisor::of(q.sched_group);
    q.kblocks_row = KIND == WGRAD ? 0 : q.nterms * (q.K / BK);
    return MOE_OK;
}

template <int KIND, int EPI> int32_t launch_as(const CUtensorMap &tmA, const CUtensorMap &tmB, const GemmParams &p, unsigned grid,
                                               cudaStream_t st, const CUtensorMap &tmO) {
    static PerDevice configured;
    if (!allow_shared(configured, grouped_gemm_kernel<KIND, EPI>, SMEM_BYTES)) return MOE_ERR_CUDA;
    if (grid == 0) return MOE_OK;
    launch_kernel(grouped_gemm_kernel<KIND, EPI>, grid, NTHREADS, SMEM_BYTES, st, tmA, tmB, tmO, p);
    MOE_LAUNCHED();
    return MOE_OK;
}
// one or two K blocks in the average segment of a weight gradient
static bool short_segments(int64_t R, int32_t nseg) { return R < 128 * (int64_t)nseg; }
template <int KIND> int32_t launch(const CUtensorMap &tmA, const CUtensorMap &tmB, const GemmParams &p_in,
                                   int64_t max_tiles, cudaStream_t st, const CUtensorMap *tmO = nullptr) {
    GemmParams p = p_in;
    p.tma_out = tmO != nullptr;
    MOE_TRY((complete_params<KIND, BM>(p, max_tiles)));
    const unsigned grid = max_tiles > 0 ? (unsigned)imin(max_tiles, sm_count()) : 0u;
    const CUtensorMap &out = tmO ? *tmO : tmA;
    if (p.out_f32) return launch_as<KIND, EPI_F32>(tmA, tmB, p, grid, st, out);
    if constexpr (KIND == ROW_BMN) {
        if (p.relu) return launch_as<KIND, EPI_BIAS | EPI_RELU>(tmA, tmB, p, grid, st, out);
        return launch_as<KIND, EPI_BIAS>(tmA, tmB, p, grid, st, out);
    } else {
        if constexpr (KIND == ROW_BK) {
            if (p.bits_in) return launch_as<KIND, EPI_BITS>(tmA, tmB, p, grid, st, out);
            if (p.mask) return launch_as<KIND, EPI_MASK>(tmA, tmB, p, grid, st, out);
        }
        if constexpr (KIND == WGRAD) {
            if (short_segments(p.R, p.nseg)) return launch_as<KIND, EPI_TWO_BOXES>(tmA, tmB, p, grid, st, out);
        }
        return launch_as<KIND, EPI_PLAIN>(tmA, tmB, p, grid, st, out);
    }
}

// The sub-block accumulating wgrad (float output)
int32_t launch_acc_wgrad(const CUtensorMap &tmA, const CUtensorMap &tmB, const GemmParams &p_in, int64_t max_tiles,
                         cudaStream_t st) {
    GemmParams p = p_in;
    MOE_TRY((complete_params<WGRAD, BM>(p, max_tiles)));
    static PerDevice configured;
    if (!allow_shared(configured, grouped_gemm_kernel<WGRAD, EPI_F32, true>, SMEM_BYTES)) return MOE_ERR_CUDA;
    if (max_tiles <= 0) return MOE_OK;
    const unsigned grid = (unsigned)imin(max_tiles, sm_count());
    launch_kernel((grouped_gemm_kernel<WGRAD, EPI_F32, true>), grid, NTHREADS, SMEM_BYTES, st, tmA, tmB, tmA, p);
    MOE_LAUNCHED();
    return MOE_OK;
}

template <int KIND, int EPI, bool MASKT = false, bool ACC = false>
int32_t launch2_as(const CUtensorMap &tmA, const CUtensorMap &tmB, const GemmParams &p_in, int64_t max_tiles,
                   cudaStream_t st, const CUtensorMap *tmM, const CUtensorMap *tmO) {
    GemmParams p = p_in;
    p.tma_out = tmO != nullptr;
    MOE_TRY((complete_params<KIND, 256>(p, max_tiles)));
    static PerDevice clusters;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeClusterDimension;
    attrs[0].val.clusterDim.x = 2; attrs[0].val.clusterDim.y = 1; attrs[0].val.clusterDim.z = 1;
    attrs[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_kernel
    attrs[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.blockDim = dim3(NTHREADS2); cfg.dynamicSmemBytes = SMEM2_BYTES; cfg.stream = st;
    cfg.attrs = attrs; cfg.numAttrs = 2;
    const int max_clusters = clusters.get([&]() {
        cfg.gridDim = dim3(2 * (sm_count() / 2));
        int n = 0;
        const auto kernel = grouped_gemm2_kernel<KIND, EPI, MASKT, ACC>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM2_BYTES) != cudaSuccess) return 0;
        return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess ? n : 0;
    });
    if (max_clusters <= 0) return MOE_ERR_CUDA;
    if (max_tiles <= 0) return MOE_OK;
#ifdef MOE_TILE_TRACE
    {   // the launch whose index (counted over the two-CTA launches of the process) equals MOE_TRACE_LAUNCH records
        const char *env = getenv("MOE_TRACE_LAUNCH");
        p.trace = env && atoi(env) == g_trace_launch_no;
        ++g_trace_launch_no;
    }
#endif
    cfg.gridDim = dim3(2 * (unsigned)imin(max_tiles, max_clusters));
    MOE_CUDA(cudaLaunchKernelEx(&cfg, (grouped_gemm2_kernel<KIND, EPI, MASKT, ACC>), tmA, tmB, tmM ? *tmM : tmA, tmO ? *tmO : tmA, p));
    MOE_LAUNCHED();
    return MOE_OK;
}

template <int KIND>
int32_t launch2(const CUtensorMap &tmA, const CUtensorMap &tmB, const GemmParams &p, int64_t max_tiles, cudaStream_t st,
                const CUtensorMap *tmM = nullptr, const CUtensorMap *tmO = nullptr) {
    if constexpr (KIND != WGRAD) {
        if (p.out_f32) return launch2_as<KIND, EPI_F32>(tmA, tmB, p, max_tiles, st, tmM, tmO);
    }
    if constexpr (KIND == ROW_BMN) {
        if (p.relu) return launch2_as<KIND, EPI_BIAS | EPI_RELU>(tmA, tmB, p, max_tiles, st, tmM, tmO);
        return launch2_as<KIND, EPI_BIAS>(tmA, tmB, p, max_tiles, st, tmM, tmO);
    } else {
        if constexpr (KIND == ROW_BK) {
            if (p.bits_in) return launch2_as<KIND, EPI_BITS>(tmA, tmB, p, max_tiles, st, tmM, tmO);
            if (p.mask) return launch2_as<KIND, EPI_MASK, true>(tmA, tmB, p, max_tiles, st, tmM, tmO);  // mask rows as TMA tiles
        }
        return launch2_as<KIND, EPI_PLAIN>(tmA, tmB, p, max_tiles, st, tmM, tmO);
    }
}

}  // namespace

bool tc_ffn_supported(const moe_config &c) {
    return c.act == MOE_BF16 && c.d % 64 == 0 && c.h % 64 == 0 && c.d >= 64 && c.h >= 64;
}


// The two-CTA kernel's 256 x 256 tiles pay off when the average segment fills them and there are more of them than SMs (cols: the wider
// side of an expert's matrices). A step with all its products on pairs / on one CTA each, us: 4000 rows x 1024 columns
// (64 tiles) 131 / 119, 8000 x 1024 (128) 155 / 152, 9000 x 832 (144) 171 / 166, but 6000 x 2048 (192) 244 / 255, 16384 x 1024 (256)
// 242 / 244, 32000 x 1024 399 / 421.
static bool use_two_cta(int64_t R, int32_t nseg, int32_t flags, int32_t cols) {
    if ((flags & MOE_FLAG_TC_ONE_CTA) || cdiv(R, 256) * cdiv(cols, 256) <= sm_count()) return false;
    return R / (nseg > 0 ? nseg : 1) >= 384;
}

// The last K block of a segment through the segment's own maps: each costs the loading thread a fence, and the call a pass that writes
// them, so that with one or two K blocks to a segment, or few tiles to a CTA, the one-CTA kernel clears the rows in shared memory
// instead (4096 experts x 64 rows: 1070 us, with maps 1187; 256 x 78: 67, 75; but 256 x 188: 93, 82; a step with 20 experts
// x 450 rows of 320 x 832, two tiles a CTA: 165, 170; on SM pairs, where clearing held the tensor cores up for a third of a
// tile, 256 x 512: 192, 138)
static bool wgrad_uses_maps(int64_t R, int32_t nseg, int32_t M, int32_t N, int32_t flags) {
    const int32_t wide = M > N ? M : N, narrow = M > N ? N : M;
    if (short_segments(R, nseg)) return false;
    return use_two_cta(R, nseg, flags, wide) || nseg * cdiv(narrow, BM) * cdiv(wide, BN) >= 4 * (int64_t)sm_count();
}
// The rows of a row product behind a segment's end are read and dropped, or, through the segment's own map, not read. That saves bytes
// of A (half of them where segments are half a tile), but the fence delays the tile: worth it only where a CTA or pair has so many tiles
// that the loads of the ones before cover it. Steps, us: 4096 experts x 64 rows, 110 tiles a CTA, 6440, without 6490; on pairs 256 x 512
// rows, 41 tiles a pair, 1420, without 1430; but 480 x 24 rows, ten tiles a CTA, 386, 374; 32 x 1024 rows, nine a pair, 353, 345; the
// two products alone at 64 x 62 rows 22.7, 16.9. On one CTA a tile longer segments gain too little. cols: the wider side, as in
// use_two_cta
static bool rows_use_maps(int64_t R, int32_t nseg, int32_t flags, int32_t cols) {
    const bool two = use_two_cta(R, nseg, flags, cols);
    if (!two && !short_segments(R, nseg)) return false;
    return (cdiv(R, two ? 256 : BM) + nseg) * cdiv(cols, BN) >= 32 * (int64_t)(two ? sm_count() / 2 : sm_count());
}

int32_t tc_segment_maps(const moe_config &c, SegmentMaps *maps, const void *xs_rows, const void *hid_rows, const void *dys_rows,
                        const void *dz_rows, const void *hid_cols, const void *dys_cols, const void *xs_cols, const void *dz_cols) {
    memset(maps, 0, sizeof(*maps));
    const int64_t R = (int64_t)c.T * c.k, rows = R > 0 ? R : 1;
    auto add = [&](SegmentMap which, const void *p, int64_t cols, int chunks) -> int32_t {
        if (!p) return MOE_OK;
        maps->made[which] = 1;
        return chunks ? map_rows_mnmajor(&maps->base[which], p, rows, cols, chunks) : map_rows_kmajor(&maps->base[which], p, rows, cols);
    };
    // boxes as in tc_row_gemm and tc_wgrad_gemm
    const bool two = use_two_cta(R, c.n, c.flags, c.d > c.h ? c.d : c.h);
    const int b2 = two && c.h >= 256 ? 2 : BN / 64, b1 = two && c.d >= 256 ? 2 : BN / 64;
    if (rows_use_maps(R, c.n, c.flags, c.d > c.h ? c.d : c.h)) {
        MOE_TRY(add(MAP_XS_ROWS, xs_rows, c.d, 0));
        MOE_TRY(add(MAP_HID_ROWS, hid_rows, c.h, 0));
        MOE_TRY(add(MAP_DYS_ROWS, dys_rows, c.d, 0));
        MOE_TRY(add(MAP_DZ_ROWS, dz_rows, c.h, 0));
    }
    if (!wgrad_uses_maps(R, c.n, c.d, c.h, c.flags)) return MOE_OK;
    MOE_TRY(add(MAP_HID_COLS, hid_cols, c.h, 2));
    MOE_TRY(add(MAP_DYS_COLS, dys_cols, c.d, b2));
    MOE_TRY(add(MAP_XS_COLS, xs_cols, c.d, 2));
    return add(MAP_DZ_COLS, dz_cols, c.h, b1);
}

// C[rows, N] = epilogue(A[rows, K] . B_e) over the segments; B_e = W[e] as [K, N] (transposed = false)
// or as [N, K] read transposed (transposed = true).
// Tile table of a ragged row GEMM: tile_prefix[e] = number of tm-row tiles of the segments before e
// (tile_prefix[nseg] = total), and one record per M tile {segment, first row, segment end, 0}; records past
// the last tile carry segment -1. One block.
__global__ void __launch_bounds__(1024) tile_table_kernel(const int32_t *__restrict__ offsets, int32_t n, int32_t tm,
                                                          int32_t max_m, int32_t *__restrict__ tile_prefix,
                                                          int4 *__restrict__ info) {
    wait_previous_kernel();
    __shared__ int32_t warp_sum[32];
    __shared__ int32_t carry;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int32_t base = 0; base < n; base += 1024) {
        const int32_t e = base + threadIdx.x;
        const int32_t v = e < n ? (offsets[e + 1] - offsets[e] + tm - 1) / tm : 0;
        int32_t inc = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t o = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += o;
        }
        if (lane == 31) warp_sum[w] = inc;
        __syncthreads();
        if (w == 0) {
            const int32_t sw = warp_sum[lane];
            int32_t si = sw;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int32_t o = __shfl_up_sync(0xffffffffu, si, off);
                if (lane >= off) si += o;
            }
            warp_sum[lane] = si - sw;
        }
        __syncthreads();
        const int32_t excl = carry + warp_sum[w] + inc - v;
        if (e < n) tile_prefix[e] = excl;
        __syncthreads();
        if (threadIdx.x == 1023) carry = excl + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) tile_prefix[n] = carry;
    __syncthreads();  // the prefix (global memory, this block's own writes) is complete
    const int32_t total = carry;
    for (int32_t mt = threadIdx.x; mt < max_m; mt += 1024) {
        if (mt >= total) { info[mt] = make_int4(-1, 0, 0, 0); continue; }
        int lo = 0, hi = n;  // last e with tile_prefix[e] <= mt (empty segments share a prefix: take the last)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (tile_prefix[mid] <= mt) lo = mid; else hi = mid;
        }
        info[mt] = make_int4(lo, offsets[lo] + (mt - tile_prefix[lo]) * tm, offsets[lo + 1], 0);
    }
}

// ints a tile table needs behind its [nseg + 1] prefix (records are 16 bytes, 16-byte aligned)
int64_t tc_tile_ws_ints(int64_t R, int64_t nseg) { return ((nseg + 1 + 3) & ~(int64_t)3) + 4 * (cdiv(R, 128) + nseg + 1); }
static int4 *tile_info_of(int32_t *tile_prefix, int32_t nseg) {
    return reinterpret_cast<int4 *>(tile_prefix + ((nseg + 1 + 3) & ~3));
}
static int32_t launch_tile_table(const int32_t *offsets, int32_t nseg, int32_t tm, int64_t R, int32_t *tile_prefix,
                                 cudaStream_t st) {
    launch_kernel(tile_table_kernel, 1, 1024, 0, st, offsets, nseg, tm, (int32_t)(cdiv(R, tm) + nseg), tile_prefix,
                                          tile_info_of(tile_prefix, nseg));
    MOE_LAUNCHED();
    return MOE_OK;
}

template <int COLS> __global__ void __launch_bounds__(256) colsum_blocks_final_kernel(const BlockSums a) {
    wait_previous_kernel();
    __shared__ float4 sh[16][16];
    block_sums_final<COLS>(a, blockIdx.x, blockIdx.y, sh);
}

int64_t tc_colsum_part_floats(int64_t R, int32_t nseg, int32_t N) { return (cdiv(R, 128) * 4 + 8 * (int64_t)nseg + 8) * N; }

// colsum_part / colsum_out: if set, out's column sums per segment (a bias gradient) are formed in the epilogue
// and reduced into colsum_out [nseg, N] (sums_left given: that may be left to the caller); colsum_part needs tc_colsum_part_floats(R, nseg, N) floats
int32_t tc_row_gemm(const void *A, const void *W, bool transposed, const int32_t *offsets, int32_t nseg, int64_t R,
                    int32_t N, int32_t K, void *out, const void *bias, const void *mask, int relu,
                    const SegmentPlan &plan, int counter, SegmentMap seg, int32_t *status, cudaStream_t st, int32_t flags,
                    float *colsum_part = nullptr, void *colsum_out = nullptr, uint32_t *bits_out = nullptr,
                    const uint32_t *bits_in = nullptr, BlockSums *sums_left = nullptr) {
    if (R == 0) {
        if (colsum_out) MOE_CUDA(cudaMemsetAsync(colsum_out, 0, sizeof(bf16) * (size_t)nseg * N, st));
        return MOE_OK;
    }
    auto finish = [&](int32_t rc, int32_t G) -> int32_t {
        if (rc != MOE_OK || !colsum_out) return rc;
        const BlockSums sums = {colsum_part, plan.prefix[0], (bf16 *)colsum_out, nseg, N, G};
        if (nseg >= 128 && R <= 128 * (int64_t)nseg) {
            launch_kernel(colsum_blocks_final_kernel<1024>, dim3((unsigned)nseg, (unsigned)cdiv(N, 1024)), 256, 0, st, sums);
        } else if (sums_left) {
            *sums_left = sums;
            return MOE_OK;
        } else {
            launch_kernel(colsum_blocks_final_kernel<64>, dim3((unsigned)nseg, (unsigned)cdiv(N, 64)), 256, 0, st, sums);
        }
        MOE_LAUNCHED();
        return MOE_OK;
    };
    CUtensorMap tmA, tmB;
    MOE_TRY(map_rows_kmajor(&tmA, A, R, K));
    GemmParams p = default_params();
    p.offsets = offsets; p.tile_prefix = plan.prefix[0]; p.tile_info = plan.info;
    p.nseg = nseg; p.M = 0; p.N = N; p.K = K; p.R = R;
    if (rows_use_maps(R, nseg, flags, N > K ? N : K)) p.seg_a = plan.maps_of(seg);
    p.out = (bf16 *)out; p.bias = (const bf16 *)bias; p.mask = (const bf16 *)mask; p.relu = relu; p.status = status;
    p.bits_out = bits_out; p.bits_in = bits_in;
    if (bits_in) p.mask = nullptr;  // the bits replace the element-wise mask tensor
    p.colsum_part = colsum_out ? colsum_part : nullptr;
    if (use_two_cta(R, nseg, flags, N > K ? N : K)) {  // segments long enough to fill 256-row tiles: SM pairs
        if (transposed) MOE_TRY(map_weight_kmajor_half(&tmB, W, nseg, N, K));
        else MOE_TRY(map_weight_mnmajor_half(&tmB, W, nseg, K, N));
        p.sched_counter = plan.counters + counter;  // tiles handed out at run time
        p.sched_table = p.tile_info;
        p.sched_group = (int32_t)cdiv(N, BN);
        const int64_t max_tiles2 = (cdiv(R, 256) + nseg) * cdiv(N, BN);
        CUtensorMap tmO;
        MOE_TRY(map_out_boxes(&tmO, out, R, N));
        if (transposed && mask && !bits_in) {  // the ReLU-mask rows come in as TMA tiles
            CUtensorMap tmM;
            MOE_TRY(map_rows_kmajor(&tmM, mask, R, N));
            return finish(launch2<ROW_BK>(tmA, tmB, p, max_tiles2, st, &tmM, &tmO), 8);
        }
        return finish(transposed ? launch2<ROW_BK>(tmA, tmB, p, max_tiles2, st, nullptr, &tmO)
                                 : launch2<ROW_BMN>(tmA, tmB, p, max_tiles2, st, nullptr, &tmO), 8);
    }
    // Half as wide tiles where whole ones leave half of the SMs without: a handful of tokens, whose time is one tile's loads
    const int64_t rows_of_tiles = cdiv(R, BM) + imin(nseg, R);
    p.tile_n = N > 128 && 2 * rows_of_tiles * cdiv(N, BN) <= sm_count() ? 128 : BN;
    if (transposed) MOE_TRY(map_weight_kmajor(&tmB, W, nseg, N, K, p.tile_n));
    else MOE_TRY(map_weight_mnmajor(&tmB, W, nseg, K, N, p.tile_n));
    const int64_t max_tiles = (cdiv(R, BM) + nseg) * cdiv(N, p.tile_n);
    CUtensorMap tmO;
    MOE_TRY(map_out_boxes(&tmO, out, R, N));
    return finish(transposed ? launch<ROW_BK>(tmA, tmB, p, max_tiles, st, &tmO) : launch<ROW_BMN>(tmA, tmB, p, max_tiles, st, &tmO), 4);
}

// dW[e] [M, N] = A_e^T . B_e, contraction over the rows of segment e; A [R, M], B [R, N].
// plan.sched (if made): the two-CTA kernel hands its tiles out at run time, longest segments first.
int32_t tc_wgrad_gemm(const void *A, const void *B, const int32_t *offsets, int32_t nseg, int64_t R, int32_t M,
                      int32_t N, void *out, int32_t *status, cudaStream_t st, int32_t flags, const SegmentPlan &plan, int counter,
                      SegmentMap seg_a, SegmentMap seg_b) {
    CUtensorMap tmA, tmB;
    GemmParams p = default_params();
    p.offsets = offsets; p.nseg = nseg; p.M = M; p.N = N; p.R = R;
    if (wgrad_uses_maps(R, nseg, M, N, flags)) { p.seg_a = plan.maps_of(seg_a); p.seg_b = plan.maps_of(seg_b); }
    p.out = (bf16 *)out; p.status = status;
    CUtensorMap tmO;  // the experts' matrices as one tall matrix (a 32-row box never straddles two: M is a multiple of 64)
    MOE_TRY(map_out_boxes(&tmO, out, (int64_t)nseg * M, N));
    if (use_two_cta(R, nseg, flags, M > N ? M : N) && M >= 256) {  // SM pairs: 256 x 256 tiles, each CTA stages half of A and half of B
        MOE_TRY(map_rows_mnmajor(&tmA, A, R > 0 ? R : 1, M, 2));
        MOE_TRY(map_rows_mnmajor(&tmB, B, R > 0 ? R : 1, N, 2));
        if (plan.sched) {
            p.sched_counter = plan.counters + counter;
            p.sched_table = plan.sched;
            p.sched_group = (int32_t)(cdiv(M, 256) * cdiv(N, BN));
        }
        return launch2<WGRAD>(tmA, tmB, p, (int64_t)nseg * cdiv(M, 256) * cdiv(N, BN), st, nullptr, &tmO);
    }
    MOE_TRY(map_rows_mnmajor(&tmA, A, R > 0 ? R : 1, M, BM / 64));
    MOE_TRY(map_rows_mnmajor(&tmB, B, R > 0 ? R : 1, N, BN / 64));
    return launch<WGRAD>(tmA, tmB, p, (int64_t)nseg * cdiv(M, BM) * cdiv(N, BN), st, &tmO);
}

int32_t tc_row_tile(int64_t R, int32_t nseg, int32_t flags, int32_t cols) { return use_two_cta(R, nseg, flags, cols) ? 256 : BM; }
bool tc_wgrad_sorted(const moe_config &c) {
    return use_two_cta((int64_t)c.T * c.k, c.n, c.flags, c.d > c.h ? c.d : c.h) && c.n > 1 && c.n <= PLAN_MAX_SORTED;
}

int32_t launch_tc_ffn(const moe_config &c, const void *xs, const int32_t *offsets, const void *W1, const void *b1,
                      const void *W2, const void *b2, void *hid, void *ys, const SegmentPlan &plan, int32_t *status_word,
                      cudaStream_t st, bool first_only, uint32_t *relu_bits) {
    const int64_t R = (int64_t)c.T * c.k;
    MOE_TRY(tc_row_gemm(xs, W1, false, offsets, c.n, R, c.h, c.d, hid, b1, nullptr, 1, plan, first_only ? PLAN_ROWS_AGAIN : PLAN_ROWS_A,
                        MAP_XS_ROWS, status_word, st, c.flags, nullptr, nullptr, relu_bits));
    if (first_only) return MOE_OK;
    return tc_row_gemm(hid, W2, false, offsets, c.n, R, c.d, c.h, ys, b2, nullptr, 0, plan, PLAN_ROWS_B, MAP_HID_ROWS, status_word, st, c.flags);
}

// ------------------------------------------------------------------------------------------
// Gate backward contractions on the tensor cores (no bit-exactness is required there):
//   dW = x^T . dlogit   and   dX_gate = dlogit . [W_g | W_noise]^T
// with the float operands split into three bf16 terms (hi + mid + lo carries 24 mantissa bits), x being
// bf16 already. dsplit is [T, 3 * n2] = (hi | mid | lo) of the [T, n2] logit gradients (n2 = 2n: clean
// columns then raw-noise columns), wsplit is [d, 3 * n2] likewise for [W_g | W_noise].
// ------------------------------------------------------------------------------------------
// ldw: row stride of Wg and Wn in floats (n for two separate [d, n] matrices; 2n when they are the two halves of the
// columns of one [d, 2n] matrix)
__global__ void __launch_bounds__(256) split_weights_kernel(const float *__restrict__ Wg,
                                                            const float *__restrict__ Wn, int32_t d, int32_t n,
                                                            bf16 *__restrict__ wsplit, int32_t ldw) {
    wait_previous_kernel();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t n2 = 2 * n;
    if (i >= (int64_t)d * n2) return;
    const int32_t q = (int32_t)(i / n2), j = (int32_t)(i % n2);
    const float v = j < n ? Wg[(int64_t)q * ldw + j] : Wn[(int64_t)q * ldw + (j - n)];
    const bf16 hi = __float2bfloat16_rn(v);
    const float r1 = v - __bfloat162float(hi);
    const bf16 mid = __float2bfloat16_rn(r1);
    const bf16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
    bf16 *row = wsplit + (int64_t)q * 3 * n2;
    row[j] = hi; row[n2 + j] = mid; row[2 * n2 + j] = lo;
}

// out (group g = blockIdx.y) = sum_c part[c * part_stride + g * d * 2n + .], split into the W_g and W_noise halves
__global__ void __launch_bounds__(256) reduce_partials_kernel(const float *__restrict__ part, int32_t nparts,
                                                              int64_t part_stride, int32_t d, int32_t n,
                                                              float *__restrict__ dWg, float *__restrict__ dWn,
                                                              int32_t ldw) {
    wait_previous_kernel();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t n2 = 2 * n;
    const int64_t total = (int64_t)d * n2;
    if (i >= total) return;
    const int64_t g = blockIdx.y;
    double s = 0.0;
    for (int32_t c = 0; c < nparts; ++c) s += (double)part[(int64_t)c * part_stride + g * total + i];
    const int32_t q = (int32_t)(i / n2), j = (int32_t)(i % n2);
    if (j < n) dWg[(g * d + q) * ldw + j] = (float)s;
    else dWn[(g * d + q) * ldw + (j - n)] = (float)s;
}

__global__ void __launch_bounds__(256) gate_parts_kernel(const GateParts a) {
    wait_previous_kernel();
    gate_parts_sum(a, blockIdx.x);
}

bool tc_gate_bwd_supported(int32_t act, int32_t d, int32_t n) {
    // dX_gate contracts over the 2n logit columns (six split terms each) in one fp32 tensor-core accumulator, which
    // truncates: beyond 2n = 4096 the result drifts past 1e-5 (measured 2e-5 at n = 8192), so very wide flat gates take
    // the fp32 SIMT contractions instead
    return act == MOE_BF16 && d % 64 == 0 && (2 * n) % 64 == 0 && 2 * n <= 4096;
}

// dW of the gate: the contraction over the tokens is cut into row ranges (one float partial per range and precision
// term, added in double afterwards), and inside a range the tensor-core accumulator is restarted every GB_ROWS_HI rows
// for the leading (hi) term: an fp32 accumulator loses low bits when a long run of same-sign terms is added (e.g. the
// gradient of a constant input feature); 128 rows keep that below 1e-5 of the result. The mid and lo terms are 2^-8
// and 2^-16 of the hi term and restart every GB_ROWS_LO rows. The restarts' sums are added in registers (see acc_tile), so only one
// partial per range goes to global memory.
// SM pairs where a tile of theirs is full: on one CTA a 64-row K block brings 48 KiB to an SM for 512 cycles of tensor work, which the L2
// does not deliver (32768 tokens, 512 x 512: 91 us, on pairs 73; 131072, 1024 x 256: 383, 271).
// Ranges: whole waves of tiles. A tile costs its K blocks and about eight more for its 128 KiB of sums, read again later at the copy
// rate; no longer than GB_ROWS_MOST rows unless there are more than three waves of the leading term's tiles.
constexpr int GB_ROWS_HI = 128, GB_ROWS_LO = 2048, GB_ROWS_LEAST = 256, GB_ROWS_MOST = 4096;
static bool gate_bwd_pairs(int32_t d, int32_t n) { return d >= 256 && 2 * n >= 256; }
static void gate_bwd_split(int64_t T, int32_t d, int32_t n, int32_t *nranges, int32_t *rows, int32_t *rows_lo) {
    const bool pairs = gate_bwd_pairs(d, n);
    const int64_t tiles = 3 * cdiv(d, pairs ? 256 : BM) * cdiv(2 * n, BN), workers = pairs ? sm_count() / 2 : sm_count();
    const int64_t most = cdiv(9 * workers, tiles);
    const int64_t rows_most = imax(GB_ROWS_MOST, cdiv(cdiv(T, most), GB_ROWS_HI) * GB_ROWS_HI);
    double least = 0.0;
    for (int64_t w = 1; w <= 9; ++w) {
        const int64_t ranges = imax(1, w * workers / tiles);
        const int64_t r = imin(rows_most, imax(GB_ROWS_LEAST, cdiv(cdiv(T, ranges), GB_ROWS_HI) * GB_ROWS_HI));
        const int64_t made = T > 0 ? cdiv(T, r) : 1, waves = cdiv(made * tiles, workers);
        const double cost = (double)waves * (r / BK + 8) + 12.0 * made * d * 2 * n / 2.2e6;  // K blocks; 2.2 MB are read in the time of one
        if (w == 1 || cost < least) {
            least = cost;
            *rows = (int32_t)r;
            *rows_lo = (int32_t)imin(r, GB_ROWS_LO);
            *nranges = (int32_t)made;
        }
    }
}

int64_t tc_gate_bwd_partials(int64_t T, int32_t d, int32_t n) {
    int32_t nr, rows, rows_lo;
    gate_bwd_split(T, d, n, &nr, &rows, &rows_lo);
    return (int64_t)3 * nr * d * 2 * n;
}

int32_t launch_tc_gate_bwd(const void *x, int64_t T, int32_t d, int32_t n, const float *Wg, const float *Wn,
                           const void *dsplit, void *wsplit, float *partials, float *dWg, float *dWn,
                           float *dX_gate, int32_t *status, cudaStream_t st, int32_t flags, int32_t ldw, GateParts *parts_left) {
    const int32_t n2 = 2 * n;
    if (T == 0 && ldw > 0) {
        for (int32_t q = 0; q < d; ++q) MOE_CUDA(cudaMemsetAsync(dWg + (int64_t)q * ldw, 0, sizeof(float) * n2, st));
        return MOE_OK;
    }
    if (T == 0) {
        MOE_CUDA(cudaMemsetAsync(dWg, 0, sizeof(float) * d * n, st));
        MOE_CUDA(cudaMemsetAsync(dWn, 0, sizeof(float) * d * n, st));
        return MOE_OK;
    }
    launch_kernel(split_weights_kernel, (unsigned)cdiv((int64_t)d * n2, 256), 256, 0, st, Wg, Wn, d, n, (bf16 *)wsplit, ldw > 0 ? ldw : n);
    MOE_LAUNCHED();
    int32_t nr, rows, rows_lo;
    gate_bwd_split(T, d, n, &nr, &rows, &rows_lo);
    {   // dW partials: contraction over the tokens, cut into row ranges, one set per precision term
        CUtensorMap tmA, tmB;
        const bool pairs = gate_bwd_pairs(d, n) && !(flags & MOE_FLAG_TC_ONE_CTA);
        MOE_TRY(map_rows_mnmajor(&tmA, x, T, d, BM / 64));
        MOE_TRY(map_rows_mnmajor(&tmB, dsplit, T, 3 * n2, (pairs ? 128 : BN) / 64));
        GemmParams p = default_params();
        p.nseg = 3 * nr; p.M = d; p.N = n2; p.R = T; p.out_f32 = partials; p.status = status;
        p.segs_term0 = nr; p.rows_per_seg0 = rows;
        p.rows_per_seg = rows; p.segs_per_term = nr; p.b_term_chunks = n2 / 64;
        p.sub_kb0 = GB_ROWS_HI / BK; p.sub_kb = rows_lo / BK; p.interleave = 3;
        if (pairs) MOE_TRY((launch2_as<WGRAD, EPI_F32, false, true>(tmA, tmB, p, (int64_t)p.nseg * cdiv(d, 256) * cdiv(n2, BN), st, nullptr, nullptr)));
        else MOE_TRY(launch_acc_wgrad(tmA, tmB, p, (int64_t)p.nseg * cdiv(d, BM) * cdiv(n2, BN), st));
        const GateParts parts = {partials, 3 * nr, d, n2, n, ldw > 0 ? ldw : n, dWg, dWn};
        if (parts_left) {
            *parts_left = parts;
        } else {
            launch_kernel(gate_parts_kernel, (unsigned)cdiv((int64_t)d * n2, 256), 256, 0, st, parts);
            MOE_LAUNCHED();
        }
    }
    {   // dX_gate: six cross terms of the two split operands, concatenated along the contraction
        CUtensorMap tmA, tmB;
        const bool pairs = T >= 256 * 74 && !(flags & MOE_FLAG_TC_ONE_CTA);  // enough 256-row tiles for every SM pair
        MOE_TRY(map_rows_kmajor(&tmA, dsplit, T, 3 * n2));
        if (pairs) MOE_TRY(map_weight_kmajor_half(&tmB, wsplit, 1, d, 3 * n2));
        else MOE_TRY(map_weight_kmajor(&tmB, wsplit, 1, d, 3 * n2));
        GemmParams p = default_params();
        p.nseg = 1; p.N = d; p.K = n2; p.R = T; p.out_f32 = dX_gate; p.status = status;
        p.nterms = 6;
        const int32_t at[6] = {2, 0, 1, 0, 1, 0}, bt[6] = {0, 2, 1, 1, 0, 0};  // smallest products first
        for (int i = 0; i < 6; ++i) { p.a_term_col[i] = at[i] * n2; p.b_term_col[i] = bt[i] * n2; }
        if (pairs) MOE_TRY(launch2<ROW_BK>(tmA, tmB, p, cdiv(T, 256) * cdiv(d, BN), st));
        else MOE_TRY(launch<ROW_BK>(tmA, tmB, p, cdiv(T, BM) * cdiv(d, BN), st));
    }
    return MOE_OK;
}

// Forward gate projection for the routing screen: clean | raw = x . (W_lo + W_mid + W_hi), smallest term first.
static void two_outputs(GemmParams &p, float *clean, float *raw, int32_t n) {
    p.out_f32 = clean; p.out2 = raw; p.split_n = n;
    p.out_words = ((reinterpret_cast<uintptr_t>(clean) | reinterpret_cast<uintptr_t>(raw)) & 15) != 0;
}
bool tc_gate_fwd_supported(int32_t act, int64_t T, int32_t d, int32_t n, int32_t flags) {
    // MOE_FLAG_GATE_SCREEN_OFF: every token through the fma chain; _ON: screen whenever the shapes allow;
    // neither: screen when the projection is large enough to pay for the extra launches
    if (flags & MOE_FLAG_GATE_SCREEN_OFF) return false;
    if (!(act == MOE_BF16 && d % 64 == 0 && (2 * n) % 64 == 0 && T >= 256)) return false;
    if (flags & MOE_FLAG_GATE_SCREEN_ON) return true;
    return (double)T * d * 2.0 * n >= 1.0e9;
}

int32_t launch_tc_gate_fwd(const void *x, int64_t T, int32_t d, int32_t n, const void *wsplit, float *clean, float *raw,
                           int32_t *status, cudaStream_t st) {
    const int32_t n2 = 2 * n;
    CUtensorMap tmA, tmB;
    MOE_TRY(map_rows_kmajor(&tmA, x, T, d));
    MOE_TRY(map_weight_mnmajor_half(&tmB, wsplit, 1, 3 * (int64_t)d, n2));
    GemmParams p = default_params();
    p.nseg = 1; p.N = n2; p.K = d; p.R = T; p.status = status;
    two_outputs(p, clean, raw, n);
    p.nterms = 3;
    for (int i = 0; i < 3; ++i) { p.a_term_col[i] = 0; p.b_term_col[i] = (2 - i) * d; }
    return launch2<ROW_BMN>(tmA, tmB, p, cdiv(T, 256) * cdiv(n2, BN), st);
}

// The same for the secondary gates of the hierarchical layer: rows = the slots (t, s1) sorted by primary group
// (xs_p [P1, d], offsets_p [a + 1]), one [d, 2b] weight pair per group. wsplit_s [3][a * d][2b] (term, group, feature);
// Sorted row r's logits go to row perm_p[r] of clean / raw [P1, b].
int32_t launch_tc_gate_fwd_grouped(const void *xs_p, int64_t P1, int32_t d, int32_t a, int32_t b, const void *wsplit_s,
                                   const int32_t *offsets_p, int32_t *tile_prefix, const int32_t *perm_p, float *clean, float *raw,
                                   int32_t *status, cudaStream_t st, int32_t flags) {
    if (P1 == 0) return MOE_OK;
    const int32_t n2 = 2 * b;
    const bool pairs = use_two_cta(P1, a, flags, n2 > d ? n2 : d);
    CUtensorMap tmA, tmB;
    MOE_TRY(map_rows_kmajor(&tmA, xs_p, P1, d));
    {   // the group is the map's last coordinate (stride d rows), the precision term an offset of a * d rows along K
        const uint64_t dims[4] = {64, (uint64_t)3 * a * d, (uint64_t)(n2 / 64), (uint64_t)a};
        const uint64_t str[3] = {(uint64_t)n2 * 2, 128, (uint64_t)d * n2 * 2};
        const uint32_t box[4] = {64, BK, pairs ? 2u : (uint32_t)(BN / 64), 1};
        MOE_TRY(make_map(&tmB, wsplit_s, 4, dims, str, box));
    }
    GemmParams p = default_params();
    p.offsets = offsets_p; p.tile_prefix = tile_prefix; p.tile_info = tile_info_of(tile_prefix, a);
    p.nseg = a; p.N = n2; p.K = d; p.R = P1; p.status = status;
    two_outputs(p, clean, raw, b);
    p.out_rows = perm_p;
    p.nterms = 3;
    for (int i = 0; i < 3; ++i) { p.a_term_col[i] = 0; p.b_term_col[i] = (2 - i) * a * d; }  // lo, mid, hi
    const int32_t tm = pairs ? 256 : BM;
    MOE_TRY(launch_tile_table(offsets_p, a, tm, P1, tile_prefix, st));
    const int64_t max_tiles = (cdiv(P1, tm) + a) * cdiv(n2, BN);
    return pairs ? launch2<ROW_BMN>(tmA, tmB, p, max_tiles, st) : launch<ROW_BMN>(tmA, tmB, p, max_tiles, st);
}

// Secondary gates of the hierarchical layer: the slots (t, s1) sorted by primary group are the rows.
// xs_p [P1, d] token rows in sorted order, dsplit_s [P1, 3 * 2b] split logit gradients in sorted order.
bool tc_hier_gate_bwd_supported(int32_t act, int32_t d, int32_t a, int32_t b) {
    return act == MOE_BF16 && d % 64 == 0 && (2 * a) % 64 == 0 && (2 * b) % 64 == 0;
}

int32_t launch_tc_hier_secondary_bwd(const void *xs_p, const void *dsplit_s, void *wsplit_s, const float *Wg_s,
                                     const float *Wn_s, const int32_t *offsets_p, int32_t *tile_prefix, int32_t a,
                                     int64_t P1, int32_t d, int32_t b, float *partials, float *dWg_s, float *dWn_s,
                                     float *dX_sec, int32_t *status, cudaStream_t st) {
    const int32_t n2 = 2 * b;
    launch_kernel(split_weights_kernel, (unsigned)cdiv((int64_t)a * d * n2, 256), 256, 0, st, Wg_s, Wn_s, a * d, b, (bf16 *)wsplit_s, b);
    MOE_LAUNCHED();
    {   // dW_s[i] = sum over the slots of group i of x[token]^T . dlogit[slot], one partial per precision term
        CUtensorMap tmA, tmB;
        MOE_TRY(map_rows_mnmajor(&tmA, xs_p, P1 > 0 ? P1 : 1, d, BM / 64));
        MOE_TRY(map_rows_mnmajor(&tmB, dsplit_s, P1 > 0 ? P1 : 1, 3 * n2, BN / 64));
        GemmParams p = default_params();
        p.offsets = offsets_p; p.nseg = 3 * a; p.off_mod = a; p.b_term_chunks = n2 / 64;
        p.M = d; p.N = n2; p.R = P1; p.out_f32 = partials; p.status = status;
        MOE_TRY(launch<WGRAD>(tmA, tmB, p, (int64_t)p.nseg * cdiv(d, BM) * cdiv(n2, BN), st));
        launch_kernel(reduce_partials_kernel, dim3((unsigned)cdiv((int64_t)d * n2, 256), (unsigned)a), 256, 0, st, 
            partials, 3, (int64_t)a * d * n2, d, b, dWg_s, dWn_s, b);
        MOE_LAUNCHED();
    }
    if (P1 > 0) {   // dX_sec[row] = dlogit[row] . [W_g | W_noise][group]^T, six cross terms
        CUtensorMap tmA, tmB;
        MOE_TRY(map_rows_kmajor(&tmA, dsplit_s, P1, 3 * n2));
        MOE_TRY(map_weight_kmajor(&tmB, wsplit_s, a, d, 3 * n2));
        MOE_TRY(launch_tile_table(offsets_p, a, BM, P1, tile_prefix, st));
        GemmParams p = default_params();
        p.offsets = offsets_p; p.tile_prefix = tile_prefix; p.tile_info = tile_info_of(tile_prefix, a);
        p.nseg = a; p.N = d; p.K = n2; p.R = P1;
        p.out_f32 = dX_sec; p.status = status;
        p.nterms = 6;
        const int32_t at[6] = {2, 0, 1, 0, 1, 0}, bt[6] = {0, 2, 1, 1, 0, 0};
        for (int i = 0; i < 6; ++i) { p.a_term_col[i] = at[i] * n2; p.b_term_col[i] = bt[i] * n2; }
        MOE_TRY(launch<ROW_BK>(tmA, tmB, p, (cdiv(P1, BM) + a) * cdiv(d, BN), st));
    }
    return MOE_OK;
}

int32_t launch_tc_ffn_bwd(const moe_config &c, const void *xs, const void *hid, const void *dys,
                          const int32_t *offsets, const void *W1, const void *W2, void *dxs, void *dW1, void *db1,
                          void *dW2, void *dz, float *colsum, const SegmentPlan &plan, int32_t *status_word,
                          cudaStream_t st, const uint32_t *relu_bits, BlockSums *db1_left) {
    const int64_t R = (int64_t)c.T * c.k;
    MOE_TRY(tc_wgrad_gemm(hid, dys, offsets, c.n, R, c.h, c.d, dW2, status_word, st, c.flags, plan, PLAN_WGRAD_A,
                          MAP_HID_COLS, MAP_DYS_COLS));
    // db1 = column sums of dz, formed in the epilogue of the GEMM that produces dz
    MOE_TRY(tc_row_gemm(dys, W2, true, offsets, c.n, R, c.h, c.d, dz, nullptr, hid, 0, plan, PLAN_ROWS_A, MAP_DYS_ROWS, status_word, st, c.flags,
                        colsum, db1, nullptr, relu_bits, db1_left));
    MOE_TRY(tc_wgrad_gemm(xs, dz, offsets, c.n, R, c.d, c.h, dW1, status_word, st, c.flags, plan, PLAN_WGRAD_B,
                          MAP_XS_COLS, MAP_DZ_COLS));
    return tc_row_gemm(dz, W1, true, offsets, c.n, R, c.d, c.h, dxs, nullptr, nullptr, 0, plan, PLAN_ROWS_B, MAP_DZ_ROWS, status_word, st, c.flags);
}

// ------------------------------------------------------------------------------------------
// The expiry path of the bounded waits, exercised on its own: one thread waits, with the helper the GEMM kernels use,
// on an mbarrier nobody arrives at. Nothing asynchronous is outstanding (no copy, no MMA, no tensor memory), so the
// kernel simply returns once the limit has passed and leaves MOE_ERR_TIMEOUT in the status word.
// ------------------------------------------------------------------------------------------
__global__ void debug_wait_kernel(int32_t *status, unsigned long long limit_ns) {
    wait_previous_kernel();
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int abort_flag;
    abort_flag = 0;
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_wait_limit(smem_u32(&bar), 0, &abort_flag, status, limit_ns);
}

int32_t launch_debug_wait(int32_t *status, unsigned long long limit_ns, cudaStream_t st) {
    launch_kernel(debug_wait_kernel, 1, 1, 0, st, status, limit_ns);
    MOE_LAUNCHED();
    return MOE_OK;
}

MOE_BOUNDS_READER(bounds_violations_ffn)

}  // namespace moe

#ifdef MOE_TILE_TRACE
extern "C" int32_t moe_debug_tile_trace(long long *host_out) {
    return cudaMemcpyFromSymbol(host_out, moe::g_tile_trace, sizeof(moe::g_tile_trace)) == cudaSuccess ? MOE_OK : MOE_ERR_CUDA;
}
#endif
