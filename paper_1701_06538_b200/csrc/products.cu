// Expert feed-forward networks on the 5th-generation tensor cores (Section 3.2, Appendix C): variable-size grouped GEMMs, bf16 operands,
// fp32 accumulation in tensor memory. A persistent kernel whose tiles come from one product or from two that do not need each other:
// hid; ys; dz and dW2; dW1 and dxs.
//
// Kinds of product:
//   ROW_BMN  rows x K activations (K-major A) times a per-expert [K, N] weight (N contiguous, "MN-major" B):
//            hid = relu(xs.W1 + b1),  ys = hid.W2 + b2
//   ROW_BK   same A, per-expert weight read transposed ([N, K], K contiguous, K-major B):
//            dz = (dys.W2^T) * [hid > 0],  dxs = dz.W1^T
//   WGRAD    contraction over the rows of a segment, both operands MN-major:  dW2 = hid^T.dys,  dW1 = xs^T.dz
//
// Two products in one launch fill each other's last wave (a step of 20 experts x 450 rows of 320 x 832: 158 us, this way 143; 32 x 1024
// rows of 512 x 1024: 359, 345). Where CTAs have many tiles these are handed out at run time: with a fixed deal CTAs finish at different
// times (the tiles of a weight gradient differ in length by the ratio of the largest to the smallest expert, and SMs
// do not all run at the same speed: distance to the L2 slices, the two dies). Weight gradients on SM pairs take the
// segments in descending size. Which CTA computes a tile does not change its result: outputs are
// bit-reproducible. (The products of a whole pass in one launch, those that read another's result waiting for counts of stored tiles
// expert by expert, gained nothing more: the counts' way through memory is as long as the gap between two launches, and tiles of four
// products side by side were 17 % slower at 4096 experts x 64 rows than one product behind the other.)
//
// A CTA has one thread or warp for each role: warp 0 bulk tensor copies into 128-byte-swizzled shared memory, warp 1
// tcgen05.mma (accumulators double buffered in tensor memory), warps 2-9 the epilogue (tcgen05.ld, bias / ReLU / mask, round to bf16;
// whole [32][64] boxes leave as bulk tensor stores, boxes cut by a segment end as guarded row stores), warp 10 draws tiles.
// PAIR: a cluster of two CTAs (an SM pair) works on a 256 x 256 tile with cta_group::2; each CTA stages its own 128 rows of A and 128
// columns of B, and has the accumulator of its 128 rows. Otherwise one CTA and 128 x 256 tiles.
// Weights are addressed through one tensor map with the expert as a coordinate, segment bounds are read on the device: no
// per-expert descriptors and no host synchronisation.
//
// Every wait on an mbarrier is bounded (2 s of %globaltimer); on expiry the CTA records MOE_ERR_TIMEOUT in the
// workspace status word, stops issuing work, drains and frees its TMEM.
#include <string.h>

#include <type_traits>

#include "sums.cuh"
#include "tc.cuh"

namespace moe {

namespace {

// What the epilogue does with an accumulator; each product has its own code (with run-time options inside one body every element pair
// became its own basic block)
enum Epilogue { EPI_PLAIN = 0, EPI_BIAS = 1, EPI_BIAS_RELU = 2, EPI_KEEP_BITS = 3, EPI_KEEP_MASK = 4 };
constexpr bool epi_bias(int e) { return e == EPI_BIAS || e == EPI_BIAS_RELU; }
constexpr bool epi_keep(int e) { return e == EPI_KEEP_BITS || e == EPI_KEEP_MASK; }
// The products of a launch are known to its kernel, which then has each one's parameters as constants and only its own code on each path (as
// one body with run-time kinds and options: dz of 256 experts x 512 rows 211 us, this way 156).
enum Set { SET_HID = 0, SET_YS = 1, SET_DZ_DW2 = 2, SET_DZ_DW2_MASK = 3, SET_DW1_DXS = 4 };  // _MASK: the caller has no mask bits
constexpr int set_size(int set) { return set == SET_HID || set == SET_YS ? 1 : 2; }
constexpr Kind set_kind(int set, int i) {
    return set == SET_HID || set == SET_YS ? ROW_BMN : (set == SET_DW1_DXS) == (i == 0) ? WGRAD : ROW_BK;
}
// Registers a thread: as few as do without spills (but for two words of ys on SM pairs), so that a launch's blocks find room beside the last ones of the launch
// before; odd widths have running sums in registers besides
constexpr int most_registers(int set, bool whole) { return !whole ? 168 : set == SET_HID || set == SET_YS ? 128 : 112; }
constexpr Epilogue set_epilogue(int set, int i) {
    if (set == SET_HID) return EPI_BIAS_RELU;
    if (set == SET_YS) return EPI_BIAS;
    return set_kind(set, i) == WGRAD || set == SET_DW1_DXS ? EPI_PLAIN : set == SET_DZ_DW2 ? EPI_KEEP_BITS : EPI_KEEP_MASK;
}
template <int SET, int I = 0, typename F> __device__ __forceinline__ void with_product(int prod, F f) {
    if constexpr (I + 1 == set_size(SET)) f(std::integral_constant<int, I>());
    else if (prod == I) f(std::integral_constant<int, I>());
    else with_product<SET, I + 1>(prod, f);
}
constexpr int MAX_PRODUCTS = 2;

struct Product {
    int32_t N, M;  // output columns; WGRAD: rows of the per-segment output
    int32_t tile_n, tiles_n, per_e, kblocks;  // columns of a tile (256 or 128), tiles beside each other, WGRAD: tiles of a segment, ROW_*: K blocks
    int32_t last_steps;                       // ROW_*: K steps of 16 in the last K block
    Divisor by_tiles_n, by_per_e;
    bf16 *out;                 // ROW_*: [R, N]; WGRAD: [nseg, M, N]
    const bf16 *bias;          // [nseg, N]
    const bf16 *mask;          // EPI_KEEP_MASK: [R, N], the result is kept where mask > 0
    const uint32_t *bits_in;   // EPI_KEEP_BITS: the same as one bit per element, [R, N / 32] words (bit j of word c: column 32 c + j)
    uint32_t *bits_out;        // EPI_BIAS_RELU: such bits of the result, or nullptr
    float *colsum_part;        // EPI_KEEP_*: column sums of the stored values over each warp's 32 rows, [32-row block][N]
    const CUtensorMap *seg_a, *seg_b;  // one map per segment that ends with it, for the box that reaches beyond; or nullptr
};
struct Products {
    Product p[MAX_PRODUCTS];
    int32_t nseg, max_row_tiles;
    const int32_t *offsets;   // [nseg + 1] segment bounds (rows)
    const int32_t *by_rank;   // [nseg + 1] row tiles of the segments before, in the order of `sched`
    const int4 *info;         // per row tile, in that order: {segment, first row, segment end, number of the tile}
    const int4 *sched;        // {segment, first row, end row, 0} in descending size, or nullptr: as they lie
    int32_t *counter;         // tiles drawn so far; nullptr: all are dealt
    int32_t *status;
    int64_t R;
};
struct ProductMaps { CUtensorMap a[MAX_PRODUCTS], b[MAX_PRODUCTS], out[MAX_PRODUCTS]; };

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

// Epilogue arithmetic of one thread's 32 accumulator columns: bias, ReLU, ReLU mask, rounding to bf16
template <int EPI>
__device__ __forceinline__ void pack32(const uint32_t (&v)[32], const uint4 (&bias_raw)[4], uint4 (&packed)[4], uint32_t keep_word) {
    const uint32_t *bw = reinterpret_cast<const uint32_t *>(bias_raw);
    uint32_t *out = reinterpret_cast<uint32_t *>(packed);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        float x0 = __uint_as_float(v[2 * j]), x1 = __uint_as_float(v[2 * j + 1]);
        if (epi_bias(EPI)) { x0 += __uint_as_float(bw[j] << 16); x1 += __uint_as_float(bw[j] & 0xffff0000u); }
        if (epi_keep(EPI)) {
            if (!((keep_word >> (2 * j)) & 1u)) x0 = 0.0f;
            if (!((keep_word >> (2 * j + 1)) & 1u)) x1 = 0.0f;
        }
        __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
        if (EPI == EPI_BIAS_RELU) h = __hmax2(h, __float2bfloat162_rn(0.0f));  // rounding keeps the sign: the same value as max before rounding
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
template <bool WHOLE> __device__ __forceinline__ void bias_load(const bf16 *bias, int32_t columns, uint4 (&out)[2][4]) {  // columns: that exist
#pragma unroll
    for (int q = 0; q < 8; ++q) out[q >> 2][q & 3] = WHOLE || 8 * q < columns ? reinterpret_cast<const uint4 *>(bias)[q] : make_uint4(0u, 0u, 0u, 0u);
}
// mask bits of a lane's row, 128 columns from col0 on (two boxes), as far as the row has them
__device__ __forceinline__ void keep_load(const Product &p, int64_t row, int32_t col0, uint2 (&keep)[2]) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
        if (col0 + 64 * u < p.N) keep[u] = *reinterpret_cast<const uint2 *>(p.bits_in + row * (p.N >> 5) + ((col0 + 64 * u) >> 5));
}
// The same from the masking tensor itself (callers without bits): the warp reads its 32 rows' 128 columns, half a warp a row, turns the
// eight values of a load into a byte, and passes the bytes through `box` to the lanes that own the rows.
__device__ __forceinline__ void keep_from_mask(const Product &p, int64_t row0, int32_t rows_valid, int32_t col0, int lane, uint8_t *box, uint2 (&keep)[2]) {
    const int32_t col = col0 + (lane & 15) * 8;
    const bool in_row = col < p.N;  // N is a multiple of eight
    const bf16 *src = p.mask + row0 * p.N + col;
    const __nv_bfloat162 zero = __float2bfloat162_rn(0.0f);
    uint4 v[16];  // all in flight together: the accumulator's registers are free yet
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int32_t r = 2 * i + (lane >> 4);
        v[i] = in_row && r < rows_valid ? *reinterpret_cast<const uint4 *>(src + (int64_t)r * p.N) : make_uint4(0u, 0u, 0u, 0u);
    }
    if (lane == 0) tma_store_wait_read();  // an earlier store may still be reading the box
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const __nv_bfloat162 *w = reinterpret_cast<const __nv_bfloat162 *>(&v[i]);
        uint32_t m = 0u;  // bit j: element 2 j, bit 16 + j: element 2 j + 1
#pragma unroll
        for (int j = 0; j < 4; ++j) m |= __hgt2_mask(w[j], zero) & (0x00010001u << j);
        box[(2 * i + (lane >> 4)) * 16 + (lane & 15)] = (uint8_t)(spread_bits(m & 0xffffu) | (spread_bits(m >> 16) << 1));
    }
    __syncwarp();
    const uint4 w = *reinterpret_cast<const uint4 *>(box + lane * 16);
    keep[0] = make_uint2(w.x, w.y);
    keep[1] = make_uint2(w.z, w.w);
    __syncwarp();
}

// One [32 rows][64 columns] box of an output tile, by one warp (a lane owns a row): tensor memory -> bias / ReLU / mask ->
// bf16 -> global memory. With eight epilogue warps an SM sub-partition has two to hide the latencies of this chain, so a
// box is taken whole: both 32-column loads are in flight together and everything behind them has twice the independent
// work (with 32-column steps the epilogue of a 256 x 256 tile took 8500 cycles, against 4900 of tensor work at K = 512).
// Whole boxes leave as bulk tensor stores through one of the warp's 4 KiB pieces of shared memory (rows of 128 bytes, 16-byte pieces
// swizzled by row); boxes cut by a segment end as guarded row stores.
struct BoxArgs {
    const CUtensorMap *tm_out;
    uint8_t *box;
    int64_t out_off, row0;      // output row of lane 0 is row0 of the matrix that starts at element out_off
    int32_t rows_valid, col0;
    int32_t map_row;            // the same row in the output's tensor map
    int64_t colsum_row;
    const bf16 *next_bias;      // of the warp's next box, or nullptr
    uint2 keep;                 // mask bits
};
__device__ __forceinline__ void load_box(uint32_t taddr, uint32_t (&v)[2][32]) {
    tc_ld_32x32(taddr, v[0]);
    tc_ld_32x32(taddr + 32, v[1]);
    tc_ld_wait();
}
template <int EPI, int BOXES, bool WHOLE> __device__ __forceinline__ void epilogue_box(const Product &p, int lane, const BoxArgs &b, uint4 (&bias)[2][4], const uint32_t (&v)[2][32]) {
    const bool row_ok = lane < b.rows_valid, staged = b.rows_valid >= 32;
    const int64_t out_row = b.row0 + lane;
    uint8_t *mine = b.box + lane * 128;
    uint4 packed[2][4];
#pragma unroll
    for (int u = 0; u < 2; ++u) pack32<EPI>(v[u], bias[u], packed[u], u ? b.keep.y : b.keep.x);
    if (epi_bias(EPI) && b.next_bias) bias_load<WHOLE>(b.next_bias, p.N - b.col0 - 64, bias);
    if (EPI == EPI_BIAS_RELU && p.bits_out && row_ok)
        *reinterpret_cast<uint2 *>(p.bits_out + out_row * (p.N >> 5) + (b.col0 >> 5)) =
            make_uint2(positive_bits(packed[0]), positive_bits(packed[1]));
    if (staged) {
        if (lane == 0) {  // an earlier store may still be reading the box
            if (BOXES > 1) tma_store_wait_read_but_one();
            else tma_store_wait_read();
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q) *reinterpret_cast<uint4 *>(mine + ((q ^ (lane & 7)) << 4)) = packed[q >> 2][q & 3];
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
            tma_store_2d(b.tm_out, smem_u32(b.box), b.col0, b.map_row);
            tma_store_commit();
        }
        if (epi_keep(EPI)) {
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
            if (WHOLE || b.col0 + 2 * lane < p.N)
                *reinterpret_cast<float2 *>(p.colsum_part + b.colsum_row * p.N + b.col0 + 2 * lane) = make_float2(s0 + u0, s1 + u1);
            __syncwarp();  // read before the next box overwrites this one
        }
        return;
    }
    if (row_ok) {
        uint4 *dst = reinterpret_cast<uint4 *>(p.out + b.out_off + out_row * p.N + b.col0);
        if (WHOLE) {
#pragma unroll
            for (int q = 0; q < 4; ++q) st_global_32B(dst + 2 * q, packed[q >> 1][2 * (q & 1)], packed[q >> 1][2 * (q & 1) + 1]);
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (b.col0 + 8 * q < p.N) dst[q] = packed[q >> 2][q & 3];
        }
    }
    if (epi_keep(EPI)) {  // sums of the rounded values, rows past the segment end count as 0; the whole warp: shuffles
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float a[32];
            const uint32_t *pw = reinterpret_cast<const uint32_t *>(packed[u]);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                a[2 * j] = row_ok ? __uint_as_float(pw[j] << 16) : 0.0f;
                a[2 * j + 1] = row_ok ? __uint_as_float(pw[j] & 0xffff0000u) : 0.0f;
            }
            const float s = warp_column_sums(a, lane);
            if (WHOLE || b.col0 + 32 * u + lane < p.N) p.colsum_part[b.colsum_row * p.N + b.col0 + 32 * u + lane] = s;
        }
    }
}

// ------------------------------------------------------------------------------------------ tiles
struct Tile {
    int32_t e, row0, row_end;  // segment; ROW_*: first row of the tile, WGRAD: of the segment; end of the segment
    int32_t prod;              // which product
    int32_t mt, n0, m0;        // ROW_*: number of the row tile; first output column; WGRAD: first output row
};
// The place of a tile id as two words: {segment, row0, row_end, product}, {mt, n0, m0, 0}; segment -1: behind the last tile. row_tiles: of all segments
template <bool PAIR, int SET> __device__ __forceinline__ void find_tile(const Products &P, int32_t id, int32_t row_tiles, int4 &a, int4 &b) {
    constexpr int TM = PAIR ? 256 : 128;
    b = make_int4(0, 0, 0, 0);
    auto inside = [&](auto I_) {
        constexpr int I = decltype(I_)::value;
        constexpr bool wgrad = set_kind(SET, I) == WGRAD;
        const Product &p = P.p[I];
        const int32_t tiles = wgrad ? P.nseg * p.per_e : row_tiles * p.tiles_n;
        int32_t rest, tn;
        if (!wgrad) {  // asked for before the number of tiles is there: one way to memory less in front of a CTA's first tile
            const int32_t t = p.by_tiles_n(id, tn);
            a = P.info[min(t, P.max_row_tiles - 1)];
        }
        if (id >= tiles) {
            id -= tiles;
            a = make_int4(-1, 0, 0, 0);
            return false;
        }
        if (wgrad) {
            const int32_t r = p.by_per_e(id, rest);
            a = P.sched ? P.sched[r] : make_int4(r, P.offsets[r], P.offsets[r + 1], 0);
            b.z = p.by_tiles_n(rest, tn) * TM;
        } else {
            b.x = a.w;
        }
        b.y = tn * p.tile_n;
        a.w = I;
        MOE_BOUNDS_NOTE(a.x >= 0 && a.x < P.nseg && a.y >= 0 && a.y <= a.z && (int64_t)a.z <= P.R);
        return true;
    };
    if (!inside(std::integral_constant<int, 0>()) && set_size(SET) > 1) inside(std::integral_constant<int, set_size(SET) - 1>());
}

// The first tile of a CTA or pair is dealt and looked up by every role. The following ones are drawn by a thread that keeps a few records ahead
// of the other roles, in a ring in shared memory (PAIR: of both CTAs). A record with segment -1 ends the sequence. What it takes to
// find a tile (a counter in memory, the tile's record) is off the other roles' paths.
// Three records, drawn when a slot is free: what is drawn early is missing elsewhere in the last wave. Tiles of one or two K blocks, which
// the operand loads have to be further ahead of: four, and one id more (4096 experts x 64 rows, a step 6520 us, with three 6560).
template <bool SHORT> constexpr int ring_slots() { return SHORT ? 4 : 3; }
template <bool PAIR, bool SHORT, int SET> struct TileRing {
    static constexpr int RING = ring_slots<SHORT>();
    const Products &P;
    const uint32_t ring, full0, empty0;
    volatile int *abort_flag;
    const bool warp_wide, arrives;  // all 32 lanes of the warp call next() together; this thread reports the slot as read
    int i;
    __device__ __forceinline__ TileRing(const Products &P_, uint32_t bars, volatile int *abort_, bool warp_wide_, bool arrives_)
        : P(P_), ring(bars + 256), full0(bars + 128), empty0(bars + 160), abort_flag(abort_), warp_wide(warp_wide_),
          arrives(arrives_), i(-1) {}
    __device__ __forceinline__ bool next(Tile &t) {
        if (i < 0) {
            int4 a, b;
            find_tile<PAIR, SET>(P, PAIR ? blockIdx.x >> 1 : blockIdx.x, P.by_rank[P.nseg], a, b);
            return set(t, a, b);
        }
        const uint32_t slot = (uint32_t)i % RING, par = ((uint32_t)i / RING) & 1u, full = full0 + 8u * slot;
        if (!mbar_wait(full, par, abort_flag, P.status)) return false;
        if (PAIR) mbar_try_wait_cluster(full, par);  // acquire at cluster scope: the record came from the other CTA's thread
        // The slot is overwritten once every reader has reported it read, so a reader's copy has to be in its registers
        // before its report leaves. The report is a relaxed arrive (a release at cluster scope would wait for the thread's
        // earlier output stores, 3 % of a step), which by itself orders nothing: with an ordinary load the assembler was
        // free to fetch the record again later instead of keeping it in registers, and one warp then now and again worked on the
        // record of four tiles ahead. Hence volatile loads (issued once, where they stand) and an arrive whose address
        // is computed from the loaded words of all lanes (sign bits that are always 0), which cannot issue before
        // those loads have returned.
        int4 a, b;
        asm volatile("ld.volatile.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w)
                     : "r"(ring + 32u * slot) : "memory");
        asm volatile("ld.volatile.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                     : "r"(ring + 32u * slot + 16u) : "memory");
        uint32_t seen = (uint32_t)a.w | (uint32_t)b.w;
        if (warp_wide) seen = __reduce_or_sync(0xffffffffu, seen);
        const uint32_t empty = empty0 + 8u * slot + ((seen >> 31) << 3);
        if (arrives) {
            if (PAIR) mbar_arrive_leader_relaxed(empty);
            else mbar_arrive(empty);
        }
        return set(t, a, b);
    }

  private:
    __device__ __forceinline__ bool set(Tile &t, const int4 &a, const int4 &b) {
        ++i;
        t.e = a.x; t.row0 = a.y; t.row_end = a.z; t.prod = a.w;
        t.mt = b.x; t.n0 = b.y; t.m0 = b.z;
        return a.x >= 0;
    }
};

// Weight gradients of other widths than multiples of 64 are summed in tensor memory over 8 K blocks, 512 rows, and these sums added in registers: a tensor
// core's accumulator drops low bits at every step of 16, over many rows more than the rounding of the result hides. Error of dW1 and dW2 against 64 bits (2-norms), as
// sums of multiply-adds, in one accumulator and this way, in 1e-3: 60000 rows of 264 x 136 1.651 and 1.589, 1.653 and 1.596, 1.651 and 1.589; 400000 of 72 x 40 1.563
// and 1.645, 1.705 and 1.947, 1.563 and 1.645. A warp has the sums of one box, so a tile of a longer segment is done 128 columns at a time; where segments are that
// long on average the tiles are that wide from the start. A backward call, us, in one accumulator and this way: 4 experts x 15000 rows of 200 x 136 301, 226; 64 x 200 of
// 72 x 2056 107, 109; 8 x 3750 of 1000 x 2008 660, 724 (by multiply-adds 9750).
constexpr int SUM_BLOCKS = 8;
template <bool WHOLE, Kind KIND> __device__ __forceinline__ bool in_parts(const Tile &t) { return !WHOLE && KIND == WGRAD && t.row_end - t.row0 > SUM_BLOCKS * BK; }

// PAIR: the two CTAs' shares of a tile
template <bool PAIR> constexpr int tile_rows() { return PAIR ? 256 : 128; }
template <bool PAIR> constexpr int stage_bytes() { return A_BYTES + (PAIR ? 128 : BN) * BK * 2; }
template <bool PAIR, int NST> constexpr int box_count() { return NST == (PAIR ? 6 : 4) ? 1 : 2; }  // staging pieces of an epilogue warp
template <bool PAIR, int NST> constexpr int data_bytes() { return NST * stage_bytes<PAIR>() + 8 * 4096 * box_count<PAIR, NST>(); }
template <bool PAIR, int NST> constexpr int shared_bytes() { return data_bytes<PAIR, NST>() + 1024 /*alignment*/ + 384 /*barriers, ring*/; }

// WHOLE: all widths are multiples of 64. Otherwise of eight, and one CTA: MN-major operands come in chunk by chunk through maps of the whole width, what lies
// behind it reads as zero and is not stored.
template <bool PAIR, int NST, int SET, bool WHOLE>
__global__ void __maxnreg__(most_registers(SET, WHOLE)) expert_products_kernel(const __grid_constant__ ProductMaps maps, const __grid_constant__ Products P) {
    constexpr bool SHORT = !PAIR && NST == 3;
    constexpr int RING = ring_slots<SHORT>(), BOXES = box_count<PAIR, NST>(), STAGE = stage_bytes<PAIR>(), TM = tile_rows<PAIR>();
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;  // 1024-B aligned for the 128-B swizzle
    uint8_t *smem = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bars = base + data_bytes<PAIR, NST>();
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (NST + s); };
    auto tfull_bar = [&](int a) { return bars + 8u * (2 * NST + a); };
    auto tempty_bar = [&](int a) { return bars + 8u * (2 * NST + 2 + a); };
    const uint32_t ring_full0 = bars + 128, ring_empty0 = bars + 160, ring = bars + 256;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + data_bytes<PAIR, NST>() + 192);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + data_bytes<PAIR, NST>() + 200);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;  // 0: issues the MMAs, owns the full / tempty / ring_empty barriers

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), PAIR ? 16 : 8); }
        // readers of a record: producer and 8 epilogue warps in each CTA, the MMA warp of the even one
        for (int q = 0; q < RING; ++q) { mbar_init(ring_full0 + 8u * q, 1); mbar_init(ring_empty0 + 8u * q, PAIR ? 19 : 10); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.a[0]) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.b[0]) : "memory");
    }
    if (warp == 1) {
        if (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void *)tmem_slot)),
                         "r"((uint32_t)TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void *)tmem_slot)),
                         "r"((uint32_t)TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync_all();  // both CTAs' barriers exist before anything is signalled across the pair
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    wait_previous_kernel();  // barriers and tensor memory are set up while the previous kernel drains

    if (warp == 0) {
        // ------------------------------------------------------------------ bulk tensor copies (both CTAs)
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            TileRing<PAIR, SHORT, SET> tiles(P, bars, abort_flag, false, true);
            Tile t;
            while (ok && tiles.next(t)) {
              with_product<SET>(t.prod, [&](auto I_) {
                constexpr int I = decltype(I_)::value;
                constexpr Kind KIND = set_kind(SET, I);
                const Product &p = P.p[I];
                const CUtensorMap *tm_a = &maps.a[I], *tm_b = &maps.b[I];
                const int width = in_parts<WHOLE, KIND>(t) ? 128 : p.tile_n;  // columns of a pass over the contraction
                const uint32_t bytes = PAIR ? 2 * STAGE : A_BYTES + width * BK * 2;
                auto stage = [&](auto load) {  // load(A's place, B's place, barrier) of one K block
                    ok = mbar_wait(empty_bar(s), ph ^ 1u, abort_flag, P.status);
                    if (!ok) return;
                    if (rank == 0) mbar_expect_tx(full_bar(s), bytes);
                    load(base + s * STAGE, base + s * STAGE + A_BYTES, full_bar(s));
                    if (++s == NST) { s = 0; ph ^= 1u; }
                };
                auto load_2d = [&](uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1) {
                    if (PAIR) tma2_load_2d(dst, tm, bar, c0, c1);
                    else tma_load_2d(dst, tm, bar, c0, c1);
                };
                auto load_3d = [&](uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1, int c2) {
                    if (PAIR) tma2_load_3d(dst, tm, bar, c0, c1, c2);
                    else tma_load_3d(dst, tm, bar, c0, c1, c2);
                };
                auto load_4d = [&](uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1, int c2, int c3) {
                    if (PAIR) tma2_load_4d(dst, tm, bar, c0, c1, c2, c3);
                    else tma_load_4d(dst, tm, bar, c0, c1, c2, c3);
                };
                if constexpr (KIND == WGRAD) {
                    const int kblocks = (t.row_end - t.row0 + BK - 1) / BK;
                    // the last block of rows through the segment's own maps, where they are made
                    const bool ragged = p.seg_a && (t.row_end - t.row0) % BK != 0;
                    if (ragged) { acquire_map(p.seg_a + t.e); acquire_map(p.seg_b + t.e); }
                    const int ca = t.m0 / 64 + 2 * (int)rank, cb = t.n0 / 64 + 2 * (int)rank;
                    auto pass = [&](int32_t n0) {
                        for (int kb = 0; kb < kblocks && ok; ++kb) {
                            const bool tail = ragged && kb == kblocks - 1;
                            const int r = t.row0 + kb * BK;
                            stage([&](uint32_t a, uint32_t b, uint32_t bar) {
                                if (WHOLE) {
                                    load_3d(a, tail ? p.seg_a + t.e : tm_a, bar, 0, r, ca);
                                    load_3d(b, tail ? p.seg_b + t.e : tm_b, bar, 0, r, cb);
                                } else {
                                    for (int c = 0; c < BM / 64; ++c) tma_load_2d(a + c * (BK * 128), tm_a, bar, t.m0 + 64 * c, r);
                                    for (int c = 0; c < width / 64; ++c) tma_load_2d(b + c * (BK * 128), tm_b, bar, n0 + 64 * c, r);
                                }
                            });
                        }
                    };
                    if constexpr (WHOLE) pass(t.n0);
                    else
                        for (int32_t n0 = t.n0; n0 < min(t.n0 + p.tile_n, p.N) && ok; n0 += width) pass(n0);
                } else {
                    const int kblocks = p.kblocks, row = t.row0 + 128 * (int)rank;
                    if (p.seg_a && row + 128 > t.row_end) {
                        tm_a = p.seg_a + t.e;
                        acquire_map(tm_a);
                    }
                    if constexpr (KIND == ROW_BMN) {
                        const int cb = t.n0 / 64 + 2 * (int)rank;
                        for (int kb = 0; kb < kblocks && ok; ++kb)
                            stage([&](uint32_t a, uint32_t b, uint32_t bar) {
                                load_2d(a, tm_a, bar, kb * BK, row);
                                if (WHOLE) load_4d(b, tm_b, bar, 0, kb * BK, cb, t.e);
                                else for (int c = 0; c < p.tile_n / 64; ++c) tma_load_3d(b + c * (BK * 128), tm_b, bar, t.n0 + 64 * c, kb * BK, t.e);
                            });
                    } else {
                        const int cb = t.n0 + 128 * (int)rank;
                        for (int kb = 0; kb < kblocks && ok; ++kb)
                            stage([&](uint32_t a, uint32_t b, uint32_t bar) {
                                load_2d(a, tm_a, bar, kb * BK, row);
                                load_3d(b, tm_b, bar, kb * BK, cb, t.e);
                            });
                    }
                }
              });
            }
            // drain: every copy this thread started must have landed before the CTA may exit
            if (!ok && !PAIR)
                for (int q = 0; q < NST; ++q) {
                    const unsigned long long t0 = global_ns();
                    while (!mbar_try_wait(full_bar(q), 0) && !mbar_try_wait(full_bar(q), 1) && global_ns() - t0 < WAIT_LIMIT_NS) {}
                }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (even CTA only)
        // PAIR: one thread runs the whole loop. Otherwise the whole warp, which may have rows to clear (see below).
        if (rank == 0 && (!PAIR || lane == 0)) {
            int s = 0, acc = 0;
            uint32_t ph = 0, acc_ph = 0;
            bool ok = true;
            TileRing<PAIR, SHORT, SET> tiles(P, bars, abort_flag, !PAIR, lane == 0);
            Tile t;
            while (ok && tiles.next(t)) {
              with_product<SET>(t.prod, [&](auto I_) {
                constexpr int I = decltype(I_)::value;
                constexpr Kind KIND = set_kind(SET, I);
                constexpr bool wgrad = KIND == WGRAD;
                const Product &p = P.p[I];
                const int kblocks = wgrad ? (t.row_end - t.row0 + BK - 1) / BK : p.kblocks;
                if (kblocks == 0) return;  // empty segment (WGRAD): the epilogue writes zeros
                constexpr int a_mn = wgrad ? 1 : 0, b_mn = KIND == ROW_BK ? 0 : 1;
                // a K step of 16 advances the start address (low descriptor bits, in 16-byte units) by 32 bytes in a
                // K-major tile and by 16 rows of 128 bytes in an MN-major one; the sum never leaves the address field
                constexpr uint64_t a_step = a_mn ? (16 * 128) >> 4 : 32 >> 4, b_step = b_mn ? (16 * 128) >> 4 : 32 >> 4;
                const int tail = wgrad ? (t.row_end - t.row0) - (kblocks - 1) * BK : BK;  // rows of the last block
                const bool parts = in_parts<WHOLE, KIND>(t);
                auto pass = [&](int32_t n0, int width) {
                    // one CTA: columns behind the output's are not computed
                    const uint32_t idesc = PAIR ? make_idesc2(a_mn, b_mn) : make_idesc(a_mn, b_mn, min(width, WHOLE ? p.N - n0 : (p.N - n0 + 15) & ~15));
                    const int part_blocks = parts ? SUM_BLOCKS : kblocks;
                    for (int part = 0; part < kblocks; part += part_blocks) {
                        ok = mbar_wait(tempty_bar(acc), acc_ph ^ 1u, abort_flag, P.status);
                        if (!ok) return;
                        tc_fence_after();
                        const uint32_t d_tmem = tmem_base + acc * BN;
                        const int part_end = parts ? min(kblocks, part + SUM_BLOCKS) : kblocks;
                        for (int kb = part; kb < part_end; ++kb) {
                            ok = mbar_wait(full_bar(s), ph, abort_flag, P.status);
                            if (!ok) break;
                            tc_fence_after();
                            const uint32_t a_src = base + s * STAGE, b_src = a_src + A_BYTES;
                            // K steps of 16 rows to issue for this block: none that lies behind the segment's end
                            const int ksteps = kb < kblocks - 1 || (WHOLE && !wgrad) ? BK / 16 : wgrad ? (tail + 15) / 16 : p.last_steps;
                            if (!PAIR && wgrad && kb == kblocks - 1 && !p.seg_a && ksteps * 16 > tail) {
                                // Without the segments' own maps (see wgrad_uses_maps) the rows behind the end, up to the end of the step that holds
                                // it, are the next segment's: zeroed in A AND in B (0 x finite = 0 would do for finite data; both keep a
                                // non-finite value of the next segment out of this segment's sums): 128-B lines in all 64-column
                                // chunks, the A tile's two chunks directly followed by the B tile's four. Eight lanes a line of one chunk,
                                // four lines at a time (as one loop over all lines, with a division for each, this was 1450 cycles a tile of 64 rows)
                                uint8_t *z = smem + s * STAGE + (tail + (lane >> 3)) * 128 + (lane & 7) * 16;
                                for (int r = lane >> 3; r < ksteps * 16 - tail; r += 4, z += 4 * 128)
#pragma unroll
                                    for (int chunk = 0; chunk < (BM + BN) / 64; ++chunk)
                                        *reinterpret_cast<uint4 *>(z + chunk * (BK * 128)) = make_uint4(0, 0, 0, 0);
                                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                                __syncwarp();
                            }
                            if (PAIR || lane == 0) {
                                const uint64_t ad = a_mn ? desc_mnmajor(a_src) : desc_kmajor(a_src), bd = b_mn ? desc_mnmajor(b_src) : desc_kmajor(b_src);
#pragma unroll
                                for (int k = 0; k < BK / 16; ++k) {
                                    if (k >= ksteps) break;
                                    if (PAIR) tc_mma2_bf16(d_tmem, ad + k * a_step, bd + k * b_step, idesc, (kb > part || k > 0) ? 1u : 0u);
                                    else tc_mma_bf16(d_tmem, ad + k * a_step, bd + k * b_step, idesc, (kb > part || k > 0) ? 1u : 0u);
                                }
                                if (PAIR) tc_commit2(empty_bar(s));  // the stage may be refilled once these MMAs have read it
                                else tc_commit(empty_bar(s));
                            }
                            if (!PAIR) __syncwarp();
                            if (++s == NST) { s = 0; ph ^= 1u; }
                        }
                        if (ok && (PAIR || lane == 0)) {  // accumulator complete
                            if (PAIR) tc_commit2(tfull_bar(acc));
                            else tc_commit(tfull_bar(acc));
                        }
                        if (!PAIR) __syncwarp();
                        if (!ok) return;
                        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
                    }
                };
                if constexpr (WHOLE || !wgrad) {
                    pass(t.n0, p.tile_n);
                } else {
                    const int width = parts ? 128 : p.tile_n;
                    for (int32_t n0 = t.n0; n0 < min(t.n0 + p.tile_n, p.N) && ok; n0 += width) pass(n0, width);
                }
              });
            }
        }
    } else if (warp == 10) {
        // ------------------------------------------------------------------ drawing tiles (even CTA, one thread)
        if (rank == 0 && lane == 0) {
            const uint32_t peer_ring = PAIR ? peer_smem_addr(ring, 1) : 0u, peer_full0 = PAIR ? peer_smem_addr(ring_full0, 1) : 0u;
            const int32_t workers = PAIR ? gridDim.x >> 1 : gridDim.x;
            const int32_t row_tiles = P.by_rank[P.nseg];
            int32_t dealt = PAIR ? blockIdx.x >> 1 : blockIdx.x, ahead = SHORT && P.counter ? atomicAdd(P.counter, 1) : 0;
            bool ok = true;
            for (int i = 0; ok; ++i) {
                const uint32_t slot = (uint32_t)i % RING;
                if (i >= RING) {  // every reader of the record this slot held has its copy
                    const uint32_t par = ((uint32_t)i / RING - 1) & 1u;
                    ok = mbar_wait(ring_empty0 + 8u * slot, par, abort_flag, P.status);
                    if (!ok) break;
                    if (PAIR) mbar_try_wait_cluster(ring_empty0 + 8u * slot, par);
                }
                int32_t id = dealt += workers;
                if (P.counter) {
                    id = workers + (SHORT ? ahead : atomicAdd(P.counter, 1));  // the first tiles are dealt
                    if (SHORT) ahead = atomicAdd(P.counter, 1);
                }
                int4 a, b;
                find_tile<PAIR, SET>(P, id, row_tiles, a, b);
                const uint32_t at = ring + 32u * slot;
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w) : "memory");
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + 16u), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
                if (PAIR) {
                    st_cluster_v4(peer_ring + 32u * slot, a);
                    st_cluster_v4(peer_ring + 32u * slot + 16u, b);
                }
                mbar_arrive(ring_full0 + 8u * slot);
                if (PAIR) mbar_arrive_cluster_addr(peer_full0 + 8u * slot);
                if (a.x < 0) break;
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
        // Two warps share each quarter of the accumulator's rows and take half of its columns each, in boxes of 64.
        const int quarter = warp & 3, half = (warp - 2) >> 2;  // TMEM lanes 32*quarter .. 32*quarter + 31 belong to this warp
        uint8_t *boxes_at = smem + NST * STAGE + (warp - 2) * (4096 * BOXES);
        int acc = 0, turn = 0;
        uint32_t acc_ph = 0;
        bool ok = true;
        TileRing<PAIR, SHORT, SET> tiles(P, bars, abort_flag, true, lane == 0);
        Tile t;
        while (ok && tiles.next(t)) {
            with_product<SET>(t.prod, [&](auto I_) {
                constexpr int I = decltype(I_)::value;
                constexpr int EPI = set_epilogue(SET, I);
                constexpr bool wgrad = set_kind(SET, I) == WGRAD;
                const Product &p = P.p[I];
                const bool have_acc = !wgrad || t.row_end > t.row0;
                const int32_t first = t.n0 + half * (p.tile_n / 2);
                const int boxes = min(p.tile_n / 128, max(0, (WHOLE ? p.N - first : p.N - first + 63) / 64));
                BoxArgs b;
                b.tm_out = &maps.out[I];
                b.out_off = wgrad ? (int64_t)t.e * p.M * p.N : 0;
                b.row0 = (wgrad ? t.m0 : t.row0) + 128 * (int)rank + quarter * 32;
                b.rows_valid = (wgrad ? p.M : t.row_end) - (int32_t)b.row0;
                b.map_row = (int32_t)b.row0 + (wgrad ? t.e * p.M : 0);
                b.colsum_row = PAIR ? (t.mt * 2 + (int)rank) * 4 + quarter : t.mt * 4 + quarter;
                uint4 bias[2][4];
                const bf16 *bias_at = nullptr;
                if (epi_bias(EPI)) {
                    bias_at = p.bias + (int64_t)t.e * p.N + first;
                    if (boxes > 0) bias_load<WHOLE>(bias_at, p.N - first, bias);
                }
                uint2 keep[2] = {make_uint2(0u, 0u), make_uint2(0u, 0u)};
                if (EPI == EPI_KEEP_BITS && lane < b.rows_valid) keep_load(p, b.row0 + lane, first, keep);
                if (EPI == EPI_KEEP_MASK) keep_from_mask(p, b.row0, b.rows_valid, first, lane, boxes_at, keep);
                auto release = [&]() {  // the warp's part of the accumulator is in registers: the buffer goes back
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if (PAIR) mbar_arrive_leader_relaxed(tempty_bar(acc));
                        else mbar_arrive(tempty_bar(acc));
                    }
                };
                const uint32_t mine = tmem_base + ((uint32_t)(quarter * 32) << 16) + half * (p.tile_n / 2);
                auto begin = [&](int u) {  // box u, ahead of its loads
                    b.col0 = first + 64 * u;
                    b.next_bias = epi_bias(EPI) && u + 1 < boxes ? bias_at + 64 : nullptr;
                    b.keep = u ? keep[1] : keep[0];
                    b.box = boxes_at + (BOXES > 1 ? turn * 4096 : 0);
                    if (b.rows_valid >= 32) turn ^= 1;  // (else nothing is stored from the box)
                };
                if (in_parts<WHOLE, set_kind(SET, I)>(t)) {  // sums of SUM_BLOCKS K blocks, added in registers: a box a warp and 128 columns
                    for (int32_t n0 = t.n0; n0 < min(t.n0 + p.tile_n, p.N); n0 += 128) {
                        uint32_t v[2][32];
                        float sum[2][32];
#pragma unroll
                        for (int j = 0; j < 64; ++j) sum[j >> 5][j & 31] = 0.0f;
                        for (int r = t.row0; r < t.row_end; r += SUM_BLOCKS * BK) {
                            ok = mbar_wait(tfull_bar(acc), acc_ph, abort_flag, P.status);
                            if (!ok) return;
                            tc_fence_after();
                            load_box(tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + half * 64, v);
                            release();
#pragma unroll
                            for (int j = 0; j < 64; ++j) sum[j >> 5][j & 31] += __uint_as_float(v[j >> 5][j & 31]);
                            if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
                        }
#pragma unroll
                        for (int j = 0; j < 64; ++j) v[j >> 5][j & 31] = __float_as_uint(sum[j >> 5][j & 31]);
                        if (n0 + half * 64 < p.N) {
                            begin(0);
                            b.col0 = n0 + half * 64;
                            epilogue_box<EPI, BOXES, WHOLE>(p, lane, b, bias, v);
                        }
                    }
                } else {
                    if (have_acc) {  // (the loads above are in flight while the warp waits for its accumulator)
                        ok = mbar_wait(tfull_bar(acc), acc_ph, abort_flag, P.status);
                        if (!ok) return;
                        tc_fence_after();
                    }
                    for (int u = 0; u < boxes; ++u) {
                        uint32_t v[2][32];
                        begin(u);
                        if (have_acc) {
                            load_box(mine + acc * BN + 64 * u, v);
                            if (u + 1 == boxes) release();
                        } else {
#pragma unroll
                            for (int j = 0; j < 64; ++j) v[j >> 5][j & 31] = 0u;
                        }
                        epilogue_box<EPI, BOXES, WHOLE>(p, lane, b, bias, v);
                    }
                    if (have_acc) {
                        if (boxes == 0) release();
                        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
                    }
                }
            });
        }
        if (lane == 0) tma_store_wait_all();  // no bulk store may outlive the CTA's shared memory
    }

    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync_all();  // the pair's MMAs read both CTAs' shared memory: leave together
    if (warp == 1) {
        tc_fence_after();
        if (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
    }
}

// ------------------------------------------------------------------------------------------ host
// bf16 output rows as [32][64] boxes
int32_t map_out_boxes(CUtensorMap *tm, const void *p, int64_t rows, int64_t cols) {
    const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows}, str[1] = {(uint64_t)cols * 2};
    const uint32_t box[2] = {64, 32};
    return tc_make_map(tm, p, 2, dims, str, box);
}

// SM pairs' 256 x 256 tiles pay off when the average segment fills them and there are more of them than SMs (cols: the wider
// side of an expert's matrices). A step with all its products on pairs / on one CTA each, us: 4000 rows x 1024 columns
// (64 tiles) 131 / 119, 8000 x 1024 (128) 155 / 152, 9000 x 832 (144) 171 / 166, but 6000 x 2048 (192) 244 / 255, 16384 x 1024 (256)
// 242 / 244, 32000 x 1024 399 / 421.
bool use_pairs(int64_t R, int32_t nseg, int32_t flags, int32_t cols) {
    if ((flags & MOE_FLAG_TC_ONE_CTA) || cdiv(R, 256) * cdiv(cols, 256) <= tc_sm_count()) return false;
    return R / (nseg > 0 ? nseg : 1) >= 384;
}
bool whole(const moe_config &c) { return c.d % 64 == 0 && c.h % 64 == 0; }
bool use_pairs(const moe_config &c) { return whole(c) && use_pairs((int64_t)c.T * c.k, c.n, c.flags, c.d > c.h ? c.d : c.h); }
// one or two K blocks in the average segment of a weight gradient
bool short_segments(int64_t R, int32_t nseg) { return R < 128 * (int64_t)nseg; }

// The last K block of a segment through the segment's own maps: each costs the loading thread a fence, and the call a pass that writes
// them, so that with one or two K blocks to a segment, or few tiles to a CTA, the one-CTA kernel clears the rows in shared memory
// instead (4096 experts x 64 rows: 1070 us, with maps 1187; 256 x 78: 67, 75; but 256 x 188: 93, 82; a step with 20 experts
// x 450 rows of 320 x 832, two tiles a CTA: 165, 170; on SM pairs, where clearing held the tensor cores up for a third of a
// tile, 256 x 512: 192, 138)
bool wgrad_uses_maps(const moe_config &c) {
    const int64_t R = (int64_t)c.T * c.k;
    const int32_t wide = c.d > c.h ? c.d : c.h, narrow = c.d > c.h ? c.h : c.d;
    if (use_pairs(c)) return true;
    if (!whole(c) || short_segments(R, c.n)) return false;
    return c.n * cdiv(narrow, BM) * cdiv(wide, BN) >= 4 * (int64_t)tc_sm_count();
}
// The rows of a row product behind a segment's end are read and dropped, or, through the segment's own map, not read. That saves bytes
// of A (half of them where segments are half a tile), but the fence delays the tile: worth it only where a CTA or pair has so many tiles
// that the loads of the ones before cover it. Steps, us: 4096 experts x 64 rows, 110 tiles a CTA, 6440, without 6490; on pairs 256 x 512
// rows, 41 tiles a pair, 1420, without 1430; but 480 x 24 rows, ten tiles a CTA, 386, 374; 32 x 1024 rows, nine a pair, 353, 345; the
// two products alone at 64 x 62 rows 22.7, 16.9. On one CTA a tile longer segments gain too little.
bool rows_use_maps(const moe_config &c) {
    const int64_t R = (int64_t)c.T * c.k;
    const bool pairs = use_pairs(c);
    if (!whole(c) || (!pairs && !short_segments(R, c.n))) return false;
    return (cdiv(R, pairs ? 256 : BM) + c.n) * cdiv(c.d > c.h ? c.d : c.h, BN) >= 32 * (int64_t)(pairs ? tc_sm_count() / 2 : tc_sm_count());
}

template <bool PAIR, int NST, int SET, bool WHOLE> int32_t launch_products_as(const ProductMaps &maps, const Products &P, int64_t tiles, cudaStream_t st) {
    static PerDevice slots;  // CTAs or pairs that run at once
    const auto kernel = expert_products_kernel<PAIR, NST, SET, WHOLE>;
    constexpr int SHARED = shared_bytes<PAIR, NST>();
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_kernel
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = 2; attrs[1].val.clusterDim.y = 1; attrs[1].val.clusterDim.z = 1;
    cfg.blockDim = dim3(NTHREADS_DRAW); cfg.dynamicSmemBytes = SHARED; cfg.stream = st;
    cfg.attrs = attrs; cfg.numAttrs = PAIR ? 2 : 1;
    const int most = slots.get([&]() {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED) != cudaSuccess) return 0;
        if (!PAIR) return tc_sm_count();
        int n = 0;
        cfg.gridDim = dim3(2 * (tc_sm_count() / 2));
        return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess ? n : 0;
    });
    if (most <= 0) return MOE_ERR_CUDA;
    if (tiles <= 0) return MOE_OK;
    cfg.gridDim = dim3((PAIR ? 2 : 1) * (unsigned)imin(tiles, most));
    MOE_CUDA(cudaLaunchKernelEx(&cfg, kernel, maps, P));
    MOE_LAUNCHED();
    return MOE_OK;
}

// The products of one launch
class ProductList {
    const moe_config &c;
    const SegmentPlan &plan;
    const int64_t R;
    const bool pairs, row_maps, wgrad_maps;
    const int tm;
    int64_t tiles = 0, product_tiles[MAX_PRODUCTS];
    int count = 0;
    int32_t *drawn;
    ProductMaps maps;

  public:
    Products P;
    ProductList(const moe_config &c_, const SegmentPlan &plan_, const int32_t *offsets, PlanCounter counter, int32_t *status)
        : c(c_), plan(plan_), R((int64_t)c_.T * c_.k), pairs(use_pairs(c_)), row_maps(rows_use_maps(c_)), wgrad_maps(wgrad_uses_maps(c_)),
          tm(pairs ? 256 : BM) {
        memset(&maps, 0, sizeof(maps));
        memset(&P, 0, sizeof(P));
        P.nseg = c.n; P.max_row_tiles = (int32_t)(cdiv(R, tm) + c.n); P.offsets = offsets; P.by_rank = plan.by_rank; P.info = plan.info; P.sched = plan.sched;
        drawn = plan.counters + counter; P.status = status; P.R = R;
    }
    // out [R, N] = epilogue(A [R, K] . W[e]), W[e] as [K, N], or [N, K] read transposed
    int32_t row(Product **made, const void *A, const void *W, bool transposed, int32_t N, int32_t K, void *out, SegmentMap seg) {
        Product &p = P.p[count];
        p.N = N; p.kblocks = (int32_t)cdiv(K, BK); p.last_steps = (int32_t)cdiv(K - (p.kblocks - 1) * BK, 16);
        // Half as wide tiles where whole ones leave half of the SMs without: a handful of tokens, whose time is one tile's loads
        const int64_t row_tiles = cdiv(R, tm) + imin(c.n, R);
        p.tile_n = !pairs && N > 128 && 2 * row_tiles * cdiv(N, BN) <= tc_sm_count() ? 128 : BN;
        p.tiles_n = (int32_t)cdiv(N, p.tile_n);
        p.by_tiles_n = Divisor::of(p.tiles_n);
        p.out = (bf16 *)out;
        if (row_maps) p.seg_a = plan.maps_of(seg);
        const int box_n = pairs ? 128 : p.tile_n;
        MOE_TRY(tc_map_rows_kmajor(&maps.a[count], A, R, K, BM));
        if (transposed) MOE_TRY(tc_map_weight_kmajor(&maps.b[count], W, c.n, N, K, box_n));
        else if (!whole(c)) MOE_TRY(tc_map_weight_kmajor(&maps.b[count], W, c.n, K, N, BK));  // (64 columns of 64 rows)
        else MOE_TRY(tc_map_weight_mnmajor(&maps.b[count], W, c.n, K, N, box_n));
        MOE_TRY(map_out_boxes(&maps.out[count], out, R, N));
        add((cdiv(R, tm) + c.n) * p.tiles_n);
        *made = &p;
        return MOE_OK;
    }
    // out[e] [M, N] = A_e^T . B_e, contraction over the rows of segment e; A [R, M], B [R, N]
    int32_t wgrad(const void *A, const void *B, int32_t M, int32_t N, void *out, SegmentMap seg_a, SegmentMap seg_b) {
        Product &p = P.p[count];
        p.N = N; p.M = M;
        p.tile_n = whole(c) || R < SUM_BLOCKS * BK * (int64_t)c.n ? BN : 128;  // (see SUM_BLOCKS)
        p.tiles_n = (int32_t)cdiv(N, p.tile_n); p.per_e = (int32_t)cdiv(M, tm) * p.tiles_n;
        p.by_tiles_n = Divisor::of(p.tiles_n); p.by_per_e = Divisor::of(p.per_e);
        p.out = (bf16 *)out;
        if (wgrad_maps) { p.seg_a = plan.maps_of(seg_a); p.seg_b = plan.maps_of(seg_b); }
        if (whole(c)) {
            MOE_TRY(tc_map_rows_mnmajor(&maps.a[count], A, R, M, 2));
            MOE_TRY(tc_map_rows_mnmajor(&maps.b[count], B, R, N, pairs ? 2 : BN / 64));
        } else {
            MOE_TRY(tc_map_rows_kmajor(&maps.a[count], A, R, M, BK));
            MOE_TRY(tc_map_rows_kmajor(&maps.b[count], B, R, N, BK));
        }
        // the experts' matrices as one tall matrix (a box that is stored whole has 32 rows of its expert)
        MOE_TRY(map_out_boxes(&maps.out[count], out, (int64_t)c.n * M, N));
        add((int64_t)c.n * p.per_e);
        return MOE_OK;
    }
    // of two products that were added the one: the other one has no tiles
    void only(int which) {
        Product &other = P.p[1 - which];
        tiles = product_tiles[which];
        other.tiles_n = other.per_e = 0;
    }
    template <int SET> int32_t launch(cudaStream_t st) {
        if (tiles >= ((int64_t)1 << 31) - ((int64_t)1 << 22)) return MOE_ERR_UNSUPPORTED;
        // Pairs draw their tiles. Single CTAs do with many tiles each (4096 experts x 64 rows, 166 and more a CTA: a step 6550 us, dealt
        // 6680); with few the thread that draws is ahead by a good part of them (256 x 78 rows, 10 and 28 a CTA: 576, dealt 570; a step of
        // 256 x 188 rows 1289, dealt 1273)
        P.counter = pairs || tiles > 64 * (int64_t)tc_sm_count() ? drawn : nullptr;
        if (!whole(c)) {
            if constexpr (SET != SET_DZ_DW2 && SET != SET_HID) return launch_products_as<false, 4, SET, false>(maps, P, tiles, st);
            return MOE_ERR_UNSUPPORTED;  // (no bits without whole words; hid: api.cu)
        }
        if (pairs) return launch_products_as<true, 6, SET, true>(maps, P, tiles, st);
        // Weight gradients of one or two K blocks a tile last as long as their epilogue, 1100 cycles a box, 420 of them waiting until the
        // store before had read the box out: a warp's boxes take turns in two 4 KiB pieces, for one operand stage less (4096 experts x
        // 64 rows, a product: 1056 and 1087 us -> 981 to 1012 and 1056 to 1076, 256 x 78 rows 61 -> 58). With three K blocks a tile the stage is
        // worth more (256 x 188 rows 83 -> 86). Sixteen epilogue warps, eight an accumulator, were no faster than the second box.
        if constexpr (set_size(SET) > 1) {
            if (short_segments(R, c.n)) return launch_products_as<false, 3, SET, true>(maps, P, tiles, st);
        }
        return launch_products_as<false, 4, SET, true>(maps, P, tiles, st);
    }

  private:
    void add(int64_t n) {
        tiles += n;
        product_tiles[count++] = n;
    }
};

}  // namespace

bool tc_ffn_supported(const moe_config &c) {
    return c.act == MOE_BF16 && c.d % 64 == 0 && c.h % 64 == 0 && c.d >= 64 && c.h >= 64;
}

// All bf16 layers: their widths are multiples of eight (a configuration's rows are whole 16-byte vectors). us a step of widths that are no multiples of 64 by
// FP32 multiply-adds and this way (hid stays with them, see api.cu): 64 experts x 200 rows of 72 x 2056 1257, 368; 20 x 300 of 120 x 1000 396, 165;
// 32 x 500 of 200 x 200 452, 181.
bool tc_ffn_takes(const moe_config &c) { return c.act == MOE_BF16; }

int32_t tc_segment_maps(const moe_config &c, SegmentMaps *maps, const void *xs_rows, const void *hid_rows, const void *dys_rows,
                        const void *dz_rows, const void *hid_cols, const void *dys_cols, const void *xs_cols, const void *dz_cols) {
    memset(maps, 0, sizeof(*maps));
    const int64_t R = (int64_t)c.T * c.k, rows = R > 0 ? R : 1;
    auto add = [&](SegmentMap which, const void *p, int64_t cols, int chunks) -> int32_t {
        if (!p) return MOE_OK;
        maps->made[which] = 1;
        return chunks ? tc_map_rows_mnmajor(&maps->base[which], p, rows, cols, chunks) : tc_map_rows_kmajor(&maps->base[which], p, rows, cols, BM);
    };
    if (rows_use_maps(c)) {
        MOE_TRY(add(MAP_XS_ROWS, xs_rows, c.d, 0));
        MOE_TRY(add(MAP_HID_ROWS, hid_rows, c.h, 0));
        MOE_TRY(add(MAP_DYS_ROWS, dys_rows, c.d, 0));
        MOE_TRY(add(MAP_DZ_ROWS, dz_rows, c.h, 0));
    }
    if (!wgrad_uses_maps(c)) return MOE_OK;
    const int b = use_pairs(c) ? 2 : BN / 64;  // boxes as in ProductList
    MOE_TRY(add(MAP_HID_COLS, hid_cols, c.h, 2));
    MOE_TRY(add(MAP_DYS_COLS, dys_cols, c.d, b));
    MOE_TRY(add(MAP_XS_COLS, xs_cols, c.d, 2));
    return add(MAP_DZ_COLS, dz_cols, c.h, b);
}

int32_t tc_row_tile(const moe_config &c) { return use_pairs(c) ? 256 : BM; }
bool tc_wgrad_sorted(const moe_config &c) { return use_pairs(c) && c.n > 1 && c.n <= PLAN_MAX_SORTED; }
bool tc_use_pairs(int64_t R, int32_t nseg, int32_t flags, int32_t cols) { return use_pairs(R, nseg, flags, cols); }

int32_t launch_tc_ffn(const moe_config &c, const void *xs, const int32_t *offsets, const void *W1, const void *b1,
                      const void *W2, const void *b2, void *hid, void *ys, const SegmentPlan &plan, int32_t *status_word,
                      cudaStream_t st, bool first_only, uint32_t *relu_bits) {
    if ((int64_t)c.T * c.k == 0) return MOE_OK;
    ProductList hidden(c, plan, offsets, PLAN_HID, status_word);
    Product *p;
    MOE_TRY(hidden.row(&p, xs, W1, false, c.h, c.d, hid, MAP_XS_ROWS));
    p->bias = (const bf16 *)b1; p->bits_out = relu_bits;
    MOE_TRY(hidden.launch<SET_HID>(st));
    return first_only ? MOE_OK : launch_tc_ys(c, offsets, W2, b2, hid, ys, plan, status_word, st);
}
int32_t launch_tc_ys(const moe_config &c, const int32_t *offsets, const void *W2, const void *b2, const void *hid, void *ys, const SegmentPlan &plan,
                     int32_t *status_word, cudaStream_t st) {
    if ((int64_t)c.T * c.k == 0) return MOE_OK;
    ProductList out(c, plan, offsets, PLAN_YS, status_word);
    Product *p;
    MOE_TRY(out.row(&p, hid, W2, false, c.d, c.h, ys, MAP_HID_ROWS));
    p->bias = (const bf16 *)b2;
    return out.launch<SET_YS>(st);
}

template <int COLS> __global__ void __launch_bounds__(256) colsum_blocks_final_kernel(const BlockSums a) {
    wait_previous_kernel();
    __shared__ float4 sh[16][16];
    block_sums_final<COLS>(a, blockIdx.x, blockIdx.y, sh);
}

int64_t tc_colsum_part_floats(int64_t R, int32_t nseg, int32_t N) { return (cdiv(R, 128) * 4 + 8 * (int64_t)nseg + 8) * N; }

int32_t launch_tc_ffn_bwd(const moe_config &c, const void *xs, const void *hid, const void *dys, const int32_t *offsets, const void *W1,
                          const void *W2, void *dxs, void *dW1, void *db1, void *dW2, void *dz, float *colsum, const SegmentPlan &plan,
                          int32_t *status_word, cudaStream_t st, const uint32_t *relu_bits, BlockSums *db1_left) {
    const int64_t R = (int64_t)c.T * c.k, w = (int64_t)c.n * c.d * c.h;
    if (R == 0) {
        MOE_CUDA(cudaMemsetAsync(dW1, 0, sizeof(bf16) * w, st));
        MOE_CUDA(cudaMemsetAsync(dW2, 0, sizeof(bf16) * w, st));
        MOE_CUDA(cudaMemsetAsync(db1, 0, sizeof(bf16) * (size_t)c.n * c.h, st));
        return MOE_OK;
    }
    ProductList by_w2(c, plan, offsets, PLAN_DZ_DW2, status_word), by_w1(c, plan, offsets, PLAN_DW1_DXS, status_word);
    Product *p;
    MOE_TRY(by_w2.row(&p, dys, W2, true, c.h, c.d, dz, MAP_DYS_ROWS));
    p->mask = (const bf16 *)hid; p->bits_in = relu_bits;
    p->colsum_part = colsum;  // db1 = column sums of dz, formed in the epilogue of the product that makes dz
    MOE_TRY(by_w2.wgrad(hid, dys, c.h, c.d, dW2, MAP_HID_COLS, MAP_DYS_COLS));
    if (relu_bits) MOE_TRY(by_w2.launch<SET_DZ_DW2>(st));
    else MOE_TRY(by_w2.launch<SET_DZ_DW2_MASK>(st));
    auto by_w1_products = [&](ProductList &list) -> int32_t {
        MOE_TRY(list.wgrad(xs, dz, c.d, c.h, dW1, MAP_XS_COLS, MAP_DZ_COLS));
        return list.row(&p, dz, W1, true, c.d, c.h, dxs, MAP_DZ_ROWS);
    };
    MOE_TRY(by_w1_products(by_w1));
    const int64_t xs_bytes = R * c.d * (int64_t)sizeof(bf16);
    if (overlap(xs, xs_bytes, dxs, xs_bytes)) {  // the caller has no use for xs any more: dxs waits until dW1 has read it
        ProductList after(c, plan, offsets, PLAN_DXS, status_word);
        MOE_TRY(by_w1_products(after));
        by_w1.only(0);
        after.only(1);
        MOE_TRY(by_w1.launch<SET_DW1_DXS>(st));
        MOE_TRY(after.launch<SET_DW1_DXS>(st));
    } else {
        MOE_TRY(by_w1.launch<SET_DW1_DXS>(st));
    }
    const BlockSums sums = {colsum, plan.prefix[0], offsets, (bf16 *)db1, c.n, c.h, tc_row_tile(c) / 32, tc_row_tile(c)};
    if (c.n >= 128 && R <= 128 * (int64_t)c.n) {
        launch_kernel(colsum_blocks_final_kernel<1024>, dim3((unsigned)c.n, (unsigned)cdiv(c.h, 1024)), 256, 0, st, sums);
    } else if (db1_left) {
        *db1_left = sums;
        return MOE_OK;
    } else {
        launch_kernel(colsum_blocks_final_kernel<64>, dim3((unsigned)c.n, (unsigned)cdiv(c.h, 64)), 256, 0, st, sums);
    }
    MOE_LAUNCHED();
    return MOE_OK;
}

MOE_BOUNDS_READER(bounds_violations_products)

}  // namespace moe
