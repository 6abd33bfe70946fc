// Dense and grouped products of the gates on the 5th-generation tensor cores: bf16 operands (float ones as three bf16 terms), fp32
// accumulation in tensor memory, float results. The forward projections of the routing screen, and the gate backward's contractions.
//
// One persistent kernel template, one CTA per SM, 128 x 256 output tiles, K blocks of 64:
//   warp 0      TMA producer: one bulk tensor copy per operand per stage into 128-byte-swizzled
//               shared memory, completion counted on an mbarrier (4 stages)
//   warp 1      MMA issuer: tcgen05.mma (cta_group::1, kind::f16, M 128, N 256, K 16), accumulator
//               in TMEM, double buffered (2 x 256 columns) so the epilogue of one tile overlaps
//               the main loop of the next; tcgen05.commit releases the stage / publishes the tile
//   warps 2-9   epilogue: tcgen05.ld (32 lanes x 32 columns per instruction), 128-byte row segments through shared memory
//
// Three operand arrangements (KIND):
//   ROW_BMN  rows x K activations (K-major A) times a [K, N] weight (N contiguous, "MN-major" B), one per group of rows: the screen's products
//   ROW_BK   same A, weight read transposed ([N, K], K contiguous, K-major B): dX_gate = dlogit.[W_g | W_noise]^T
//   WGRAD    contraction over rows, both operands MN-major: dW = x^T.dlogit
// The experts' own products are in products.cu.
//
// Every wait on an mbarrier is bounded (2 s of %globaltimer); on expiry the CTA records
// MOE_ERR_TIMEOUT in the workspace status word, stops issuing work, drains and frees its TMEM.
#include <stdlib.h>
#include <string.h>

#include <type_traits>

#include "sums.cuh"
#include "tc.cuh"

namespace moe {

namespace {

constexpr int MAX_TERMS = 8;

struct GemmParams {
    const int32_t *offsets;      // [nseg + 1] segment bounds (rows); nullptr = uniform segments
    const int32_t *tile_prefix;  // ROW_* with offsets: [nseg + 1] prefix of the M tiles
    const int4 *tile_info;       // ROW_* with offsets: per M tile {segment or -1, first row, segment end, 0}
    // set by the launchers: N tiles per row of tiles, WGRAD tiles per segment, number of tile ids, K blocks of a ROW tile
    int32_t tiles_n, per_e, total_tiles, kblocks_row;
    Divisor by_tiles_n, by_per_e, by_mod, by_terms, by_interleave;  // tiles_n, per_e, off_mod, segs_per_term, interleave
    int32_t nseg;
    int32_t M;  // WGRAD: rows of the per-segment output; ROW_*: unused
    int32_t N;  // output columns
    int32_t K;  // ROW_*: contraction length of one term; WGRAD: unused (segment rows)
    float *out_f32;  // ROW_*: [R, N]; WGRAD: [nseg, M, N]
    // results of two matrices side by side: columns from split_n on go to out2, both with rows of split_n (a multiple of 32);
    // out_rows: where an output row goes (rows sorted by group); out_words: rows that do not start on 16 bytes
    float *out2;
    const int32_t *out_rows;
    int32_t split_n, out_words;
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
    // ROW_*: the contraction is the concatenation of nterms pieces of length K; piece i reads A
    // columns a_term_col[i] + [0, K) and B columns b_term_col[i] + [0, K)
    int32_t nterms;
    int32_t a_term_col[MAX_TERMS], b_term_col[MAX_TERMS];
};

// One [32 rows][64 columns] box of an output tile, by one warp (a lane owns a row): tensor memory -> global memory by way of the warp's 4 KiB of
// shared memory, 128-byte row segments at a time. A box is taken whole, so that both 32-column loads are in flight together.
// release() hands the accumulator back; it is called once the box is in registers.
struct BoxArgs {
    uint8_t *box;
    uint32_t taddr;             // tensor-memory address of the box
    int64_t out_off, row0;      // output row of lane 0 is row0 of the matrix that starts at element out_off
    int32_t rows_valid, col0;
    bool have_acc;
};
template <typename Release>
__device__ __forceinline__ void epilogue_box(const GemmParams &p, int lane, const BoxArgs &b, Release release) {
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
    const int my_piece = lane & 7, my_sub = lane >> 3;  // lane l moves piece l % 8 of row 4 * i + l / 8
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
        t.n0 = tn * BN;
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
        t.n0 = tn * BN;
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
// ACC (WGRAD with float output over long uniform row ranges, the gate backward): the contraction of a tile is cut
// into sub-blocks of p.sub_kb0 / p.sub_kb K blocks (first term / other terms). Each sub-block is accumulated in TMEM on
// its own (an fp32 tensor-core accumulator truncates, and a long run of same-sign terms loses low bits: 128 rows keep
// that below 1e-5), handed to the epilogue like a tile, and added there, with rounding to nearest, to running sums in
// registers (a lane's row of the warp's 128 columns; the cap of 168 registers makes the compiler spill 96 bytes of other
// values, 132 on SM pairs); the sums go to global memory once per tile. (With the sums in shared memory, which left room for two operand
// stages, a K block took 1850 cycles: the latency of its loads.)
template <int KIND, bool ACC = false>
__global__ void __launch_bounds__(NTHREADS, 1)
grouped_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;  // 1024-B aligned for the 128-B swizzle
    uint8_t *smem = smem_raw + (base - smem_u32(smem_raw));
    constexpr int NST = STAGES;
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
                for (int kb = 0; kb < t.kblocks && ok; ++kb) {
                    ok = mbar_wait(empty_bar(s), ph ^ 1u, abort_flag, p.status);
                    if (!ok) break;
                    const uint32_t a_dst = base + s * STAGE_BYTES, b_dst = a_dst + A_BYTES;
                    mbar_expect_tx(full_bar(s), A_BYTES + BN * BK * 2);
                    if (KIND == WGRAD) {
                        const int r = t.row0 + kb * BK;
                        tma_load_3d(a_dst, &tmA, full_bar(s), 0, r, t.m0 / 64);
                        tma_load_3d(b_dst, &tmB, full_bar(s), 0, r, t.b_chunk);
                    } else {
                        tma_load_2d(a_dst, &tmA, full_bar(s), p.a_term_col[term] + kk, t.row0);
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
            const uint32_t idesc = make_idesc(KIND == WGRAD ? 1 : 0, KIND == ROW_BK ? 0 : 1, min(BN, p.N - t.n0));
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
                    // The rows behind the end, up to the end of the step that holds it, are the next segment's: zeroed in A AND in B (0 x finite = 0 would do for finite data; both keep a
                    // non-finite value of the next segment out of this segment's sums): 128-B lines in all 64-column
                    // chunks, the A tile's two chunks directly followed by the B tile's four.
                    if (p.offsets && nz > 0) {
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
        int acc = 0;
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
            const int32_t first = t.n0 + half * (BN / 2);
            const int boxes = min(2, max(0, (p.N - first) / 64));  // N is a multiple of 64
            BoxArgs b;
            b.out_off = KIND == WGRAD ? (int64_t)t.e * p.M * p.N : 0;
            b.row0 = (KIND == WGRAD ? t.m0 : t.row0) + quarter * 32;
            b.rows_valid = (KIND == WGRAD ? p.M : t.row_end) - (int32_t)b.row0;
            b.have_acc = have_acc;
            b.box = smem + NST * STAGE_BYTES + 1024 + (warp - 2) * 4096;
            if (have_acc) {
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
                b.taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + half * (BN / 2) + 64 * u;
                epilogue_box(p, lane, b, [&]() { if (u + 1 == boxes) release(); });
            }
            if (have_acc) {
                if (boxes == 0) release();
                if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
            }
        }
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
// Two-CTA variant: a cluster of two CTAs (an SM pair) works on a
// 256 x 256 tile with tcgen05.mma cta_group::2 (M 256). Each CTA stages its own 128 rows of A and its
// own 128 columns of B (32 KiB per stage instead of 48, six stages), the pair's tensor cores exchange
// the B halves, and each CTA keeps the accumulator of its 128 rows in its own TMEM. The even CTA of
// the pair issues the MMAs; the loads of both CTAs count on its "full" barrier; tcgen05.commit
// releases a stage / publishes an accumulator in both CTAs at once; the odd CTA's epilogue warps
// hand their accumulator buffer back with an arrive on the even CTA's barrier.
// ------------------------------------------------------------------------------------------
template <int KIND, bool ACC>
__global__ void __launch_bounds__(NTHREADS, 1)
grouped_gemm2_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const GemmParams p) {
    constexpr int NST = STAGES2;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bars = base + DATA2_BYTES;  // [stages][float staging or mask tile] then the barriers
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (NST + s); };
    auto tfull_bar = [&](int a) { return bars + 8u * (2 * NST + a); };
    auto tempty_bar = [&](int a) { return bars + 8u * (2 * NST + 2 + a); };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + DATA2_BYTES + 240);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + DATA2_BYTES + 248);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();  // 0: issues the MMAs, owns the full / tempty barriers
    const int64_t cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 16); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
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
            uint32_t ph = 0;
            bool ok = true;
            TileIter<KIND, 256> it(p, (int32_t)cluster_id, (int32_t)n_clusters);
            Tile t;
            while (ok && it.next(t)) {
                int term = 0, kk = 0;  // ROW_*: piece of the contraction and column inside it
                for (int kb = 0; kb < t.kblocks && ok; ++kb) {
                    ok = mbar_wait(empty_bar(s), ph ^ 1u, abort_flag, p.status);
                    if (!ok) break;
                    const uint32_t a_dst = base + s * STAGE2_BYTES, b_dst = a_dst + A2_BYTES;
                    if (KIND == WGRAD) {
                        const int r = t.row0 + kb * BK;
                        if (rank == 0) mbar_expect_tx(full_bar(s), 2 * STAGE2_BYTES);
                        tma2_load_3d(a_dst, &tmA, full_bar(s), 0, r, t.m0 / 64 + 2 * (int)rank);
                        tma2_load_3d(b_dst, &tmB, full_bar(s), 0, r, t.b_chunk + 2 * (int)rank);
                    } else {
                        if (rank == 0) mbar_expect_tx(full_bar(s), 2 * STAGE2_BYTES);
                        tma2_load_2d(a_dst, &tmA, full_bar(s), p.a_term_col[term] + kk, t.row0 + 128 * (int)rank);
                        if (KIND == ROW_BMN)
                            tma2_load_4d(b_dst, &tmB, full_bar(s), 0, p.b_term_col[term] + kk, t.n0 / 64 + 2 * (int)rank, t.e);
                        else
                            tma2_load_3d(b_dst, &tmB, full_bar(s), p.b_term_col[term] + kk, t.n0 + 128 * (int)rank, t.e);
                        kk += BK;
                        if (kk == p.K) { kk = 0; ++term; }
                    }
                    if (++s == NST) { s = 0; ph ^= 1u; }
                }
            }
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
            TileIter<KIND, 256> it(p, (int32_t)cluster_id, (int32_t)n_clusters);
            Tile t;
            while (ok && it.next(t)) {
                if (t.kblocks == 0) continue;  // empty segment (WGRAD): the epilogue writes zeros
                const int sub = !ACC ? t.kblocks : t.e < p.segs_term0 ? p.sub_kb0 : p.sub_kb;  // K blocks per accumulator
                int kin = 0;                                                                  // the block's place among them
                ok = mbar_wait(tempty_bar(acc), acc_ph ^ 1u, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                uint32_t d_tmem = tmem_base + acc * BN;
                const int tail_valid = KIND == WGRAD ? (t.row_end - t.row0) - (t.kblocks - 1) * BK : BK;  // rows of the last block
                for (int kb = 0; kb < t.kblocks; ++kb) {
                    ok = mbar_wait(full_bar(s), ph, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a_src = base + s * STAGE2_BYTES, b_src = a_src + A2_BYTES;
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
                    if (++s == NST) { s = 0; ph ^= 1u; }
                }
                if (ok) tc_commit2(tfull_bar(acc));
                if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        int acc = 0;
        uint32_t acc_ph = 0;
        bool ok = true;
        TileIter<KIND, 256> it(p, (int32_t)cluster_id, (int32_t)n_clusters);
        Tile t;
        while (ok && it.next(t)) {
            const bool have_acc = t.kblocks > 0;
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
            b.out_off = KIND == WGRAD ? (int64_t)t.e * p.M * p.N : 0;
            b.row0 = (KIND == WGRAD ? t.m0 : t.row0) + 128 * (int)rank + quarter * 32;
            b.rows_valid = (KIND == WGRAD ? p.M : t.row_end) - (int32_t)b.row0;
            b.have_acc = have_acc;
            b.box = smem + NST * STAGE2_BYTES + (warp - 2) * 4096;
            if (have_acc) {
                ok = mbar_wait(tfull_bar(acc), acc_ph, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
            }
            auto release = [&]() {  // the warp's part of the accumulator is in registers: the buffer goes back
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_leader_relaxed(tempty_bar(acc));
            };
            for (int u = 0; u < boxes; ++u) {
                b.col0 = first + 64 * u;
                b.taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + half * (BN / 2) + 64 * u;
                epilogue_box(p, lane, b, [&]() { if (u + 1 == boxes) release(); });
            }
            if (have_acc) {
                if (boxes == 0) release();
                if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
            }
        }
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
GemmParams default_params() {
    GemmParams p;
    memset(&p, 0, sizeof(p));
    p.nterms = 1;
    p.segs_per_term = 1;
    return p;
}

// Derived tile counts the device code divides by; ids are 32-bit.
template <int KIND, int TM> int32_t complete_params(GemmParams &q, int64_t max_tiles) {
    if (max_tiles >= ((int64_t)1 << 31) - ((int64_t)1 << 22)) return MOE_ERR_UNSUPPORTED;
    q.tiles_n = (int32_t)cdiv(q.N, BN);
    q.per_e = KIND == WGRAD ? (int32_t)cdiv(q.M, TM) * q.tiles_n : 1;
    q.total_tiles = (int32_t)max_tiles;
    q.by_tiles_n = Divisor::of(q.tiles_n); q.by_per_e = Divisor::of(q.per_e); q.by_mod = Divisor::of(q.off_mod);
    q.by_terms = Divisor::of(q.segs_per_term); q.by_interleave = Divisor::of(q.interleave);
    q.kblocks_row = KIND == WGRAD ? 0 : q.nterms * (q.K / BK);
    return MOE_OK;
}

template <int KIND, bool ACC = false> int32_t launch(const CUtensorMap &tmA, const CUtensorMap &tmB, const GemmParams &p_in, int64_t max_tiles,
                                                     cudaStream_t st) {
    GemmParams p = p_in;
    MOE_TRY((complete_params<KIND, BM>(p, max_tiles)));
    static PerDevice configured;
    if (!allow_shared(configured, grouped_gemm_kernel<KIND, ACC>, SMEM_BYTES)) return MOE_ERR_CUDA;
    if (max_tiles <= 0) return MOE_OK;
    launch_kernel((grouped_gemm_kernel<KIND, ACC>), (unsigned)imin(max_tiles, tc_sm_count()), NTHREADS, SMEM_BYTES, st, tmA, tmB, p);
    MOE_LAUNCHED();
    return MOE_OK;
}

template <int KIND, bool ACC = false>
int32_t launch2(const CUtensorMap &tmA, const CUtensorMap &tmB, const GemmParams &p_in, int64_t max_tiles, cudaStream_t st) {
    GemmParams p = p_in;
    MOE_TRY((complete_params<KIND, 256>(p, max_tiles)));
    static PerDevice clusters;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeClusterDimension;
    attrs[0].val.clusterDim.x = 2; attrs[0].val.clusterDim.y = 1; attrs[0].val.clusterDim.z = 1;
    attrs[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_kernel
    attrs[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = SMEM2_BYTES; cfg.stream = st;
    cfg.attrs = attrs; cfg.numAttrs = 2;
    const int max_clusters = clusters.get([&]() {
        cfg.gridDim = dim3(2 * (tc_sm_count() / 2));
        int n = 0;
        const auto kernel = grouped_gemm2_kernel<KIND, ACC>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM2_BYTES) != cudaSuccess) return 0;
        return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess ? n : 0;
    });
    if (max_clusters <= 0) return MOE_ERR_CUDA;
    if (max_tiles <= 0) return MOE_OK;
    cfg.gridDim = dim3(2 * (unsigned)imin(max_tiles, max_clusters));
    MOE_CUDA(cudaLaunchKernelEx(&cfg, (grouped_gemm2_kernel<KIND, ACC>), tmA, tmB, p));
    MOE_LAUNCHED();
    return MOE_OK;
}

}  // namespace

// ------------------------------------------------------------------------------------------ host
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
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
int32_t tc_make_map(CUtensorMap *tm, const void *base, int rank, const uint64_t *dims, const uint64_t *strides,
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
// rows x cols activations, K-major operand: box 64 (cols) x box_rows
int32_t tc_map_rows_kmajor(CUtensorMap *tm, const void *p, int64_t rows, int64_t cols, int box_rows) {
    const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows}, str[1] = {(uint64_t)cols * 2};
    const uint32_t box[2] = {64, (uint32_t)box_rows};
    return tc_make_map(tm, p, 2, dims, str, box);
}
// rows x cols activations, MN-major operand (contraction over rows): dims (64, rows, cols/64)
int32_t tc_map_rows_mnmajor(CUtensorMap *tm, const void *p, int64_t rows, int64_t cols, int chunks) {
    const uint64_t dims[3] = {64, (uint64_t)rows, (uint64_t)(cols / 64)}, str[2] = {(uint64_t)cols * 2, 128};
    const uint32_t box[3] = {64, BK, (uint32_t)chunks};
    return tc_make_map(tm, p, 3, dims, str, box);
}
// per-expert weight [n, K, N] used as MN-major B: dims (64, K, N/64, n)
int32_t tc_map_weight_mnmajor(CUtensorMap *tm, const void *p, int64_t n, int64_t K, int64_t N, int tile_n) {
    const uint64_t dims[4] = {64, (uint64_t)K, (uint64_t)(N / 64), (uint64_t)n};
    const uint64_t str[3] = {(uint64_t)N * 2, 128, (uint64_t)K * N * 2};
    const uint32_t box[4] = {64, BK, (uint32_t)tile_n / 64, 1};
    return tc_make_map(tm, p, 4, dims, str, box);
}
// per-expert weight [n, N, K] used as K-major B: dims (K, N, n)
int32_t tc_map_weight_kmajor(CUtensorMap *tm, const void *p, int64_t n, int64_t N, int64_t K, int tile_n) {
    const uint64_t dims[3] = {(uint64_t)K, (uint64_t)N, (uint64_t)n};
    const uint64_t str[2] = {(uint64_t)K * 2, (uint64_t)N * K * 2};
    const uint32_t box[3] = {64, (uint32_t)tile_n, 1};
    return tc_make_map(tm, p, 3, dims, str, box);
}

int tc_sm_count() {
    static PerDevice count;
    const int n = count.get([]() {
        int dev = 0, v = 0;
        return cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? v : 0;
    });
    return n > 0 ? n : 148;
}

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
    const int64_t tiles = 3 * cdiv(d, pairs ? 256 : BM) * cdiv(2 * n, BN), workers = pairs ? tc_sm_count() / 2 : tc_sm_count();
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
        MOE_TRY(tc_map_rows_mnmajor(&tmA, x, T, d, BM / 64));
        MOE_TRY(tc_map_rows_mnmajor(&tmB, dsplit, T, 3 * n2, (pairs ? 128 : BN) / 64));
        GemmParams p = default_params();
        p.nseg = 3 * nr; p.M = d; p.N = n2; p.R = T; p.out_f32 = partials; p.status = status;
        p.segs_term0 = nr; p.rows_per_seg0 = rows;
        p.rows_per_seg = rows; p.segs_per_term = nr; p.b_term_chunks = n2 / 64;
        p.sub_kb0 = GB_ROWS_HI / BK; p.sub_kb = rows_lo / BK; p.interleave = 3;
        if (pairs) MOE_TRY((launch2<WGRAD, true>(tmA, tmB, p, (int64_t)p.nseg * cdiv(d, 256) * cdiv(n2, BN), st)));
        else MOE_TRY((launch<WGRAD, true>(tmA, tmB, p, (int64_t)p.nseg * cdiv(d, BM) * cdiv(n2, BN), st)));
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
        MOE_TRY(tc_map_rows_kmajor(&tmA, dsplit, T, 3 * n2, BM));
        if (pairs) MOE_TRY(tc_map_weight_kmajor(&tmB, wsplit, 1, d, 3 * n2, 128));
        else MOE_TRY(tc_map_weight_kmajor(&tmB, wsplit, 1, d, 3 * n2, BN));
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
    MOE_TRY(tc_map_rows_kmajor(&tmA, x, T, d, BM));
    MOE_TRY(tc_map_weight_mnmajor(&tmB, wsplit, 1, 3 * (int64_t)d, n2, 128));
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
    const bool pairs = tc_use_pairs(P1, a, flags, n2 > d ? n2 : d);
    CUtensorMap tmA, tmB;
    MOE_TRY(tc_map_rows_kmajor(&tmA, xs_p, P1, d, BM));
    {   // the group is the map's last coordinate (stride d rows), the precision term an offset of a * d rows along K
        const uint64_t dims[4] = {64, (uint64_t)3 * a * d, (uint64_t)(n2 / 64), (uint64_t)a};
        const uint64_t str[3] = {(uint64_t)n2 * 2, 128, (uint64_t)d * n2 * 2};
        const uint32_t box[4] = {64, BK, pairs ? 2u : (uint32_t)(BN / 64), 1};
        MOE_TRY(tc_make_map(&tmB, wsplit_s, 4, dims, str, box));
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
        MOE_TRY(tc_map_rows_mnmajor(&tmA, xs_p, P1 > 0 ? P1 : 1, d, BM / 64));
        MOE_TRY(tc_map_rows_mnmajor(&tmB, dsplit_s, P1 > 0 ? P1 : 1, 3 * n2, BN / 64));
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
        MOE_TRY(tc_map_rows_kmajor(&tmA, dsplit_s, P1, 3 * n2, BM));
        MOE_TRY(tc_map_weight_kmajor(&tmB, wsplit_s, a, d, 3 * n2, BN));
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
