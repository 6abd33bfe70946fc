// The segment plan of a call (see plan.cu) as device code: one piece of it per block, by segment_plan_kernel or by blocks of their own in the
// launch that finds the segments (route.cu).
#pragma once

#include "moe_internal.cuh"
#include "moments.cuh"

namespace moe {

struct PlanArgs {
    SegmentPlan plan;
    int32_t n;
    int32_t *status;   // cleared if given
    Cv2Job cv2[2];
    int32_t map_block0;  // first block of the tensor maps
    int32_t rows;        // of the mapped tensors: no map ends behind them, whatever the offsets say
    SegmentMaps maps;
};
constexpr int MAPS_PER_BLOCK = 64;  // two per warp
inline int64_t plan_blocks(const PlanArgs &a) {
    int64_t maps = 0;
    for (int i = 0; i < SEGMENT_MAPS; ++i) maps += a.maps.made[i] ? a.n : 0;
    return a.map_block0 + cdiv(maps, MAPS_PER_BLOCK);
}
// Segments are put in order by counting, for each, the larger ones, or from so many on by a bitonic sort: the plan of a backward call, us, counted and sorted: 257
// segments 9.6, 9.2; 512 14.8, 9.6; 1024 46.8, 12.7; 2048 174, 21.5. (256 counted: 6.9.)
constexpr int PLAN_SORT_FROM = 257;
__host__ __device__ inline int32_t sort_places(int32_t n) {  // n, filled up to a power of two
    int32_t places = 1;
    while (places < n) places *= 2;
    return places;
}
// ints of shared memory a piece of the plan needs: the lengths of n sorted segments and their order (sorted: 64-bit keys), or the maps under construction
inline int64_t plan_shared_ints(int32_t n) {
    const int64_t ints = n >= PLAN_SORT_FROM ? 2 * (int64_t)sort_places(n) : 2 * (int64_t)n;
    return ints > MAPS_PER_BLOCK * 32 ? ints : MAPS_PER_BLOCK * 32;
}

__device__ __forceinline__ int32_t *on_128_bytes(int32_t *shared) {
    return shared + ((128u - ((uint32_t)__cvta_generic_to_shared(shared) & 127u)) & 127u) / 4u;
}

// exclusive prefix of the tiles of bm rows of segments of rows(i) rows; returns the total to every thread (1024 threads)
template <typename Rows>
static __device__ __forceinline__ int32_t tile_prefix_block(Rows rows, int32_t n, int32_t bm, int32_t *prefix, int32_t *sh /* [32] */) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t carry = 0;
    for (int32_t base = 0; base < n; base += 1024) {
        const int32_t e = base + threadIdx.x;
        const int32_t v = e < n ? (rows(e) + bm - 1) / bm : 0;
        int32_t inc = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t o = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += o;
        }
        __syncthreads();
        if (lane == 31) sh[w] = inc;
        __syncthreads();
        const int32_t sw = sh[lane];
        int32_t si = sw;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t o = __shfl_up_sync(0xffffffffu, si, off);
            if (lane >= off) si += o;
        }
        const int32_t before = __shfl_sync(0xffffffffu, si - sw, w);
        if (e < n) prefix[e] = carry + before + inc - v;
        carry += __shfl_sync(0xffffffffu, si, 31);
    }
    if (threadIdx.x == 0) prefix[n] = carry;
    return carry;
}

// Piece `block` of the plan, by 1024 threads; offsets: global or shared memory; cnt: plan_shared_ints(n), on 128 bytes.
// Pieces 0..3: tile prefixes (0: the order by size, the records, the counters and the status word as well); 4, 5: loss gradients; from
// map_block0 on: the segments' tensor maps
__device__ __forceinline__ void plan_piece(const PlanArgs &a, int32_t block, const int32_t *offsets, int32_t *cnt, int32_t *sh /* [32] */,
                                           double *moments /* [32] */) {
    const int32_t n = a.n;
    if (block >= a.map_block0) {
        const int w = threadIdx.x >> 5;
        for (int q = 0; q < MAPS_PER_BLOCK / 32; ++q) {
            int64_t i = (int64_t)(block - a.map_block0) * MAPS_PER_BLOCK + 32 * q + w;
            int which = 0;  // the (i / n)-th map that is wanted
            for (; which < SEGMENT_MAPS; ++which) {
                if (!a.maps.made[which]) continue;
                if (i < n) break;
                i -= n;
            }
            if (which < SEGMENT_MAPS)
                write_segment_map(a.maps.base[which], a.plan.maps + (int64_t)which * n + i, min(offsets[i + 1], a.rows), (uint32_t *)cnt + 64 * w + 32 * q);
        }
        return;
    }
    if (block < PLAN_HEIGHTS) {
        const int which = block;
        if (which == 0) {
            if (threadIdx.x < PLAN_COUNTERS && a.plan.counters) a.plan.counters[threadIdx.x] = 0;
            if (threadIdx.x == 0 && a.status) *a.status = 0;
        }
        if (a.plan.bm[which] == 0) return;
        const int32_t bm = a.plan.bm[which];
        auto rows_of = [&](int32_t e) { return offsets[e + 1] - offsets[e]; };
        if (which != 0 || !a.plan.info) {
            tile_prefix_block(rows_of, n, bm, a.plan.prefix[which], sh);
            return;
        }
        int32_t *by_rank = a.plan.by_rank, *order = cnt + n;
        const bool sorted = a.plan.sched != nullptr;
        int32_t total;
        if (sorted) {  // rank by descending size, equal sizes by index
            if (n < PLAN_SORT_FROM) {  // `lanes` lanes a segment, each compares with its share of the others
                int32_t lanes = 1;
                while (lanes < 32 && 2 * lanes * n <= 1024) lanes *= 2;
                for (int32_t e = threadIdx.x; e < n; e += 1024) cnt[e] = rows_of(e);
                __syncthreads();
                const int32_t share = threadIdx.x & (lanes - 1);
                for (int32_t e0 = 0; e0 < n; e0 += 1024 / lanes) {
                    const int32_t e = e0 + threadIdx.x / lanes, mine = e < n ? cnt[e] : 0;
                    int32_t rank = 0;
                    for (int32_t o = share; o < n; o += lanes) rank += (cnt[o] > mine || (cnt[o] == mine && o < e)) ? 1 : 0;
                    for (int32_t s = 1; s < lanes; s <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, s);
                    if (e < n && share == 0) order[rank] = e;
                }
            } else {
                const int32_t places = sort_places(n);  // at most two a thread
                uint64_t *keys = reinterpret_cast<uint64_t *>(cnt);
                for (int32_t e = threadIdx.x; e < places; e += 1024) keys[e] = e < n ? (uint64_t)~(uint32_t)rows_of(e) << 32 | (uint32_t)e : ~0ull;
                for (int32_t run = 2; run <= places; run *= 2)
                    for (int32_t apart = run / 2; apart > 0; apart /= 2) {
                        __syncthreads();
                        if (threadIdx.x < places / 2) {
                            const int32_t low = threadIdx.x & (apart - 1), i = 2 * ((int32_t)threadIdx.x - low) + low;
                            const uint64_t x = keys[i], y = keys[i + apart];
                            if ((x > y) == ((i & run) == 0)) {
                                keys[i] = y;
                                keys[i + apart] = x;
                            }
                        }
                    }
                __syncthreads();
                uint64_t mine[2];
                for (int32_t q = 0; q < 2; ++q) mine[q] = (int32_t)threadIdx.x + 1024 * q < n ? keys[threadIdx.x + 1024 * q] : 0;
                __syncthreads();  // lengths and order take the keys' place
                for (int32_t q = 0; q < 2; ++q) {
                    const int32_t r = threadIdx.x + 1024 * q;
                    if (r >= n) break;
                    order[r] = (int32_t)(uint32_t)mine[q];
                    cnt[order[r]] = (int32_t)~(uint32_t)(mine[q] >> 32);
                }
            }
            __syncthreads();
            for (int32_t r = threadIdx.x; r < n; r += 1024) {
                const int32_t e = order[r];
                a.plan.sched[r] = make_int4(e, offsets[e], offsets[e + 1], 0);
            }
            total = tile_prefix_block([&](int32_t r) { return cnt[order[r]]; }, n, bm, by_rank, sh);
        } else {
            by_rank = a.plan.prefix[0];
            total = tile_prefix_block(rows_of, n, bm, by_rank, sh);
        }
        __syncthreads();  // the prefix (global memory, this block's own writes) is complete
        if (sorted)
            for (int32_t r = threadIdx.x; r < n; r += 1024) a.plan.prefix[0][order[r]] = by_rank[r];
        for (int32_t mt = threadIdx.x; mt < total; mt += 1024) {
            int lo = 0, hi = n;  // last rank with by_rank <= mt (empty segments share a prefix: take the last)
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (by_rank[mid] <= mt) lo = mid; else hi = mid;
            }
            const int32_t e = sorted ? order[lo] : lo;
            a.plan.info[mt] = make_int4(e, offsets[e] + (mt - by_rank[lo]) * bm, offsets[e + 1], mt);
        }
    } else if (block < PLAN_HEIGHTS + 2) {
        const Cv2Job &job = a.cv2[block - PLAN_HEIGHTS];
        if (job.v) cv2_grad_block(job, moments);
    }
}

}  // namespace moe
