// What the kernels of one call need to know about the expert segments, worked out once per call by one launch: tile prefixes
// for up to four tile heights, the tile records and the run-time counters of the tensor-core GEMMs, the segments in
// descending size (weight gradients hand out their longest tiles first), and in the backward pass the gradients of the two
// balancing losses with respect to Importance and Load. Each is the work of one block; as launches of their own they were
// nine of the 23 of a small backward pass, 2 to 4 us each.
#include <string.h>

#include "moe_internal.cuh"
#include "moments.cuh"

namespace moe {

namespace {

struct PlanArgs {
    SegmentPlan plan;
    const int32_t *offsets;
    int32_t n, max_m;  // max_m: tile records of plan.info
    int32_t *status;   // cleared if given
    Cv2Job cv2[2];
    int32_t map_block0;  // first block of the tensor maps
    SegmentMaps maps;
};
constexpr int MAPS_PER_BLOCK = 64;  // two per warp

// exclusive prefix of the segments' tiles of bm rows; returns the total to every thread (1024 threads)
__device__ int32_t tile_prefix_block(const int32_t *offsets, int32_t n, int32_t bm, int32_t *prefix, int32_t *sh /* [32] */) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t carry = 0;
    for (int32_t base = 0; base < n; base += 1024) {
        const int32_t e = base + threadIdx.x;
        const int32_t v = e < n ? (offsets[e + 1] - offsets[e] + bm - 1) / bm : 0;
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

// blocks 0..3: tile prefixes (0: the records, the counters and the status word as well); 4, 5: loss gradients; from 6 on:
// 1024 segments each of the order by size; from map_block0 on: the segments' tensor maps
__global__ void __launch_bounds__(1024) segment_plan_kernel(const __grid_constant__ PlanArgs a) {
    wait_previous_kernel();
    __shared__ int32_t sh[32];
    __shared__ double moments[32];
    __shared__ __align__(128) int32_t cnt[PLAN_MAX_SORTED];
    const int32_t *offsets = a.offsets;
    const int32_t n = a.n;
    if ((int32_t)blockIdx.x >= a.map_block0) {
        const int w = threadIdx.x >> 5;
        for (int q = 0; q < MAPS_PER_BLOCK / 32; ++q) {
            int64_t i = (int64_t)(blockIdx.x - a.map_block0) * MAPS_PER_BLOCK + 32 * q + w;
            int which = 0;  // the (i / n)-th map that is wanted
            for (; which < SEGMENT_MAPS; ++which) {
                if (!a.maps.made[which]) continue;
                if (i < n) break;
                i -= n;
            }
            if (which < SEGMENT_MAPS)
                write_segment_map(a.maps.base[which], a.plan.maps + (int64_t)which * n + i, offsets[i + 1], (uint32_t *)cnt + 64 * w + 32 * q);
        }
        return;
    }
    if (blockIdx.x < PLAN_HEIGHTS) {
        const int which = blockIdx.x;
        if (which == 0) {
            if (threadIdx.x < PLAN_COUNTERS && a.plan.counters) a.plan.counters[threadIdx.x] = 0;
            if (threadIdx.x == 0 && a.status) *a.status = 0;
        }
        if (a.plan.bm[which] == 0) return;
        int32_t *prefix = a.plan.prefix[which];
        const int32_t bm = a.plan.bm[which], total = tile_prefix_block(offsets, n, bm, prefix, sh);
        if (which != 0 || !a.plan.info) return;
        __syncthreads();  // the prefix (global memory, this block's own writes) is complete
        for (int32_t mt = threadIdx.x; mt < a.max_m; mt += 1024) {
            if (mt >= total) { a.plan.info[mt] = make_int4(-1, 0, 0, 0); continue; }
            int lo = 0, hi = n;  // last e with prefix[e] <= mt (empty segments share a prefix: take the last)
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (prefix[mid] <= mt) lo = mid; else hi = mid;
            }
            a.plan.info[mt] = make_int4(lo, offsets[lo] + (mt - prefix[lo]) * bm, offsets[lo + 1], 0);
        }
    } else if (blockIdx.x < PLAN_HEIGHTS + 2) {
        const Cv2Job &job = a.cv2[blockIdx.x - PLAN_HEIGHTS];
        if (job.v) cv2_grad_block(job, moments);
    } else if (a.plan.sched) {  // rank by descending size, equal sizes by index
        for (int32_t e = threadIdx.x; e < n; e += 1024) cnt[e] = offsets[e + 1] - offsets[e];
        __syncthreads();
        const int32_t e = (blockIdx.x - PLAN_HEIGHTS - 2) * 1024 + threadIdx.x;
        if (e >= n) return;
        const int32_t mine = cnt[e];
        int32_t rank = 0;
        for (int32_t o = 0; o < n; ++o) rank += (cnt[o] > mine || (cnt[o] == mine && o < e)) ? 1 : 0;
        a.plan.sched[rank] = make_int4(e, offsets[e], offsets[e + 1], 0);
    }
}

}  // namespace

static int64_t align4(int64_t v) { return (v + 3) & ~(int64_t)3; }
int64_t plan_ints(int64_t R, int64_t n) { return PLAN_HEIGHTS * align4(n + 1) + 4 * (cdiv(R, 128) + n + 1) + 4 * n + PLAN_COUNTERS + 32 + SEGMENT_MAPS * 32 * n; }  // 32: the maps start on 128 bytes

SegmentPlan plan_at(int32_t *ws, int64_t R, int64_t n) {
    SegmentPlan p;
    for (int i = 0; i < PLAN_HEIGHTS; ++i) { p.prefix[i] = ws + i * align4(n + 1); p.bm[i] = 0; }
    p.info = reinterpret_cast<int4 *>(ws + PLAN_HEIGHTS * align4(n + 1));
    p.sched = p.info + cdiv(R, 128) + n + 1;
    p.counters = reinterpret_cast<int32_t *>(p.sched + n);
    p.n = (int32_t)n;
    p.maps = reinterpret_cast<CUtensorMap *>((reinterpret_cast<uintptr_t>(p.counters + PLAN_COUNTERS) + 127) & ~(uintptr_t)127);
    return p;
}

int32_t launch_segment_plan(const SegmentPlan &plan, const int32_t *offsets, int32_t n, int64_t R, int32_t *status,
                            cudaStream_t st, const SegmentMaps *maps, const Cv2Job *jobs) {
    PlanArgs a;
    memset(&a, 0, sizeof(a));
    a.plan = plan; a.offsets = offsets; a.n = n; a.status = status;
    a.max_m = plan.info && plan.bm[0] ? (int32_t)(cdiv(R, plan.bm[0]) + n) : 0;
    a.cv2[0] = jobs ? jobs[0] : Cv2Job{nullptr, 0, 0.0f, nullptr};
    a.cv2[1] = jobs ? jobs[1] : Cv2Job{nullptr, 0, 0.0f, nullptr};
    unsigned blocks = PLAN_HEIGHTS + (plan.sched ? 2u + (unsigned)cdiv(n, 1024) : jobs ? 2u : 0u);
    a.map_block0 = (int32_t)blocks;
    if (maps && plan.maps) {
        a.maps = *maps;
        int64_t count = 0;
        for (int i = 0; i < SEGMENT_MAPS; ++i) count += maps->made[i] ? n : 0;
        blocks += (unsigned)cdiv(count, MAPS_PER_BLOCK);
    }
    launch_kernel(segment_plan_kernel, blocks, 1024, 0, st, a);
    MOE_LAUNCHED();
    return MOE_OK;
}

}  // namespace moe
