// What the kernels of one call need to know about the expert segments, worked out once per call by one launch: tile prefixes
// for up to four tile heights, the tile records and the run-time counters of the tensor-core GEMMs, the segments in
// descending size (weight gradients: the longest tiles first), and in the backward pass the gradients of the two
// balancing losses with respect to Importance and Load. Each is the work of one block; as launches of their own they were
// nine of the 23 of a small backward pass, 2 to 4 us each. The forward pass has it done by further blocks of the launch that finds the
// segments (route.cu) where that takes one pass over them.
#include <string.h>

#include "plan.cuh"

namespace moe {

__global__ void __launch_bounds__(1024) segment_plan_kernel(const __grid_constant__ PlanArgs a, const int32_t *__restrict__ offsets) {
    wait_previous_kernel();
    extern __shared__ __align__(128) int32_t plan_sh[];
    __shared__ int32_t sh[32];
    __shared__ double moments[32];
    plan_piece(a, blockIdx.x, offsets, on_128_bytes(plan_sh), sh, moments);
}

static int64_t align4(int64_t v) { return (v + 3) & ~(int64_t)3; }
int64_t plan_ints(int64_t R, int64_t n) { return PLAN_HEIGHTS * align4(n + 1) + 4 * (cdiv(R, 128) + n + 1) + 4 * n + PLAN_COUNTERS + 32 + SEGMENT_MAPS * 32 * n; }  // 32: the maps start on 128 bytes

SegmentPlan plan_at(int32_t *ws, int64_t R, int64_t n) {
    SegmentPlan p;
    for (int i = 0; i < PLAN_HEIGHTS; ++i) { p.prefix[i] = ws + i * align4(n + 1); p.bm[i] = 0; }
    p.info = reinterpret_cast<int4 *>(ws + PLAN_HEIGHTS * align4(n + 1));
    p.sched = p.info + cdiv(R, 128) + n + 1;
    p.by_rank = p.prefix[2];
    p.counters = reinterpret_cast<int32_t *>(p.sched + n);
    p.n = (int32_t)n;
    p.maps = reinterpret_cast<CUtensorMap *>((reinterpret_cast<uintptr_t>(p.counters + PLAN_COUNTERS) + 127) & ~(uintptr_t)127);
    return p;
}

void fill_plan(PlanArgs *a, const SegmentPlan &plan, int32_t n, int64_t R, int32_t *status, const SegmentMaps *maps, const Cv2Job *jobs) {
    memset(a, 0, sizeof(*a));
    a->plan = plan; a->n = n; a->status = status;
    if (jobs) { a->cv2[0] = jobs[0]; a->cv2[1] = jobs[1]; }
    a->map_block0 = PLAN_HEIGHTS + (jobs ? 2 : 0);
    a->rows = (int32_t)R;
    if (maps && plan.maps) a->maps = *maps;
}

int32_t launch_segment_plan(const PlanArgs &a, const int32_t *offsets, cudaStream_t st) {
    const size_t shared = plan_shared_ints(a.plan.sched ? a.n : 0) * sizeof(int32_t) + 128;  // at most 16 KiB: PLAN_MAX_SORTED keys
    launch_kernel(segment_plan_kernel, (unsigned)plan_blocks(a), 1024, shared, st, a, offsets);
    MOE_LAUNCHED();
    return MOE_OK;
}

}  // namespace moe
