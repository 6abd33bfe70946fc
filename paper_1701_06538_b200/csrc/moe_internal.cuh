// Internal declarations shared by the translation units of the library (not part of the ABI).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "moe.h"
#include "per_device.h"

#define MOE_TRY(expr)                                \
    do {                                             \
        int32_t st_ = (expr);                        \
        if (st_ != MOE_OK) return st_;               \
    } while (0)

#define MOE_CUDA(expr)                               \
    do {                                             \
        if ((expr) != cudaSuccess) return MOE_ERR_CUDA; \
    } while (0)

#define MOE_LAUNCHED()                                           \
    do {                                                         \
        ::moe::count_launch();                                   \
        if (cudaGetLastError() != cudaSuccess) return MOE_ERR_CUDA; /* consumed: reported once */ \
    } while (0)

// Checking build (-DMOE_BOUNDS_CHECK, the stand-in for a memory checker): every place where a value read from memory
// becomes an index reports a value outside its range to a counter of the translation unit (never a trap; the access
// itself is skipped by the guards that are always compiled in). moe_debug_bounds_violations adds the counters up.
#ifdef MOE_BOUNDS_CHECK
static __device__ unsigned long long g_tu_bounds_violations = 0ull;
#define MOE_BOUNDS_NOTE(ok)                                                  \
    do {                                                                     \
        if (!(ok)) atomicAdd(&g_tu_bounds_violations, 1ull);                 \
    } while (0)
#define MOE_BOUNDS_READER(fn)                                                                                   \
    unsigned long long fn() {                                                                                   \
        unsigned long long v = 0;                                                                               \
        return cudaMemcpyFromSymbol(&v, g_tu_bounds_violations, sizeof(v)) == cudaSuccess ? v : ~0ull;          \
    }
#else
#define MOE_BOUNDS_NOTE(ok) do {} while (0)
#define MOE_BOUNDS_READER(fn) unsigned long long fn() { return 0ull; }
#endif

namespace moe {

// Kernels are launched with programmatic stream serialization: the next kernel's launch is processed while its predecessor
// drains, and before it touches memory every kernel waits until the predecessor has finished and its writes are visible.
// The order of memory accesses stays that of the stream. It saves 1.5 us a launch: a step of 39 small kernels 183 -> 122 us, one
// of 50 large ones (32768 tokens, 256 experts) 1773 -> 1715 us. Letting the successor start earlier
// (griddepcontrol.launch_dependents at the head of a kernel) was slower: 128 and 1820 us.
__device__ __forceinline__ void wait_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... Params, typename... Args>
void launch_kernel(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);  // errors: MOE_LAUNCHED reads them
}

void count_launch();  // diagnostics: kernels launched by this library so far (api.cu)
// per translation unit: out-of-range indices seen by the checking build (0 in the regular build)
unsigned long long bounds_violations_route();
unsigned long long bounds_violations_losses();
unsigned long long bounds_violations_hier();
unsigned long long bounds_violations_gate();
unsigned long long bounds_violations_gate_bwd();
unsigned long long bounds_violations_ffn();
unsigned long long bounds_violations_products();

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f32<bf16>(float v) { return __float2bfloat16_rn(v); }

static inline size_t act_bytes(int32_t act) { return act == MOE_BF16 ? 2 : 4; }
static inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
static inline int64_t imin(int64_t a, int64_t b) { return a < b ? a : b; }
static inline int64_t imax(int64_t a, int64_t b) { return a > b ? a : b; }
// whether two buffers share memory
static inline bool overlap(const void *a, int64_t a_bytes, const void *b, int64_t b_bytes) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + (uintptr_t)b_bytes && y < x + (uintptr_t)a_bytes;
}
static inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 31) == 0; }  // 32 bytes: the epilogues use 256-bit stores

// In the place of work that rides along with a launch, where none does: the parameters and registers of the work cost the launch's own
// (moe_combine of 32768 x 512, one slot: 14.1 us with them, 9.3 without; 1000 x 512: 1.67, 1.55)
struct Nothing {};
template <typename Ride> constexpr bool rides() { return !std::is_same<Ride, Nothing>::value; }

// Carves 256-byte aligned pieces out of a workspace. With base == nullptr it only measures,
// so the size queries and the calls that use the workspace run the same code.
struct Carver {
    char *base;
    size_t off;
    explicit Carver(void *b) : base(static_cast<char *>(b)), off(0) {}
    template <typename T> T *take(int64_t count) {
        size_t bytes = (static_cast<size_t>(count < 0 ? 0 : count) * sizeof(T) + 255) & ~size_t(255);
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += bytes;
        return p;
    }
    void *take_bytes(int64_t bytes) { return take<char>(bytes); }
};

// Every workspace begins with a 256-byte header; word 0 is the status word of bounded waits.
static const int64_t kWsHeader = 256;

// ----------------------------------------------------------------------------- gating (gate.cu)
// Projection clean = rows.W0, raw = rows.W1 with the fixed fused-multiply-add chain.
// Ungrouped: offsets == nullptr, rows are tokens 0..M-1, outputs [M, n0].
// Grouped (secondary gates): sorted row r belongs to segment e (offsets[e] <= r < offsets[e+1]),
// reads token perm[r] / kdiv, uses W0 + e*d*n0, and writes output row perm[r].
int32_t launch_projection(const void *x, int32_t act, int64_t M, int32_t d, int32_t n0, const float *W0,
                          const float *W1, float *out0, float *out1, const int32_t *offsets, int32_t nseg,
                          const int32_t *perm, int32_t kdiv, int32_t *tile_prefix, cudaStream_t st,
                          const int32_t *row_count = nullptr, int32_t *clear = nullptr);
// The hierarchical gate (Eq. 12), written where a secondary gate's row (the slot t * k1 + s1) gets its result: flat expert id i * b + j and
// product gate, slots primary-major. idx == nullptr: not a secondary gate.
struct HierMerge {
    int32_t *idx;
    float *gates;
    const int32_t *idx_p;
    const float *g_p;
    int32_t b;
    __device__ __forceinline__ void put(int64_t slot, int32_t k2, int s, int32_t j, float g) const {
        idx[slot * k2 + s] = idx_p[slot] * b + j;
        gates[slot * k2 + s] = g_p[slot] * g;
    }
};
// Noisy logits, top-k, masked softmax for `rows` rows of n columns.
int32_t launch_gate_select(const float *clean, const float *raw, const float *noise, int64_t rows, int32_t n,
                           int32_t k, int32_t *idx, float *gates, float *kth_vals, int32_t *kth_idx,
                           cudaStream_t st, const int32_t *row_list = nullptr, const int32_t *row_count = nullptr,
                           const void *row_span = nullptr, const void *chain_list = nullptr, const HierMerge &merge = HierMerge{});
// Tensor-core screening of the routing (see gate.cu): weights split / norms, then the screening select.
int32_t launch_gate_screen_prepare(const void *x, int64_t T, int32_t d, int32_t n, const float *Wg, const float *Wn, void *wsplit,
                                   float *wnorm, float *xnorm, int32_t *unsafe_count, float *wt /* [2n, d]: columns as rows */,
                                   cudaStream_t st, int32_t groups = 1, bool with_xnorm = true, int32_t *clear = nullptr);
// The screen of the products in clean / raw. Rows it cannot certify: unsafe_list / unsafe_count[0] = rows whose selection is
// repeated (unsafe_low: the bound that picks their candidate columns; unsafe_span: where their candidates stand); chain_list
// (int2 {row, column code}, unsafe_count[1] entries, at most 2 * SCREEN_MAX_CAND per row) = single fma chains to
// recompute; full_list / unsafe_count[2] = rows with more candidates than that, which take the whole projection.
constexpr int SCREEN_MAX_CAND = 16;
int32_t launch_gate_screen(const float *noise, const float *xnorm, const float *wnorm, int32_t d, int64_t T, int32_t n, int32_t k,
                           int32_t *idx, float *gates, float *clean, float *raw, float *kth_vals, int32_t *kth_idx, int32_t *unsafe_list,
                           float *unsafe_low, int32_t *unsafe_count, void *chain_list, int32_t *full_list, void *unsafe_span,
                           cudaStream_t st, const int32_t *perm, int32_t kdiv, const int32_t *group_of,
                           const HierMerge &merge = HierMerge{});
int32_t launch_gate_chains(const void *x, int32_t d, int32_t n, const float *Wt, const void *chain_list, const int32_t *chain_count,
                           float *clean, float *raw, cudaStream_t st, int32_t kdiv = 1);  // Wt [2n, d] (per group); token = output row / kdiv
bool tc_gate_fwd_supported(int32_t act, int64_t T, int32_t d, int32_t n, int32_t flags);
// clean | raw [T, n] (float) = x . [W_g | W_noise] from the three-term split wsplit [3, d, 2n]
int32_t launch_tc_gate_fwd(const void *x, int64_t T, int32_t d, int32_t n, const void *wsplit, float *clean, float *raw,
                           int32_t *status, cudaStream_t st);

// ----------------------------------------------------------------------------- routing (route.cu)
int64_t dispatch_ws_elems(int64_t R, int32_t n);  // int32 elements of scratch
// plan: the segment plan, in the same launches if they can (*planned says so)
int32_t launch_dispatch_index(const int32_t *topk_idx, int64_t R, int32_t n, int32_t *perm, int32_t *inv_perm,
                              int32_t *counts, int32_t *offsets, int32_t *scratch, cudaStream_t st,
                              const struct PlanArgs *plan = nullptr, bool *planned = nullptr);
// sums: the loss sums over the batch, by blocks of their own in the same launch (one launch after it completes them:
// level_reduce, by combine or by itself)
int32_t launch_dispatch_rows(const void *x, int32_t act, int64_t T, int32_t k, int32_t d, const int32_t *inv_perm,
                             void *xs, cudaStream_t st, const struct LevelSums *sums = nullptr);
// keep != nullptr: the layer epilogue of Appendix C (sigmoid, dropout through the packed keep bits [T, d/8] with the
// kept activations scaled by keep_scale = 1 / (1 - DropProb), residual xres added); see route.cu
int32_t launch_combine(const void *ys, int32_t act, const float *gates, const int32_t *inv_perm, int64_t T,
                       int32_t k, int32_t d, void *y, cudaStream_t st, const void *xres = nullptr,
                       const uint8_t *keep = nullptr, float keep_scale = 1.0f, const struct LevelSums *sums = nullptr);
int32_t launch_combine_bwd(const void *dY, const void *ys, int32_t act, const float *gates,
                           const int32_t *inv_perm, int64_t T, int32_t k, int32_t d, float *dgates, void *dys,
                           cudaStream_t st, const uint8_t *keep = nullptr, float keep_scale = 1.0f,
                           const int32_t *topk_idx = nullptr, const float *dimp = nullptr, int32_t n = 0);
// (dimp [n]: the gradient of the Importance loss, added to the gate gradients of the experts in topk_idx)
// out_f32 = sum_s dxs[inv_perm[t*k+s]] (+ add_f32 if given); written as float or, if out_act
// is given instead, rounded to the act type. sec: float rows [T * k1, d] of the secondary gates, added to add_f32 (which is
// given then); perm: row of a slot, or nullptr
struct SecondaryRows { const float *rows; const int32_t *perm; int32_t k1; };
// tail: sums that earlier launches have left, by blocks of their own
int32_t launch_dispatch_bwd(const void *dxs, int32_t act, const int32_t *inv_perm, int64_t T, int32_t k,
                            int32_t d, const float *add_f32, float *out_f32, void *out_act, cudaStream_t st,
                            const void *add_act = nullptr, const SecondaryRows &sec = SecondaryRows{},
                            const struct BackwardTail *tail = nullptr);
// The segment of tile `b` of a ragged product {segment, first row, segment end, tile inside the segment}, or segment -1 behind the last
// tile, looked up by the whole block (barriers): every thread looks at its share of the segments, so that a block waits for
// one round of loads (a binary search over the prefix waits for one per step, 2 of the 5 us of a block with little to do). With more
// than four segments a thread the search is less work (12288 blocks of 256 threads, 4096 segments: 80 us, this way 96; the float
// products of 24 rows of 64 in 480 segments, 64 threads a block: 101, 122; with 256 segments of 500 rows 77, this way 74). sh: one int4
__device__ __forceinline__ int4 segment_of_tile(const int32_t *__restrict__ tile_prefix, const int32_t *__restrict__ offsets, int32_t nseg,
                                                int32_t b, int4 *sh) {
    if (threadIdx.x == 0) *sh = make_int4(-1, 0, 0, 0);
    __syncthreads();
    if (nseg > 4 * (int32_t)blockDim.x) {
        if (threadIdx.x == 0 && b < tile_prefix[nseg]) {
            int32_t lo = 0, hi = nseg;
            while (hi - lo > 1) {
                const int32_t mid = (lo + hi) >> 1;
                if (tile_prefix[mid] <= b) lo = mid; else hi = mid;
            }
            *sh = make_int4(lo, offsets[lo], offsets[lo + 1], b - tile_prefix[lo]);
        }
        __syncthreads();
        return *sh;
    }
    for (int32_t q = threadIdx.x; q < nseg; q += blockDim.x) {
        const int32_t p0 = tile_prefix[q], p1 = tile_prefix[q + 1], o0 = offsets[q], o1 = offsets[q + 1];
        if (p0 <= b && b < p1) *sh = make_int4(q, o0, o1, b - p0);
    }
    __syncthreads();
    return *sh;
}
// tile_prefix[e] = sum_{e' < e} ceil(count_e' / bm), e = 0..n
int32_t launch_tile_prefix(const int32_t *offsets, int32_t n, int32_t bm, int32_t *tile_prefix, cudaStream_t st);

// ----------------------------------------------------------------------------- per-call segment plan (plan.cu)
// Longest segments first for up to PLAN_MAX_SORTED of them, two keys a thread of one block. More are taken as they lie, which costs nothing: a backward call
// of 2049 x 400 rows of 256 x 256 871 us, 1299 with Zipf loads; 2048, in order, 890 and 1254.
constexpr int PLAN_HEIGHTS = 4, PLAN_COUNTERS = 8, PLAN_MAX_SORTED = 2048;
enum PlanCounter { PLAN_HID = 0, PLAN_YS, PLAN_DZ_DW2, PLAN_DW1_DXS, PLAN_DXS };  // the tiles drawn so far, by launch of expert products
// Tensor maps of a call's expert products whose rows end with a segment, one per segment: what lies behind a segment's last row reads
// as zero, whatever follows it in memory. ROWS: K-major operand of a row product, COLS: operand of a weight gradient
// (contraction over the rows).
enum SegmentMap { MAP_XS_ROWS = 0, MAP_HID_ROWS, MAP_DYS_ROWS, MAP_DZ_ROWS, MAP_HID_COLS, MAP_DYS_COLS, MAP_XS_COLS, MAP_DZ_COLS, SEGMENT_MAPS };
struct SegmentMaps {
    CUtensorMap base[SEGMENT_MAPS];  // of the whole tensors
    int32_t made[SEGMENT_MAPS];      // which of them are wanted
};
struct SegmentPlan {
    CUtensorMap *maps;              // [SEGMENT_MAPS][n], or nullptr
    int32_t n;
    const CUtensorMap *maps_of(SegmentMap which) const { return maps ? maps + (int64_t)which * n : nullptr; }
    int32_t *prefix[PLAN_HEIGHTS];  // [n + 1] number of tiles of bm[i] rows in the segments before
    int32_t bm[PLAN_HEIGHTS];       // 0: prefix not made
    // Tensor-core products take the segments by rank: by descending size (sched), or as they lie
    int4 *sched;         // {segment, first row, end row, 0} by rank, or nullptr
    int32_t *by_rank;    // [n + 1] tiles of bm[0] rows in the segments before, by rank (prefix[0] if sched is not made); prefix[0] is its copy by
                         // segment, without an end
    int4 *info;          // a record per tile of by_rank, or nullptr: {segment, first row, segment end, number of the tile}
    int32_t *counters;   // [PLAN_COUNTERS], zeroed
    const int32_t *prefix_of(int32_t height) const {
        for (int i = 0; i < PLAN_HEIGHTS; ++i)
            if (bm[i] == height) return prefix[i];
        return nullptr;
    }
};
struct Cv2Job { const float *v; int32_t m; float scale; float *out; };  // out = scale * dCV^2(v)/dv
int64_t plan_ints(int64_t R, int64_t n);
SegmentPlan plan_at(int32_t *ws, int64_t R, int64_t n);
struct PlanArgs;  // plan.cuh
// status: cleared if given; maps: base maps of the operands, or nullptr; jobs: two, or nullptr
void fill_plan(PlanArgs *a, const SegmentPlan &plan, int32_t n, int64_t R, int32_t *status, const SegmentMaps *maps = nullptr,
               const Cv2Job *jobs = nullptr);
int32_t launch_segment_plan(const PlanArgs &a, const int32_t *offsets, cudaStream_t st);
// One segment's map, by a warp: a copy of `base` whose rows (dimension 1) end at `rows`. sh: 128 bytes, 128-byte aligned
__device__ __forceinline__ void write_segment_map(const CUtensorMap &base, CUtensorMap *out, int32_t rows, uint32_t *sh) {
    const int lane = threadIdx.x & 31;
    sh[lane] = reinterpret_cast<const uint32_t *>(&base)[lane];
    __syncwarp();
    const uint32_t at = (uint32_t)__cvta_generic_to_shared(sh);
    if (lane == 0)
        asm volatile("tensormap.replace.tile.global_dim.shared::cta.b1024.b32 [%0], 1, %1;" ::"r"(at), "r"(rows > 1 ? rows : 1) : "memory");
    __syncwarp();
    asm volatile("tensormap.cp_fenceproxy.global.shared::cta.tensormap::generic.release.gpu.sync.aligned [%0], [%1], 128;" ::"l"(out), "r"(at)
                 : "memory");
}

// ----------------------------------------------------------------------------- losses (losses.cu)
// where the fused forward wants second copies of the stage's results (nullptr: none), and of the expert counts
struct LossOut {
    float *losses, *importance, *load;
    int32_t *counts;
    const int32_t *counts_src;
    int32_t n, n_load;  // lengths of importance / counts and of load
};
struct LossFinal { float w_imp, w_load; float *losses; LossOut copy; };
int64_t losses_ws_floats(int64_t rows, int32_t n);
// Column sums over rows of the gate mass (importance) and of P(x, i) (load), and with fin.losses set the two losses: per-chunk sums
// by one launch, an ordered pass over the chunks by the next.
struct LevelSums {
    const int32_t *idx;
    const float *gates, *clean, *raw, *kth_vals;
    int64_t rows;
    int32_t n, k, chunks;
    float *part_imp, *part_load;
    int32_t *ticket;
    float *importance, *load;  // nullptr: not wanted (with fin.losses both are)
    LossFinal fin;
};
LevelSums level_sums(const int32_t *idx, const float *gates, const float *clean, const float *raw, const float *kth_vals, int64_t rows,
                     int32_t n, int32_t k, float *importance, float *load, float *scratch, const LossFinal *fin = nullptr);
int32_t launch_level_sums(const LevelSums &sums, cudaStream_t st);   // both launches
constexpr int LEVEL_RIDE_MAX = 256;  // columns up to which the sums go along with other launches
int32_t launch_cv2(const float *importance, int32_t n_imp, const float *load, int32_t n_load, float w_imp,
                   float w_load, float *losses, cudaStream_t st, const LossOut &copy);
int32_t launch_cv2_grads(const Cv2Job *jobs /* two */, cudaStream_t st);

// ----------------------------------------------------------------------------- hierarchical pieces (hier.cu)
int32_t launch_hier_split_idx(const int32_t *topk_idx, int64_t T, int32_t k1, int32_t k2, int32_t a, int32_t b,
                              int32_t *idx_p, int32_t *idx_s, cudaStream_t st);
int32_t launch_segment_sum(const float *vals, const int32_t *perm, const int32_t *offsets, int32_t nseg, float *out,
                           cudaStream_t st);
int64_t grouped_sums_ws_floats(int64_t rows, int32_t nseg, int32_t n);
// Load_i of every group, then Load_H, the two losses of the complete vectors and the copies (Eq. 14; `load` as laid out in load_h_bwd_kernel,
// its Load_primary part is complete already)
int32_t launch_grouped_load(const int32_t *idx_s, const float *clean, const float *raw, const float *kth_vals,
                            const int32_t *perm, const int32_t *offsets, const int32_t *counts_p, int32_t a, int64_t rows, int32_t b,
                            int32_t k, const float *importance, float *load, float *scratch, const LossFinal &fin, cudaStream_t st);
int32_t launch_load_h_bwd(const float *load, const float *dload_h, int32_t a, int32_t b, float *dload,
                          cudaStream_t st);
int32_t launch_hier_gate_product_bwd(const float *gates, float *dgates, int64_t T, int32_t k1, int32_t k2,
                                     cudaStream_t st);
int32_t launch_add_slot_rows(const float *dX_sec, int64_t T, int32_t k1, int32_t d, float *dX_gate, cudaStream_t st);
int32_t launch_add_gathered(float *dgates, const int32_t *topk_idx, const float *dimp, int64_t R, int32_t n,
                            cudaStream_t st);

// ----------------------------------------------------------------------------- gate backward (gate_bwd.cu)
// dlogit [rows, 2n] = (dclean | draw) from the saved gate tensors, or (dsplit given) its three-term bf16 split.
int32_t launch_gate_logit_grads(const float *noise, const float *clean, const float *raw, const int32_t *idx,
                                const float *gates, const float *kth_vals, const int32_t *kth_idx,
                                const float *dgates, const float *dload, const int32_t *dload_row_group,
                                int64_t rows, int32_t n, int32_t k, float *dlogit, void *dsplit,
                                const int32_t *split_row_index, cudaStream_t st, const struct ColumnSums *beside = nullptr);
// beside: tile sums of a bias gradient, by blocks of their own in the same launch

// ----------------------------------------------------------------------------- SIMT grouped GEMM (gemm_simt.cu)
enum GemmType { G_F32 = 0, G_BF16 = 1 };
struct SimtGemm {
    // C(i,j) = epilogue( sum_kk A(i,kk) * B(kk,j) ), strides in elements; one index of A and of B is contiguous, j of C is.
    const void *A, *B;
    void *C;
    int32_t ta, tb, tc;  // GemmType of A, B, C
    int64_t sa_i, sa_k, sb_k, sb_j, sc_i;
    // mode 0: output rows follow the segments (M_e = count_e, K fixed); A, C advance by rows,
    //         B by expert (b_e). mode 1: contraction over the segment rows (K_e = count_e);
    //         A, B advance by rows (their k index), C by expert (c_e).
    int32_t mode;
    const int32_t *offsets;  // nullptr: a single problem of M x N x K
    int32_t nseg;
    int64_t M, N, K;
    int64_t b_e, c_e;
    const void *bias;  // [nseg, N] of type tc, or nullptr
    int32_t relu;      // 1: max(.,0)
    const void *mask;  // mode 0: same shape/type as C; result multiplied by [mask > 0]
    // a second matrix continues B / C along its contiguous index from b_split / c_split on (same strides): the two gating
    // matrices [W_g | W_noise] and their gradients. b_k_contiguous: B's contraction index is the contiguous one (needed
    // where both strides are 1)
    const void *B2;
    void *C2;
    int64_t b_split, c_split;
    int32_t b_k_contiguous;
    int32_t *clear;            // status word, cleared if given
    const int32_t *row_count;  // mode 0 without segments: number of rows, read on the device (at most M)
    // optional row gathers through a permutation: mode 0: A row i reads row a_row_index[i] / a_row_div
    // and C row i is written at c_row_index[i]; mode 1: the contraction index r reads A row
    // a_row_index[r] / a_row_div and B row b_row_index[r].
    const int32_t *a_row_index;
    int32_t a_row_div;
    const int32_t *b_row_index;
    const int32_t *c_row_index;
};
// A product of float experts (few_rows.cu) over R rows; plan: with tile prefixes of heights 16 / 32 / 64
int32_t launch_float_expert_product(const SimtGemm &g, const struct SegmentPlan &plan, int64_t R, cudaStream_t st);
// partial sums of a gate's weight gradient [nparts][d][cols], to be added into dW (columns before split) and dW2 (the others), rows ld apart
struct GateParts {
    const float *part;
    int32_t nparts, d, cols, split, ld;
    float *dW, *dW2;
};
// The two products of a gate's backward pass (gate_products.cu). Rows [rows] are tokens, or slots (token = slot / row_div) in an order `perm` sorted by
// group; the groups' matrices stand one behind the other
struct GateProduct {
    const void *x;
    int32_t act, d, n, groups, row_div;
    const float *dlogit;          // [rows, n or 2 n], not sorted
    const float *W, *W2;          // [d, n] per group; W2: of the logits from n on, or nullptr
    float *dW, *dW2, *dX;         // dX [rows, d], not sorted
    int64_t rows;
    const int32_t *offsets, *perm;  // nullptr: one group
};
bool gate_rows_supported(const GateProduct &p);  // whether to
bool gate_wgrad_supported(const GateProduct &p);
int32_t launch_gate_rows(const GateProduct &p, int32_t *tile_prefix, cudaStream_t st);
int32_t launch_gate_wgrad(const GateProduct &p, float *part, cudaStream_t st, GateParts *parts_left = nullptr);
// dW (and dW2) of every group = the slices' results [splits][groups][d][cols] added in double, in slice order (gemm_simt.cu)
int32_t launch_slices_sum(float *part, int32_t splits, int32_t groups, int32_t d, int32_t cols, int32_t n, float *dW, float *dW2, cudaStream_t st);
// Mode 1 over segments: K is the number of rows of all segments. part: simt_wgrad_splits(M, N, nseg, K) * nseg * M * N
// floats let a product with few tiles be cut along its contraction (float results only)
int32_t simt_wgrad_splits(int64_t M, int64_t N, int32_t nseg, int64_t K);
int32_t launch_simt_gemm(const SimtGemm &g, int32_t *tile_prefix, cudaStream_t st, float *part = nullptr,
                         const SegmentPlan *plan = nullptr,   // plan: tile prefixes made already (heights 16 / 32 / 64)
                         GateParts *parts_left = nullptr);    // given: slices' results of a product over one segment are left to be added
constexpr int COLSUM_ROWS = 128;   // height of the tiles of ColumnSums::tile_prefix
constexpr int COLSUM_MANY = 1024;  // segments from which the pass over the tiles looks at 256 columns a block
// out[e, j] = sum over the rows of segment e of in[r, j]   (out, in of the act type): sums of tiles, then an ordered pass over them
struct ColumnSums {
    const void *in;
    void *out;
    int32_t act, nseg, N;
    int64_t R;
    const int32_t *offsets, *tile_prefix;
    float *part;  // colsum_ws_floats
    __device__ __forceinline__ void put(int32_t e, int32_t j, float v) const {
        if (act == MOE_BF16) static_cast<bf16 *>(out)[(int64_t)e * N + j] = from_f32<bf16>(v);
        else static_cast<float *>(out)[(int64_t)e * N + j] = v;
    }
};
int64_t colsum_ws_floats(int64_t R, int32_t n, int32_t N);
static inline int64_t column_tiles(const ColumnSums &a) { return cdiv(a.R, COLSUM_ROWS) + a.nseg; }
static inline int64_t column_slabs(const ColumnSums &a) { return cdiv(a.N, a.act == MOE_BF16 ? 256 : 128); }  // of 32 lanes x one 16-byte vector
int32_t launch_segment_colsum(const ColumnSums &a, cudaStream_t st);  // the tiles
int32_t launch_segment_colsum_final(const ColumnSums &a, cudaStream_t st);
// out[e, j] = sum of segment e's blocks of 32-row column sums, G blocks a tile
struct BlockSums {
    const float *part;
    const int32_t *first_tile, *offsets;
    bf16 *out;
    int32_t nseg, N, G, tile_rows;
};
// What the fused backward leaves for its last launch (0 blocks: nothing)
struct BackwardTail {
    GateParts parts;
    BlockSums blocks;
    ColumnSums columns[2];
    int32_t parts_blocks, block_blocks, column_blocks[2];
    int64_t total() const { return (int64_t)parts_blocks + block_blocks + column_blocks[0] + column_blocks[1]; }
};
// blocks up to which they go along with the rows' (whose registers leave two on an SM in bf16, one of one slot); more take one launch of their own
// (32768 rows x 512, 256 experts, 9216 blocks: 111 us together, 83 apart; 3001 rows x 320, 20 experts, 510 blocks: 10 us, apart 16)
constexpr int64_t TAIL_RIDE_MAX = 8 * 148;

// ----------------------------------------------------------------------------- tensor-core experts (ffn_tc.cu)
bool tc_ffn_supported(const moe_config &c);  // with mask bits
bool tc_ffn_takes(const moe_config &c);
// base maps of the operands that are given (nullptr: not wanted)
int32_t tc_segment_maps(const moe_config &c, SegmentMaps *maps, const void *xs_rows, const void *hid_rows, const void *dys_rows,
                        const void *dz_rows, const void *hid_cols, const void *dys_cols, const void *xs_cols, const void *dz_cols);
int32_t tc_row_tile(const moe_config &c);    // tile height of the row products: what plan.bm[0] has to be
bool tc_wgrad_sorted(const moe_config &c);   // the backward products want plan.sched
// first_only: only hid = relu(xs.W1 + b1) (the recomputation of the hidden activations in the backward pass)
int32_t launch_tc_ys(const moe_config &c, const int32_t *offsets, const void *W2, const void *b2, const void *hid, void *ys, const SegmentPlan &plan,
                     int32_t *status_word, cudaStream_t st);  // the second product alone
int32_t launch_tc_ffn(const moe_config &c, const void *xs, const int32_t *offsets, const void *W1, const void *b1,
                      const void *W2, const void *b2, void *hid, void *ys, const SegmentPlan &plan, int32_t *status_word,
                      cudaStream_t st, bool first_only = false, uint32_t *relu_bits = nullptr);
// relu_bits [R, h / 32]: one bit per hidden activation (set where hid > 0), written by the first expert GEMM if given;
// the backward then masks dz with these bits instead of reading hid again as a mask (16 times less traffic)

// ----------------------------------------------------------------------------- float experts on the tensor cores (products_f32.cu)
bool tc_float_supported(const moe_config &c, bool backward);
// three bf16 terms of a call's operands, [rows][3 columns]: rows of xs, hid, dys, dz; matrices W1 [n d][3 h], W2 [n h][3 d]
struct FloatTerms { void *xs, *hid, *dys, *dz, *W1, *W2; };
int32_t launch_float_ys(const moe_config &c, const int32_t *offsets, const void *hid, const void *W2, const void *b2, void *ys, const SegmentPlan &plan,
                        const FloatTerms &t, int32_t *status, cudaStream_t st);
// The column sums of dys and dz are the caller's
int32_t launch_float_ffn_bwd(const moe_config &c, const void *xs, const void *hid, const void *dys, const int32_t *offsets, const void *W1,
                             const void *W2, void *dxs, void *dW1, void *dW2, void *dz, const SegmentPlan &plan, const FloatTerms &t,
                             int32_t *status, cudaStream_t st);

// ----------------------------------------------------------------------------- strictly balanced gating (balanced.cu)
int32_t launch_exclusive_scan(const int32_t *counts, int32_t n, int32_t *out, cudaStream_t st,
                              int32_t *tile_sums = nullptr /* cdiv(n + 1, 4096) ints: long inputs in parallel */);  // route.cu
int64_t balanced_ws_bytes(int64_t T, int32_t n);
int32_t launch_balanced_gate(const void *x, int32_t act, int64_t T, int32_t d, int32_t n, int32_t k, const float *Wg,
                             const float *thr, float *logits, float *probs, uint32_t *mask_bits, int32_t *tok_of_row,
                             int32_t *offsets, float *den, int32_t *tok_ptr, int32_t *tok_rows, float *loss,
                             int32_t *thr_counts, void *ws, cudaStream_t st);
int32_t launch_balanced_gather(const void *x, int32_t act, const int32_t *tok_of_row, int64_t R, int64_t T, int32_t d,
                               void *xs, cudaStream_t st);
int32_t launch_balanced_combine(const void *ys, int32_t act, const float *p, const float *den, const int32_t *tok_ptr,
                                const int32_t *tok_rows, int64_t T, int64_t R, int32_t n, int32_t m, int32_t d, void *y,
                                cudaStream_t st);
int32_t launch_balanced_combine_bwd(const void *dY, const void *ys, int32_t act, const float *p, const float *den,
                                    const int32_t *tok_of_row, int64_t R, int64_t T, int32_t n, int32_t m, int32_t d,
                                    float *dG_row, void *dys, cudaStream_t st);
// dc [T, n] float, or (dsplit given) its three-term bf16 split [T, 3n] = (hi | mid | lo) for the tensor-core contractions
int32_t launch_balanced_gate_bwd(const float *p, const uint32_t *mask_bits, const float *den, const float *thr,
                                 const int32_t *tok_ptr, const int32_t *tok_rows, const float *dG_row,
                                 const int32_t *thr_counts, float w, int64_t T, int32_t n, int32_t m, float *dc,
                                 void *dsplit, float *dthr, cudaStream_t st);
int32_t launch_balanced_dispatch_bwd(const void *dxs, int32_t act, const int32_t *tok_ptr, const int32_t *tok_rows,
                                     const float *dX_gate, int64_t T, int64_t R, int32_t d, void *dX, cudaStream_t st);

int32_t launch_debug_wait(int32_t *status, unsigned long long limit_ns, cudaStream_t st);

// ----------------------------------------------------------------------------- optimiser step (optim.cu)
int64_t adam_ws_floats(int32_t n, int32_t d, int32_t h);
int32_t launch_expert_adam(int32_t act, int32_t n, int32_t d, int32_t h, void *W1, void *b1, void *W2, void *b2,
                           const void *dW1, const void *db1, const void *dW2, const void *db2, float *state, float lr,
                           float beta2, float eps, int32_t step, float *ws, cudaStream_t st);

bool tc_gate_bwd_supported(int32_t act, int32_t d, int32_t n);
int64_t tc_gate_bwd_partials(int64_t T, int32_t d, int32_t n);  // floats of partial-sum scratch
int32_t launch_tc_gate_bwd(const void *x, int64_t T, int32_t d, int32_t n, const float *Wg, const float *Wn,
                           const void *dsplit, void *wsplit, float *partials, float *dWg, float *dWn,
                           float *dX_gate, int32_t *status, cudaStream_t st, int32_t flags, int32_t ldw = 0,
                           GateParts *parts_left = nullptr);
// (ldw > 0: Wg / Wn, dWg / dWn are the left and right column halves of one [d, 2n] matrix with row stride ldw)
int32_t launch_tc_gate_fwd_grouped(const void *xs_p, int64_t P1, int32_t d, int32_t a, int32_t b, const void *wsplit_s,
                                   const int32_t *offsets_p, int32_t *tile_prefix, const int32_t *perm_p, float *clean, float *raw,
                                   int32_t *status, cudaStream_t st, int32_t flags);
bool tc_hier_gate_bwd_supported(int32_t act, int32_t d, int32_t a, int32_t b);
int32_t launch_tc_hier_secondary_bwd(const void *xs_p, const void *dsplit_s, void *wsplit_s, const float *Wg_s,
                                     const float *Wn_s, const int32_t *offsets_p, int32_t *tile_prefix, int32_t a,
                                     int64_t P1, int32_t d, int32_t b, float *partials, float *dWg_s, float *dWn_s,
                                     float *dX_sec, int32_t *status, cudaStream_t st);
int64_t tc_tile_ws_ints(int64_t R, int64_t nseg);  // int32s of a [nseg + 1] tile prefix followed by its tile table
int64_t tc_colsum_part_floats(int64_t R, int32_t nseg, int32_t N);  // scratch of the fused bias-gradient sums
// db2 (column sums of dys) is the caller's; db1_left given: the last pass over db1's block sums may be, too
int32_t launch_tc_ffn_bwd(const moe_config &c, const void *xs, const void *hid, const void *dys,
                          const int32_t *offsets, const void *W1, const void *W2, void *dxs, void *dW1, void *db1,
                          void *dW2, void *dz, float *colsum, const SegmentPlan &plan, int32_t *status_word,
                          cudaStream_t st, const uint32_t *relu_bits = nullptr, BlockSums *db1_left = nullptr);

}  // namespace moe
