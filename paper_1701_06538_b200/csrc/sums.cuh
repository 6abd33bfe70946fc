// Sums that finish the gradients of biases and gates as device code, by blocks of 256 threads: launches of their own in the stage calls,
// beside other work in the fused backward (the tile sums of a bias gradient, bound by memory, with the logit gradients, bound by
// arithmetic: gate_bwd.cu; everything that is left with the last launch: route.cu).
#pragma once

#include "moe_internal.cuh"

namespace moe {

// One block per 128-row tile and per slab of 32 * V columns (V = elements of a 16-byte vector): lane l owns V adjacent
// columns, warp w the tile's rows w, w + 8, ..., read with 16-byte loads, four rows in flight; the eight warps' sums are
// added in warp order. A segment of one tile is finished here.
template <typename XT> __device__ __forceinline__ void column_sums_partial(const ColumnSums &a, int32_t b, int32_t slab) {
    const XT *__restrict__ in = static_cast<const XT *>(a.in);
    const int32_t nseg = a.nseg, N = a.N;
    constexpr int V = 16 / sizeof(XT);
    __shared__ float sh[8][32 * V];
    __shared__ int4 tile_at;
    const int4 at = segment_of_tile(a.tile_prefix, a.offsets, nseg, b, &tile_at);
    const int lo = at.x;
    if (lo < 0) return;
    const int64_t r0 = at.y + (int64_t)at.w * COLSUM_ROWS;
    const int64_t r1 = min(r0 + (int64_t)COLSUM_ROWS, (int64_t)at.z);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t j = (slab * 32 + lane) * V;
    float s[V];
#pragma unroll
    for (int u = 0; u < V; ++u) s[u] = 0.0f;
    if (j + V <= N) {  // N is a multiple of V wherever rows are 16-byte aligned
        int64_t r = r0 + w;
        for (; r + 24 < r1; r += 32) {
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = *reinterpret_cast<const uint4 *>(in + (r + 8 * q) * N + j);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const XT *e = reinterpret_cast<const XT *>(&v[q]);
#pragma unroll
                for (int u = 0; u < V; ++u) s[u] += to_f32(e[u]);
            }
        }
        for (; r < r1; r += 8) {
            const uint4 v = *reinterpret_cast<const uint4 *>(in + r * N + j);
            const XT *e = reinterpret_cast<const XT *>(&v);
#pragma unroll
            for (int u = 0; u < V; ++u) s[u] += to_f32(e[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < V; ++u) sh[w][lane * V + u] = s[u];
    __syncthreads();
    for (int c = threadIdx.x; c < 32 * V; c += 256) {
        const int32_t col = slab * 32 * V + c;
        if (col < N) {
            float t = sh[0][c];
#pragma unroll
            for (int q = 1; q < 8; ++q) t += sh[q][c];
            if (at.z - at.y <= COLSUM_ROWS) static_cast<XT *>(a.out)[(int64_t)lo * N + col] = from_f32<XT>(t);
            else a.part[(int64_t)b * N + col] = t;
        }
    }
}

// Sum of a segment's tile sums (a segment of one tile is complete already, which with thousands of experts most are: a
// block then looks at COLS = 256 columns, 32 at a time): a block takes 32 columns, its eight warps the tiles b0 + w, b0 + w + 8, ...
// (eight loads in flight: the largest expert of a skewed batch has hundreds of tiles), the eight sums are added in warp order.
template <int COLS> __device__ __forceinline__ void column_sums_final(const ColumnSums &a, int32_t e, int32_t slab, float (&sh)[8][32]) {
    const float *__restrict__ part = a.part;
    const int32_t *__restrict__ tile_prefix = a.tile_prefix;
    const int32_t N = a.N, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t b0 = tile_prefix[e], b1 = tile_prefix[e + 1];
    if (b1 - b0 == 1) return;
    for (int32_t c = 0; c < COLS; c += 32) {
        const int32_t j0 = slab * COLS + c, j = j0 + lane;
        if (COLS > 32 && j0 >= N) break;
        float s = 0.0f;
        if (j < N) {
            int32_t b = b0 + w;
            for (; b + 8 * 7 < b1; b += 64) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = part[(int64_t)(b + 8 * u) * N + j];
#pragma unroll
                for (int u = 0; u < 8; ++u) s += v[u];
            }
            for (; b < b1; b += 8) s += part[(int64_t)b * N + j];
        }
        if (COLS > 32) __syncthreads();  // sh may still be read for the columns before
        sh[w][lane] = s;
        __syncthreads();
        if (w == 0 && j < N) {
            float t = sh[0][lane];
#pragma unroll
            for (int u = 1; u < 8; ++u) t += sh[u][lane];
            a.put(e, j, t);
        }
    }
}

// Sum of the epilogue's 32-row column sums over each segment (bias gradient), G blocks per M tile.
// A thread block takes 64 columns of one segment: 16 column lanes (four adjacent columns each, 16-byte loads) by 16 row
// lanes; row lane q takes the blocks b = b0 + q, b0 + q + 16, ... (eight loads in flight: the largest expert of a skewed
// batch has over a thousand blocks and sets this kernel's duration) and the 16 sums are added in lane order: the
// result does not depend on timing. A block takes COLS columns: 64, or, where a segment has about one tile (thousands of
// experts), 1024: a segment of at most 16 blocks is then added by one thread per four columns, in the same order. (Both
// in one kernel cost the narrow form a loop and spills: 61 us instead of 41 at 128 experts x 4096 columns.)
template <int COLS> __device__ __forceinline__ void block_sums_final(const BlockSums &a, int32_t e, int32_t slab, float4 (&sh)[16][16]) {
    const float *__restrict__ part = a.part;
    bf16 *__restrict__ out = a.out;
    const int32_t N = a.N, G = a.G, q = threadIdx.x >> 4, cl = threadIdx.x & 15;
    const int32_t b0 = a.first_tile[e] * G, b1 = b0 + (a.offsets[e + 1] - a.offsets[e] + a.tile_rows - 1) / a.tile_rows * G;
    auto store = [&](int32_t j, const float4 &t) {
        const __nv_bfloat162 o0 = __floats2bfloat162_rn(t.x, t.y), o1 = __floats2bfloat162_rn(t.z, t.w);
        uint2 pk;
        pk.x = *reinterpret_cast<const uint32_t *>(&o0); pk.y = *reinterpret_cast<const uint32_t *>(&o1);
        *reinterpret_cast<uint2 *>(out + (int64_t)e * N + j) = pk;
    };
    if (COLS > 64 && b1 - b0 <= 16) {
        const int32_t j = slab * COLS + threadIdx.x * 4;
        if (j >= N) return;
        float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
        for (int32_t b = b0; b < b1; ++b) {
            const float4 v = *reinterpret_cast<const float4 *>(part + (int64_t)b * N + j);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        store(j, s);
        return;
    }
    for (int32_t c = 0; c < COLS; c += 64) {
        const int32_t j = slab * COLS + c + cl * 4;
        if (COLS > 64 && slab * COLS + c >= N) break;
        const bool in_row = j < N;  // (N is a multiple of four)
        float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        int32_t b = in_row ? b0 + q : b1;
        for (; b + 16 * 7 < b1; b += 16 * 8) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = *reinterpret_cast<const float4 *>(part + (int64_t)(b + 16 * u) * N + j);
#pragma unroll
            for (int u = 0; u < 8; ++u) { s.x += v[u].x; s.y += v[u].y; s.z += v[u].z; s.w += v[u].w; }
        }
        for (; b < b1; b += 16) {
            const float4 v = *reinterpret_cast<const float4 *>(part + (int64_t)b * N + j);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        if (COLS > 64) __syncthreads();  // sh may still be read for the columns before
        sh[q][cl] = s;
        __syncthreads();
        if (q == 0 && in_row) {
            float4 t = sh[0][cl];
#pragma unroll
            for (int u = 1; u < 16; ++u) { t.x += sh[u][cl].x; t.y += sh[u][cl].y; t.z += sh[u][cl].z; t.w += sh[u][cl].w; }
            store(j, t);
        }
    }
}

// dW = the partial sums of a gate's weight gradient added in double, in order
__device__ __forceinline__ void gate_parts_sum(const GateParts &a, int32_t block) {
    const int64_t i = (int64_t)block * 256 + threadIdx.x, total = (int64_t)a.d * a.cols;
    if (i >= total) return;
    double s = 0.0;
    int32_t c = 0;
    for (; c + 8 <= a.nparts; c += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = a.part[(int64_t)(c + u) * total + i];
#pragma unroll
        for (int u = 0; u < 8; ++u) s += (double)v[u];
    }
    for (; c < a.nparts; ++c) s += (double)a.part[(int64_t)c * total + i];
    const int32_t q = (int32_t)(i / a.cols), j = (int32_t)(i % a.cols);
    if (j < a.split) a.dW[(int64_t)q * a.ld + j] = (float)s;
    else a.dW2[(int64_t)q * a.ld + (j - a.split)] = (float)s;
}

// what a fused backward has left for its last launch, in order of its blocks
__device__ __forceinline__ void run_backward_tail(const BackwardTail &t, int32_t block) {
    __shared__ union { float f[8][32]; float4 v[16][16]; } sh;
    if (block < t.parts_blocks) return gate_parts_sum(t.parts, block);
    block -= t.parts_blocks;
    if (block < t.block_blocks) {
        const int32_t slabs = (t.blocks.N + 63) / 64;
        return block_sums_final<64>(t.blocks, block / slabs, block % slabs, sh.v);
    }
    block -= t.block_blocks;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (block < t.column_blocks[q]) {
            const int32_t slabs = (t.columns[q].N + 31) / 32;
            return column_sums_final<32>(t.columns[q], block / slabs, block % slabs, sh.f);
        }
        block -= t.column_blocks[q];
    }
}

}  // namespace moe
