// Sixteen bytes from global to shared memory without a register in between, several groups in flight; and multiply-adds in pairs
#pragma once

#include <stdint.h>

namespace moe {

__device__ __forceinline__ void copy16(void *to, const void *from) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}
__device__ __forceinline__ void copy4(void *to, const void *from) {  // the same with four bytes
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}
// else zeros (`from` is not read, but valid)
__device__ __forceinline__ void copy16(void *to, const void *from, bool live) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy4(void *to, const void *from, bool live) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from), "r"(live ? 4 : 0) : "memory");
}
// zeros by a store: copies of zeros from one address go one by one
__device__ __forceinline__ void zero16(void *to) { *reinterpret_cast<uint4 *>(to) = make_uint4(0u, 0u, 0u, 0u); }
__device__ __forceinline__ void zero4(void *to) { *reinterpret_cast<uint32_t *>(to) = 0u; }
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }  // all but the last N groups are there

// two fused multiply-adds with one instruction (each rounded as fmaf rounds it): c += a * b
__device__ __forceinline__ void fma_two(float &c0, float &c1, float a, float b0, float b1) {
    asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%2, %2};\n mov.b64 b, {%3, %4};\n mov.b64 c, {%0, %1};\n"
        " fma.rn.f32x2 c, a, b, c;\n mov.b64 {%0, %1}, c;\n}"
        : "+f"(c0), "+f"(c1) : "f"(a), "f"(b0), "f"(b1));
}

}  // namespace moe
