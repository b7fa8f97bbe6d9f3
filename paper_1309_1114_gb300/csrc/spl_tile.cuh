// spl_tile.cuh -- shared-memory access by address for the additive passes
// (spl_tile.cu) and the general absorption pass (spl_absorb.cu).
#pragma once
#include "spl_geom.cuh"

namespace spl {

// Bits 0, 4, ..., 28 of v gathered into the low byte.
__device__ __forceinline__ unsigned every_fourth(unsigned v) {
    v &= 0x11111111u;
    v = (v | (v >> 3)) & 0x03030303u;
    v = (v | (v >> 6)) & 0x000f000fu;
    return (v | (v >> 12)) & 0xffu;
}

// Shared memory by 32-bit address, and 16-byte asynchronous copies into it.
__device__ __forceinline__ float4 lds4(unsigned a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void lds2x2(unsigned a, f32x2 &u, f32x2 &v) {
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(u), "=l"(v) : "r"(a));
}
__device__ __forceinline__ uint4 ldsu4(unsigned a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts2x2(unsigned a, f32x2 u, f32x2 v) {
    asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(a), "l"(u), "l"(v) : "memory");
}
__device__ __forceinline__ void sts2(unsigned a, f32x2 u) {
    asm volatile("st.shared.b64 [%0], %1;" ::"r"(a), "l"(u) : "memory");
}
__device__ __forceinline__ unsigned lds_u8(unsigned a) {
    unsigned v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ unsigned lds_u16(unsigned a) {
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u8(unsigned a, unsigned v) {
    asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

__device__ __forceinline__ void cp_async16(unsigned dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

}  // namespace spl
