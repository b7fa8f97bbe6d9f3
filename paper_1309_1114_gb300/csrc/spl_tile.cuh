// spl_tile.cuh -- shared-memory access by address for the additive passes
// (spl_tile.cu), and the band geometry of the general absorption pass
// (spl_absorb.cu).
#pragma once
#include "spl_geom.cuh"

namespace spl {

template <int T>
struct Shape {
    // A tile is cut into 8 row bands, one per warp: BW columns x BH rows.
    static constexpr int BW = T == 64 ? 64 : 16;
    static constexpr int BH = T * T / (8 * BW);
    static constexpr int NBX = T / BW;             // bands across the tile
    // lanes along a band row: 8 for T = 32, so that a lane's two columns
    // share each row-pair load and the column table is read 16 bytes at a time
    static constexpr int LW = T == 32 ? 8 : (BW < 32 ? BW : 32);
    // a lane's columns: col + CSTEP k, k < CPL, col = band column + CMUL * (lane % LW)
    static constexpr int CSTEP = T == 32 ? 1 : 32;
    static constexpr int CMUL = T == 32 ? 2 : 1;
    static constexpr int G = 32 / LW;              // lane groups (rows split between them)
    static constexpr int CPL = BW / LW;            // columns per lane
    static constexpr int RPL = BH / G;             // rows per lane
    static constexpr int P = 32;                   // particles per tabulated batch
    static constexpr int PER = T / 8;              // table columns (and rows) per thread
    static constexpr bool PAIRED = RPL % 2 == 0;   // rows two at a time (FP32x2)
    // row stride of the column table: 8 entries of padding put the two
    // particles that a half-warp's 64-bit stores reach in different banks
    static constexpr int WXS = T + 8;
};

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
