// lbm_load.cuh -- loads of data that is written while the reading kernel may
// already be resident.
#pragma once

namespace lbmk {

// Value at p, where another grid or CTA may have written during this kernel's
// life: kernels launched as programmatic dependents start before the grid
// before them ends, and a persistent kernel reads what other CTAs stored before
// a barrier. The read-only path (__ldg, or plain loads through a const
// __restrict__ parameter) is defined only for data that nobody writes while the
// kernel runs, and its loads may be moved ahead of a wait. These are served by
// the coherent L2 and, as volatile assembly that may touch memory, stay behind
// the wait or barrier before them and ahead of the stores after them.
__device__ __forceinline__ float ld_live(const float* p) {
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_live(const float2* p) {
    float2 v;
    asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float4 ld_live(const float4* p) {
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double ld_live(const double* p) {
    double v;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned ld_live(const unsigned* p) {
    unsigned v;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned short ld_live(const unsigned short* p) {
    unsigned short v;
    asm volatile("ld.global.cg.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
    return v;
}

}  // namespace lbmk
