// Packed FP32 arithmetic: two FP32 values in one 64-bit register pair, each
// operation one instruction on both (add/fma.rn.f32x2, round to nearest,
// the same bits as two scalar operations).  On GB300 a packed FMA issues at the
// rate of a scalar one (measured: 16 independent FMAs per warp and iteration
// take 16.3 cycles of a scheduler either way), so it halves the issue slots and
// doubles the FP32 rate of work that comes in pairs.
#pragma once
#include <stdint.h>

namespace sphg {

typedef unsigned long long f2;  // (lo, hi)

__device__ __forceinline__ f2 f2_make(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f2 f2_dup(float v) { return f2_make(v, v); }
__device__ __forceinline__ float f2_lo(f2 a) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
    return lo;
}
__device__ __forceinline__ float f2_hi(f2 a) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
    return hi;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// approximate reciprocal and reciprocal square root of normal arguments (the
// callers keep them away from zero and the subnormals, so flushing changes nothing)
__device__ __forceinline__ float rcp_fast(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float rsqrt_fast(float a) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

}  // namespace sphg
