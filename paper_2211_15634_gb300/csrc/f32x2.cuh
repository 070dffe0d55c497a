// Packed FP32 arithmetic (f32x2) for the kernels that step two rows of four nodes per thread.
#pragma once

#include <cuda_runtime.h>

namespace psd {

// Two FP32 values in one 64-bit register pair, one instruction for both.
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_make(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float f2_lo(f2 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float f2_hi(f2 v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// a - b as a fused multiply-add by -1: one rounding, the difference's (sub.f32x2 was slower)
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) { return f2_fma(b, 0xbf800000bf800000ull, a); }
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) { return f2_fma(a, 0x3f8000003f800000ull, b); }

struct V4 {  // four nodes of a row
    f2 a, b;
};
__device__ __forceinline__ V4 v4_sub(V4 x, V4 y) { return V4{f2_sub(x.a, y.a), f2_sub(x.b, y.b)}; }
struct ZCoef2 {
    f2 dtlam, ax, ay, az;
};

// Four nodes of a row 32 apart, from f.
__device__ __forceinline__ V4 v4_load32(const float *f) {
    return V4{f2_make(f[0], f[32]), f2_make(f[64], f[96])};
}

}  // namespace psd
