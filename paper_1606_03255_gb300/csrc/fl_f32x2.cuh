// fl_f32x2.cuh -- packed pairs of floats (the f32x2 instructions of sm_100 and
// later): one instruction issues two independent single-precision operations.
// Measured on GB300: fma.rn.f32x2 1.79 warp instructions per SM and clock, i.e.
// the same arithmetic rate as scalar fma at half the issue slots, which is what
// kernels bound by instruction issue gain from.  Each half is rounded exactly
// as the scalar operation.
#pragma once

#include <cuda_runtime.h>

namespace fl {

struct f2 {
    unsigned long long v;
};

__device__ __forceinline__ f2 f2_make(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f2 f2_dup(float x) { return f2_make(x, x); }
__device__ __forceinline__ float f2_lo(f2 a) {
    return __uint_as_float((unsigned)a.v);
}
__device__ __forceinline__ float f2_hi(f2 a) {
    return __uint_as_float((unsigned)(a.v >> 32));
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

}  // namespace fl
