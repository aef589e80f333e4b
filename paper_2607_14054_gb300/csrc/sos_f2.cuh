// Pairs of FP32 values in one 64-bit register and the packed arithmetic on
// them (PTX fma/add/mul.rn.f32x2): one instruction does two independent FP32
// operations, each rounded exactly as its scalar form.  The FMA pipe takes a
// packed instruction in two cycles and a scalar one in one (measured 0.49 and
// 0.95 warp instructions per clock and scheduler), so the arithmetic rate is
// the same, but half the issue slots carry it and the other half are left for
// shuffles, loads and selects.
#pragma once

#include <cuda_runtime.h>

namespace sosf {

using f2x = unsigned long long;  // (low, high) FP32 pair

__device__ __forceinline__ f2x f2_pack(float a, float b) {
    f2x d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ f2x f2_dup(float a) { return f2_pack(a, a); }
__device__ __forceinline__ void f2_unpack(f2x v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ float f2_a(f2x v) {
    float a, b;
    f2_unpack(v, a, b);
    return a;
}
__device__ __forceinline__ float f2_b(f2x v) {
    float a, b;
    f2_unpack(v, a, b);
    return b;
}
__device__ __forceinline__ f2x f2_fma(f2x a, f2x b, f2x c) {
    f2x d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2x f2_add(f2x a, f2x b) {
    f2x d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2x f2_mul(f2x a, f2x b) {
    f2x d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

}  // namespace sosf
