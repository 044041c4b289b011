// packed.cuh -- two FP32 lanes in one 64-bit register: one packed instruction
// evaluates an operation for two interactions, which halves the FP32
// instructions a scheduler issues.  Each lane is rounded as the scalar
// instruction.  FTZ: subnormal operands and results count as zero.
#pragma once

namespace fdps {

typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pk(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_up(f2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
template <bool FTZ = false>
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 d;
    if (FTZ)
        asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    else
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
template <bool FTZ = false>
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 d;
    if (FTZ)
        asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    else
        asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
template <bool FTZ = false>
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 d;
    if (FTZ)
        asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    else
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
template <bool FTZ = false>
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 d;
    if (FTZ)
        asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    else
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// rsqrtf for arguments that are no subnormals: the bare MUFU operation
__device__ __forceinline__ float rsqrt_normal(float v) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

}  // namespace fdps
