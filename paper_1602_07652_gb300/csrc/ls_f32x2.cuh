// ls_f32x2.cuh -- pairs of FP32 values in one 64-bit register and the packed instructions of
// sm_100+ on them (add/sub/mul/fma .rn.f32x2: two IEEE single-precision operations, each
// rounded to nearest, in one instruction).  Device code only.
#pragma once

namespace {

struct F2 {
    unsigned long long r;
};
__device__ __forceinline__ F2 f2(float lo, float hi) {
    F2 o;
    asm("mov.b64 %0, {%1, %2};" : "=l"(o.r) : "f"(lo), "f"(hi));
    return o;
}
__device__ __forceinline__ F2 f2s(float a) { return f2(a, a); }
__device__ __forceinline__ void f2split(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.r));
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 o;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(o.r) : "l"(a.r), "l"(b.r));
    return o;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
    F2 o;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(o.r) : "l"(a.r), "l"(b.r));
    return o;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 o;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(o.r) : "l"(a.r), "l"(b.r));
    return o;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {  // a b + c
    F2 o;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(o.r) : "l"(a.r), "l"(b.r), "l"(c.r));
    return o;
}
__device__ __forceinline__ F2 neg2(F2 a) {  // flips both sign bits
    F2 o;
    asm("xor.b64 %0, %1, 0x8000000080000000;" : "=l"(o.r) : "l"(a.r));
    return o;
}

}  // namespace
