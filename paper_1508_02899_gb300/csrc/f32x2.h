// Two FP32 lanes in one 64-bit register pair, and the packed IEEE arithmetic of sm_100 and
// later (add/sub/mul/fma.rn.f32x2: each lane rounded exactly as the scalar instruction), used by
// the packed two-lane sweeps of the 1D and 2D steps.
#pragma once

namespace lat {

typedef unsigned long long f2;  // lane 0 in the low word

__device__ __forceinline__ f2 pk(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float lo(f2 v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return a;
}
__device__ __forceinline__ float hi(f2 v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return b;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// a - b lane by lane with scalar instructions (same rounding as sub2), for the difference of
// consecutive diffusion fluxes of the packed 1D sweep: the toolchain contracts a packed product into
// the packed add or subtract that takes it (one rounding less, other bits than the scalar sweep's).
// Later kernels form such products as fma2(a, b, an opaque zero) instead, which costs nothing.
__device__ __forceinline__ f2 sub2s(f2 a, f2 b) {
    return pk(__fsub_rn(lo(a), lo(b)), __fsub_rn(hi(a), hi(b)));
}
__device__ __forceinline__ f2 max0(f2 v) { return pk(fmaxf(lo(v), 0.f), fmaxf(hi(v), 0.f)); }
__device__ __forceinline__ f2 min0(f2 v) { return pk(fminf(lo(v), 0.f), fminf(hi(v), 0.f)); }
// Minimum and maximum that are NaN where an operand is.
__device__ __forceinline__ float min_nan(float a, float b) {
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// max(0, min(a, b, c)) where a > 0, min(0, max(a, b, c)) where a < 0, zero where a = 0, lane by lane:
// the limited increment of the sign of a, by three-input instructions.
__device__ __forceinline__ float lim_min(float a, float b, float c) {
    float lo3, hi3;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(lo3) : "f"(a), "f"(b), "f"(c));
    asm("max.f32 %0, %1, %2, %3;" : "=f"(hi3) : "f"(a), "f"(b), "f"(c));
    return fmaxf(fminf(hi3, 0.f), lo3);
}
__device__ __forceinline__ f2 lim_min2(f2 a, f2 b, f2 c) {
    return pk(lim_min(lo(a), lo(b), lo(c)), lim_min(hi(a), hi(b), hi(c)));
}
// Hides a value from the compiler's constant folding and hoisting.
__device__ __forceinline__ f2 opaque2(f2 v) {
    asm volatile("mov.b64 %0, %0;" : "+l"(v));
    return v;
}
// Koren's limiter in two lanes (lim_inc's value up to the sign of a zero).  zero2 is an opaque zero: a
// product that only feeds a packed add or subtract is formed as fma2(a, b, zero2), which keeps the
// toolchain from contracting it into that instruction (the scalar kernels round it).
struct LimPair {
    f2 mu2, third2, sixth2, zero2;
};
__device__ __forceinline__ LimPair lim_pair(float mu) {
    return LimPair{pk(mu, mu), pk(float(1.0 / 3.0), float(1.0 / 3.0)),
                   pk(float(1.0 / 6.0), float(1.0 / 6.0)), opaque2(0ull)};
}
__device__ __forceinline__ f2 lim_inc_x2(f2 dp, f2 dm, const LimPair& k) {
    return lim_min2(dp, fma2(dm, k.sixth2, mul2(dp, k.third2)), mul2(k.mu2, dm));
}

}  // namespace lat
