// pair.cuh -- two values of one type worked on together.  Two floats share a
// 64-bit register pair and go through Blackwell's packed FP32 instructions
// (add/mul/fma .rn.f32x2: one instruction for two correctly rounded results, the
// same rounding as the scalar ones); two doubles are two scalar operations.
#pragma once

#include <cuda_runtime.h>

namespace fem {

template <typename T>
struct Pair;

template <>
struct Pair<float> {
    unsigned long long v;
};
template <>
struct Pair<double> {
    double x, y;
};

__device__ __forceinline__ Pair<float> pair(float lo, float hi) {
    Pair<float> r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float pair_lo(Pair<float> p) { return __uint_as_float((unsigned)p.v); }
__device__ __forceinline__ float pair_hi(Pair<float> p) { return __uint_as_float((unsigned)(p.v >> 32)); }
__device__ __forceinline__ Pair<float> operator+(Pair<float> a, Pair<float> b) {
    Pair<float> r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Pair<float> pfma(Pair<float> a, Pair<float> b, Pair<float> c) {
    Pair<float> r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// a b + 0: a plain mul.rn.f32x2 followed by an addition was fused by the assembler in
// one kernel and not in another, and builds have to agree bit for bit.
__device__ __forceinline__ Pair<float> operator*(Pair<float> a, Pair<float> b) { return pfma(a, b, Pair<float>{0ull}); }
__device__ __forceinline__ Pair<float> operator-(Pair<float> a, Pair<float> b) {
    Pair<float> r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Pair<float> operator-(Pair<float> a) { return Pair<float>{0ull} - a; }

__device__ __forceinline__ Pair<double> pair(double lo, double hi) { return {lo, hi}; }
__device__ __forceinline__ double pair_lo(Pair<double> p) { return p.x; }
__device__ __forceinline__ double pair_hi(Pair<double> p) { return p.y; }
__device__ __forceinline__ Pair<double> operator+(Pair<double> a, Pair<double> b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Pair<double> operator-(Pair<double> a, Pair<double> b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ Pair<double> operator*(Pair<double> a, Pair<double> b) { return {a.x * b.x, a.y * b.y}; }
__device__ __forceinline__ Pair<double> operator-(Pair<double> a) { return {-a.x, -a.y}; }
__device__ __forceinline__ Pair<double> pfma(Pair<double> a, Pair<double> b, Pair<double> c) {
    return {fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
}

}  // namespace fem
