// Two FP32 values in a 64-bit register: one fma.rn.f32x2 issues two FMAs (the FMA rate and
// the roundings are those of scalar FMAs; half the issue slots stay free for loads).
#pragma once

namespace mpiffl {

using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ f32x2 dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// The same names on one value, for kernels that take one line or two.
template <bool TWO>
struct Lines;
template <>
struct Lines<true> {
    using V = f32x2;
    static __device__ __forceinline__ V pair(float a, float b) { return pack2(a, b); }
    static __device__ __forceinline__ V dup(float a) { return dup2(a); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return fma2(a, b, c); }
    static __device__ __forceinline__ V add(V a, V b) { return add2(a, b); }
    static __device__ __forceinline__ float2 parts(V v) { return unpack2(v); }
};
template <>
struct Lines<false> {
    using V = float;
    static __device__ __forceinline__ V pair(float a, float) { return a; }
    static __device__ __forceinline__ V dup(float a) { return a; }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return fmaf(a, b, c); }
    static __device__ __forceinline__ V add(V a, V b) { return a + b; }
    static __device__ __forceinline__ float2 parts(V v) { return make_float2(v, 0.f); }
};

}  // namespace mpiffl
