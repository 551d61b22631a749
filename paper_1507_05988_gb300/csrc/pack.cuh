// pack.cuh -- packed pairs of FP32 values: the same quantity of two rows (row
// stage) or two lines (Cartesian line stage) in the halves of one 64-bit register
// pair, one add/mul/fma.rn.f32x2 per operation of both (each half an IEEE
// single operation; constants and coefficients are shared by the halves).
#pragma once
#include "fcn_device.cuh"

namespace fcn {
namespace {

// Two FP32 values handled by one packed instruction.
struct alignas(8) pk2 {
    float a, b;
};
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
__device__ __forceinline__ pk2 operator+(pk2 p, pk2 q) {
    const float2 r = __fadd2_rn(make_float2(p.a, p.b), make_float2(q.a, q.b));
    return {r.x, r.y};
}
__device__ __forceinline__ pk2 operator*(pk2 p, pk2 q) {
    const float2 r = __fmul2_rn(make_float2(p.a, p.b), make_float2(q.a, q.b));
    return {r.x, r.y};
}
__device__ __forceinline__ pk2 vfma(pk2 p, pk2 q, pk2 c) {
    const float2 r = __ffma2_rn(make_float2(p.a, p.b), make_float2(q.a, q.b), make_float2(c.a, c.b));
    return {r.x, r.y};
}
#else
__device__ __forceinline__ pk2 operator+(pk2 p, pk2 q) { return {p.a + q.a, p.b + q.b}; }
__device__ __forceinline__ pk2 operator*(pk2 p, pk2 q) { return {p.a * q.a, p.b * q.b}; }
__device__ __forceinline__ pk2 vfma(pk2 p, pk2 q, pk2 c) { return {fmaf(p.a, q.a, c.a), fmaf(p.b, q.b, c.b)}; }
#endif
__device__ __forceinline__ pk2 operator-(pk2 p) { return {-p.a, -p.b}; }
__device__ __forceinline__ pk2 operator-(pk2 p, pk2 q) { return p + (-q); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }

// V: the value type a thread computes with (float, double or pk2), T =
// Pack<V>::S its scalar, L = Pack<V>::L the problems (rows, pulses) it
// carries.
template <typename V>
struct Pack {
    using S = V;
    static constexpr int L = 1;
    __device__ __forceinline__ static V splat(V s) { return s; }
};
template <>
struct Pack<pk2> {
    using S = float;
    static constexpr int L = 2;
    __device__ __forceinline__ static pk2 splat(float s) { return {s, s}; }
};

}  // namespace
}  // namespace fcn
