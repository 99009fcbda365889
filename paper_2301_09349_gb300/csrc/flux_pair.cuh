// Packed FP32x2 arithmetic of the marching fluid stages (flux_ym.cuh,
// flux_zm.cu): a float2 holds the same quantity of two faces or cells, and
// every operation is one explicit rounding (nothing is left to contraction).
#pragma once

#include "common.cuh"

namespace ibmk {
namespace {

__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return fsub2_ftz(a, b); }
__device__ __forceinline__ float2 operator*(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sp(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(rcp_ftz(a.x), rcp_ftz(a.y)); }
__device__ __forceinline__ float2 rsqrt2(float2 a) { return make_float2(rsqrtf(a.x), rsqrtf(a.y)); }
__device__ __forceinline__ float2 abs2(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ float2 max2(float2 a, float2 b) {
    return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y));
}
// products with a constant, lane by lane: a packed one would need the constant
// twice in a register pair, which costs moves
__device__ __forceinline__ float2 cmul(float c, float2 a) {
    return make_float2(__fmul_rn(c, a.x), __fmul_rn(c, a.y));
}
__device__ __forceinline__ float2 cfma(float c, float2 a, float2 b) {
    return make_float2(__fmaf_rn(c, a.x, b.x), __fmaf_rn(c, a.y, b.y));
}
__device__ __forceinline__ float2 fabs_fma(float2 a, float2 b, float2 u) {   // a b + |u|
    return make_float2(__fmaf_rn(a.x, b.x, fabsf(u.x)), __fmaf_rn(a.y, b.y, fabsf(u.y)));
}
__device__ __forceinline__ float vlh1(float a, float b) {
    const float ab = __fmul_rn(a, b);
    const float q = __fmul_rn(ab, rcp_ftz(__fadd_rn(a, b)));
    return ab > 0.0f ? q : 0.0f;
}
// half the van Leer slope, ab / (a + b) where ab > 0: the face states are
// w +- psi/2, and the factor 2 of psi = 2ab/(a+b) and the 1/2 cancel exactly
__device__ __forceinline__ float2 vlh2(float2 a, float2 b) {
    const float2 ab = a * b;
    const float2 q = ab * rcp2(a + b);
    return make_float2(ab.x > 0.0f ? q.x : 0.0f, ab.y > 0.0f ? q.y : 0.0f);
}

__device__ __forceinline__ float2 cadd(float c, float2 a) {
    return make_float2(__fadd_rn(a.x, c), __fadd_rn(a.y, c));
}

// The same operations on one face or cell.
struct F1 {
    float x;
};
__device__ __forceinline__ F1 operator+(F1 a, F1 b) { return {__fadd_rn(a.x, b.x)}; }
__device__ __forceinline__ F1 operator-(F1 a, F1 b) { return {__fsub_rn(a.x, b.x)}; }
__device__ __forceinline__ F1 operator*(F1 a, F1 b) { return {__fmul_rn(a.x, b.x)}; }
__device__ __forceinline__ F1 fma2(F1 a, F1 b, F1 c) { return {__fmaf_rn(a.x, b.x, c.x)}; }
__device__ __forceinline__ F1 rcp2(F1 a) { return {rcp_ftz(a.x)}; }
__device__ __forceinline__ F1 rsqrt2(F1 a) { return {rsqrtf(a.x)}; }
__device__ __forceinline__ F1 abs2(F1 a) { return {fabsf(a.x)}; }
__device__ __forceinline__ F1 max2(F1 a, F1 b) { return {fmaxf(a.x, b.x)}; }
__device__ __forceinline__ F1 cadd(float c, F1 a) { return {__fadd_rn(a.x, c)}; }
__device__ __forceinline__ F1 cmul(float c, F1 a) { return {__fmul_rn(c, a.x)}; }
__device__ __forceinline__ F1 cfma(float c, F1 a, F1 b) { return {__fmaf_rn(c, a.x, b.x)}; }
__device__ __forceinline__ F1 fabs_fma(F1 a, F1 b, F1 u) { return {__fmaf_rn(a.x, b.x, fabsf(u.x))}; }
__device__ __forceinline__ F1 vlh2(F1 a, F1 b) { return {vlh1(a.x, b.x)}; }

// Step-size rates of two cells, or one, of a 2D FP32 grid from their conserved
// states: s = sum_d (|u_d| + c)/h + 4 nu / h^2; p the pressure.  The one formula
// of the march, the first step size and the forced cells: every operation is an
// explicit rounding, so all of them give a state the same step size, bit for
// bit (a run continued from its own state repeats the uninterrupted one).
struct RateK {
    float gamma, gm1, s2, km, kr, ih;   // FloatConsts, ih = 1/h
};
__device__ __forceinline__ RateK rate_k(const FloatConsts &c) {
    return RateK{c.gamma, c.gm1, c.s2, c.km, c.kr, c.inv_h};
}
template <typename V>
__device__ __forceinline__ V rate_2d(const RateK &k, const V (&u)[4], V &p) {
    const V inv = rcp2(u[0]);
    const V vx = u[1] * inv, vy = u[2] * inv;
    const V rk = fma2(u[1], vx, u[2] * vy);   // rho |u|^2
    p = cmul(k.gm1, cfma(-0.5f, rk, u[3]));
    const V T = p * inv, c2 = cmul(k.gamma, T), Tf = T + T;
    const V y = cadd(k.s2, Tf);
    const V m = cmul(k.km, Tf) * (Tf * rsqrt2(Tf * y * y));   // 2 mu / h
    const V snd = c2 * rsqrt2(c2);
    return cfma(k.ih, cfma(2.0f, snd, abs2(vx) + abs2(vy)), cmul(k.kr, m) * inv);
}
__device__ __forceinline__ bool rate_ok(float rho, float p, float s) {
    return rho > 0.0f && p > 0.0f && s <= 3.0e38f;
}

}  // namespace
}  // namespace ibmk
