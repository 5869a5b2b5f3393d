// Device helpers shared by the FD stage kernels (one launch per stage) and
// the temporally blocked FD kernel (all stages of a step in one launch): the
// WENO-5 interface value (Sec. 2, Jiang-Shu), lane arithmetic and periodic
// index wrapping.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace lbm {

// Pairs of values evaluated together (V holds two). For float they map to
// the packed FP32x2 instructions of sm_100+ (one instruction, two results);
// for double they are two scalar operations.
template <typename T>
struct Pr;

template <>
struct Pr<float> {
    using V = float2;
    static constexpr int N = 2;
    static __device__ __forceinline__ V mk(float a, float b) { return make_float2(a, b); }
    static __device__ __forceinline__ V sp(float a) { return make_float2(a, a); }
    static __device__ __forceinline__ float get(V a, int h) { return h ? a.y : a.x; }
    static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
    static __device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
    static __device__ __forceinline__ V neg(V a) { return make_float2(-a.x, -a.y); }
    static __device__ __forceinline__ V sub(V a, V b) { return __fadd2_rn(a, neg(b)); }
    // a product that enters a sum as rounded: the compiler may fuse a packed
    // product and a packed sum into one multiply-add, differently where the
    // product is used once or twice; an added zero keeps them apart
    static __device__ __forceinline__ V mulr(V a, V b) { return __ffma2_rn(a, b, make_float2(0.f, 0.f)); }
    // with a literal c: scalar instructions, whose immediate operand is read
    // from the instruction
    static __device__ __forceinline__ V mulc(V a, float c) { return make_float2(__fmul_rn(a.x, c), __fmul_rn(a.y, c)); }
    static __device__ __forceinline__ V fmac(V a, float c, V b) {
        return make_float2(__fmaf_rn(a.x, c, b.x), __fmaf_rn(a.y, c, b.y));
    }
    static __device__ __forceinline__ V rcp(V b) { return make_float2(fast_rcp(b.x), fast_rcp(b.y)); }
    // once per node, not per face: refined by a Newton step r + r (1 - b r), to
    // within an ulp of 1 / b (a division in the moments cost 9 velocities 4%)
    static __device__ __forceinline__ V rcp_node(V b) {
        const V r = rcp(b);
        return fma(fma(neg(b), r, make_float2(1.f, 1.f)), r, r);
    }
};

template <>
struct Pr<double> {
    using V = double2;
    static constexpr int N = 2;
    static __device__ __forceinline__ V mk(double a, double b) { return make_double2(a, b); }
    static __device__ __forceinline__ V sp(double a) { return make_double2(a, a); }
    static __device__ __forceinline__ V add(V a, V b) { return make_double2(a.x + b.x, a.y + b.y); }
    static __device__ __forceinline__ V mul(V a, V b) { return make_double2(a.x * b.x, a.y * b.y); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return make_double2(::fma(a.x, b.x, c.x), ::fma(a.y, b.y, c.y)); }
    static __device__ __forceinline__ V neg(V a) { return make_double2(-a.x, -a.y); }
    static __device__ __forceinline__ V sub(V a, V b) { return make_double2(a.x - b.x, a.y - b.y); }
    static __device__ __forceinline__ V mulr(V a, V b) { return make_double2(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y)); }
    static __device__ __forceinline__ V mulc(V a, double c) { return make_double2(a.x * c, a.y * c); }
    static __device__ __forceinline__ V fmac(V a, double c, V b) { return fma(a, sp(c), b); }
    static __device__ __forceinline__ V rcp(V b) { return make_double2(fast_rcp(b.x), fast_rcp(b.y)); }
};

// What a lane of the stage kernels computes with: for float two nodes at a
// time (Pr<float>), for double one node (N = 1; mk keeps the first value).
template <typename T>
struct Lanes;

template <>
struct Lanes<float> : Pr<float> {};

template <>
struct Lanes<double> {
    using V = double;
    static constexpr int N = 1;
    static __device__ __forceinline__ V mk(double a, double) { return a; }
    static __device__ __forceinline__ V sp(double a) { return a; }
    static __device__ __forceinline__ double get(V a, int) { return a; }
    // contraction-proof: the same operations in every instantiation
    static __device__ __forceinline__ V add(V a, V b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ V mul(V a, V b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __fma_rn(a, b, c); }
    static __device__ __forceinline__ V neg(V a) { return -a; }
    static __device__ __forceinline__ V sub(V a, V b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ V mulr(V a, V b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ V mulc(V a, double c) { return __dmul_rn(a, c); }
    static __device__ __forceinline__ V fmac(V a, double c, V b) { return __fma_rn(a, c, b); }
    static __device__ __forceinline__ V rcp(V b) { return fast_rcp(b); }
    static __device__ __forceinline__ V rcp_node(V b) { return fast_rcp(b); }
};

// WENO-5 interface value (Jiang-Shu) of the face i+1/2 from the four node
// differences d1 .. d4 = f_{i-2} - f_{i-1}, ..., f_{i+1} - f_{i+2} of its
// upwind-ordered stencil (exact for close values; this sign needs no
// negations below).
//   candidates, relative to f_i: q0 = (2 d1 - 5 d2)/6, q1 = -(d2 + 2 d3)/6,
//   q2 = (d4 - 4 d3)/6;
//   smoothness (13/12 t^2 + 1/4 u^2 of the three stencils, t, u their second
//   and first differences): 3/4 beta_0 = d1^2 - 11/4 d1 d2 + 5/2 d2^2, 3/4
//   beta_1 = d2^2 - 5/4 d2 d3 + d3^2, 3/4 beta_2 = d4^2 - 11/4 d4 d3 + 5/2 d3^2.
//   Completing the square leaves the same term 39/64 d2^2 in beta_0 and
//   beta_1 (and 39/64 d3^2 in beta_2): with F(d) = 39/64 d^2 + 3/4 eps,
//     s0 = (d1 - 11/8 d2)^2 + F(d2), s1 = (d3 - 5/8 d2)^2 + F(d2),
//     s2 = (d4 - 11/8 d3)^2 + F(d3),  s_r = 3/4 (eps + beta_r):
//   sums of squares (no cancellation) and F is shared, between two candidates
//   and with the next face along the axis.
//   weights alpha_r = d_r / (eps + beta_r)^2, d = (1/10, 6/10, 3/10), face =
//   sum alpha_r q_r / sum alpha_r; a common factor on every alpha_r drops
//   out, so numerator and denominator are multiplied by s0^2 s1^2 s2^2: one
//   reciprocal per face.
// Returns 3 (face - f_i): a small number next to f_i, so its rounding is small
// next to the flux differences it feeds. 15 operations and a reciprocal, plus
// 10 for the s_r and 4 for the differences (the textbook form takes 64).
template <typename P, typename T>
__device__ __forceinline__ typename P::V weno5_f(typename P::V d, typename P::V eps_s) {
    return P::fma(P::mulc(d, T(39.0 / 64.0)), d, eps_s);
}
template <typename P, typename T>
__device__ __forceinline__ typename P::V weno5_diff(typename P::V d1, typename P::V d2, typename P::V d3,
                                                    typename P::V d4, typename P::V f2, typename P::V f3) {
    using V = typename P::V;
    const V x0 = P::fmac(d2, T(-1.375), d1);
    const V x1 = P::fmac(d2, T(-0.625), d3);
    const V x2 = P::fmac(d3, T(-1.375), d4);
    V s0 = P::fma(x0, x0, f2), s1 = P::fma(x1, x1, f2), s2 = P::fma(x2, x2, f3);
    s0 = P::mul(s0, s0);
    s1 = P::mul(s1, s1);
    s2 = P::mul(s2, s2);
    const V q0 = P::fmac(d2, T(-2.5), d1);   // 3 (q0 - f_i)
    const V q1 = P::fmac(d2, T(0.5), d3);    // -3 (q1 - f_i)
    const V q2 = P::fmac(d4, T(-0.25), d3);  // -3/2 (q2 - f_i)
    const V a = P::mulc(s0, T(6)), b = P::mul(a, s1);
    const V num = P::fma(s2, P::fma(P::neg(a), q1, P::mul(s1, q0)), P::neg(P::mul(b, q2)));
    const V den = P::fmac(b, T(0.5), P::mul(s2, P::fmac(s0, T(6), s1)));
    return P::mulr(num, P::rcp(den));
}
template <typename P, typename T>
__device__ __forceinline__ typename P::V weno5_vals(typename P::V a, typename P::V b, typename P::V c, typename P::V d,
                                                    typename P::V e, typename P::V eps_s) {
    using V = typename P::V;
    const V d1 = P::sub(a, b), d2 = P::sub(b, c), d3 = P::sub(c, d), d4 = P::sub(d, e);
    return weno5_diff<P, T>(d1, d2, d3, d4, weno5_f<P, T>(d2, eps_s), weno5_f<P, T>(d3, eps_s));
}

__device__ __forceinline__ int wrapi(int i, int n) {
    i %= n;
    return i < 0 ? i + n : i;
}

// The same for an i that is mostly within one period of [0, n).
__device__ __forceinline__ int wrap_near(int i, int n) {
    if (i < 0) i += n;
    else if (i >= n) i -= n;
    return (unsigned)i < (unsigned)n ? i : wrapi(i, n);
}

}  // namespace lbm
