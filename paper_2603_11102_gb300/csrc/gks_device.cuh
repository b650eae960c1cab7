// gks_device.cuh -- device building blocks shared by the forward stencil
// (gks_stencil.cu) and its adjoint (gks_adjoint.cu): physical constants,
// WENO5-JS, the tangential Gauss-point stencils, the closed-form
// gas-kinetic flux, and the TMA / mbarrier helpers. Internal header.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "gks_ds.cuh"
#include "gks_internal.h"

namespace gks {
namespace dev {

template <typename R>
struct Phys {
    R lambda, theta, mu, off, sqlam, kE;
};

template <typename R>
Phys<R> make_phys(const Ctx &c)
{
    Phys<R> p;
    p.lambda = (R)c.lambda;
    p.theta = (R)c.theta;
    p.mu = (R)c.mu;
    p.off = (R)c.off;
    p.sqlam = (R)sqrt(c.lambda);
    p.kE = (R)(1.0 / (2.0 * sqrt(3.14159265358979323846 * c.lambda)));
    return p;
}

// |U|^2 of a cell for the CFL time step, with every operation rounded
// explicitly so that each kernel that forms it gets the same bits: FP32C from
// hi + lo in FP32, FP64 from the state. max_u2 keeps a NaN.
__device__ __forceinline__ float cell_u2f(const float h[4], const float l[4])
{
    const float r = __fadd_rn(h[0], l[0]), a = __fadd_rn(h[1], l[1]);
    const float b = __fadd_rn(h[2], l[2]), c = __fadd_rn(h[3], l[3]);
    const float m2 = __fadd_rn(__fadd_rn(__fmul_rn(a, a), __fmul_rn(b, b)), __fmul_rn(c, c));
    return __fdiv_rn(m2, __fmul_rn(r, r));
}
__device__ __forceinline__ double cell_u2(const double w[4])
{
    const double m2 = __dadd_rn(__dadd_rn(__dmul_rn(w[1], w[1]), __dmul_rn(w[2], w[2])), __dmul_rn(w[3], w[3]));
    return __ddiv_rn(m2, __dmul_rn(w[0], w[0]));
}
__device__ __forceinline__ double max_u2(double a, double b) { return (b > a || b != b) ? b : a; }
__device__ __forceinline__ float max_u2f(float a, float b) { return (b > a || b != b) ? b : a; }

// Block-wide max of v (blockDim.x * blockDim.y threads, a multiple of 32,
// at most 1024) folded into *bits (a non-negative double) by one atomicMax,
// left out when *bits is already no smaller (it only grows during the launch).
__device__ __forceinline__ void block_max_to(double v, unsigned long long *bits)
{
    __shared__ double red[32];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, nw = (blockDim.x * blockDim.y) >> 5;
    for (int o = 16; o > 0; o >>= 1) v = max_u2(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < nw; ++w) v = max_u2(v, red[w]);
        const unsigned long long b = (unsigned long long)__double_as_longlong(v);
        if (b > *(volatile unsigned long long *)bits) atomicMax(bits, b);
    }
}

// Direction d: normal axis d, tangential axes t1, t2.
__host__ __device__ inline int tan1(int d) { return d == 0 ? 1 : 0; }
__host__ __device__ inline int tan2(int d) { return d == 2 ? 1 : 2; }

// WENO5-JS (Sec. 2): eps_w = 1e-6, power 2, linear weights 1/10, 6/10, 3/10
// on the candidate stencils (a,b,c), (b,c,d), (c,d,e) for the right face of
// the centre cell c.
// Both face values of the centre cell of q[0..4] (cells -2..2) from one set
// of Jiang-Shu smoothness indicators: the value at the right face (+1/2) and,
// with the stencils mirrored, at the left face (-1/2). The mirrored
// indicators are the same numbers in reverse order, so they are computed
// once. With s_k = (eps + beta_k)^2 the weights d_k / s_k are scaled by
// 10 s0 s1 s2 (linear weights 1/10, 6/10, 3/10 -> 1, 6, 3) and the 1/6 of the
// candidate polynomials moves into the one division per face value.
template <typename R>
__device__ __forceinline__ void weno5_pair(const R q[5], R &right, R &left)
{
    const R c13 = R(13.0 / 12.0), qq = R(0.25);
    const R a = q[0], b = q[1], c = q[2], d = q[3], e = q[4];
    R t = a - R(2) * b + c, u = a - R(4) * b + R(3) * c;
    R s0 = R(1e-6) + (c13 * t * t + qq * u * u);
    t = b - R(2) * c + d; u = b - d;
    R s1 = R(1e-6) + (c13 * t * t + qq * u * u);
    t = c - R(2) * d + e; u = R(3) * c - R(4) * d + e;
    R s2 = R(1e-6) + (c13 * t * t + qq * u * u);
    s0 *= s0; s1 *= s1; s2 *= s2;
    const R w02 = R(6) * (s0 * s2), s01 = s0 * s1, s12 = s1 * s2;
    // right face: candidates 6 p_k on (a,b,c), (b,c,d), (c,d,e)
    {
        const R p0 = R(2) * a - R(7) * b + R(11) * c;
        const R p1 = -b + R(5) * c + R(2) * d;
        const R p2 = R(2) * c + R(5) * d - e;
        const R w2 = R(3) * s01;
        right = (s12 * p0 + w02 * p1 + w2 * p2) / (R(6) * (s12 + w02 + w2));
    }
    // left face: candidates on (e,d,c), (d,c,b), (c,b,a) with indicators s2, s1, s0
    {
        const R p0 = R(2) * e - R(7) * d + R(11) * c;
        const R p1 = -d + R(5) * c + R(2) * b;
        const R p2 = R(2) * c + R(5) * b - a;
        const R w2 = R(3) * s12;
        left = (s01 * p0 + w02 * p1 + w2 * p2) / (R(6) * (s01 + w02 + w2));
    }
}

// erf(z), exp(-z^2) - 1 and exp(-z^2) of the half-space moments, z =
// sqrt(lambda) U. For |z| <= 1/2 (|U| up to 7 U_ref at Ma 0.1), with t = z^2:
//   erf z = z E(t),  exp(-t) - 1 = -t X(-t),
// E and X in FP64 and double-single as polynomials of least deviation on 0 <=
// t <= 1/4 (Chebyshev fits of the two Maclaurin series), of degree 8 (within
// 4.3e-18 and 7.3e-18), 8 multiply-adds less per pair than the truncated series
// of the same accuracy. exp = 1 + expm1. Beyond 1/2 the library functions.
template <typename T>
__device__ __forceinline__ void half_space_polys(T t, T x, T &E, T &X)
{
    constexpr double ce[9] = {1.4725865480556743912e-6, -0.000014845849259707869768, 0.00012053335124353740746,
                              -0.00085482977536749668828, 0.0052239773730214700169, -0.026866170632887929351,
                              0.11283791670925353147, -0.37612638903183473544, 1.1283791670955125696};
    constexpr double cx[9] = {2.4634585655528519648e-6, 0.000024667266113234713626, 0.00019837907206591588519,
                              0.001388883962567040931, 0.0083333329084976221444, 0.041666666646060813782,
                              0.166666666666165589, 0.49999999999999530577, 0.99999999999999999276};
    E = T(ce[0]);
    X = T(cx[0]);
#pragma unroll
    for (int k = 1; k < 9; ++k) {
        E = fma(E, t, T(ce[k]));
        X = fma(X, x, T(cx[k]));
    }
}
// FP32: the truncated Maclaurin series themselves (n = 0..6 and 1..7, first
// dropped terms below 4e-10 and 2e-9 relative). Shorter polynomials of the same
// accuracy round differently, and the FP32C gradients follow (WenoWindow).
template <typename T>
__device__ __forceinline__ void half_space_series32(T t, T x, T &E, T &X)
{
    constexpr double k = 1.1283791670955126;   // 2 / sqrt(pi)
    constexpr double ce[7] = {k / (720.0 * 13.0), -k / (120.0 * 11.0), k / (24.0 * 9.0), -k / (6.0 * 7.0),
                              k / (2.0 * 5.0), -k / 3.0, k};
    constexpr double cx[7] = {1.0 / 5040.0, 1.0 / 720.0, 1.0 / 120.0, 1.0 / 24.0, 1.0 / 6.0, 0.5, 1.0};
    E = T(ce[0]);
    X = T(cx[0]);
#pragma unroll
    for (int i = 1; i < 7; ++i) {
        E = fma(E, t, T(ce[i]));
        X = fma(X, x, T(cx[i]));
    }
}
__device__ __forceinline__ void half_space_terms(double z, double &e, double &m1, double &ex)
{
    const double t = z * z, x = -t;
    if (fabs(z) <= 0.5) {
        double E, X;
        half_space_polys(t, x, E, X);
        e = E * z;
        m1 = X * x;
        ex = fma(X, x, 1.0);
    } else {
        e = erf(z);
        m1 = expm1(x);
        ex = exp(x);
    }
}
__device__ __forceinline__ void half_space_terms(float z, float &e, float &m1, float &ex)
{
    const float t = __fmul_rn(z, z), x = -t;
    if (fabsf(z) <= 0.5f) {
        float E, X;
        half_space_series32(t, x, E, X);
        e = __fmul_rn(E, z);
        m1 = __fmul_rn(X, x);
        ex = __fadd_rn(1.0f, m1);
    } else {
        e = erff(z);
        m1 = expm1f(x);
        ex = expf(x);
    }
}

// Value conversion between a storage type and a compute type (identity, or
// double <-> double-single).
template <typename T>
__device__ __forceinline__ T cvt(double x) { return (T)x; }
template <>
__device__ __forceinline__ dsf cvt<dsf>(double x) { return to_ds(x); }
template <typename T>
__device__ __forceinline__ T cvt(float x) { return (T)x; }
template <typename T>
__device__ __forceinline__ T cvt(dsf x) { return (T)to_double(x); }
template <>
__device__ __forceinline__ dsf cvt<dsf>(dsf x) { return x; }

// Double-single: the FP64 polynomials in double-single arithmetic for
// |z| <= 1/2; beyond, the FP64 library functions.
__device__ __forceinline__ void half_space_terms(dsf z, dsf &e, dsf &m1, dsf &ex)
{
    if (fabsf(z.hi) <= 0.5f) {
        const dsf t = z * z, x = -t;
        dsf E, X;
        half_space_polys(t, x, E, X);
        e = E * z;
        m1 = X * x;
        ex = dsf(1.0) + m1;
    } else {
        double de, dm, dx;
        half_space_terms(to_double(z), de, dm, dx);
        e = to_ds(de);
        m1 = to_ds(dm);
        ex = to_ds(dx);
    }
}

// Equilibrium state at a face (local frame) of an FP64 grid, where rho is
// stored whole (ph.off = 0): the u>0 half of the left Maxwellian plus the u<0
// half of the right one.
__device__ __forceinline__ void face_equilibrium(const Phys<double> &ph, const double Ql[4], const double Qr[4],
                                                 double Q0[4])
{
    const double Ul = Ql[1] / Ql[0], Ur = Qr[1] / Qr[0];
    double el, er, ml, mr, xl, xr;
    half_space_terms(ph.sqlam * Ul, el, ml, xl);
    half_space_terms(ph.sqlam * Ur, er, mr, xr);
    const double Pl = fma(0.5, el, 0.5);    // <u^0>_{u>0} of the left state
    const double Pr = fma(-0.5, er, 0.5);   // <u^0>_{u<0} of the right state
    const double El = ph.kE * xl, Er = ph.kE * xr;
    Q0[0] = fma(Ql[0], Pl, Qr[0] * Pr);
    Q0[1] = fma(Ql[1], Pl, Qr[1] * Pr) + fma(Ql[0], El, -(Qr[0] * Er));
    Q0[2] = fma(Ql[2], Pl, Qr[2] * Pr);
    Q0[3] = fma(Ql[3], Pl, Qr[3] * Pr);
}

// Quartic through 5 face averages q[-2..2], at the Gauss points -g, +g of
// the centre cell, g = 1/(2 sqrt 3) (index space):
//   value(+-g) = E +- O, derivative(+-g) = Do +- De with s_k = q_k + q_-k,
//   a_k = q_k - q_-k and
//   E  = q0 + (s1 - 2 q0)/1080 - (s2 - 2 q0)/4320,
//   O  = (25 sqrt3 / 216) a1 - (7 sqrt3 / 432) a2,
//   Do = (2/3) a1 - (1/12) a2,
//   De = (13 sqrt3 / 54)(s1 - 2 q0) - (sqrt3 / 54)(s2 - 2 q0).
// NEG: the derivatives negated.
template <typename R, bool NEG = false>
__device__ __forceinline__ void tan_val_der(R qm2, R qm1, R q0, R qp1, R qp2, R &vm, R &vp, R &dm,
                                            R &dp)
{
    constexpr double s = NEG ? -1.0 : 1.0;
    const R d1 = fma(q0, R(-2.0), qp1 + qm1), d2 = fma(q0, R(-2.0), qp2 + qm2);
    const R a1 = qp1 - qm1, a2 = qp2 - qm2;
    const R E = fma(d1, R(1.0 / 1080.0), fma(d2, R(-1.0 / 4320.0), q0));
    const R O = fma(a1, R(0.20046884346862007), a2 * R(-0.028065638085606807));
    const R Do = fma(a1, R(s * 2.0 / 3.0), a2 * R(s * -1.0 / 12.0));
    const R De = fma(d1, R(s * 0.41697519441472974), d2 * R(s * -0.032075014954979206));
    vm = E - O;
    vp = E + O;
    dm = Do - De;
    dp = Do + De;
}

// The values alone as two 5-weight dot products (all on the FMA pipe). Used
// for rows that vanish identically in a uniform state (normal slopes,
// tangential derivatives), where the weights not summing exactly to one in
// floating point is harmless. NEG: the negated values (the density slopes as
// gk_flux takes them), from negated weights.
template <typename R, bool NEG = false>
__device__ __forceinline__ void tan_val_direct(R qm2, R qm1, R q0, R qp1, R qp2, R &vm, R &vp)
{
    constexpr double s = NEG ? -1.0 : 1.0;
    const R w0 = R(s * (-1.0 / 4320.0 + 0.028065638085606807)), w1 = R(s * (1.0 / 1080.0 - 0.20046884346862007));
    const R w2 = R(s * 719.0 / 720.0);
    const R w3 = R(s * (1.0 / 1080.0 + 0.20046884346862007)), w4 = R(s * (-1.0 / 4320.0 - 0.028065638085606807));
    vp = fma(w4, qp2, fma(w3, qp1, fma(w2, q0, fma(w1, qm1, w0 * qm2))));
    vm = fma(w0, qp2, fma(w1, qp1, fma(w2, q0, fma(w3, qm1, w4 * qm2))));
}

// ---- Packed FP32 pairs ----
//
// Two independent FP32 values that go through the same arithmetic (the two
// t2 Gauss points of a face) as one float2: the FP32x2 add, multiply and
// fused multiply-add of sm_100 and later do both in one instruction, which
// halves the issue slots of the arithmetic (the FP32 kernels are bound by
// instruction issue, not by the FMA pipe). Every operation is rounded
// explicitly, each lane exactly as its scalar counterpart (__fadd_rn,
// __fmul_rn, __fmaf_rn); nothing is contracted implicitly.
struct f2 {
    float2 v;
    f2() = default;
    __device__ __forceinline__ f2(float2 a) : v(a) {}
    __device__ __forceinline__ f2(float a, float b) : v(make_float2(a, b)) {}
    __device__ __forceinline__ explicit f2(float a) : v(make_float2(a, a)) {}   // both lanes
    __device__ __forceinline__ explicit f2(double a) : f2((float)a) {}
};
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return f2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return f2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }
// a - b as a + (-1) b: the product is exact, so one rounding as in __fsub_rn
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return fma(b, f2(-1.0f), a); }
// a sign costs nothing: the packed instructions negate their operands
__device__ __forceinline__ f2 operator-(f2 a) { return f2(-a.v.x, -a.v.y); }
__device__ __forceinline__ f2 &operator+=(f2 &a, f2 b) { return a = a + b; }
__device__ __forceinline__ f2 &operator-=(f2 &a, f2 b) { return a = a - b; }

// Two double-single values side by side (hi and lo parts as packed pairs):
// every operation is lane by lane the double-single operation of gks_ds.cuh
// (the same FP32 operations in the same order, so the same bits), with one
// packed instruction doing both lanes. Used for the flux of double-single
// grids at two Gauss points at once.
struct dsf2 {
    f2 hi, lo;
    dsf2() = default;
    __device__ __forceinline__ dsf2(f2 h, f2 l) : hi(h), lo(l) {}
    __device__ __forceinline__ dsf2(dsf a, dsf b) : hi(a.hi, b.hi), lo(a.lo, b.lo) {}
    __device__ __forceinline__ explicit dsf2(dsf a) : hi(a.hi), lo(a.lo) {}           // both lanes
    __device__ __forceinline__ explicit dsf2(double x) : dsf2(dsf(x)) {}
    __device__ __forceinline__ explicit dsf2(int x) : dsf2(dsf(x)) {}
    __device__ __forceinline__ dsf lane(int k) const
    {
        return k == 0 ? dsf(hi.v.x, lo.v.x) : dsf(hi.v.y, lo.v.y);
    }
};
__device__ __forceinline__ dsf2 two_sum(f2 a, f2 b)
{
    const f2 s = a + b;
    const f2 bb = s - a;
    return dsf2(s, (a - (s - bb)) + (b - bb));
}
// two_sum(a, -b): the same bits, with the negations folded into exact
// subtractions
__device__ __forceinline__ dsf2 two_diff(f2 a, f2 b)
{
    const f2 s = a - b;
    const f2 bb = s - a;
    return dsf2(s, (a - (s - bb)) - (b + bb));
}
__device__ __forceinline__ dsf2 fast_two_sum(f2 a, f2 b)
{
    const f2 s = a + b;
    return dsf2(s, b - (s - a));
}
__device__ __forceinline__ dsf2 operator+(dsf2 a, dsf2 b)
{
    dsf2 s = two_sum(a.hi, b.hi);
    const dsf2 t = two_sum(a.lo, b.lo);
    s = fast_two_sum(s.hi, s.lo + t.hi);
    return fast_two_sum(s.hi, s.lo + t.lo);
}
__device__ __forceinline__ dsf2 operator-(dsf2 a, dsf2 b)
{
    dsf2 s = two_diff(a.hi, b.hi);
    const dsf2 t = two_diff(a.lo, b.lo);
    s = fast_two_sum(s.hi, s.lo + t.hi);
    return fast_two_sum(s.hi, s.lo + t.lo);
}
__device__ __forceinline__ dsf2 operator-(dsf2 a) { return dsf2(-a.hi, -a.lo); }
__device__ __forceinline__ dsf2 operator*(dsf2 a, dsf2 b)
{
    const f2 p = a.hi * b.hi;
    f2 e = fma(a.hi, b.hi, -p);
    e = fma(a.hi, b.lo, e);
    e = fma(a.lo, b.hi, e);
    return fast_two_sum(p, e);
}
__device__ __forceinline__ dsf2 operator/(dsf2 a, dsf2 b)
{
    const f2 q1(__fdiv_rn(a.hi.v.x, b.hi.v.x), __fdiv_rn(a.hi.v.y, b.hi.v.y));
    const dsf2 r = a - b * dsf2(q1, f2(0.0f));
    const f2 q2(__fdiv_rn(r.hi.v.x, b.hi.v.x), __fdiv_rn(r.hi.v.y, b.hi.v.y));
    return fast_two_sum(q1, q2);
}
__device__ __forceinline__ dsf2 &operator+=(dsf2 &a, dsf2 b) { return a = a + b; }

__device__ __forceinline__ dsf2 &operator*=(dsf2 &a, dsf2 b) { return a = a * b; }
// a b + c with the product left unnormalised (exact high product, its error
// and the cross terms apart): 21 operations against the 27 of product and sum
// at the same error (1.0 to 1.06 times its rms over the sizes of c; leaving
// out the low parts' exact sum as well, 18 operations, was 1.2 times it at
// 1.04x the speed). Face state of a 96^3 double-single step 1.58 -> 1.41 ms,
// fluxes 1.33 -> 1.22 ms.
__device__ __forceinline__ dsf2 fma(dsf2 a, dsf2 b, dsf2 c)
{
    const f2 p = a.hi * b.hi;
    f2 e = fma(a.hi, b.hi, -p);
    e = fma(a.hi, b.lo, e);
    e = fma(a.lo, b.hi, e);
    const dsf2 s = two_sum(p, c.hi), t = two_sum(e, c.lo);
    const dsf2 r = fast_two_sum(s.hi, s.lo + t.hi);
    return dsf2(r.hi, r.lo + t.lo);
}

// half_space_terms of two double-single arguments: the polynomials of both lanes
// as pairs when both lie in |z| <= 1/2, else lane by lane (the same bits as
// the scalar double-single version either way).
__device__ __forceinline__ void half_space_terms(dsf2 z, dsf2 &e, dsf2 &m1, dsf2 &ex)
{
    if (fabsf(z.hi.v.x) <= 0.5f && fabsf(z.hi.v.y) <= 0.5f) {
        const dsf2 t = z * z, x = -t;
        dsf2 E, X;
        half_space_polys(t, x, E, X);
        e = E * z;
        m1 = X * x;
        ex = dsf2(1.0) + m1;
    } else {
        dsf e0, e1, m0, m1_, x0, x1;
        half_space_terms(z.lane(0), e0, m0, x0);
        half_space_terms(z.lane(1), e1, m1_, x1);
        e = dsf2(e0, e1);
        m1 = dsf2(m0, m1_);
        ex = dsf2(x0, x1);
    }
}

// face_equilibrium in double-single (an FP64 grid: ph.off = 0) with the left
// and right half-space terms evaluated as one pair.
__device__ __forceinline__ void face_equilibrium_ds2(const Phys<dsf> &ph, const dsf2 L[2], const dsf2 R[2], dsf2 Q0[2])
{
    // lanes (left, right) of rho and m_n
    const dsf2 r(L[0].lane(0), R[0].lane(0));
    const dsf2 U = dsf2(L[0].lane(1), R[0].lane(1)) / r;
    dsf2 e, m1, x;
    half_space_terms(dsf2(ph.sqlam) * U, e, m1, x);
    const dsf Pl = dsf(0.5) + scale_pow2(e.lane(0), 0.5f);   // <u^0>_{u>0} of the left state
    const dsf Pr = dsf(0.5) - scale_pow2(e.lane(1), 0.5f);   // <u^0>_{u<0} of the right state
    const dsf2 rE = r * (dsf2(ph.kE) * x);
    Q0[0] = L[0] * dsf2(Pl) + R[0] * dsf2(Pr);
    Q0[1] = L[1] * dsf2(Pl) + R[1] * dsf2(Pr);
    const dsf mn = Q0[0].lane(1) + (rE.lane(0) - rE.lane(1));
    Q0[0] = dsf2(Q0[0].lane(0), mn);
}

// ---- FP32 face state on packed pairs ----

// Approximate reciprocal per lane (1 ulp; one instruction: the arguments, a
// density or a sum of squared smoothness indicators of at least 1e-24, are
// never subnormal, so the flush of subnormal inputs changes nothing).
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ f2 wrcp(f2 x) { return f2(rcp_approx(x.v.x), rcp_approx(x.v.y)); }

// half_space_terms of two FP32 arguments: the polynomials of both lanes as
// pairs when both lie in |z| <= 1/2 (the same operations per lane as the
// scalar version, so the same bits), else lane by lane.
__device__ __forceinline__ void half_space_terms(f2 z, f2 &e, f2 &m1, f2 &ex)
{
    if (fabsf(z.v.x) <= 0.5f && fabsf(z.v.y) <= 0.5f) {
        const f2 t = z * z, x = t * f2(-1.0f);
        f2 E, X;
        half_space_series32(t, x, E, X);
        e = E * z;
        m1 = X * x;
        ex = f2(1.0f) + m1;
    } else {
        half_space_terms(z.v.x, e.v.x, m1.v.x, ex.v.x);
        half_space_terms(z.v.y, e.v.y, m1.v.y, ex.v.y);
    }
}

// WENO5-JS along a march, in differences. With the first differences
// D_{k+1/2} = q_{k+1} - q_k, the second ones S_k = D_{k+1/2} - D_{k-1/2} and
// the third ones T_{k+1/2} = S_{k+1} - S_k, the face values of cell i are the
// centre candidate plus what the outer two add to it,
//   right = q_i + D_{i+1/2}/2 - S_i/6 - w0 T_{i-1/2}/3 - w2 T_{i+1/2}/6,
//   left  = q_i - D_{i-1/2}/2 - S_i/6 + v0 T_{i+1/2}/3 + v2 T_{i-1/2}/6
// (w0, w2 and, mirrored, v0, v2 the weights of the outer candidates), and the
// indicators are those of weno5_pair over 13/12 (the weights depend on their
// ratios only): beta = S^2 + (3/13) u^2 with u = S_{i-1} + 2 D_{i-1/2},
// D_{i-1/2} + D_{i+1/2} and S_{i+1} - 2 D_{i+1/2}. A cell that enters the
// march brings one new difference of each order and one new square, where
// the 5-cell form redoes them for every cell: 33 operations per cell and
// component against 81. The FP64 face state is bound by the FP64 pipe and
// follows the count (6 launches of a 96^3 step: 7.92 -> 4.67 ms), the
// double-single one too (2.38 -> 1.66 ms). Written without a product that
// feeds an addition, so that no contraction is left to
// the compiler and a face's bits do not depend on its position in the march.
template <typename T>
struct WenoMarch {
    T c, d;             // cells i, i + 1
    T Dm, D0, Sm, S0;   // D_{i-1/2}, D_{i+1/2}, S_{i-1}, S_i
    T Tm;               // T_{i-1/2}
    T bm, b0;           // eps + S_{i-1}^2, eps + S_i^2

    // cells i - 2 .. i + 1
    __device__ __forceinline__ void start(T q0, T q1, T q2, T q3)
    {
        const T eps(12e-6 / 13.0);
        c = q2;
        d = q3;
        Dm = q2 - q1;
        D0 = q3 - q2;
        Sm = Dm - (q1 - q0);
        S0 = D0 - Dm;
        Tm = S0 - Sm;
        bm = fma(Sm, Sm, eps);
        b0 = fma(S0, S0, eps);
    }

    // normal slope times the centre distance at the face between i - 1 and i
    // (12 x the quartic's derivative is 15 D - (D_{-1} + D + D_{+1}) = 12 D - T)
    __device__ __forceinline__ T slope() const { return fma(Tm, T(-1.0 / 12.0), Dm); }

    // cell e = q_{i+2} enters: the right- and left-face values of cell i;
    // then i + 1 becomes the centre
    __device__ __forceinline__ void push(T e, T &right, T &left)
    {
        const T eps(12e-6 / 13.0), k(3.0 / 13.0), half(0.5), nhalf(-0.5);
        const T D1 = e - d, S1 = D1 - D0, Tp = S1 - S0;
        const T b1 = fma(S1, S1, eps);
        const T u0 = fma(Dm, T(2.0), Sm), u1 = Dm + D0, u2 = fma(D0, T(-2.0), S1);
        T s0 = fma(u0 * k, u0, bm), s1 = fma(u1 * k, u1, b0), s2 = fma(u2 * k, u2, b1);
        s0 = s0 * s0;
        s1 = s1 * s1;
        s2 = s2 * s2;
        const T s02 = s0 * s2, s01 = s0 * s1, s12 = s1 * s2;
        // 3 x the sums of the weights (s12 : 6 s02 : 3 s01 and mirrored)
        const T w1 = s02 * T(18.0);
        const T dr = fma(s12, T(3.0), fma(s01, T(9.0), w1)), dl = fma(s01, T(3.0), fma(s12, T(9.0), w1));
        const T a = s12 * Tm, b = s01 * Tp;
        const T cs = fma(S0, T(-1.0 / 6.0), c);
        sub_quotients(fma(b, T(1.5), a), dr, fma(D0, half, cs), right, fma(a, T(1.5), b), dl, fma(Dm, nhalf, cs), left);
        c = d;
        d = e;
        Dm = D0;
        D0 = D1;
        Sm = S0;
        S0 = S1;
        Tm = Tp;
        bm = b0;
        b0 = b1;
    }

    // r = cr - nr / dr, l = cl + nl / dl
    static __device__ __forceinline__ void sub_quotients(T nr, T dr, T cr, T &r, T nl, T dl, T cl, T &l);
};
// One FP64 division for both faces (the denominators are sums of 8th powers
// of differences above 1e-23; where their product overflows, each by itself).
template <>
__device__ __forceinline__ void WenoMarch<double>::sub_quotients(double nr, double dr, double cr, double &r, double nl,
                                                                 double dl, double cl, double &l)
{
    const double p = dr * dl;
    double ir, il;
    if (__double2hiint(p) < 0x7ff00000) {
        const double ip = 1.0 / p;
        ir = ip * dl;
        il = ip * dr;
    } else {
        ir = 1.0 / dr;
        il = 1.0 / dl;
    }
    r = fma(-nr, ir, cr);
    l = fma(nl, il, cl);
}
template <>
__device__ __forceinline__ void WenoMarch<dsf2>::sub_quotients(dsf2 nr, dsf2 dr, dsf2 cr, dsf2 &r, dsf2 nl, dsf2 dl,
                                                               dsf2 cl, dsf2 &l)
{
    r = cr - nr / dr;
    l = cl + nl / dl;
}

// weno5_pair of two components at once, every multiply-add fused explicitly
// and the constant factors folded into the candidates:
//  - the indicators are those of weno5_pair divided by 13/12 (the weights
//    depend on their ratios only): s_k = (eps 12/13 + t_k^2 + (3/13) u_k^2)^2,
//    with u_0 = t_0 + 2 (c - b) and u_2 = t_2 + 2 (c - d);
//  - the right-face weights times 10 s0 s1 s2 / 3 are s1 s2 / 3, 2 s0 s2 and
//    s0 s1 (mirrored for the left face), so with the candidates P_k = the
//    integer-coefficient ones divided by 18, 3 and 6 the face value is
//    (s12 P0 + s02 P1 + s01 P2) / (s12 / 3 + 2 s02 + s01).
__device__ __forceinline__ void weno5_pair2(const f2 q[5], f2 &right, f2 &left)
{
    const f2 m2(-2.0f), two(2.0f), eps(float(12e-6 / 13.0)), k(float(3.0 / 13.0));
    const f2 a = q[0], b = q[1], c = q[2], d = q[3], e = q[4];
    f2 t = fma(b, m2, a) + c, u = fma(c - b, two, t);
    f2 s0 = fma(t, t, fma(u * k, u, eps));
    t = fma(c, m2, b) + d;
    u = b - d;
    f2 s1 = fma(t, t, fma(u * k, u, eps));
    t = fma(d, m2, c) + e;
    u = fma(c - d, two, t);
    f2 s2 = fma(t, t, fma(u * k, u, eps));
    s0 = s0 * s0;
    s1 = s1 * s1;
    s2 = s2 * s2;
    const f2 s02 = s0 * s2, s01 = s0 * s1, s12 = s1 * s2;
    const f2 third(float(1.0 / 3.0));
    const f2 c3 = c * third, c53 = c * f2(float(5.0 / 3.0)), c1118 = c * f2(float(11.0 / 18.0));
    const f2 k19(float(1.0 / 9.0)), k718(float(-7.0 / 18.0)), k23(float(2.0 / 3.0)), km13(float(-1.0 / 3.0));
    const f2 k56(float(5.0 / 6.0)), km16(float(-1.0 / 6.0));
    {
        // right face: candidates on (a,b,c), (b,c,d), (c,d,e)
        const f2 P0 = fma(a, k19, fma(b, k718, c1118));
        const f2 P1 = fma(b, km13, fma(d, k23, c53));
        const f2 P2 = fma(e, km16, fma(d, k56, c3));
        right = fma(s12, P0, fma(s02, P1, s01 * P2)) * wrcp(fma(s12, third, fma(s02, two, s01)));
    }
    {
        // left face: the mirrored candidates with indicators s2, s1, s0
        const f2 P0 = fma(e, k19, fma(d, k718, c1118));
        const f2 P1 = fma(d, km13, fma(b, k23, c53));
        const f2 P2 = fma(a, km16, fma(b, k56, c3));
        left = fma(s01, P0, fma(s02, P1, s12 * P2)) * wrcp(fma(s01, third, fma(s02, two, s12)));
    }
}

// The 5-cell window of a march of FP32 component pairs, with WenoMarch's
// interface. The differences of WenoMarch, 33 operations per cell and
// component against 53, are hardly faster here, where the march waits on its
// loads (face state of a 384x256x256 step 1.84 ms against 1.83 with the window,
// of 128^3 0.206 against 0.214), and every value of an FP32C state then rounds
// differently, and with it the gradients: the FP32 rounding of the face values
// is seen through the curvature of the weights, 4e-6 of the root mean square of
// an inflow-speed gradient, a sum that nearly cancels. The rounding of this
// path is part of its results (tests/test_gpu_fp32c_rounding.py).
struct WenoWindow {
    f2 w[5];   // cells i - 2 .. i + 2; before a push the first 4 are i - 2 .. i + 1

    __device__ __forceinline__ void start(f2 q0, f2 q1, f2 q2, f2 q3)
    {
        w[0] = q0; w[1] = q1; w[2] = q2; w[3] = q3;
    }
    // 12 x the normal slope times the centre distance at the face between i - 1 and i
    __device__ __forceinline__ f2 slope12() const
    {
        return fma(w[3] - w[0], f2(-1.0f), (w[2] - w[1]) * f2(15.0f));
    }
    __device__ __forceinline__ void push(f2 e, f2 &right, f2 &left)
    {
        w[4] = e;
        weno5_pair2(w, right, left);
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = w[k + 1];
    }
};

// face_equilibrium with the components paired as (rho, m_n) and (m_t1, m_t2)
// (index 0 and 1 of L, R and Q0) and the half-space terms of the left and
// right states as one pair (lane 0 left, lane 1 right).
__device__ __forceinline__ void face_equilibrium2(const Phys<float> &ph, const f2 L[2], const f2 R[2], f2 Q0[2])
{
    const f2 r = f2(ph.off) + f2(L[0].v.x, R[0].v.x);
    const f2 U = f2(L[0].v.y, R[0].v.y) * wrcp(r);
    f2 e, m1, x;
    half_space_terms(f2(ph.sqlam) * U, e, m1, x);
    // (<u^0>_{u>0} of the left state, <u^0>_{u<0} of the right one)
    const f2 P = fma(e, f2(0.5f, -0.5f), f2(0.5f));
    const f2 E = f2(ph.kE) * x;
    const float d0 = (0.5f * ph.off) * (e.v.x - e.v.y);
    const float d1 = fmaf(L[0].v.x, E.v.x, -(R[0].v.x * E.v.y)) + (ph.kE * ph.off) * (m1.v.x - m1.v.y);
    const f2 Pl(P.v.x), Pr(P.v.y);
    Q0[0] = fma(R[0], Pr, fma(L[0], Pl, f2(d0, d1)));
    Q0[1] = fma(R[1], Pr, L[1] * Pl);
}

// Gas-kinetic flux at one Gauss point (local frame: index 0 normal, 1 and 2
// tangential), or at two at once (T = f2, dsf2). The moments of f = g0 (1 -
// tau (a1 u + a2 v + a3 w + A) + A t) with the coefficients solved from the
// slopes and compatibility (Appendix) reduce to a closed form (Chapman-Enskog
// structure, tau p = mu):
//   a.u + A = (1/theta) d_i U_j (c_i c_j - theta delta_ij),   c = u - U,
//   A = A0 + A_j c_j, A0 = -U.grad ln rho - div U,
//   A_k = -d_k ln rho - 2 lambda U_i d_i U_k,
//   F0 = (m_n, m_n U_k + p' delta_nk - mu (d_n U_k + d_k U_n)),
//   F1 = rho (A0 U_n + theta A_n, A0 (U_n U_k + theta delta_nk) + theta (A_k U_n + A_n U_k)),
// with p' = theta (rho - off): the constant theta off cancels in L. It is
// evaluated with rho multiplied through, so that a single reciprocal (for U)
// is left and rho drops out of F1:
//   H_ik = rho d_i U_k = d_i m_k - U_k d_i rho,
//   B = -rho A0 = H_kk + U.grad rho,   C_k = -rho theta A_k = theta d_k rho + U_i H_ik,
//   X = U_n B + C_n = -F1[0],
//   -F1[k] = U_k X + U_n C_k + delta_nk theta B   (n: U_n X + C_n U_n + theta B),
// 52 operations against the 77 of the form with G_ik = d_i U_k, A0 and A_k.
// The density slopes Dn[0], D1[0] and D2[0] come negated (the t2 pass gives
// them so for nothing), F1 is returned negated (nF1): no operation is spent
// on a sign. D1 and D2 are index-space tangential slopes; ih1, ih2 turn them
// into physical ones. What bounds the kernels that call it is the FMA pipe
// (FP32, double-single) or the FP64 pipe, so operations are what counts (x and
// y face fluxes of a 384x256x256 FP32C step 2.97 -> 2.77 ms, of a 96^3 FP64
// step 5.59 -> 5.00 ms).
template <typename T>
struct FluxPhys {
    T off, th, nth, nmu;
};
template <typename T>
__device__ __forceinline__ FluxPhys<T> flux_phys(const Phys<T> &p)
{
    return {p.off, p.theta, -p.theta, -p.mu};
}
__device__ __forceinline__ FluxPhys<f2> flux_phys_f2(const Phys<float> &p)
{
    return {f2(p.off), f2(p.theta), f2(-p.theta), f2(-p.mu)};
}
__device__ __forceinline__ FluxPhys<dsf2> flux_phys_ds2(const Phys<dsf> &p)
{
    return {dsf2(p.off), dsf2(p.theta), dsf2(-p.theta), dsf2(-p.mu)};
}
// rho and 1 / rho; FP64 grids store rho whole (off = 0)
__device__ __forceinline__ f2 whole_rho(f2 off, f2 q) { return off + q; }
__device__ __forceinline__ double whole_rho(double, double q) { return q; }
__device__ __forceinline__ dsf2 whole_rho(dsf2, dsf2 q) { return q; }
__device__ __forceinline__ double inverse(double a) { return 1.0 / a; }
__device__ __forceinline__ f2 inverse(f2 a) { return wrcp(a); }
__device__ __forceinline__ dsf2 inverse(dsf2 a) { return dsf2(1.0) / a; }

template <typename T, bool NEED_F0>
__device__ __forceinline__ void gk_flux(const FluxPhys<T> &ph, const T q[4], const T Dn[4], const T D1[4],
                                        const T D2[4], T ih1, T ih2, T F0[4], T nF1[4])
{
    const T inv = inverse(whole_rho(ph.off, q[0]));
    const T U0 = q[1] * inv, U1 = q[2] * inv, U2 = q[3] * inv;
    const T V1 = U1 * ih1, V2 = U2 * ih2;
    const T H00 = fma(U0, Dn[0], Dn[1]), H01 = fma(U1, Dn[0], Dn[2]), H02 = fma(U2, Dn[0], Dn[3]);
    const T H10 = fma(U0, D1[0], D1[1]), H11 = fma(U1, D1[0], D1[2]), H12 = fma(U2, D1[0], D1[3]);
    const T H20 = fma(U0, D2[0], D2[1]), H21 = fma(U1, D2[0], D2[2]), H22 = fma(U2, D2[0], D2[3]);
    const T S = fma(V2, D2[0], fma(V1, D1[0], U0 * Dn[0]));   // -U.grad rho
    const T B = fma(ih2, H22, fma(ih1, H11, H00)) - S;
    const T C0 = fma(ph.nth, Dn[0], fma(U0, H00, fma(V1, H10, V2 * H20)));
    const T C1 = fma(ph.nth * ih1, D1[0], fma(U0, H01, fma(V1, H11, V2 * H21)));
    const T C2 = fma(ph.nth * ih2, D2[0], fma(U0, H02, fma(V1, H12, V2 * H22)));
    if (NEED_F0) {
        const T nm = ph.nmu * inv;
        F0[0] = q[1];
        F0[1] = fma(q[1], U0, fma(ph.th, q[0], (H00 + H00) * nm));
        F0[2] = fma(q[1], U1, fma(ih1, H10, H01) * nm);
        F0[3] = fma(q[1], U2, fma(ih2, H20, H02) * nm);
    }
    const T X = fma(U0, B, C0);
    nF1[0] = X;
    nF1[1] = fma(U0, X, fma(C0, U0, ph.th * B));
    nF1[2] = fma(U1, X, U0 * C1);
    nF1[3] = fma(U2, X, U0 * C2);
}

// ---- Double-single sums of products ----
//
// The t1 and t2 passes of double-single grids are sums of products with
// constant weights, wanted at the two Gauss points -g, +g: both at once in the
// lanes of a pair, the stencil's values broadcast (which costs nothing), every
// product and every partial sum of the high parts exact, the errors in one low
// part (Ogita, Rump and Oishi's Dot2, SIAM J. Sci. Comput. 2005): 12
// operations a term where a double-single product and sum take 28. The terms
// are added in the order of their size, the cell's own value last, so that the
// low part is rounded at the size of the corrections: against 64 bits the
// values' error is 0.6 times that of the double-single chains (1.2e-15 rms of
// a cell's value), the derivatives' 0.07 to 1 times. Face fluxes of a 96^3
// step 2.09 -> 1.33 ms, z faces and update 1.22 -> 0.84 ms.
struct Dot2 {
    f2 s, e;
    // the first product
    __device__ __forceinline__ Dot2(dsf q, double wm, double wp)
    {
        const f2 h(q.hi), wh((float)wm, (float)wp), wl((float)(wm - (double)(float)wm), (float)(wp - (double)(float)wp));
        s = wh * h;
        e = fma(wh, f2(q.lo), fma(wl, h, fma(wh, h, -s)));
    }
    __device__ __forceinline__ void add(dsf q, double wm, double wp)
    {
        const Dot2 p(q, wm, wp);
        const dsf2 t = two_sum(s, p.s);
        s = t.hi;
        e += t.lo + p.e;
    }
    __device__ __forceinline__ dsf2 value() const { return two_sum(s, e); }
    __device__ __forceinline__ dsf2 plus(dsf c) const
    {
        const dsf2 t = two_sum(f2(c.hi), s);
        return two_sum(t.hi, t.lo + (e + f2(c.lo)));
    }
};
// tan_val_direct (negated with NEG) of double-single values.
template <bool NEG>
__device__ __forceinline__ dsf2 ds_val_direct(const dsf q[5])
{
    constexpr double g = NEG ? -1.0 : 1.0;
    constexpr double w0 = g * (-1.0 / 4320.0 + 0.028065638085606807), w1 = g * (1.0 / 1080.0 - 0.20046884346862007);
    constexpr double w2 = g * (-1.0 / 720.0);   // less the value itself
    constexpr double w3 = g * (1.0 / 1080.0 + 0.20046884346862007), w4 = g * (-1.0 / 4320.0 - 0.028065638085606807);
    Dot2 d(q[2], w2, w2);
    d.add(q[0], w4, w0);
    d.add(q[4], w0, w4);
    d.add(q[1], w3, w1);
    d.add(q[3], w1, w3);
    return d.plus(NEG ? -q[2] : q[2]);
}
// tan_val_der of double-single values from the centre value c and the 4
// differences D of neighbouring cells (exactly c, and slopes exactly zero, in
// a uniform state): values and derivatives (negated with NEG).
template <bool NEG>
__device__ __forceinline__ void ds_val_der(dsf c, const dsf D[4], dsf2 &val, dsf2 &der)
{
    constexpr double o1 = 0.20046884346862007, o2 = 0.028065638085606807, a = 1.0 / 1080.0, b = 1.0 / 4320.0;
    constexpr double e1 = 0.41697519441472974, e2 = 0.032075014954979206, g = NEG ? -1.0 : 1.0;
    // per value weight W_k of cell k the difference D_k takes the sum of the
    // weights beyond it: -(W_-2), -(W_-2 + W_-1), W_1 + W_2, W_2
    Dot2 v(D[0], b + o2, b - o2);
    v.add(D[3], -b + o2, -b - o2);
    v.add(D[1], b + o2 - a - o1, b - o2 - a + o1);
    v.add(D[2], a - o1 - b + o2, a + o1 - b - o2);
    val = v.plus(c);
    Dot2 d(D[0], g * (-1.0 / 12.0 - e2), g * (-1.0 / 12.0 + e2));
    d.add(D[3], g * (-1.0 / 12.0 + e2), g * (-1.0 / 12.0 - e2));
    d.add(D[1], g * (7.0 / 12.0 + e1 - e2), g * (7.0 / 12.0 - e1 + e2));
    d.add(D[2], g * (7.0 / 12.0 - e1 + e2), g * (7.0 / 12.0 + e1 - e2));
    der = d.value();
}

// A block takes consecutive positions of the extended face plane, t1 fastest,
// whatever its width: 32 x 8 blocks leave a fifth of the lanes idle on the
// 132 x 132 positions of a 128^3 grid and half of them on 36 x 36.
__device__ __forceinline__ bool face_position(unsigned p, int n1, int n2, int &a, int &b)
{
    const unsigned r = p / (unsigned)(n1 + 4);
    a = (int)(p - r * (unsigned)(n1 + 4)) - 2;
    b = (int)r - 2;
    return b < n2 + 2;
}

constexpr int TX = 32, TY = 8;              // face tile
constexpr int SQ_W = TX + 4, SQ_H = TY + 4; // tile with the tangential halo
constexpr int SQ_N = 8 * SQ_H * SQ_W;
constexpr int ST_ROWS = SQ_H * TX;          // rows of the t1 pass
constexpr int ST_N = 24 * ST_ROWS;

// 8 consecutive values of a shared-memory row from a 16-byte aligned address,
// and 4 consecutive values to one.
__device__ __forceinline__ void lds8(const double *p, double q[8])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double2 a = reinterpret_cast<const double2 *>(p)[i];
        q[2 * i] = a.x;
        q[2 * i + 1] = a.y;
    }
}
__device__ __forceinline__ void sts4(double *p, const double q[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(q[0], q[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(q[2], q[3]);
}
__device__ __forceinline__ void lds8(const dsf *p, dsf q[8])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 a = reinterpret_cast<const float4 *>(p)[i];
        q[2 * i] = dsf(a.x, a.y);
        q[2 * i + 1] = dsf(a.z, a.w);
    }
}
__device__ __forceinline__ void sts4(dsf *p, const dsf q[4])
{
    reinterpret_cast<float4 *>(p)[0] = make_float4(q[0].hi, q[0].lo, q[1].hi, q[1].lo);
    reinterpret_cast<float4 *>(p)[1] = make_float4(q[2].hi, q[2].lo, q[3].hi, q[3].lo);
}

static_assert(TX * TY == 256 && TY == 8 && SQ_H == 12 && TX == 32, "t1-pass task split assumes 32 x 8 tiles");

// Physical row of row r (0 <= r < 2 SQ_H) of a tile's t1 results, a ring of
// SQ_H rows.
__device__ __forceinline__ int ring_row(int r) { return r < SQ_H ? r : r - SQ_H; }

// One task of the t1 pass: a group of 4 columns of row r of a face-box tile,
// values and t1-derivatives of Q0 (kind 0) or values of the normal slope of
// component v at the two t1 Gauss points, into row rp of st. It reads 8
// consecutive values and writes 4 columns.
template <typename R, typename C>
__device__ __forceinline__ void t1_task(const R *sq, C *st, int kind, int v, int r, int rp, int cg)
{
    constexpr int ROWS = SQ_H * TX;
    C q[8];
    lds8(sq + ((kind * 4 + v) * SQ_H + r) * SQ_W + 4 * cg, q);
    C *o = st + rp * TX + 4 * cg;
    if constexpr (std::is_same<C, dsf>::value) {
        dsf x[4][4];
        if (kind == 0) {
            dsf D[7];
#pragma unroll
            for (int i = 0; i < 7; ++i) D[i] = q[i + 1] - q[i];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                dsf2 val, der;
                ds_val_der<false>(q[i + 2], D + i, val, der);
                x[0][i] = val.lane(0);
                x[1][i] = val.lane(1);
                x[2][i] = der.lane(0);
                x[3][i] = der.lane(1);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) sts4(o + (v * 4 + k) * ROWS, x[k]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const dsf2 val = ds_val_direct<false>(q + i);
                x[0][i] = val.lane(0);
                x[1][i] = val.lane(1);
            }
            sts4(o + (16 + v * 2 + 0) * ROWS, x[0]);
            sts4(o + (16 + v * 2 + 1) * ROWS, x[1]);
        }
    } else if (kind == 0) {
        C vm[4], vp[4], dm[4], dp[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) tan_val_der(q[i], q[i + 1], q[i + 2], q[i + 3], q[i + 4], vm[i], vp[i], dm[i], dp[i]);
        sts4(o + (v * 4 + 0) * ROWS, vm);
        sts4(o + (v * 4 + 1) * ROWS, vp);
        sts4(o + (v * 4 + 2) * ROWS, dm);
        sts4(o + (v * 4 + 3) * ROWS, dp);
    } else {
        C vm[4], vp[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) tan_val_direct(q[i], q[i + 1], q[i + 2], q[i + 3], q[i + 4], vm[i], vp[i]);
        sts4(o + (16 + v * 2 + 0) * ROWS, vm);
        sts4(o + (16 + v * 2 + 1) * ROWS, vp);
    }
}

// t1 pass of the last H rows of a face-box tile into the ring of rows, whose
// first tile row stands at `off`: 64 H equal tasks, H / 4 per thread; the
// lanes of a warp share the kind and the component and take 4 rows. The
// double-single task is long and not unrolled (one copy for every H).
template <typename R, typename C>
__device__ __forceinline__ void tile_t1_pass(const R *sq, C *st, int tid, int H, int off)
{
    const int per = H >> 2, lane = tid & 31;
    auto round = [&](int j) {
        const int wt = (tid >> 5) + 8 * j, kv = H == TY ? wt >> 1 : wt / 3, r = SQ_H - H + 4 * (wt - kv * per) + (lane >> 3);
        t1_task(sq, st, kv >> 2, kv & 3, r, ring_row(r + off), lane & 7);
    };
    if constexpr (std::is_same<C, dsf>::value) {
#pragma unroll 1
        for (int j = 0; j < per; ++j) round(j);
    } else {
        round(0);
        round(1);
        if (H == SQ_H) round(2);
    }
}

// ---- FP32 component pairs ----
//
// FP32 face boxes and t1-pass rows hold the components as pairs (rho, m_n)
// and (m_t1, m_t2), 8 bytes per position: the face-state kernel's packed
// values are stored as they are (4 stores per face instead of 8), and the t1
// and t2 passes run on both components of a pair at once. Face-box tile: 4
// pair arrays (Q0 of both pairs, then their normal slopes) of H x SQ_W; rows:
// 12 pair arrays of H x TX, 4 P + {0, 1} Q0 of pair P at the two t1 Gauss
// points, 4 P + {2, 3} its t1 slopes there, 8 + 2 P + {0, 1} its normal slope.
// The face state of a 384x256x256 step took 2.15 ms with 8 separate stores
// and takes 1.90 ms with 4 paired ones.

// t1 pass of a face-box tile: 64 SQ_H equal tasks (pair, row, group of 2
// columns), SQ_H / 4 per thread: 6 pairs in by 128-bit loads, 2 columns out by
// one 128-bit store per array (consecutive lanes, consecutive 16 bytes: no
// bank conflict; groups of 4 columns would store 32 bytes apart).
__device__ __forceinline__ void tile_t1_pass_f2(const float2 *sq, float2 *st, int tid)
{
    static_assert(SQ_H % 4 == 0, "a warp's tasks share the pair");
    constexpr int NV = 16 * SQ_H, ROWS = SQ_H * TX;
#pragma unroll
    for (int j = 0; j < SQ_H / 4; ++j) {
        const int task = tid + j * 256, p = task / NV, rem = task - p * NV, r = rem >> 4, cg = rem & 15;
        const float4 *in = reinterpret_cast<const float4 *>(sq + (p * SQ_H + r) * SQ_W + 2 * cg);
        f2 q[6];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float4 x = in[i];
            q[2 * i] = f2(x.x, x.y);
            q[2 * i + 1] = f2(x.z, x.w);
        }
        float2 *o = st + r * TX + 2 * cg;
        f2 v[4][2];
        if (p < 2) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
                tan_val_der(q[i], q[i + 1], q[i + 2], q[i + 3], q[i + 4], v[0][i], v[1][i], v[2][i], v[3][i]);
            o += 4 * p * ROWS;
        } else {
#pragma unroll
            for (int i = 0; i < 2; ++i) tan_val_direct(q[i], q[i + 1], q[i + 2], q[i + 3], q[i + 4], v[0][i], v[1][i]);
            o += (8 + 2 * (p - 2)) * ROWS;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < 2 || p < 2)
                *reinterpret_cast<float4 *>(o + k * ROWS) = make_float4(v[k][0].v.x, v[k][0].v.y, v[k][1].v.x, v[k][1].v.y);
    }
}

// tan_val_direct and tan_val_der of a component pair, with the two Gauss
// points (not the components) in the lanes of the results, as the flux takes
// them: x0 and x1 of the pair's two components, value (-g, +g). Everything up
// to the last operation runs on both components at once; that one is scalar
// and writes its lane in place (no moves). NEG: component 0 negated, by the
// operand signs of the last operation.
template <bool NEG>
__device__ __forceinline__ void pair_val_direct(const f2 p[5], f2 &x0, f2 &x1)
{
    constexpr float w0 = float(-1.0 / 4320.0 + 0.028065638085606807), w1 = float(1.0 / 1080.0 - 0.20046884346862007);
    constexpr float w2 = float(719.0 / 720.0);
    constexpr float w3 = float(1.0 / 1080.0 + 0.20046884346862007), w4 = float(-1.0 / 4320.0 - 0.028065638085606807);
    const f2 a = fma(f2(w3), p[3], fma(f2(w2), p[2], fma(f2(w1), p[1], f2(w0) * p[0])));
    const f2 b = fma(f2(w1), p[3], fma(f2(w2), p[2], fma(f2(w3), p[1], f2(w4) * p[0])));
    x0 = NEG ? f2(__fmaf_rn(-w0, p[4].v.x, -b.v.x), __fmaf_rn(-w4, p[4].v.x, -a.v.x))
             : f2(__fmaf_rn(w0, p[4].v.x, b.v.x), __fmaf_rn(w4, p[4].v.x, a.v.x));
    x1 = f2(__fmaf_rn(w0, p[4].v.y, b.v.y), __fmaf_rn(w4, p[4].v.y, a.v.y));
}
template <bool NEG>
__device__ __forceinline__ void pair_val_der(const f2 p[5], f2 &x0, f2 &x1, f2 &d0, f2 &d1)
{
    const f2 s1 = fma(p[2], f2(-2.0f), p[3] + p[1]), s2 = fma(p[2], f2(-2.0f), p[4] + p[0]);
    const f2 a1 = p[3] - p[1], a2 = p[4] - p[0];
    const f2 E = fma(s1, f2(float(1.0 / 1080.0)), fma(s2, f2(float(-1.0 / 4320.0)), p[2]));
    const f2 O = fma(a1, f2(float(0.20046884346862007)), a2 * f2(float(-0.028065638085606807)));
    const f2 Do = fma(a1, f2(float(2.0 / 3.0)), a2 * f2(float(-1.0 / 12.0)));
    const f2 De = fma(s1, f2(float(0.41697519441472974)), s2 * f2(float(-0.032075014954979206)));
    x0 = f2(__fsub_rn(E.v.x, O.v.x), __fadd_rn(E.v.x, O.v.x));
    x1 = f2(__fsub_rn(E.v.y, O.v.y), __fadd_rn(E.v.y, O.v.y));
    d0 = NEG ? f2(__fsub_rn(De.v.x, Do.v.x), __fadd_rn(-Do.v.x, -De.v.x))
             : f2(__fsub_rn(Do.v.x, De.v.x), __fadd_rn(Do.v.x, De.v.x));
    d1 = f2(__fsub_rn(Do.v.y, De.v.y), __fadd_rn(Do.v.y, De.v.y));
}

// The t2 pass of face (tx, ty) of a tile at t1 Gauss point m: values and t2
// slopes of Q0, values of the t1 slopes and of the normal slope at the two t2
// Gauss points (the lanes). NEG: the density's slopes negated, as gk_flux takes
// them.
template <bool NEG>
__device__ __forceinline__ void t2_pass_f2(const float2 *st, int m, int tx, int ty, f2 q[4], f2 dn[4], f2 d1[4], f2 d2[4])
{
    const float2 *s = st + ty * TX + tx;
    f2 p[5];
#pragma unroll
    for (int P = 0; P < 2; ++P) {
#pragma unroll
        for (int i = 0; i < 5; ++i) p[i] = f2(s[(4 * P + m) * ST_ROWS + i * TX]);
        if (P == 0)
            pair_val_der<NEG>(p, q[0], q[1], d2[0], d2[1]);
        else
            pair_val_der<false>(p, q[2], q[3], d2[2], d2[3]);
#pragma unroll
        for (int i = 0; i < 5; ++i) p[i] = f2(s[(4 * P + 2 + m) * ST_ROWS + i * TX]);
        if (P == 0)
            pair_val_direct<NEG>(p, d1[0], d1[1]);
        else
            pair_val_direct<false>(p, d1[2], d1[3]);
#pragma unroll
        for (int i = 0; i < 5; ++i) p[i] = f2(s[(8 + 2 * P + m) * ST_ROWS + i * TX]);
        if (P == 0)
            pair_val_direct<NEG>(p, dn[0], dn[1]);
        else
            pair_val_direct<false>(p, dn[2], dn[3]);
    }
}

template <typename R>
constexpr size_t flux_smem_bytes()
{
    return (size_t)(SQ_N + ST_N) * sizeof(R) + 2 * sizeof(unsigned long long);
}

// ---- TMA and mbarrier helpers (sm_90+ PTX) ----

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// One bulk tensor copy of the (TX+4) x (TY+4) x 1 x 8 face box starting at
// (c0, c1, c2, 0) into dst; completion is signalled on bar with the byte
// count.
__device__ __forceinline__ void tma_load_tile(const CUtensorMap *map, void *dst, uint64_t *bar, int c0, int c1,
                                              int c2, uint32_t bytes)
{
    const uint32_t b = smem_u32(bar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(0), "r"(b)
        : "memory");
}

// 4- or 8-byte asynchronous copy global -> shared (completion through
// cp.async groups), and the group fences.
__device__ __forceinline__ void cp_async(float *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)),
                 "l"((unsigned long long)__cvta_generic_to_global(src))
                 : "memory");
}
__device__ __forceinline__ void cp_async(double *dst, const double *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)),
                 "l"((unsigned long long)__cvta_generic_to_global(src))
                 : "memory");
}
__device__ __forceinline__ void cp_async(dsf *dst, const dsf *src)
{
    cp_async(reinterpret_cast<double *>(dst), reinterpret_cast<const double *>(src));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Wait for phase `parity` of bar; gives up after ~1 s of SM clock and
// returns false (the caller raises FLAG_TIMEOUT).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity)
{
    const uint32_t b = smem_u32(bar);
    const long long t0 = clock64();
    while (true) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(b), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > (1LL << 31)) return false;
    }
}


}  // namespace dev
}  // namespace gks
