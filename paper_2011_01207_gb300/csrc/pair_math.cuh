// Radial functions of atom pairs, shared by the real-space kernels.
//
// Screened:  B_0 = erfc(beta r)/r,  B_n = [(2n-1) B_{n-1} + (2 beta^2)^n e^{-beta^2 r^2}/(beta sqrt(pi))] / r^2
// Coulomb:   U_n = (2n-1)!! / r^(2n+1)
// Thole:     s = a r^3 / sqrt(alpha_i alpha_j),  1 - lambda_3 = e^-s, 1 - lambda_5 = (1+s) e^-s,
//            1 - lambda_7 = (1 + s + 3/5 s^2) e^-s, 1 - lambda_9 = (1 + s + 18/35 s^2 + 9/35 s^3) e^-s
// Kernel:    R_n = B_n - (1 - sigma lambda_{2n+1}) U_n  (sigma = 1, or 0 for excluded pairs)
//
// In FP32 a thread of a pair kernel holds two target atoms and meets one source atom at a time, so
// every quantity of the two pairs is a two-vector, and its operations are the f32x2 ones of sm_100
// and later, two per issue slot (the kernels are bound by issue). In FP64, where the pipe is the
// bound and registers are short, a thread holds one target and the "vectors" are plain numbers.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

// erfc(x), x >= 0, in FP32: e^{-x^2} times a polynomial of degree six in
// t = 1 / (1 + 0.4 x) without constant term, the form of Abramowitz & Stegun 7.1.26 one degree
// higher; the coefficients are a minimax fit (linear programming on 900 points of [0, 5], absolute
// error weighted as erfc's) made for this file. In FP32 it stays within 2.0e-7 of erfc (rms 2.7e-8 on
// [0, 4.5]; 7.1.26: 3.2e-7, 8.0e-8). FP64: the library erfc.
#define AP_ERFC_P 0.4f
__device__ constexpr float ERFC_C[6] = {0.232319036f, 0.159588671f, 0.473249716f, -0.376376784f, 0.712111243f, -0.200891881f};

// ---- the targets' vectors ----------------------------------------------------------------
template <class T> struct Vec;
template <> struct Vec<float> {
    typedef float2 type;
    static constexpr int W = 2;
    static __device__ __forceinline__ float get(float2 v, int h) { return h ? v.y : v.x; }
};
template <> struct Vec<double> {
    typedef double type;
    static constexpr int W = 1;
    static __device__ __forceinline__ double get(double v, int) { return v; }
};
__device__ __forceinline__ float2 splat2(float a) { return make_float2(a, a); }
__device__ __forceinline__ double splat2(double a) { return a; }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long ra, rb, rd;
    memcpy(&ra, &a, 8);
    memcpy(&rb, &b, 8);
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    float2 d;
    memcpy(&d, &rd, 8);
    return d;
}
__device__ __forceinline__ double add2(double a, double b) { return a + b; }
__device__ __forceinline__ double mul2(double a, double b) { return a * b; }
__device__ __forceinline__ double fma2(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double sub2(double a, double b) { return a - b; }
// vector minus, times a number every target shares: two scalar operations cost less than making
// the pair (b, b) for a packed one
__device__ __forceinline__ float2 sub1(float2 a, float b) { return make_float2(a.x - b, a.y - b); }
__device__ __forceinline__ double sub1(double a, double b) { return a - b; }
__device__ __forceinline__ float2 mul1(float2 a, float b) { return make_float2(a.x * b, a.y * b); }
__device__ __forceinline__ double mul1(double a, double b) { return a * b; }

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 ex2_2(float2 a) { return make_float2(ex2_approx(a.x), ex2_approx(a.y)); }
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(rcp_approx(a.x), rcp_approx(a.y)); }
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 rsqrt2(float2 a) { return make_float2(rsqrt_approx(a.x), rsqrt_approx(a.y)); }

// ---- constants and radial terms ----------------------------------------------------------
template <class T>
struct PairConsts {
    T beta;            // Ewald beta
    T c[5];            // c[n] = (2 beta^2)^n / (beta sqrt(pi)), n = 1..4 (c[0] unused)
    T thole_a;
    T rc2;             // cutoff^2
    int n;             // real atoms; slots >= n are padding
};
template <class T>
inline PairConsts<T> make_consts(const ap_ctx *ctx) {
    PairConsts<T> pc;
    const ap_params &P = ctx->prm;
    const double b = P.ewald_beta;
    double p = 1.0 / (b * AP_SQRT_PI);
    pc.beta = (T)b;
    pc.c[0] = 0;
    for (int k = 1; k <= 4; ++k) {
        p *= 2.0 * b * b;
        pc.c[k] = (T)p;
    }
    pc.thole_a = (T)P.thole_a;
    pc.rc2 = (T)(P.cutoff * P.cutoff);
    pc.n = ctx->n;
    return pc;
}

// Constants in the form the radial terms use. FP32: the exponents are taken to base 2
// (e^-y = 2^(-y log2 e)), so each exponential is one multiply-add and one 2^x. All signs are those
// of -R_n.
template <class T> struct RadialConsts;
template <> struct RadialConsts<float> {
    float2 ce;        // -beta^2 log2(e): e^{-beta^2 r^2} = 2^{ce r^2}
    float2 pb;        // AP_ERFC_P beta: t = 1 / (1 + pb r)
    float2 c[4];      // -(2 beta^2)^n / (beta sqrt(pi)), n = 1..4
    float2 nl2e;      // -log2(e)
    float ta;         // Thole a
    __device__ __forceinline__ explicit RadialConsts(const PairConsts<float> &pc) {
        const float l2e = 1.4426950408889634f;
        ce = splat2(-pc.beta * pc.beta * l2e);
        pb = splat2(AP_ERFC_P * pc.beta);
        for (int k = 0; k < 4; ++k) c[k] = splat2(-pc.c[k + 1]);
        nl2e = splat2(-l2e);
        ta = pc.thole_a;
    }
};
template <> struct RadialConsts<double> {
    PairConsts<double> pc;
    double ta;
    __device__ __forceinline__ explicit RadialConsts(const PairConsts<double> &p) : pc(p), ta(p.thole_a) {}
};

// g = e^{-beta^2 r^2} (zero where pen says so) and poly = -erfc(beta r) / g, from r^2 and r
__device__ __forceinline__ void screening(const RadialConsts<float> &k, float2 r2, float2 r, float2 pen, float2 &g, float2 &poly) {
    g = ex2_2(fma2(r2, k.ce, pen));
    const float2 t = rcp2(fma2(k.pb, r, splat2(1.0f)));
    poly = splat2(-ERFC_C[5]);
#pragma unroll
    for (int n = 4; n >= 0; --n) poly = fma2(poly, t, splat2(-ERFC_C[n]));
    poly = mul2(poly, t);
}

// -R_1..-R_N from r^2 and the Thole products tw = a w_target w_source:
//   Mu[n] with sigma = 1, and with EX also Md[n] with sigma = 0 where exa, exb say so.
// pen is 0 for a pair that counts and AP_OUT for one that does not (out of range): added to both
// exponents it makes both exponentials, and with them every R_n, exactly zero, at no cost.
// With R_n = B_n - o_n U_n and o_1 = e, o_n = o_(n-1) + d_n (e = e^-s, d_2 = s e, d_3 = (3/5) s^2 e,
// d_4 = ((9/35) s - (3/35)) s^2 e):
//   R_n = [(2n-1) (R_(n-1) - d_n U_(n-1)) + c_n e^{-beta^2 r^2}] / r^2
// so one chain serves for B_n and the damping together; with sigma = 0 (o_n = 1) every d_n is 0.
#define AP_OUT -1e5f
template <int N, bool EX>
__device__ __forceinline__ void radial(const RadialConsts<float> &k, float2 r2, float2 tw, float2 pen, bool exa, bool exb,
                                       float2 *Mu, float2 *Md) {
    const float2 rinv = rsqrt2(r2);
    const float2 r = mul2(r2, rinv), rinv2 = mul2(rinv, rinv);
    float2 g, poly;
    screening(k, r2, r, pen, g, poly);
    const float2 b1 = mul2(g, mul2(fma2(poly, rinv, k.c[0]), rinv2));   // -B_1
    const float2 s = mul2(mul2(r2, r), tw);
    const float2 e = ex2_2(fma2(s, k.nl2e, pen));
    float2 u = mul2(rinv, rinv2);
    Mu[0] = fma2(e, u, b1);
    float2 x;
    if (EX) {
        x = add2(b1, u);
        Md[0] = make_float2(exa ? x.x : Mu[0].x, exb ? x.y : Mu[0].y);
    }
    float2 d = mul2(s, e);
    float2 s2e;
    if (N > 2) s2e = mul2(s, d);
#pragma unroll
    for (int n = 1; n < N; ++n) {
        const float2 cg = mul2(k.c[n], g), f = splat2((float)(2 * n + 1));
        if (n == 2) d = mul2(s2e, splat2(0.6f));
        if (n == 3) d = mul2(s2e, fma2(s, splat2(9.0f / 35.0f), splat2(-3.0f / 35.0f)));
        Mu[n] = mul2(fma2(f, fma2(d, u, Mu[n - 1]), cg), rinv2);
        if (EX) {
            x = mul2(fma2(f, x, cg), rinv2);
            Md[n] = make_float2(exa ? x.x : Mu[n].x, exb ? x.y : Mu[n].y);
        }
        if (n + 1 < N) u = mul2(mul2(u, f), rinv2);
    }
}

template <int N, bool EX>
__device__ __forceinline__ void radial(const RadialConsts<double> &k, double r2, double tw, double pen, bool ex, bool,
                                       double *Mu, double *Md) {
    const double rinv = rsqrt(r2), r = r2 * rinv, rinv2 = rinv * rinv;
    const double x = k.pc.beta * r, e2 = exp(-x * x);
    const bool out = pen < 0.0;
    double b = erfc(x) * rinv, u = rinv;
    const double s = tw * r2 * r, e = exp(-s);
    double o[4];
    o[0] = e;
    if (N > 1) o[1] = (1.0 + s) * e;
    if (N > 2) o[2] = (1.0 + s + 0.6 * s * s) * e;
    if (N > 3) o[3] = (1.0 + s + s * s * (18.0 / 35.0 + (9.0 / 35.0) * s)) * e;
#pragma unroll
    for (int n = 0; n < N; ++n) {
        b = ((2 * n + 1) * b + k.pc.c[n + 1] * e2) * rinv2;
        u = (2 * n + 1) * u * rinv2;
        Mu[n] = out ? 0.0 : o[n] * u - b;
        if (EX) Md[n] = ex ? u - b : Mu[n];
    }
}

// Exact FP32 -> FP64 conversion with integer operations only (FP64 instructions issue at a
// small fraction of the FP32 rate on this part): the sign, the exponent rebased from 127 to
// 1023 and the 23 mantissa bits moved to the top of the 52. Zero and subnormal inputs
// (below 1.2e-38) give a signed zero; infinities and NaNs keep their class.
__device__ __forceinline__ double f2d_exact(float x) {
    const unsigned u = __float_as_uint(x);
    const unsigned e = (u >> 23) & 0xffu, s = u & 0x80000000u, m = u & 0x7fffffu;
    unsigned hi = s | ((e + 896u) << 20) | (m >> 3);
    hi = e == 0u ? s : hi;
    hi = e == 0xffu ? (s | 0x7ff00000u | (m >> 3)) : hi;
    const unsigned lo = e == 0u ? 0u : (m << 29);
    return __hiloint2double((int)hi, (int)lo);
}

// Compensated FP32 sum hi + lo: each addition is Knuth's TwoSum (the rounding error of
// hi + x, recovered exactly in FP32, is added to lo), so the pair carries ~48 bits.
struct F2 {
    float hi, lo;
};
__device__ __forceinline__ void f2_add(F2 &a, float x) {
    const float t = a.hi + x;
    const float z = t - a.hi;
    a.lo += (a.hi - (t - z)) + (x - z);
    a.hi = t;
}
__device__ __forceinline__ float add2(float a, float b) { return a + b; }
__device__ __forceinline__ float sub2(float a, float b) { return a - b; }
// the same for float2s (two sums at once) and floats, adding hi + lo of another such sum
template <class V>
__device__ __forceinline__ void f2_merge(V &hi, V &lo, V ohi, V olo) {
    const V t = add2(hi, ohi), z = sub2(t, hi), err = add2(sub2(hi, sub2(t, z)), sub2(ohi, z));
    lo = add2(add2(lo, olo), err);
    hi = t;
}
template <class V>
__device__ __forceinline__ void f2_add(V &hi, V &lo, V x) {
    const V t = add2(hi, x), z = sub2(t, hi);
    lo = add2(lo, add2(sub2(hi, sub2(t, z)), sub2(x, z)));
    hi = t;
}

// A target's sum to its accumulator slot: FP64, or (fixed) 64-bit fixed point. Every slot is
// written by one thread, from sums formed in a fixed order, so both are reproducible.
template <class T>
__device__ __forceinline__ void store_acc(double *p, T v, int fixed) {
    if (fixed) *reinterpret_cast<long long *>(p) = ap_to_fx((double)v);
    else *p = (double)v;
}
