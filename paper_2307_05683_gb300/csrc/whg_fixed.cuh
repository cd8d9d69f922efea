// whg_fixed.cuh -- the Kepler drift's universal-variable solver in 64-bit
// fixed point on the integer pipe.
//
// Why.  An FP64 warp instruction holds its sub-partition's pipe for 64 cycles
// (76 with all four sub-partitions busy).  A 64 x 64 -> 64-bit fixed-point
// product is three 32-bit multiply-adds, 17-19 cycles of the integer pipe, 41
// cycles from operand to result against 64, and keeps 62 bits instead of 53.
// So the solver, which was 125 of the 153 FP64 instructions of a drift, runs
// here in integers, more accurately than in doubles, and leaves the FP64
// pipe to the vectors.
//
// The dimensionless equation.  With s = X r0/h,
//     a = eta0 h/r0^2,  m = mu h^2/r0^3,  V = v^2 h^2/r0^2,
//     B = beta h^2/r0^2 = 2 m - V,  b = zeta0 h^2/r0^3 = V - m,  z = B s^2,
//     g2 = s^2 c2(z),  g3 = s^3 c3(z),  g1 = s - B g3,  g0 = 1 - B g2,
// Kepler's equation and its derivative are
//     phi(s) = s - 1 + a g2 + b g3 = 0,   R(s) = r/r0 = 1 + a g1 + b g2,
// and the Lagrange coefficients
//     f - 1 = -m g2,  g/h = 1 - m g3,  gdot - 1 = -m g2/R,
//     fdot = -(mu h/r0^3) g1/R.
// Every quantity is of order one or less whatever the orbit's scale, so fixed
// point loses nothing; the factors m and mu h/r0^3 in front of the
// coefficients enter as normalized significands, which keeps the relative
// precision of a slow outer planet's coefficients.
//
// Solution: a starting value from two FP32 Halley steps (an error of ~2^-22,
// as any FP64 Halley phase only supplies the Newton phase's start), one
// evaluation of both series at it in fixed point, the third-order step
//     d = d0 - d0^2 R'/(2 R),  d0 = -phi/R,
// and the g_n carried to s + d by their Taylor series (dg_n/ds = g_{n-1})
// through d^2.  d is accepted below 2^-19, where the neglected d^3 terms are
// below 2^-59; the start is taken low by 2^-20.5 so that d > 0.
//
// With the series cut at z^T, dg_3/ds = g_2 and dg_1/ds = g_0 still hold, but
// dg_2/ds = g_1 + tau, tau = z^(T+1) s/(2T+3)!.  For T = 8 tau d is below 2^-67;
// for T = 6 it reaches 2^-53 (z = 2), always of one sign, so G_2 and the step
// (slope R + a tau) take it along, tau in FP32: without, 1 - f and 1 - gdot were off by
// -0.9 2^-53 in the mean for 1.75 < z < 2, with it by -0.03 2^-53, as everywhere.
//
// The result's error is ~2^-58 (of h for g, which at the domain's edge is up to
// 64 times smaller) before the coefficients are rounded to doubles, below what
// the FP64 solver's own roundings left: over the whole domain rms 0.43 2^-53
// against 1.5 to 2.7 2^-53, and at most 1.2 2^-53 against 16 2^-53 (g 4.4 against 230).  Products are
// rounded about their mean (mulhi's constant), not truncated: a drift of
// 2^-60 per step would add up over 1e9 steps.
//
// Measured on 4096 8-planet systems, 1000 steps: 14.44 ms with the solver in
// FP64 (238 FP64 instructions per planet and step, 153 of them the drift's),
// 7.64 ms with this one (106, 21).
//
// Domain: |a| < 1, |b|, B < 2, z < 2, 9/16 < s < 7/4, 1/2 < R < 2, V < 1.9999 m
// (a bound orbit): every step of up to about P/6 on a near-circular orbit, or
// of up to half the pericentre timescale on an eccentric one.  Outside it, or
// where the start is not within reach, solve() returns false and the caller
// runs the FP64 solver.  Formats: Qn is an integer of value x 2^n; operands of
// mulhi stay below 2^63.
#pragma once

#include <math.h>
#include <stdint.h>

#if defined(__CUDACC__)
#define WHG_HD __host__ __device__ __forceinline__
#else
#define WHG_HD inline
#endif

namespace whg {
namespace fixed {

typedef unsigned long long u64;
typedef long long i64;
typedef unsigned int u32;
typedef int i32;

#if defined(__CUDA_ARCH__)
__device__ __forceinline__ u32 hi32(u64 x) { return (u32)(x >> 32); }
__device__ __forceinline__ u64 bits_of(double x) { return (u64)__double_as_longlong(x); }
__device__ __forceinline__ double from_bits(u64 b) { return __longlong_as_double((i64)b); }
__device__ __forceinline__ u32 umulhi(u32 a, u32 b) { return __umulhi(a, b); }
__device__ __forceinline__ i32 smulhi(i32 a, i32 b) { return __mulhi(a, b); }
__device__ __forceinline__ int clz32(u32 x) { return __clz((int)x); }
__device__ __forceinline__ float rcp_f32(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ u32 f32_to_u32(float x) { return __float2uint_rz(x); }
__device__ __forceinline__ float u32_to_f32(u32 x) { return __uint2float_rz(x); }
__device__ __forceinline__ float bits_to_f32(u32 b) { return __uint_as_float(b); }
__device__ __forceinline__ u32 f32_bits(float x) { return __float_as_uint(x); }
__device__ __forceinline__ u64 umulhi64(u64 a, u64 b) { return __umul64hi(a, b); }
__device__ __forceinline__ float rsqrt_f32(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
#else
// Host forms of the same operations (the fixed-point code is checked on the
// CPU against extended precision).
inline u32 hi32(u64 x) { return (u32)(x >> 32); }
inline u64 bits_of(double x)
{
    union { double d; u64 u; } c;
    c.d = x;
    return c.u;
}
inline double from_bits(u64 b)
{
    union { double d; u64 u; } c;
    c.u = b;
    return c.d;
}
inline u32 umulhi(u32 a, u32 b) { return (u32)(((u64)a * b) >> 32); }
inline i32 smulhi(i32 a, i32 b) { return (i32)(((i64)a * b) >> 32); }
inline int clz32(u32 x) { return x ? __builtin_clz(x) : 32; }
inline float rcp_f32(float x) { return 1.0f / x; }
inline u32 f32_to_u32(float x) { return x > 0.0f ? (x < 4294967040.0f ? (u32)x : 0xffffffffu) : 0u; }
inline float u32_to_f32(u32 x) { return (float)(x & (x >> 24 ? ~((1u << (32 - __builtin_clz(x) - 24)) - 1u) : ~0u)); }
inline float bits_to_f32(u32 b)
{
    union { float f; u32 u; } c;
    c.u = b;
    return c.f;
}
inline u32 f32_bits(float x)
{
    union { float f; u32 u; } c;
    c.f = x;
    return c.u;
}
inline u64 umulhi64(u64 a, u64 b) { return (u64)(((unsigned __int128)a * b) >> 64); }
inline float rsqrt_f32(float x) { return 1.0f / sqrtf(x); }
#endif

// Float operations that are never contracted: every kernel that inlines this
// code computes the same bits.
#if defined(__CUDA_ARCH__)
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
inline float add(float a, float b) { volatile float r = a + b; return r; }
inline float sub(float a, float b) { volatile float r = a - b; return r; }
inline float mul(float a, float b) { volatile float r = a * b; return r; }
inline float fma(float a, float b, float c) { return fmaf(a, b, c); }
#endif

// High word of a b, a, b < 2^63, to about one unit: the product of the low
// words is left out (1/4 unit on average) and the rest truncated (1/2), and
// K 2^-32 units are added so that the error's mean is zero (default 3/4).
template <u64 K = 0xC0000000ull>
WHG_HD u64 mulhi(u64 a, u64 b)
{
    const u32 ah = hi32(a), al = (u32)a, bh = hi32(b), bl = (u32)b;
    u64 t = (u64)al * bh + K;
    t += (u64)ah * bl;
    return (u64)ah * bh + (t >> 32);
}

// The same for b = bh 2^32: the product with a 32-bit operand, rounded.
WHG_HD u64 mulhi32(u64 a, u32 bh)
{
    const u64 t = (u64)(u32)a * bh + 0x80000000ull;
    return (u64)hi32(a) * bh + (t >> 32);
}

// Significand with its leading one at bit 62, of a positive normal double.
WHG_HD u64 significand62(u64 bits) { return ((bits & 0x000fffffffffffffull) | 0x0010000000000000ull) << 10; }

WHG_HD int exponent_of(u64 bits) { return (int)(hi32(bits) >> 20) & 0x7ff; }

// n 2^-s as a double, rounded to nearest (ties, one in 2^(11 - lz), to even:
// upward they would bias the result by 2^-60); 2^32 <= n < 2^63, the result
// normal.
WHG_HD double to_double(u64 n, int s)
{
    const int lz = clz32(hi32(n)) - 1;
    n <<= lz;                                        // leading one at bit 62: rounding cannot leave the word
    const u64 r = (n + (0x1ffull + ((u32)(n >> 10) & 1u))) >> 10;   // at bit 52; a carry moves into the exponent
    return from_bits(r + ((u64)(u32)(1023 + 61 - lz - s) << 52));
}

// A double as an integer on a grid: its significand (leading one at bit 62)
// shifted right by sh (truncated; 0 from 63 on), with the sign.
WHG_HD i64 to_fixed(u64 bits, int sh)
{
    const u64 m = significand62(bits) >> (sh > 63 ? 63 : sh);
    return (i64)(bits >> 63 ? 0ull - m : m);
}

WHG_HD int larger(int a, int b) { return a > b ? a : b; }

WHG_HD int smaller(int a, int b) { return a < b ? a : b; }

// 2^k as a float, 0 below 2^-126 and infinity from 2^128 on (solve's exponent
// guards let k reach about +-1000: a speed of 2^300, a step of 2^150).
WHG_HD float power2(int k) { return bits_to_f32(k < -126 ? 0u : (u32)(smaller(k, 128) + 127) << 23); }

// Series coefficients 4^k/n! as round(4^k 2^q / n!), from an exact division.
constexpr u64 coef(int k, int n, int q)
{
    // (2^(q + 2k)) / n! by long division in base 2^32 of a 128-bit numerator
    unsigned __int128 num = (unsigned __int128)1 << (q + 2 * k);
    unsigned __int128 den = 1;
    for (int i = 2; i <= n; ++i) den *= (unsigned)i;
    return (u64)((num + den / 2) / den);
}

// Stumpff functions through z^T (T = 6, 8) for x = z/4 < 1/2 in Q64: c2 in
// Q64, c3 in Q65.  Horner steps p_k = 4^k/(2k+n)! - x p_{k+1}; the tail
// (k >= 6), whose terms are below 2^-24 and enter with x^6, in 32 bits.
template <int T>
WHG_HD void stumpff(u64 x, u64& c2, u64& c3)
{
    const u32 xh = hi32(x);
    u32 t2, t3;                                      // scales 2^55 and 2^58
    if (T == 8) {
        t2 = (u32)coef(8, 18, 55);
        t3 = (u32)coef(8, 19, 58);
        t2 = (u32)coef(7, 16, 55) - umulhi(xh, t2);
        t3 = (u32)coef(7, 17, 58) - umulhi(xh, t3);
        t2 = (u32)coef(6, 14, 55) - umulhi(xh, t2);
        t3 = (u32)coef(6, 15, 58) - umulhi(xh, t3);
    } else {
        t2 = (u32)coef(6, 14, 55);
        t3 = (u32)coef(6, 15, 58);
    }
    u64 p2 = coef(5, 12, 64) - (((u64)xh * t2) >> 23);
    u64 p3 = coef(5, 13, 65) - (((u64)xh * t3) >> 25);
    p2 = coef(4, 10, 64) - mulhi(x, p2);
    p3 = coef(4, 11, 65) - mulhi(x, p3);
    p2 = coef(3, 8, 64) - mulhi(x, p2);
    p3 = coef(3, 9, 65) - mulhi(x, p3);
    p2 = coef(2, 6, 64) - mulhi(x, p2);
    p3 = coef(2, 7, 65) - mulhi(x, p3);
    p2 = coef(1, 4, 64) - mulhi(x, p2);
    p3 = coef(1, 5, 65) - mulhi(x, p3);
    c2 = 0x7fffffffffffffffull - mulhi(x, p2);
    c3 = coef(0, 3, 65) - mulhi(x, p3);
}

// Two Halley steps in FP32 for phi(s) = 0, from s.
WHG_HD float halley(float s, float a, float b, float B)
{
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int it = 0; it < 2; ++it) {
        const float u = mul(s, s), z = mul(-B, u);
        float c2 = (float)(1.0 / 3628800.0), c3 = (float)(1.0 / 39916800.0);
        c2 = fma(z, c2, (float)(1.0 / 40320.0));
        c3 = fma(z, c3, (float)(1.0 / 362880.0));
        c2 = fma(z, c2, (float)(1.0 / 720.0));
        c3 = fma(z, c3, (float)(1.0 / 5040.0));
        c2 = fma(z, c2, (float)(1.0 / 24.0));
        c3 = fma(z, c3, (float)(1.0 / 120.0));
        c2 = fma(z, c2, 0.5f);
        c3 = fma(z, c3, (float)(1.0 / 6.0));
        const float g2 = mul(u, c2), g3 = mul(mul(s, u), c3), g1 = fma(-B, g3, s), g0 = fma(-B, g2, 1.0f);
        const float F = add(sub(s, 1.0f), fma(a, g2, mul(b, g3)));
        const float R = fma(a, g1, fma(b, g2, 1.0f));
        const float R1 = fma(a, g0, mul(b, g1));
        s = fma(-mul(F, R), rcp_f32(fma(R, R, mul(-0.5f, mul(F, R1)))), s);
    }
    return s;
}

WHG_HD float start(float a, float b, float B)
{
    const float s = fma(-1.0f / 6.0f, b, fma(0.5f, fma(a, a, -a), 1.0f));
    return halley(s < 0.6f ? 0.6f : (s > 1.7f ? 1.7f : s), a, b, B);
}

struct Solution {
    double fm1n;             // 1 - f
    double g;                // g
    double fdn;              // -fdot
    double gdm1n;            // 1 - gdot
    double s, g1, g2, g3, Ri;   // s, g_n and r0/r at the solution (with VALS, for the adjoint's tape)
};

// Leading one to bit 62 (n >= 2^32), the exponent adjusted.
WHG_HD u64 normalize(u64 n, int& e)
{
    const int sh = clz32(hi32(n)) - 1;
    e -= sh;
    return n << sh;
}

// Right shift of a significand to fixed point: 0..63 (a value too small for
// the format becomes 0).
WHG_HD int shift63(int n) { return n > 63 ? 63 : n; }

// Solve for a drift of h under mu from r0^2, eta0 = Q.v and v^2; false outside
// the domain (o is then undefined).
template <int T, bool VALS>
WHG_HD bool solve(double mu, double h, double r0sq, double eta0, double v2, Solution& o)
{
    const u64 rb = bits_of(r0sq), eb = bits_of(eta0), vb = bits_of(v2), hb = bits_of(h), mb = bits_of(mu);
    const int er = exponent_of(rb), ee = exponent_of(eb), ev = exponent_of(vb), eh = exponent_of(hb),
              emu = exponent_of(mb);
    // r0 within 2^+-100, h within 2^+-150, mu within 2^+-100 of one: every
    // result is a normal double; inf and NaN are outside.  (A zero or subnormal
    // eta0 or v^2 counts as 2^-1023, which its fixed-point form rounds to 0.)
    if ((u32)(er - 823) > 400u || larger(ee, ev) > 1623 || (u32)(eh - 873) > 300u || (u32)(emu - 923) > 200u)
        return false;
    const bool neg = (eb >> 63) != 0;

    // 1/r0 = r 2^(-62 - half), r = mant^(-1/2) with r0^2 = mant 4^half, mant in
    // [1, 4): FP32 seed y = My 2^-24, e = 1 - mant y^2 in Q60, y (1 + e/2 + 3 e^2/8)
    const int odd = (er + 1) & 1, half = (er - 1023 - odd) / 2;
    const u64 rx = significand62(rb) >> (1 - odd);                       // mant 2^61
    const float yf = rsqrt_f32(mul(u32_to_f32(hi32(rx)), 1.0f / 536870912.0f));
    const u32 My = f32_to_u32(mul(yf, 16777216.0f));
    const i64 ey = (i64)((1ull << 60) - mulhi(rx, ((u64)My * My) << 15));
    const i32 eyh = (i32)(ey >> 13);                                     // Q47
    const i64 U = (ey >> 1) + ((3 * (((i64)eyh * eyh) >> 34)) >> 3);     // Q60
    const u64 r = ((u64)My << 38) + (u64)(((i64)My * U + 0x200000) >> 22);

    // dimensionless parameters, in FP32 for the domain and the start
    const u64 hM = significand62(hb), muM = significand62(mb);
    const float s30 = 1.0f / 1073741824.0f;
    const float hf = mul(u32_to_f32(hi32(hM)), s30), hy = mul(hf, yf), hy2 = mul(hy, hy);
    const int kw = eh - 1023 - half;
    const u64 vM = significand62(vb), eM = significand62(eb);
    const float mf = mul(mul(mul(u32_to_f32(hi32(muM)), s30), mul(yf, hy2)), power2(emu - 1023 + 2 * kw - half));
    const float Vf = mul(mul(mul(u32_to_f32(hi32(vM)), s30), hy2), power2(larger(ev - 1023 + 2 * kw, -200)));
    const float am = mul(mul(mul(u32_to_f32(hi32(eM)), s30), mul(hy, yf)), power2(larger(ee - 1023 + kw - half, -200)));
    const float af = neg ? -am : am, bf = sub(Vf, mf), Bf = fma(2.0f, mf, -Vf);
    // (comparisons that are false for NaN)
    if (!(Vf < mul(1.9998f, mf) && Vf < 3.99f && mf < 3.99f && am < 0.999f && bf < 1.999f && bf > -1.999f && Bf < 1.999f))
        return false;

    // and as significands x 2^exponent (each product's error is ~2^-59 of it)
    const u64 wM = mulhi(hM, r) << 2;                                    // h/r0 = wM 2^(eh - 1085 - half)
    const u64 kM = mulhi(wM, r) << 2;                                    // h/r0^2 = kM 2^(eh - 1085 - 2 half)
    const u64 w2M = mulhi(wM, wM) << 1;                                  // (h/r0)^2 = w2M 2^(2 eh - 2107 - 2 half)
    const u64 nM = mulhi(muM, r) << 2;                                   // mu/r0 = nM 2^(emu - 1085 - half)
    int ej = emu + eh - 2106 - 3 * half, em = emu + 2 * eh - 3128 - 3 * half;
    int ea = ee + eh - 2106 - 2 * half, eV = ev + 2 * eh - 3128 - 2 * half;
    const u64 jM = normalize(mulhi(nM, kM), ej);                         // mu h/r0^3 = jM 2^(ej)
    const u64 mM = normalize(mulhi(nM, w2M), em);                        // m = mM 2^(em)
    const u64 aM = normalize(mulhi(eM, kM), ea);                         // |a| = aM 2^(ea)
    const u64 VM = normalize(mulhi(vM, w2M), eV);                        // V = VM 2^(eV)

    // parameters in fixed point: |a| in Q62, m and V in Q61
    const u64 one60 = 1ull << 60, one62 = 1ull << 62;
    const u64 amag = aM >> shift63(-62 - ea), mq = mM >> shift63(-61 - em), Vq = VM >> shift63(-61 - eV);
    const u64 a1 = neg ? one62 - amag : one62 + amag;                    // a + 1, Q62
    const u64 b2 = Vq - mq + one62;                                      // b + 2, Q61
    i64 Bs = (i64)(2 * mq - Vq);                                         // Q61
    Bs = Bs < 0 ? 0 : Bs;
    const u64 B = (u64)Bs << 1;                                          // Q62
    const float sf = start(af, bf, Bf);
    const float zf = mul(Bf, mul(sf, sf));
    if (!(sf > 0.5625f && sf < 1.75f && zf < 1.99f)) return false;
    const u32 sh = f32_to_u32(mul(sf, 1073741824.0f)) - 724u;                // Q30, 2^-20.5 low

    // series and g_n at the start
    const u64 u = (u64)sh * sh;                                          // s^2, Q60
    const u64 x = mulhi(B, u) << 4;                                      // z/4, Q64
    u64 c2, c3;
    stumpff<T>(x, c2, c3);
    const u64 g2 = mulhi(u, c2);                                         // Q60
    const u64 g3 = mulhi32(mulhi(u, c3) << 2, sh);                       // Q61
    const u64 g2w = g2 << 2, g3w = g3 << 2;                              // Q62, Q63
    const u64 g1 = ((u64)sh << 32) - (mulhi(B, g3w) << 1);               // Q62
    const u64 g0 = one62 - (mulhi(B, g2w) << 2);                         // Q62

    // phi (Q60, <= 0 at the low start) and R (Q60)
    const i64 nphi = (i64)(one60 - ((u64)sh << 30) - (mulhi(a1, g2w) - g2) - (mulhi(b2, g3w) - g3));
    u64 R = one60 + (mulhi(a1, g1) - (g1 >> 2)) + ((mulhi(b2, g2w) - g2) << 1);
    const i32 ah = (i32)hi32(a1) - (i32)(1u << 30), bh = (i32)hi32(b2) - (i32)(1u << 30);    // Q30, Q29
    u32 tau = 0;                                                         // Q55
    if (T == 6) {
        const float z2 = mul(zf, zf), z4 = mul(z2, z2);
        tau = f32_to_u32(mul(mul(mul(z4, z2), mul(zf, sf)), (float)(36028797018963968.0 / 1307674368000.0)));
        R += (u64)((i64)smulhi(ah, (i32)tau) * 128);
    }
    if (!(nphi >= 0 && nphi < (1ll << 41) && R > (one60 >> 1) + (one60 >> 6) && R < (one60 << 1) - (one60 >> 6)))
        return false;

    // 1/R to ~2^-44: FP32 seed and one Newton correction
    const u32 y0 = f32_to_u32(mul(rcp_f32(u32_to_f32((u32)(R >> 29))), 72057594037927936.0f));   // Q25
    const i64 D = (i64)(0ull - R * (u64)y0);                             // (1 - R y0) 2^85
    const u64 y = ((u64)y0 << 37) + (u64)(((i64)(i32)y0 * (i64)(i32)(D >> 32)) >> 16);       // Q62

    // the step d (Q62), with its second-order term in 32 bits
    const u64 d0 = mulhi((u64)nphi << 4, y);
    const u32 dh = (u32)(d0 >> 18);                                      // Q44
    const u32 d2 = (u32)(((u64)dh * dh) >> 21);                          // d^2/2, Q68
    const u32 g0h = hi32(g0), g1h = hi32(g1), Bh = hi32(B), yh = hi32(y);   // Q30
    const i32 R1 = smulhi(ah, (i32)g0h) + 2 * smulhi(bh, (i32)g1h);      // dR/ds, Q28
    const u64 d = d0 - (u64)(i64)smulhi(smulhi(R1, (i32)yh), (i32)d2);

    // g_n at s + d (mulhi's constants also make up for the truncated shifts)
    const u64 G3 = g3 + (mulhi<0x100000000ull>(d, g2w) << 1) + (umulhi(d2, g1h) >> 5);   // Q61
    const u64 G2 = g2 + mulhi<0x140000000ull>(d, g1) + (umulhi(d2, g0h) >> 6) + (umulhi(dh, tau) >> 7);   // Q60
    const u64 G1 = g1 + (mulhi(d, g0) << 2) - (umulhi(d2, umulhi(Bh, g1h)) >> 2);            // Q62
    const u64 G2w = G2 << 2;
    const u64 Rn = one60 + (mulhi<0xA0000000ull>(a1, G1) - (G1 >> 2)) + ((mulhi(b2, G2w) - G2) << 1);       // Q60

    // 1/R at s + d from y: y (1 + e + e^2), |e| < 2^-20
    const i64 d1 = (i64)(one60 - mulhi(Rn << 2, y));                     // Q60
    if (!(d1 < (1ll << 40) && d1 > -(1ll << 40))) return false;
    const i64 e1 = d1 >> 13;                                             // Q47
    const i64 t = d1 + (((i64)(i32)e1 * (i32)e1) >> 34);                    // Q60
    const u64 yn = y + mulhi(((u64)t << 4) + (1ull << 48), y) - (y >> 16);                  // Q62

    const u64 mg3 = mulhi(mq, G3 << 2);                                  // Q60
    if (mg3 >= one60 - (one60 >> 6)) return false;
    const u64 mg2 = mulhi(mM, G2w);                                      // x 2^(em + 2)
    const u64 jg1 = mulhi(jM, G1);                                       // x 2^(ej + 2)
    o.fm1n = to_double(mg2, -2 - em);
    o.gdm1n = to_double(mulhi(mg2, yn), -4 - em);
    o.g = to_double(mulhi(hM, (one60 - mg3) << 2), 1083 - eh);
    o.fdn = to_double(mulhi(jg1, yn), -4 - ej);
    if (VALS) {
        o.s = to_double(((u64)sh << 32) + d, 62);
        o.g1 = to_double(G1, 62);
        o.g2 = to_double(G2, 60);
        o.g3 = to_double(G3, 61);
        o.Ri = to_double(yn, 62);
    }
    return true;
}

}  // namespace fixed
}  // namespace whg
