// whg_interact.cuh -- arithmetic of the interaction kick and of the GR term in
// pairs of floats: the scalar parts, host and device (interact() in
// whg_device.cuh runs them over a warp's lanes).
//
// Why.  The pair sums and the GR term were 64 FP64 instructions per planet and
// step, each holding the FP64 pipe for 64-76 cycles; an FP32 instruction
// takes one cycle.  A kick changes a velocity by a small part of itself, so
// its terms do not need the velocity's own 53 bits: a float pair (hi + lo, 48
// bits, error-free products by FMA) leaves an error of 2^-46 of a term rms
// (2^-43 at most), below 2^-56 of the velocity for any kick this form accepts
// (2^-10 of the velocity), against the 2^-54 that each of the FP64 form's seven
// additions to the velocity made.  The error's mean is +2^-48 of the term (the
// low bits of squares are not random): as if the kicks' masses were larger by 3e-15,
// action and reaction alike.  The kick's terms are summed
// apart from the velocity and reach it in one FP64 addition.  Against an 80-bit
// reference the states after 1000 steps of Solar-System-shaped systems are off
// by 8.0e-13 in the mean, 1.12e-12 with everything in FP64.
//
// Positions go onto a system's common 58-bit grid (block exponent EQ, the largest
// of its planets' coordinates, taken anew from every step's state) and are
// held as three 20-bit chunks in floats, so that differences of positions are
// exact: three subtractions, and two FMAs, one addition and one more FMA to
// the float pair.  A pair too close for the grid, or too strong for the
// accumulation, is reported and the caller redoes the sub-step in FP64.
//
// Measured, 8-planet systems: 4096 x 1000 steps 7.64 -> 5.38 ms, 2^20 x 20 40.8 ->
// 28.3 ms, 65,536 compact systems x 400 25.5 -> 18.1 ms; 106 -> 41 FP64
// instructions per planet and step.  (The same sub-step in 64-bit integers
// took 3100 instructions a warp and step against 2250, and 7.2 ms.)
//
// Units: D = d 2^(17 - EQ), |D| < 2^19; velocity changes are in 2^(2 (EQ - 17)).
#pragma once

#include "whg_fixed.cuh"

namespace whg {
namespace pairs {

using fixed::i32;
using fixed::i64;
using fixed::u32;
using fixed::u64;

using fixed::add;
using fixed::fma;
using fixed::mul;
using fixed::sub;

struct Pair {
    float h, l;
};

// A coordinate on the grid: chunks of 18 (signed), 20 and 20 bits as floats
// 1.5 2^23 + c2, 2^23 + c1, 2^23 + c0, whose differences are those of the chunks.
struct Coord {
    float c2, c1, c0;
};

WHG_HD Coord chunks(i64 X)
{
    const u32 hi = (u32)((u64)X >> 32), lo = (u32)(u64)X;
    Coord c;
    c.c2 = fixed::bits_to_f32(0x4B400000u + (u32)((i32)hi >> 8));
    c.c1 = fixed::bits_to_f32(0x4B000000u | (((hi << 12) | (lo >> 20)) & 0xfffffu));
    c.c0 = fixed::bits_to_f32(0x4B000000u | (lo & 0xfffffu));
    return c;
}

// D = h + m 2^-20 + l 2^-40 as a float pair (exact but for the last bits of l).
WHG_HD Pair joined(float h, float m, float l)
{
    const float s20 = 1.0f / 1048576.0f, s40 = s20 * s20;
    Pair r;
    r.h = fma(m, s20, h);
    r.l = fma(l, s40, fma(m, s20, sub(h, r.h)));
    return r;
}

WHG_HD Pair difference(const Coord& a, const Coord& b) { return joined(sub(a.c2, b.c2), sub(a.c1, b.c1), sub(a.c0, b.c0)); }

WHG_HD Pair own(const Coord& a)
{
    return joined(sub(a.c2, 12582912.0f), sub(a.c1, 8388608.0f), sub(a.c0, 8388608.0f));
}

// Sum of two floats and its error.
WHG_HD Pair two_sum(float a, float b)
{
    Pair r;
    r.h = add(a, b);
    const float t = sub(r.h, a);
    r.l = add(sub(a, sub(r.h, t)), sub(b, t));
    return r;
}

struct Separation {
    Pair x, y, z;
    float r2, r2l, y1, s, es, e;  // |D|^2 (a float pair); y1 ~ |D|^-1, s + es = y1^2, e = 1 - |D|^2 y1^2 to 2^-46
};

WHG_HD Separation separation(const Pair& x, const Pair& y, const Pair& z)
{
    Separation p;
    p.x = x;
    p.y = y;
    p.z = z;
    const float px = mul(x.h, x.h), py = mul(y.h, y.h), pz = mul(z.h, z.h);
    const Pair a = two_sum(px, py), b = two_sum(a.h, pz);
    float lo = add(a.l, b.l);
    lo = add(lo, fma(x.h, x.h, -px));
    lo = add(lo, fma(y.h, y.h, -py));
    lo = add(lo, fma(z.h, z.h, -pz));
    lo = fma(add(x.h, x.h), x.l, lo);
    lo = fma(add(y.h, y.h), y.l, lo);
    lo = fma(add(z.h, z.h), z.l, lo);
    p.r2 = b.h;
    p.r2l = lo;
    p.y1 = fixed::rsqrt_f32(b.h);
    p.s = mul(p.y1, p.y1);
    p.es = fma(p.y1, p.y1, -p.s);
    p.e = fma(-lo, p.s, fma(-b.h, p.es, fma(-b.h, p.s, 1.0f)));
    return p;
}

// |D|^-3 = y^3 (1 + 3e/2 + 15 e^2/8) and |D|^-4 = y^4 (1 + 2e + 3 e^2).
WHG_HD Pair inverse_cube(const Separation& p)
{
    Pair r;
    r.h = mul(p.s, p.y1);
    const float err = fma(p.es, p.y1, fma(p.s, p.y1, -r.h));
    r.l = fma(r.h, mul(p.e, fma(1.875f, p.e, 1.5f)), err);
    return r;
}

WHG_HD Pair inverse_fourth(const Separation& p)
{
    Pair r;
    r.h = mul(p.s, p.s);
    const float err = fma(add(p.s, p.s), p.es, fma(p.s, p.s, -r.h));
    r.l = fma(r.h, mul(p.e, fma(3.0f, p.e, 2.0f)), err);
    return r;
}

// a b to ~2^-46.
WHG_HD Pair product(const Pair& a, const Pair& b)
{
    Pair r;
    r.h = mul(a.h, b.h);
    r.l = fma(a.l, b.h, fma(a.h, b.l, fma(a.h, b.h, -r.h)));
    return r;
}

// s + (h + l), the sum kept to ~2^-47 of itself.
WHG_HD void accumulate(Pair& s, float h, float l)
{
    const Pair t = two_sum(s.h, h);
    s.h = t.h;
    s.l = add(s.l, add(t.l, l));
}

// a + b to ~2^-47 of the larger, the same bits as b + a.
WHG_HD Pair sum(const Pair& a, const Pair& b)
{
    const Pair t = two_sum(a.h, b.h);
    Pair r;
    r.h = t.h;
    r.l = add(t.l, add(a.l, b.l));
    return r;
}

// a - b, never contracted with the product that a may be.
#if defined(__CUDA_ARCH__)
__device__ __forceinline__ double sub64(double a, double b) { return __dsub_rn(a, b); }
#else
inline double sub64(double a, double b) { volatile double r = a - b; return r; }
#endif

// A constant as a float and the rest of it (24 + 24 bits).
WHG_HD Pair split(double x)
{
    Pair r;
    r.h = (float)x;
    r.l = (float)sub64(x, (double)r.h);
    return r;
}

// f 2^k as a double from the bit fields (0 and FP32 subnormals give 0).
WHG_HD double widen(float f, int k)
{
    const u32 b = fixed::f32_bits(f);
    const u32 ex = (b >> 23) & 0xffu;
    const u32 hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + ((u32)(896 + k) << 20));
    return fixed::from_bits(ex == 0u ? 0ull : (((u64)hi << 32) | (u64)(b << 29)));
}

}  // namespace pairs
}  // namespace whg
