// 62-bit fixed-point arithmetic of the 1D integrator (device), and the same on
// the host for its tests.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

namespace pmf {

// A 62-bit fixed-point number as two 31-bit limbs, h 2^31 + l with
// 0 <= l < 2^31.  a b 2^-62 of two such numbers (|a|, |b| < 2^62) is
// a.h b.h + 2 (hi(a.h b.l) + hi(a.l b.h)), hi = the upper 32 bits of a 64-bit
// product: the two cross products keep 30 bits each and the product of the low
// limbs is dropped.  Both round down: the result is 0 to 5 units low, 2 1/4 on
// average (1 for each cross product, 1/4 for the low limbs), and what is added
// to it makes up for that average (step_of, q_offset).
struct Limbs {
    int h, l;
};
__host__ __device__ __forceinline__ Limbs limbs(long long v) { return {(int)(v >> 31), (int)(v & 0x7fffffff)}; }
__host__ __device__ __forceinline__ int mul_hi(int a, int b)
{
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int)(((long long)a * b) >> 32);
#endif
}
__host__ __device__ __forceinline__ int mad_hi(int a, int b, int c)
{
#ifdef __CUDA_ARCH__
    int d;
    asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
#else
    return (int)((unsigned)mul_hi(a, b) + (unsigned)c);
#endif
}
__host__ __device__ __forceinline__ long long mad_wide(int a, int b, long long c)  // wraps
{
#ifdef __CUDA_ARCH__
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (long long)((unsigned long long)((long long)a * b) + (unsigned long long)c);
#endif
}
__host__ __device__ __forceinline__ long long mul62_add(Limbs a, Limbs b, long long c)
{
    return mad_wide(mad_hi(a.l, b.h, mul_hi(a.h, b.l)), 2, mad_wide(a.h, b.h, c));
}

struct FixedStep {
    Limbs ca;      // cA 4^b 2^62
    long long cb;  // (cB - 1) 2^62, and the mean that w would be low by
};
__host__ __device__ __forceinline__ long long round_ll(double v)
{
#ifdef __CUDA_ARCH__
    return __double2ll_rn(v);
#else
    return llrint(v);
#endif
}
__host__ __device__ __forceinline__ FixedStep step_of(double cA, double cB1, int b)
{
    FixedStep f{limbs(round_ll(scalbn(cA, 62 + 2 * b))), round_ll(scalbn(cB1, 62))};
    // w = ca y + cb is 2 1/4 low, and by ca times the 2 1/3 that y = x^2 is (its low limb is squared)
    if (cA != 0.0) f.cb += (long long)(2.75f + 2.3333f * (float)f.ca.h * 0x1p-31f);
    return f;
}
// The mean of a step's last product, x w, in 1/256 units.  With cA = 0 w is a
// constant: a limb of zero loses nothing, and its low limb's mean is itself.
__host__ __device__ __forceinline__ int q_offset256(double cA, double cB1)
{
    if (cA != 0.0) return 576;
    const Limbs w = limbs(round_ll(scalbn(cB1, 62)));
    return 256 * ((w.h != 0) + (w.l != 0)) + (w.l >> 24);
}
// Its share in step n's q_n: whole units, o256 over any 256 steps.
__host__ __device__ __forceinline__ int q_offset(int o256, long long n)
{
    const int i = (int)(n & 255);
    return ((o256 * (i + 1)) >> 8) - ((o256 * i) >> 8);
}
// One step, X' = X + Q + X w, w = (cB - 1) + cA x^2: three products, 19
// integer instructions with the sums folded into the multiply-adds (64-bit
// products by limbs cost twice that, most of it shifts and splits).  Sums wrap
// where a trajectory leaves the range; the caller discards that tile.
__host__ __device__ __forceinline__ long long fixed_step(const FixedStep &f, long long X, long long q)
{
    const Limbs x = limbs(X);
    const Limbs y = limbs(mad_wide(mul_hi(x.h, x.l), 4, (long long)x.h * x.h));
    const Limbs w = limbs(mul62_add(f.ca, y, f.cb));
    return mul62_add(w, x, (long long)((unsigned long long)X + (unsigned long long)q));
}
// Top bit set: X outside [-2^62, 2^62).  (Unsigned: the sum of a position above
// the range is meant to carry into the top bit.)
__host__ __device__ __forceinline__ unsigned range_guard(long long X)
{
    return (unsigned)((unsigned long long)X >> 32) + 0x40000000u;
}

// Which b (|x| < 2^b) a simulation's fixed point takes.  It depends on the
// model, the run's parameters and the simulation's own trap centres alone, so a
// window's trajectory has the same bits in every launch that holds it.
constexpr int kNoRange = -1000;  // FP64 instead
struct RangeRule {
    double hold = 0, pad = 0;    // 2^b > max(|trap centre|, hold) + pad: start and wells, six widths of the trap
    double width = 0, well = 0;  // |x| is of the order of max(width, min(|trap centre|, well))
    unsigned long long fits = 0; // bit b + 30: no step from inside the range wraps a 64-bit sum
};
__host__ __device__ __forceinline__ long long double_bits(double v)
{
#ifdef __CUDA_ARCH__
    return __double_as_longlong(v);
#else
    long long b;
    memcpy(&b, &v, sizeof(b));
    return b;
#endif
}
// e with v < 2^e (v >= 0), and max and min of non-negative numbers, on the integer pipe.
__host__ __device__ __forceinline__ int exponent_above(double v) { return (int)(double_bits(v) >> 52) - 1022; }
__host__ __device__ __forceinline__ double max_bits(double a, double b) { return double_bits(a) > double_bits(b) ? a : b; }
__host__ __device__ __forceinline__ double min_bits(double a, double b) { return double_bits(a) < double_bits(b) ? a : b; }
// far, near: largest and smallest |trap centre| of the simulation.  A step of the
// fixed point is off by 1.2 units of 2^(b-62) rms, one of FP64 by |x| 2^-53.7, so FP64 is
// as close where 2^b = 256 |x| (measured without wells, 2^b / width 128, 256,
// 512: 0.48, 0.90, 1.8 times FP64's error); the line is at half of that.
__host__ __device__ __forceinline__ int fixed_range(const RangeRule &r, double far, double near)
{
    const int b = exponent_above(max_bits(far, r.hold) + r.pad);
    const double size = max_bits(r.width, min_bits(near, r.well));
    return b >= -30 && b <= 30 && ((r.fits >> (b + 30)) & 1) && b <= exponent_above(size) + 6 ? b : kNoRange;
}

}  // namespace pmf
