// 62-bit fixed-point arithmetic of the 1D integrator (device), and the same on
// the host for its tests.
#pragma once

#include <cuda_runtime.h>

namespace pmf {

// A 62-bit fixed-point number as two 31-bit limbs, h 2^31 + l with
// 0 <= l < 2^31.  a b 2^-62 of two such numbers (|a|, |b| < 2^62) is
// a.h b.h + 2 (hi(a.h b.l) + hi(a.l b.h)), hi = the upper 32 bits of a 64-bit
// product, within 5 units: the two cross products keep 30 bits each and the
// product of the low limbs is dropped.
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
    long long cb;  // (cB - 1) 2^62
};
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

}  // namespace pmf
