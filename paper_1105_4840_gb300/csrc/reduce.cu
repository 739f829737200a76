// FP64 reductions of the recorded x samples into the paper's estimators.
//
// Stage 1 (a team of 1, 2, 4 or 8 warps per (window i, replica r), two passes
// over the samples):
//   work increments of Eq. (9),
//   w = k/2 (lambda_{i+1} - lambda_i)(lambda_{i+1} + lambda_i - 2 x),
//   the replica's minimum m_ir, the max-shifted exponential sum
//   S_ir = sum exp(-(w - m_ir)/kT) (Eq. (12)), and the shifted moments
//   sum (x - lambda_i), sum (x - lambda_i)^2.
// Stage 2 (one CTA per window): merge the replicas (log-sum-exp aware),
//   the per-window JE increment, the Eq. (14) and Eq. (13) increments and
//   the delete-one-replica jackknife.
// Stage 3 (the last CTA of stage 2): prefix sums over windows into the
//   profiles and the combined estimate of Sec. V.
// The windows are independent (Sec. II: rho(W_mech) is the product of the
// rho(x_i)), so the average of exp(-W_mech/kT) over all combinations of
// samples is the product of the per-window averages.
//
// What bounds the three stages on small and ordinary paths is the latency of
// FP64 operations (64 cycles each for one warp of this GPU), so stages 2 and 3
// spend as few of them in sequence as they can and run independent ones on
// different warps.  21 windows x 32 replicas x 3600 samples, back to back:
// four launches (layout, partials, windows, profiles) 65.6 us, now 28.7 us;
// 5 x 4 x 256: 49.2 us, now 16.4 to 18.4 us from one call of the measurement to
// the next; 64 x 512 x 1801: 724 us, now 272 us.
#include <math.h>
#include <stddef.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "internal.h"

namespace pmf {

struct Partial {
    double m, S, n, sdx, sdx2;
};
static_assert(sizeof(Partial) == kPartialDoubles * sizeof(double), "partials are exported as 5 doubles");
struct WindowOut {
    double je, fl, g, wmean, varw, n, jk_je, jk_fl, mean, var;
};

__device__ __forceinline__ void neumaier(double &s, double &c, double v)
{
    const double t = s + v;
    if (fabs(s) >= fabs(v)) c += (s - t) + v;
    else c += (v - t) + s;
    s = t;
}

template <int NT> __device__ double block_sum(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0) {
        for (int q = 0; q < NT / 32; ++q) t += red[q];
        red[NT / 32] = t;
    }
    __syncthreads();
    return red[NT / 32];
}

template <int NT> __device__ double block_min(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = red[0];
        for (int q = 1; q < NT / 32; ++q) t = fmin(t, red[q]);
        red[NT / 32] = t;
    }
    __syncthreads();
    return red[NT / 32];
}

constexpr int kPartialThreads = 256;

// ---- the exponential of stage 1 in double-float arithmetic on the FP32 pipe
//
// GB300's FP64 unit retires 1/64 of the FP32 rate, and an FP64 exp per
// sample made stage 1 FP64-bound.  The exponent is linear in x: with the
// work increment w = k/2 (lambda_{i+1} - lambda_i)(lambda_{i+1} + lambda_i - 2x)
// and its minimum at the sample x_ref (the largest x when lambda_{i+1} >
// lambda_i, the smallest otherwise), -(w - min w)/kT = c (x - x_ref) <= 0 with
// c = k (lambda_{i+1} - lambda_i)/kT.  x - x_ref is exact as a pair of floats
// (TwoSum), c (x - x_ref) is formed as a pair of floats, and exp of that pair
// follows Tang's table-driven method (P. T. P. Tang, ACM TOMS 15 (1989)
// 144-157): a = n ln2/32 + r with |r| <= ln2/64, exp(a) = 2^(n div 32)
// 2^((n mod 32)/32) (1 + p(r)), p the Taylor series of e^r - 1 to r^6 (the
// next term is below 2e-18), 2^(j/32) as a pair of floats from the FP64 exp2,
// ln2/32 split in three floats whose first has 12 significant bits so that
// n times it is exact.  The relative error of a term, weighted by its size,
// stays near 1e-14; terms below e^-80 of the largest are dropped (the largest
// is 1).

__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e)
{
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ void fast_two_sum_f(float a, float b, float &s, float &e)  // |a| >= |b|
{
    s = a + b;
    e = b - (s - a);
}

// Passed by value: 2^(j/32) as hi + lo, 32 / ln 2, and ln2/32 = l1 + l2 + l3
// with 12 significant bits in l1.
struct ExpTable {
    float hi[32], lo[32];
    float inv_l, l1, l2, l3;
};

const ExpTable &exp_table()
{
    static const ExpTable table = [] {
        ExpTable t;
        for (int j = 0; j < 32; ++j) {
            const double v = std::exp2(j / 32.0);
            t.hi[j] = (float)v;
            t.lo[j] = (float)(v - (double)t.hi[j]);
        }
        // ln 2 as the double nearest to it plus the remainder
        const double ln2_hi = 0.6931471805599453, ln2_lo = 2.319046813846299558e-17;
        const double l = ln2_hi / 32.0;  // exact: a power-of-two scaling
        t.inv_l = (float)(32.0 / ln2_hi);
        const float lf = (float)l;
        uint32_t bits;
        std::memcpy(&bits, &lf, 4);
        bits &= ~0xFFFu;
        std::memcpy(&t.l1, &bits, 4);
        const double r1 = l - (double)t.l1;
        t.l2 = (float)r1;
        t.l3 = (float)((r1 - (double)t.l2) + ln2_lo / 32.0);
        return t;
    }();
    return table;
}

// exp(ah + al) for ah + al <= 0 as a pair of floats eh + el (tab: 2^(j/32)
// = tab_hi[j] + tab_lo[j]).
__device__ __forceinline__ void exp_ff(float ah, float al, const ExpTable &k, const float *tab_hi,
                                       const float *tab_lo, float &eh, float &el)
{
    // nearest integer to ah 32 / ln 2 (at most 3700 in size) by the addition of 1.5 2^23
    const float big = fmaf(ah, k.inv_l, 12582912.f);
    const float kf = big - 12582912.f;
    const int n = __float_as_int(big) - 0x4B400000;
    // r = a - n ln2/32: n l1 is exact and close to ah, n l2 exact as p2 + e2
    const float t1 = fmaf(-kf, k.l1, ah);
    const float p2 = kf * k.l2;
    const float e2 = fmaf(kf, k.l2, -p2);
    float rh, rl;
    two_sum_f(t1, -p2, rh, rl);
    rl += (al - e2) - kf * k.l3;
    fast_two_sum_f(rh, rl, rh, rl);
    // e^r - 1 = r + r^2/2 + r^3 (1/6 + r (1/24 + r (1/120 + r/720)))
    const float sh = rh * rh;
    const float sl = fmaf(rh, rh, -sh) + 2.f * rh * rl;
    const float q = rh * sh * fmaf(rh, fmaf(rh, fmaf(rh, 1.f / 720.f, 1.f / 120.f), 1.f / 24.f), 1.f / 6.f);
    float ph, pl;
    two_sum_f(rh, 0.5f * sh, ph, pl);
    pl += (rl + 0.5f * sl) + q;
    fast_two_sum_f(ph, pl, ph, pl);
    // 2^(j/32) (1 + p), then the power of two 2^(n div 32) (exact)
    const int j = n & 31, m = n >> 5;
    const float th = tab_hi[j], tl = tab_lo[j];
    const float uh = th * ph;
    const float ul = fmaf(th, ph, -uh) + (th * pl + tl * ph);
    float hh, hl;
    two_sum_f(th, uh, hh, hl);
    hl += tl + ul;
    const float sc = __int_as_float((m + 127) << 23);
    const bool drop = ah < -80.f;
    eh = drop ? 0.f : hh * sc;
    el = drop ? 0.f : hl * sc;
}

// Running sum h + l of float pairs: h carries the sum, l the rounding errors
// of h (TwoSum, exact) and the low parts.
__device__ __forceinline__ void ff_sum(float &h, float &l, float bh, float bl)
{
    float e;
    two_sum_f(h, bh, h, e);
    l += e + bl;
}

// Per-thread sums kept as pairs of floats and flushed into FP64 every
// kFlushSamples terms: within a flush the pair's error stays near
// kFlushSamples x 2^-47 of the partial sum, and the FP64 unit does a few
// operations per flush instead of several per sample.
constexpr int kFlushSamples = 16;

// (double)f by integer operations (a conversion takes a turn of the FP64
// unit); FP32 denormals are zero here as everywhere in this library's build.
__device__ __forceinline__ double widen(float f)
{
    const int b = __float_as_int(f), e = b & 0x7f800000;
    const int hi = (b & 0x80000000) | (((b & 0x7fffffff) >> 3) + (e == 0x7f800000 ? 0x70000000 : 0x38000000));
    return e == 0 ? __hiloint2double(b & 0x80000000, 0) : __hiloint2double(hi, b << 29);
}

// Per-window constants of stage 1, set once per CTA by one thread (the FP64
// unit is the scarce one: per-thread setup in FP64 would cost more than the
// samples themselves at a few samples per thread).
struct WindowConsts {
    double hkd, ssum;  // w = hkd (ssum - 2 x)
    double lo;         // lambda_i - (float)lambda_i
    float ch, cl;      // c = 2 hkd / kT as a pair of floats
    float li;          // (float)lambda_i
};

__device__ __forceinline__ long long samples_of(const ReduceLayout &L, int w) { return L.tw ? L.tw[w] : L.t_max; }
__device__ __forceinline__ long long offset_of(const ReduceLayout &L, int w)
{
    return L.off_w ? L.off_w[w] : (long long)w * L.replicas * L.t_max;
}

// Doubles in the order of their bits as signed integers (no NaN): compared
// on the integer pipe.
__device__ __forceinline__ long long order_key(double v)
{
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double from_order_key(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}

// Warp sums of three doubles in six additions instead of fifteen: the first
// two exchanges also sort the quantities over the lanes.  a's sum is in lanes
// 0..7, b's in 8..15, c's in 16..23.
__device__ __forceinline__ double warp_sum3(double a, double b, double c, int lane)
{
    const bool up = lane & 16, mid = lane & 8;
    double p = up ? c : a, q = up ? 0.0 : b;
    p += __shfl_xor_sync(0xffffffffu, up ? a : c, 16);
    q += __shfl_xor_sync(0xffffffffu, up ? b : 0.0, 16);
    double v = mid ? q : p;
    v += __shfl_xor_sync(0xffffffffu, mid ? p : q, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Warp sums of two doubles in five additions: a's in lanes 0..15, b's in 16..31.
__device__ __forceinline__ double warp_sum2(double a, double b, int lane)
{
    const bool up = lane & 16;
    double v = up ? b : a;
    v += __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// CTA (w, chunk): replicas [chunk x per, (chunk + 1) x per) of window w, 8 / G
// at a time by teams of G warps.  First pass: x_ref, the sample at which w is
// smallest (the largest x if w falls with x, else the smallest); second pass
// (mostly from cache): the exponential sum and the sums of q = x - (float)
// lambda_i (exact as a pair of floats) and q^2; the rest of lambda_i enters
// their totals in FP64.  About 100 FP32 operations a sample bound the large
// stores, latency (loads, the FP64 trees) the small.
// Five CTAs per SM for the large teams (672 replicas of 3600 samples then run
// in one wave: 32.8 -> 30.7 us in all); four, with 64 registers, for a warp per
// replica (64 x 512 x 1801: 274 us, five 283).
template <int G>
__global__ void __launch_bounds__(kPartialThreads, G >= 4 ? 5 : 4) partial_kernel(const ReduceLayout L, const __grid_constant__ ExpTable tab,
                                                                  int per, Partial *out)
{
    constexpr int kTeams = kPartialThreads / 32 / G, kTeamThreads = 32 * G;
    __shared__ float tab_hi[32], tab_lo[32];
    __shared__ WindowConsts wc;
    __shared__ float red_max[kPartialThreads / 32];
    __shared__ double red[kPartialThreads / 32][3];
    const int w = blockIdx.x, R = L.replicas, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int team = warp / G, tid = threadIdx.x - team * kTeamThreads;
    const long long T = samples_of(L, w), off = offset_of(L, w);
    const double li = L.lambda[w], ln = w + 1 < L.n_windows ? L.lambda[w + 1] : li;
    const float sgn = order_key(ln) < order_key(li) ? -1.f : 1.f;
    // for the combination behind this grid, which touches it after this grid's end
    if (L.counter != nullptr && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) *L.counter = 0;
    if (threadIdx.x < 32) {
        tab_hi[threadIdx.x] = tab.hi[threadIdx.x];
        tab_lo[threadIdx.x] = tab.lo[threadIdx.x];
    } else if (threadIdx.x == kPartialThreads - 1) {
        wc.hkd = 0.5 * L.k * (ln - li);
        wc.ssum = ln + li;
        const double c = 2.0 * wc.hkd / L.kT;
        wc.ch = (float)c;
        wc.cl = (float)(c - (double)wc.ch);
        wc.li = (float)li;
        wc.lo = li - (double)wc.li;
    }
    // The combination may be launched meanwhile (its CTAs wait for this grid's
    // end).  Not with one-warp teams, the rule for grids that fill the chip for
    // long: 64 x 512 x 1801 samples took 322 us with it, 272 without.
    if (G > 1) cudaTriggerProgrammaticLaunchCompletion();
    const int r0 = blockIdx.y * per, r1 = min(R, r0 + per);
    for (int rb = r0; rb < r1; rb += kTeams) {
        const int r = rb + team;
        const bool live = r < r1;
        const float *x = L.x + off + (long long)r * T;
        float mx = -INFINITY;
        if (live) {
#pragma unroll 8
            for (long long t = tid; t < T; t += kTeamThreads) mx = fmaxf(mx, sgn * x[t]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (G > 1 && lane == 0) red_max[warp] = mx;
        if (G > 1 || rb == r0) __syncthreads();  // the constants and the table are there, and the team's maxima
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (G > 1) mx = fmaxf(mx, red_max[team * G + g]);
        const float xref = sgn * mx;
        const float ch = wc.ch, cl = wc.cl, li_h = wc.li;
        double S = 0, s1 = 0, s2 = 0;
        if (live) {
            // blocks of kFlushSamples; the flush stands outside the sample
            // loop so that its FP64 operations are not speculated per sample
            // (they were: 87 % of the FP64 pipe, 802 us for 64 x 512 x 1801)
            for (long long tb = tid; tb < T; tb += (long long)kFlushSamples * kTeamThreads) {
                float Sh = 0, Sl = 0, ah1 = 0, al1 = 0, ah2 = 0, al2 = 0;
                const long long te = min(T, tb + (long long)kFlushSamples * kTeamThreads);
#pragma unroll 4
                for (long long t = tb; t < te; t += kTeamThreads) {
                    const float xv = x[t];
                    float dh, dl;
                    two_sum_f(xv, -xref, dh, dl);  // x - x_ref exactly
                    float ah = ch * dh;
                    float al = fmaf(ch, dh, -ah) + (ch * dl + cl * dh);
                    fast_two_sum_f(ah, al, ah, al);
                    float eh, el;
                    exp_ff(ah, al, tab, tab_hi, tab_lo, eh, el);
                    ff_sum(Sh, Sl, eh, el);
                    float qh, ql;
                    two_sum_f(xv, -li_h, qh, ql);
                    ff_sum(ah1, al1, qh, ql);
                    const float ph = qh * qh;
                    ff_sum(ah2, al2, ph, fmaf(qh, qh, -ph) + 2.f * qh * ql);
                }
                S += widen(Sh);
                s1 += widen(ah1);
                s2 += widen(ah2);
                S += widen(Sl);
                s1 += widen(al1);
                s2 += widen(al2);
            }
        }
        double v = warp_sum3(S, s1, s2, lane);
        if (G > 1) {
            if ((lane & 7) == 0 && lane < 24) red[warp][lane >> 3] = v;
            __syncthreads();
            if (tid < 32) {
                const int q = lane >> 3;  // lanes 0, 8, 16: the three totals
                if (q < 3)
#pragma unroll
                    for (int g = 1; g < G; ++g) v += red[warp + g][q];
            }
        }
        if (live && tid < 32) {
            const double n = (double)T;
            const double a1 = __shfl_sync(0xffffffffu, v, 8), a2 = __shfl_sync(0xffffffffu, v, 16);
            // sums of (x - lambda_i) and its square from those of q = x - lambda_i + lo
            if (lane == 0)
                out[(size_t)w * R + r] =
                    T == 0 ? Partial{INFINITY, 0.0, 0.0, 0.0, 0.0}
                           : Partial{wc.hkd * (wc.ssum - 2.0 * (double)xref), v, n, a1 - n * wc.lo,
                                     a2 - wc.lo * (2.0 * a1 - n * wc.lo)};
        }
        if (G > 1 && rb + kTeams < r1) __syncthreads();  // red_max and red are free again
    }
}

constexpr int kWindowThreads = 256;

// Replica counts up to this keep the per-replica exponential sums E[r] in
// shared memory; larger ones recompute them in the jackknife loop.
constexpr int kWindowSmemReplicas = 16384;

// Error-free sum of two doubles: s + e == a + b exactly (Knuth's TwoSum).
__device__ __forceinline__ void two_sum(double a, double b, double &s, double &e)
{
    s = a + b;
    const double bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Block-wide sum of compensated pairs (s, c) (each thread's Neumaier sum):
// the pairs are merged with TwoSum so the result hi + lo keeps the
// compensation; hi is the correctly rounded total up to O(n eps^2).
template <int NT> __device__ void block_sum_pair(double s, double c, double *red, double &hi, double &lo)
{
    for (int o = 16; o > 0; o >>= 1) {
        const double s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
        double t, e;
        two_sum(s, s2, t, e);
        s = t;
        c = c + c2 + e;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) {
        red[2 * warp] = s;
        red[2 * warp + 1] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ts = red[0], tc = red[1];
        for (int q = 1; q < NT / 32; ++q) {
            double t, e;
            two_sum(ts, red[2 * q], t, e);
            ts = t;
            tc = tc + red[2 * q + 1] + e;
        }
        const double h = ts + tc;
        red[2 * (NT / 32)] = h;
        red[2 * (NT / 32) + 1] = tc - (h - ts);
    }
    __syncthreads();
    hi = red[2 * (NT / 32)];
    lo = red[2 * (NT / 32) + 1];
}

// Sum of the replicas' exponential sums without replica r, from the
// compensated total hi + lo of all of them: (hi - e_r) + lo.  The terms are
// non-negative, so the only cancellation is e_r close to the total, and then
// hi - e_r is exact (Sterbenz: e_r >= hi / 2) and the result carries the
// total's own accuracy; otherwise hi - e_r >= hi / 2 rounds once.  O(1) per
// replica instead of re-summing the other R - 1 terms.
__device__ __forceinline__ double sum_without(double hi, double lo, double e_r)
{
    const double v = (hi - e_r) + lo;
    return v > 0.0 ? v : 0.0;
}

// Sum over the warps of half a CTA of a value that each warp holds in the lanes
// of slot q (lane / width); every thread of the half gets all of them.
constexpr int kHalf = kWindowThreads / 2, kHalfWarps = kHalf / 32;

__device__ __forceinline__ void half_sync(int half) { asm volatile("bar.sync %0, %1;" ::"r"(1 + half), "r"(kHalf) : "memory"); }

struct CombineArgs {
    const Partial *P;
    WindowOut *wo;
    double *out;
    unsigned *counter;       // windows finished; set to 0 in every call before this grid starts
    double beta_h, beta_l;   // 1 / kT
    double k_beta, half_beta2;  // k / kT, 1 / (2 kT^2)
    double jk, inv_r;        // (R - 1) / R, 1 / R
    int log2_r;              // ceil(log2 R)
};

// The profiles are prefix sums over the windows of the per-window increments
// (and a prefix minimum of the sample counts).  One warp per quantity: a lane
// adds up s / 32 consecutive windows, the lanes' totals are scanned, and the
// lane writes its windows' values; the warps' chains run side by side.
__device__ void profile(const ReduceLayout &L, const CombineArgs &A)
{
    const int s = L.n_windows, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = (s + 31) / 32, j0 = lane * k, j1 = min(s, j0 + k);
    const double *wo = reinterpret_cast<const double *>(A.wo);
    constexpr int kFields = sizeof(WindowOut) / sizeof(double);
    auto field = [&](int j, int f) { return __ldcg(wo + (size_t)j * kFields + f); };
    auto col = [&](int f) { return A.out + (size_t)f * s; };
    // the lane's exclusive prefix of the other lanes' windows, field f
    auto before = [&](int f) {
        double own = 0.0;
        for (int j = j0; j < j1; ++j)
            if (j > 0) own += field(j - 1, f);
        double pre = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, pre, o);
            if (lane >= o) pre += u;
        }
        pre = __shfl_up_sync(0xffffffffu, pre, 1);
        return lane == 0 ? 0.0 : pre;
    };
    // inclusive prefix of field f from the point after lambda_1, fn(j, value)
    auto scan = [&](int f, auto fn) {
        double run = before(f);
        for (int j = j0; j < j1; ++j) {
            if (j > 0) run += field(j - 1, f);
            fn(j, run);
        }
    };
    enum { kJe, kFl, kG, kWMean, kVarW, kN, kJkJe, kJkFl, kMean, kVar };  // order of WindowOut
    static_assert(offsetof(WindowOut, mean) == kMean * sizeof(double) && offsetof(WindowOut, jk_je) == kJkJe * sizeof(double),
                  "WindowOut order");
    switch (warp) {
    case 0: {
        double fl = before(kFl);
        scan(kJe, [&](int j, double je) {
            if (j > 0) fl += field(j - 1, kFl);
            col(kResJE)[j] = je;
            col(kResCom)[j] = 0.5 * (je + fl);
            col(kResUnc)[j] = 0.5 * (je - fl);
        });
        break;
    }
    case 1:
        scan(kFl, [&](int j, double v) {
            col(kResFluct)[j] = v;
            col(kResAccForce)[j] = j > 0 ? v / (L.lambda[j] - L.lambda[0]) : 0.0;
        });
        break;
    case 2: scan(kG, [&](int j, double v) { col(kResG)[j] = v; }); break;
    case 3: scan(kWMean, [&](int j, double v) { col(kResWMean)[j] = v; }); break;
    case 4: scan(kJkJe, [&](int j, double v) { col(kResSeJE)[j] = j > 0 ? sqrt(v) : 0.0; }); break;
    case 5: scan(kJkFl, [&](int j, double v) { col(kResSeFluct)[j] = j > 0 ? sqrt(v) : 0.0; }); break;
    case 6: {
        double q = INFINITY;  // smallest sample count of the windows before
        for (int j = j0; j < j1; ++j)
            if (j > 0) q = fmin(q, field(j - 1, kN));
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, q, o);
            if (lane >= o) q = fmin(q, u);
        }
        double Q = __shfl_up_sync(0xffffffffu, q, 1);
        if (lane == 0) Q = INFINITY;
        scan(kVarW, [&](int j, double v) {
            if (j > 0) Q = fmin(Q, field(j - 1, kN));
            // v / Q + v^2 / (2 kT^2 (Q - 1)) over the common denominator
            const double Q1 = Q - 1.0;
            col(kResVarZW)[j] = (j > 0 && Q > 1) ? v * fma(v * A.half_beta2, Q, Q1) / (Q * Q1) : (j > 0 ? NAN : 0.0);
        });
        break;
    }
    default:
        for (int j = lane; j < s; j += 32) {
            const double var = field(j, kVar);
            col(kResLambda)[j] = L.lambda[j];
            col(kResMeanX)[j] = field(j, kMean);
            col(kResVarX)[j] = var;
            col(kResGamma2)[j] = A.k_beta * var;
        }
    }
}

// One CTA per window, in two halves that work side by side: warps 0 - 3 on the
// exponential sums, 4 - 7 on the moments.  The compensated total of the
// exponential sums comes from an exact split instead of a tree of TwoSums:
// every e_r is cut at a common bit (adding and subtracting 1.5 2^K, 2 R max e <=
// 2^K <= 8 R max e): the upper parts add up without rounding, the lower ones, at most
// 2^(K-53) each, to within (R / 128 + 11) 4 R^2 2^-106 of the total (2^-90 at R =
// 32, 2^-62 at 65536), below what a double shows of it.  Leaving out the largest
// term may leave next to nothing, so its lower part is kept apart from the others'
// sum: what is left then has a sum's own relative rounding however small it is, and for
// every other r the rest holds the largest term.  (With the lower parts in one sum
// a replica 61 kT above 31 others left 1e-5 wrong, one 75 kT above nothing at all.)
// The jackknife's sums are taken about the full estimate,
// which lies between the leave-one-out values, so one pass serves mean and
// spread.  The last CTA to finish turns the windows into the profiles.
template <bool SMEM>
__global__ void __launch_bounds__(kWindowThreads) combine_kernel(const ReduceLayout L, const CombineArgs A)
{
    extern __shared__ double E[];  // [replicas] when SMEM
    __shared__ long long red_key[2][kHalfWarps];
    __shared__ double red[2][kHalfWarps][3], red_q[2][kHalfWarps][2];
    __shared__ double sh_log, sh_top[2];  // (the largest term's upper and lower part)
    __shared__ int sh_last;
    const int w = blockIdx.x, R = L.replicas, lane = threadIdx.x & 31;
    const int half = threadIdx.x >= kHalf, t = threadIdx.x - half * kHalf, hw = t >> 5;
    const Partial *p = A.P + (size_t)w * R;
    cudaGridDependencySynchronize();  // the partials are there (returns at once after an ordinary launch)
    const bool active = hw * 32 < R;  // the other warps hold no replica and keep off the FP64 unit
    double m = 0.0;
    int top = 0;  // the replica of the largest term (to 2^-20; half 0)
    // replica r's exponential sum brought to the window's common shift m
    auto e_of = [&](int r) {
        if (!(p[r].n > 0)) return 0.0;
        const double a = m - p[r].m;
        return p[r].S * exp(fma(a, A.beta_h, a * A.beta_l));
    };
    // max over the half's threads of an integer key
    auto half_max = [&](long long key, int slot) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
        if (lane == 0) red_key[slot][hw] = key;
        half_sync(0);
#pragma unroll
        for (int g = 0; g < kHalfWarps; ++g) key = max(key, red_key[slot][g]);
        return key;
    };
    if (half == 0) {
        long long key = order_key(-INFINITY);
        for (int r = t; r < R; r += kHalf)
            if (p[r].n > 0) key = max(key, order_key(-p[r].m));
        m = -from_order_key(half_max(key, 0));
        double e0 = 0.0;  // this thread's first term
        long long emax = 0;
        for (int r = t; r < R; r += kHalf) {
            const double e = e_of(r);
            if (r == t) e0 = e;
            if (SMEM) E[r] = e;
            emax = max(emax, (__double_as_longlong(e) & ~0xffffffffLL) | r);
        }
        emax = half_max(emax, 1);
        top = (int)(emax & 0xffffffffLL);
        if (active) {
            // 1.5 2^K with 2^K >= 2 R max e (NaN and overflowing terms end up in the sums either way)
            const int K = min(max((int)(emax >> 52) - 1023 + 2 + A.log2_r, -1022), 1023);
            const double cut = __hiloint2double(((K + 1023) << 20) | 0x80000, 0);
            double hi = 0.0, lo = 0.0;
            for (int r = t; r < R; r += kHalf) {
                const double e = r == t ? e0 : (SMEM ? E[r] : e_of(r));
                const double u = (e + cut) - cut;
                hi += u;
                if (r == top) {
                    sh_top[0] = u;
                    sh_top[1] = e - u;
                } else {
                    lo += e - u;
                }
            }
            const double v = warp_sum2(hi, lo, lane);
            if ((lane & 15) == 0) red[0][hw][lane >> 4] = v;
        }
    } else if (active) {
        double sn = 0, s1 = 0, c1 = 0, s2 = 0, c2 = 0;
        for (int r = t; r < R; r += kHalf) {
            if (r == t) {
                sn = p[r].n;
                s1 = p[r].sdx;
                s2 = p[r].sdx2;
            } else {
                sn += p[r].n;
                neumaier(s1, c1, p[r].sdx);
                neumaier(s2, c2, p[r].sdx2);
            }
        }
        if (R > kHalf) {
            s1 += c1;
            s2 += c2;
        }
        const double v = warp_sum3(sn, s1, s2, lane);
        if ((lane & 7) == 0 && lane < 24) red[1][hw][lane >> 3] = v;
    }
    __syncthreads();
    auto total = [&](int h, int q) {
        double v = red[h][0][q];
#pragma unroll
        for (int g = 1; g < kHalfWarps; ++g)
            if (g * 32 < R) v += red[h][g][q];
        return v;
    };
    const bool jk = R >= 2, closing = hw == kHalfWarps - 1;  // each half's last warp: the window's own values
    double q1 = 0, q2 = 0;  // jackknife: sums of the leave-one-out values minus the full estimate, and of their squares
    double lf = 0.0;
    if (half == 0) {
        double Shi = 0, Slo = 0, n = 0, th = 0, rest = 0;
        if (active || closing) {
            th = total(0, 0);
            rest = total(0, 1);
            const double tl = rest + sh_top[1];
            n = total(1, 0);
            Shi = th + tl;
            Slo = tl - (Shi - th);
        }
        auto log_without = [&](int r) {
            const double e = SMEM ? E[r] : e_of(r);
            // (from half the total on; selects, not a branch: two FP64 operations either way)
            const bool most = r == top && __double2hiint(Shi) - __double2hiint(e) < 1 << 20;
            return log(sum_without(most ? th : Shi, most ? rest : Slo, most ? sh_top[0] : e) / (n - p[r].n));
        };
        if (closing && lane == 0) sh_log = log((Shi + Slo) / n);  // beside the leave-one-out logarithms
        double l0 = 0.0;
        if (jk && t < R) l0 = log_without(t);
        half_sync(0);
        lf = sh_log;
        if (jk)
            for (int r = t; r < R; r += kHalf) {
                const double v = L.kT * (lf - (r == t ? l0 : log_without(r)));
                q1 += v;
                q2 += v * v;
            }
    } else if (active || closing) {
        const double li = L.lambda[w], ln = w + 1 < L.n_windows ? L.lambda[w + 1] : li, d = ln - li;
        const double n = total(1, 0), sdx = total(1, 1), kd = -L.k * d;
        const double mdx = sdx / n;
        const double fl = kd * mdx;
        if (jk)
            for (int r = t; r < R; r += kHalf) {
                const double v = kd * (sdx - p[r].sdx) / (n - p[r].n) - fl;
                q1 += v;
                q2 += v * v;
            }
        if (closing && lane == 0) {
            const double mean = li + mdx, var = total(1, 2) / n - mdx * mdx;
            WindowOut &o = A.wo[w];
            o.fl = fl;
            o.g = L.k * d * d / 2.0 * (1.0 - A.k_beta * var) + fl;
            o.wmean = 0.5 * L.k * d * (ln + li - 2.0 * mean);
            o.varw = L.k * L.k * d * d * var;
            o.n = n;
            o.mean = mean;
            o.var = var;
        }
    }
    if (active) {
        const double v = warp_sum2(q1, q2, lane);
        if ((lane & 15) == 0) red_q[half][hw][lane >> 4] = v;
    }
    half_sync(half);
    if (t == 0) {
        double a = red_q[half][0][0], b = red_q[half][0][1];
#pragma unroll
        for (int h = 1; h < kHalfWarps; ++h)
            if (h * 32 < R) {
                a += red_q[half][h][0];
                b += red_q[half][h][1];
            }
        const double spread = jk ? A.jk * fmax(b - a * a * A.inv_r, 0.0) : NAN;
        if (half == 0) {
            A.wo[w].je = m - L.kT * lf;
            A.wo[w].jk_je = spread;
        } else {
            A.wo[w].jk_fl = spread;
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) sh_last = atomicAdd(A.counter, 1u) == (unsigned)L.n_windows - 1;
    __syncthreads();
    if (!sh_last) return;
    __threadfence();
    profile(L, A);
}

// ---------------------------------------------------------------------------
// Eq. (5) and Eq. (15).  The free energy of turning the trap on at lambda_1,
// dF(lambda_1, k) = kT ln < exp(u / kT) >, u = k/2 (x_1 - lambda_1)^2, over the
// first window's samples, and the state free energy
// G(lambda_j, lambda_1) = dF^JE(lambda_j, lambda_1, k) - dF(lambda_1, k).
// Stage 1 (one CTA per replica of the first window): the replica's
// max-shifted sum in the form of the JE partials with w = -u:
// m = min w = -max u, S = sum exp(-(w - m)/kT) = sum exp((u - max u)/kT).
// Stage 2 (one CTA): the turn-on estimate, G at every profile point, and the
// delete-one-replica jackknife (the first window's replica r is left out of
// its JE increment and of the turn-on average together; the other windows'
// jackknife variances of their increments are added).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kPartialThreads) turn_on_partial_kernel(const ReduceLayout L, Partial *out)
{
    __shared__ double red[kPartialThreads / 32 + 1];
    const int r = blockIdx.x;
    const long long T = L.tw[0];
    const float *x = L.x + L.off_w[0] + (long long)r * T;
    const double l1 = L.lambda[0], hk = 0.5 * L.k, beta = 1.0 / L.kT;
    double m = INFINITY, S = 0;
    for (long long t = threadIdx.x; t < T; t += kPartialThreads) {
        const double d = (double)x[t] - l1;
        const double wv = -hk * d * d;
        if (wv < m) {
            S = (m == INFINITY ? 0.0 : S * exp((wv - m) * beta)) + 1.0;
            m = wv;
        } else {
            S += exp((m - wv) * beta);
        }
    }
    const double mb = block_min<kPartialThreads>(m, red);
    const double St = m == INFINITY ? 0.0 : S * exp((mb - m) * beta);
    const double Sb = block_sum<kPartialThreads>(St, red);
    if (threadIdx.x == 0) out[r] = Partial{mb, Sb, (double)T, 0.0, 0.0};
}

// The window's exponential sums of the replicas on a common shift: the
// shift (minimum of the replicas' minima) and the compensated total.
template <int NT>
__device__ void common_shift_sum(const Partial *p, int R, double kT, double *red, double &m, double &hi, double &lo,
                                 double &n)
{
    double mm = INFINITY;
    for (int r = threadIdx.x; r < R; r += NT)
        if (p[r].n > 0) mm = fmin(mm, p[r].m);
    m = block_min<NT>(mm, red);
    double se = 0, ce = 0, sn = 0;
    for (int r = threadIdx.x; r < R; r += NT) {
        neumaier(se, ce, p[r].n > 0 ? p[r].S * exp(-(p[r].m - m) / kT) : 0.0);
        sn += p[r].n;
    }
    block_sum_pair<NT>(se, ce, red, hi, lo);
    n = block_sum<NT>(sn, red);
}

__global__ void __launch_bounds__(kWindowThreads) state_kernel(const ReduceLayout L, const Partial *P, const Partial *Pt,
                                                               const WindowOut *wo, double *out)
{
    __shared__ double red[2 * (kWindowThreads / 32 + 1)];
    const int R = L.replicas, s = L.n_windows;
    const double kT = L.kT;
    double m0, S0h, S0l, n, mt, Sth, Stl, nt;
    common_shift_sum<kWindowThreads>(P, R, kT, red, m0, S0h, S0l, n);   // first window, Eq. (12)
    common_shift_sum<kWindowThreads>(Pt, R, kT, red, mt, Sth, Stl, nt);  // first window, Eq. (5)
    const double on = kT * log((Sth + Stl) / nt) - mt;
    // leave-one-out values of the first window: its JE increment minus the
    // turn-on estimate (g), and the turn-on estimate alone (t)
    auto e_of = [&](const Partial &q, double mm) { return q.n > 0 ? q.S * exp(-(q.m - mm) / kT) : 0.0; };
    double vg = 0, vt = 0;
    const bool jk = R >= 2;
    if (jk) {
        for (int r = threadIdx.x; r < R; r += kWindowThreads) {
            const double nm = n - P[r].n;
            const double t = kT * log(sum_without(Sth, Stl, e_of(Pt[r], mt)) / nm) - mt;
            const double je = m0 - kT * log(sum_without(S0h, S0l, e_of(P[r], m0)) / nm);
            vg += je - t;
            vt += t;
        }
    }
    const double mg = block_sum<kWindowThreads>(vg, red) / R;
    const double mtt = block_sum<kWindowThreads>(vt, red) / R;
    double qg = 0, qt = 0;
    if (jk) {
        for (int r = threadIdx.x; r < R; r += kWindowThreads) {
            const double nm = n - P[r].n;
            const double t = kT * log(sum_without(Sth, Stl, e_of(Pt[r], mt)) / nm) - mt;
            const double je = m0 - kT * log(sum_without(S0h, S0l, e_of(P[r], m0)) / nm);
            qg += (je - t - mg) * (je - t - mg);
            qt += (t - mtt) * (t - mtt);
        }
    }
    const double var_g = (R - 1.0) / R * block_sum<kWindowThreads>(qg, red);
    const double var_t = (R - 1.0) / R * block_sum<kWindowThreads>(qt, red);
    if (threadIdx.x == 0) {
        double je = 0, v = var_g;
        for (int j = 0; j < s; ++j) {
            if (j > 0) je += wo[j - 1].je;
            if (j > 1) v += wo[j - 1].jk_je;
            out[j] = je - on;                                              // G(lambda_j, lambda_1)
            out[s + j] = jk ? sqrt(j == 0 ? var_t : v) : NAN;              // its standard error
        }
        out[2 * s] = on;                                                   // dF(lambda_1, k), Eq. (5)
    }
}

cudaError_t state_launch(const ReduceLayout &L, void *scratch, void *turn_partials, double *out, cudaStream_t st)
{
    const Partial *P = static_cast<const Partial *>(scratch);
    const WindowOut *wo =
        reinterpret_cast<const WindowOut *>(static_cast<const char *>(scratch) + partial_bytes(L.n_windows, L.replicas));
    Partial *Pt = static_cast<Partial *>(turn_partials);
    turn_on_partial_kernel<<<L.replicas, kPartialThreads, 0, st>>>(L, Pt);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    state_kernel<<<1, kWindowThreads, 0, st>>>(L, P, Pt, wo, out);
    return cudaGetLastError();
}

constexpr size_t kCounterBytes = 256;

size_t reduce_scratch_bytes(int n_windows, int replicas)
{
    return sizeof(Partial) * (size_t)n_windows * replicas + sizeof(WindowOut) * (size_t)n_windows + kCounterBytes;
}

unsigned *reduce_counter(void *buffer, size_t bytes)
{
    return reinterpret_cast<unsigned *>(static_cast<char *>(buffer) + bytes - kCounterBytes);
}

cudaError_t partials_launch(const ReduceLayout &L, void *P, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // Warps per replica: as few as keep 24 warps on every SM, but no more
    // than leave a thread four samples.  Replicas per CTA: one turn of its
    // teams, more where that is more CTAs than fit at once (8 per SM), so that
    // the window's constants are set less often.
    // 24 or 16 warps: 30.7, 32.8 us for 21 x 32 x 3600 samples (ordinary launches).
    const long long n = (long long)L.n_windows * L.replicas;
    int G = 1;
    while (G < 8 && n * G < 24LL * sms && 64 * G * 4 <= L.t_max) G *= 2;
    const int teams = kPartialThreads / 32 / G;
    const long long turns = std::min(8LL, std::max(1LL, n / ((long long)teams * 8 * sms)));
    const int per = teams * (int)turns;
    const dim3 grid(L.n_windows, (L.replicas + per - 1) / per);
    Partial *out = static_cast<Partial *>(P);
    const ExpTable &tab = exp_table();
    if (G == 1) partial_kernel<1><<<grid, kPartialThreads, 0, st>>>(L, tab, per, out);
    else if (G == 2) partial_kernel<2><<<grid, kPartialThreads, 0, st>>>(L, tab, per, out);
    else if (G == 4) partial_kernel<4><<<grid, kPartialThreads, 0, st>>>(L, tab, per, out);
    else partial_kernel<8><<<grid, kPartialThreads, 0, st>>>(L, tab, per, out);
    return cudaGetLastError();
}

// behind_partials: the stream's last operation is this call's partials launch,
// whose tail the combination's launch overlaps (it waits for that grid before it
// reads): 5 x 4 x 256 samples 20.5 -> 17.3 us (first measured; see the top of the file), 21 x 32 x 3600 30.7 -> 28.7 us.
// Behind anything else (gathered partials) an ordinary launch.
template <typename K>
static cudaError_t launch_combine(K kernel, size_t smem, bool behind_partials, cudaStream_t st, const ReduceLayout &L,
                                  const CombineArgs &A)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)L.n_windows);
    cfg.blockDim = dim3(kWindowThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = behind_partials ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, L, A);
}

cudaError_t combine_launch(const ReduceLayout &L, const void *P, void *window_scratch, double *out, cudaStream_t st,
                           bool behind_partials)
{
    if (L.counter == nullptr) return cudaErrorInvalidValue;
    if (!behind_partials) {  // (the partials' grid zeroes it otherwise)
        cudaError_t e = cudaMemsetAsync(L.counter, 0, sizeof(unsigned), st);
        if (e != cudaSuccess) return e;
    }
    CombineArgs A;
    A.P = static_cast<const Partial *>(P);
    A.wo = static_cast<WindowOut *>(window_scratch);
    A.out = out;
    A.counter = L.counter;
    A.beta_h = 1.0 / L.kT;
    A.beta_l = -std::fma(A.beta_h, L.kT, -1.0) * A.beta_h;
    A.k_beta = L.k / L.kT;
    A.half_beta2 = 1.0 / (2.0 * L.kT * L.kT);
    A.inv_r = 1.0 / L.replicas;
    A.jk = (L.replicas - 1.0) / L.replicas;
    A.log2_r = 0;
    while ((1LL << A.log2_r) < L.replicas) ++A.log2_r;
    if (L.replicas <= kWindowSmemReplicas) {
        const size_t smem = sizeof(double) * (size_t)L.replicas;
        if (smem > 40 * 1024) {
            cudaError_t e =
                cudaFuncSetAttribute(combine_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        return launch_combine(combine_kernel<true>, smem, behind_partials, st, L, A);
    }
    return launch_combine(combine_kernel<false>, 0, behind_partials, st, L, A);
}

// Constant-velocity pulling, record j (one block each): over the replicas,
// the Jarzynski average of the accumulated work, its mean and variance (the
// second-order cumulant estimate) and the mean reaction coordinate.
__global__ void __launch_bounds__(kWindowThreads) smd_stats_kernel(const double *W, const float *x, int R, long long T,
                                                                   double kT, double *out)
{
    __shared__ double red[kWindowThreads / 32 + 1];
    const long long j = blockIdx.x;
    double m = INFINITY;
    for (int r = threadIdx.x; r < R; r += kWindowThreads) m = fmin(m, W[(size_t)r * T + j]);
    m = block_min<kWindowThreads>(m, red);
    double se = 0, ce = 0, sw = 0, cw = 0, sx = 0, cx = 0;
    for (int r = threadIdx.x; r < R; r += kWindowThreads) {
        const double w = W[(size_t)r * T + j];
        neumaier(se, ce, exp(-(w - m) / kT));
        neumaier(sw, cw, w);
        neumaier(sx, cx, (double)x[(size_t)r * T + j]);
    }
    const double S = block_sum<kWindowThreads>(se + ce, red);
    const double mean = block_sum<kWindowThreads>(sw + cw, red) / R;
    const double mx = block_sum<kWindowThreads>(sx + cx, red) / R;
    double sv = 0, cv = 0;
    for (int r = threadIdx.x; r < R; r += kWindowThreads) {
        const double d = W[(size_t)r * T + j] - mean;
        neumaier(sv, cv, d * d);
    }
    const double var = block_sum<kWindowThreads>(sv + cv, red) / R;
    if (threadIdx.x == 0) {
        out[0 * T + j] = m - kT * log(S / R);
        out[1 * T + j] = mean - var / (2.0 * kT);
        out[2 * T + j] = mean;
        out[3 * T + j] = var;
        out[4 * T + j] = mx;
    }
}

cudaError_t smd_stats_launch(const double *W, const float *x, int R, long long T, double kT, double *out,
                             cudaStream_t st)
{
    if (T < 1) return cudaSuccess;
    smd_stats_kernel<<<(unsigned)T, kWindowThreads, 0, st>>>(W, x, R, T, kT, out);
    return cudaGetLastError();
}

size_t partial_bytes(int n_windows, int replicas) { return sizeof(Partial) * (size_t)n_windows * replicas; }

cudaError_t reduce_launch(const ReduceLayout &L, void *scratch, double *out, cudaStream_t st)
{
    void *P = scratch;
    void *wo = static_cast<char *>(scratch) + partial_bytes(L.n_windows, L.replicas);
    cudaError_t e = partials_launch(L, P, st);
    if (e != cudaSuccess) return e;
    return combine_launch(L, P, wo, out, st, true);
}

__global__ void work_increment_kernel(const ReduceLayout L, double *out)
{
    const int w = blockIdx.y, r = blockIdx.z;
    const long long T = L.tw[w];
    const double li = L.lambda[w], ln = L.lambda[w + 1];
    const double hkd = 0.5 * L.k * (ln - li), ssum = ln + li;
    const long long base = L.off_w[w] + (long long)r * T;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < T; t += (long long)gridDim.x * blockDim.x)
        out[base + t] = hkd * (ssum - 2.0 * (double)L.x[base + t]);
}

__global__ void work_paired_kernel(const ReduceLayout L, long long T, double *out)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long n = (long long)L.replicas * T;
    if (idx >= n) return;
    double W = 0.0;
    for (int i = 0; i + 1 < L.n_windows; ++i) {
        const double li = L.lambda[i], ln = L.lambda[i + 1];
        W += 0.5 * L.k * (ln - li) * (ln + li - 2.0 * (double)L.x[L.off_w[i] + idx]);
        out[(size_t)i * n + idx] = W;
    }
}

cudaError_t work_samples_launch(const ReduceLayout &L, int mode, long long samples_per_replica, double *out,
                                cudaStream_t st)
{
    if (mode == 0) {
        const int bx = (int)((samples_per_replica + 255) / 256 > 64 ? 64 : (samples_per_replica + 255) / 256);
        work_increment_kernel<<<dim3(bx > 0 ? bx : 1, L.n_windows - 1, L.replicas), 256, 0, st>>>(L, out);
    } else {
        const long long n = (long long)L.replicas * samples_per_replica;
        work_paired_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(L, samples_per_replica, out);
    }
    return cudaGetLastError();
}


// ---------------------------------------------------------------------------
// Allocation-free variant of the reduction (pmf_free_energy_noalloc).
//
// Its scratch (replica partials, window results, sample offsets) lives in one
// file-scope device array of fixed size instead of memory obtained from
// cudaMalloc.  Every GPU that loads the library holds this array until the
// process exits, and every call on that GPU reuses it: two calls whose work
// overlaps on the GPU (different streams, or a second call before the first
// has finished) write the same scratch and race.  Each call rewrites every entry
// it later reads, the counter of finished windows too, so whatever an overlap
// left there ends with the calls that overlapped.
// ---------------------------------------------------------------------------

namespace {

constexpr size_t kNoAllocPartialBytes = sizeof(Partial) * (size_t)kNoAllocMaxWindowReplicas;
constexpr size_t kNoAllocWindowBytes = sizeof(WindowOut) * (size_t)kNoAllocMaxWindows;
constexpr size_t kNoAllocBytes = kNoAllocPartialBytes + kNoAllocWindowBytes + kCounterBytes;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Host side: the array's name is only a host stand-in; its device address is
// looked up with that device current and cached per device, together with
// the unique id of the CUDA context it was looked up in.  A later call in
// another context of the same device (after cudaDeviceReset, the module and
// its array are loaded again, maybe elsewhere) looks the address up again.
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
void *g_noalloc_addr[kMaxDevices] = {};
unsigned long long g_noalloc_ctx[kMaxDevices] = {};

// Unique id of the calling thread's current context (driver entry points
// cuCtxGetCurrent / cuCtxGetId, reached through the runtime so the library
// links no driver library); 0 if it cannot be had.
unsigned long long current_context_id()
{
    using GetCurrent = int (*)(void **);
    using GetId = int (*)(void *, unsigned long long *);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<GetCurrent>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetId>(f);
    });
    void *ctx = nullptr;
    unsigned long long id = 0;
    if (get_current && get_id && get_current(&ctx) == 0 && ctx && get_id(ctx, &id) == 0) return id;
    return 0;
}

cudaError_t noalloc_scratch(void **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    const unsigned long long ctx = current_context_id();
    if (g_noalloc_addr[dev] == nullptr || ctx == 0 || ctx != g_noalloc_ctx[dev]) {
        // (the lookup makes the device's primary context current if no
        // runtime call has done so yet; the id is read again after it)
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_addr[dev] = p;
        g_noalloc_ctx[dev] = current_context_id();
    }
    *out = g_noalloc_addr[dev];
    return cudaSuccess;
}

}  // namespace

cudaError_t noalloc_set_counter(unsigned value, cudaStream_t st)
{
    void *base = nullptr;
    cudaError_t e = noalloc_scratch(&base);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(reduce_counter(base, kNoAllocBytes), &value, sizeof(value), cudaMemcpyHostToDevice, st)) != cudaSuccess)
        return e;
    return cudaStreamSynchronize(st);
}

cudaError_t reduce_noalloc_launch(const float *x, const double *lambda, int n_windows, int replicas,
                                  long long samples_per_window, double k, double kT, double *out, cudaStream_t st)
{
    void *base = nullptr;
    cudaError_t e = noalloc_scratch(&base);
    if (e != cudaSuccess) return e;
    unsigned char *b = static_cast<unsigned char *>(base);
    Partial *P = reinterpret_cast<Partial *>(b);
    WindowOut *wo = reinterpret_cast<WindowOut *>(b + kNoAllocPartialBytes);
    ReduceLayout L;
    L.x = x;
    L.lambda = lambda;
    L.t_max = samples_per_window;  // no per-window arrays: every window alike
    L.counter = reduce_counter(base, kNoAllocBytes);
    L.n_windows = n_windows;
    L.replicas = replicas;
    L.k = k;
    L.kT = kT;
    if ((e = partials_launch(L, P, st)) != cudaSuccess) return e;
    return combine_launch(L, P, wo, out, st, true);
}

}  // namespace pmf
