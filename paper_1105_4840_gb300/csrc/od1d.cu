// Overdamped Langevin particle in the 1D double well, FP64, one thread per
// simulation: the PPP of Sec. III (ii) (and the sequential protocol and
// constant-velocity pulling) on the model
// H(lambda, x) = a (x^2 - 1)^2 + k/2 (x - lambda)^2 (kT units).
//   x_{n+1} = x_n + F(x_n) dt / gamma + sqrt(2 kT dt / gamma) xi_n,
// F = -dH/dx, xi_n = normal (n mod 4) of the Philox block (0, uid, n div 4, 0).
// Regrouped, x_{n+1} = x_n (cA x_n^2 + cB) + q_n with cA = -4a dt/gamma,
// cB = 1 + (4a - k) dt/gamma and q_n = k lambda_n dt/gamma + amp xi_n.  q_n
// does not depend on the trajectory, so a parallel pre-pass computes it for
// a block of steps of every simulation; the integration is one dependent
// chain per simulation, and its latency per step is the time of the run.
//
// Arithmetic of the chain.  This GPU's FP64 unit takes 64 cycles per operation
// of a warp, dependent or not, so the three FP64 operations of a step cost 192
// cycles.  Where the launch's parameters bound the motion, the chain runs in
// 62-bit fixed point on the integer pipe instead (IMAD.WIDE: 5 cycles):
// X = x 2^S with |x| < 2^b, S = 62 - b, and
//   X' = X + Q + X w,  w = (cB - 1) + cA 4^b (X 2^-62)^2,
// products of 62-bit numbers within a few units of 2^(b-62) (9e-19 for the
// double well's b = 2), 1/128 of the FP64 rounding of a position near 1.  The
// products round down; left alone that drift adds up to 2 1/4 units /
// (k dt/gamma) where no well contracts the map faster (a = 0, k = 1, dt = 1e-3,
// b = 4: 7.5e-15 against FP64's 1.2e-15), so its mean is added to the terms
// that are there anyway, cB - 1 and q_n (the same case: 6e-17).  A simulation that leaves |x| < 2^b
// redoes the tile of steps it left in, and runs on, in FP64.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "fixed62.h"
#include "internal.h"

namespace pmf {

struct Od1dArgs {
    double x0, k;
    const double *lambda;
    const long long *nsteps_w, *nequil_w, *off_w, *tw;
    double *state;              // [n_rep][2]: x and the accumulated pulling work
    const double *start;
    float *xout;
    int *err;
    long long c0, c1;           // this launch's steps
    int replicas, stride, n_rep;
    uint32_t uid_base;
    unsigned long long seed;
    int sequential;             // sequential protocol: window = step / window_steps
    long long window_steps;
    double *wout;               // constant-velocity pulling: work at the records
    double smd_vdt;             //   trap advance per step after the equilibration
    long long *noise;           // [c1 - c0][n_rep] q_n of this launch's steps (fixed: q_n 2^S, else the double's bits)
    int fixed, range_log2;      // fixed point: on, and b
    int q_off;                  // fixed point: mean of the last product's rounding (q_offset256)
    double cA, cB1;             // -4a dt/gamma, (4a - k) dt/gamma
    double amp, ck;             // sqrt(2 kT dt/gamma), k dt/gamma; fixed: times 2^S (set on the host: per thread
                                // they took a sixth of the pre-pass's FP64 operations)
};

// Trap centre during step n of simulation rep: its window's lambda (the
// window of step n in the sequential protocol), or, when pulled, lambda_1
// advanced by vdt per step after the equilibration.
__device__ __forceinline__ double trap_centre(const Od1dArgs &a, int rep, long long n)
{
    if (a.wout) {
        const long long nequil = a.nequil_w[0];
        return n > nequil ? a.lambda[0] + a.smd_vdt * (double)(n - nequil) : a.lambda[0];
    }
    return a.lambda[a.sequential ? (int)(n / a.window_steps) : rep / a.replicas];
}

// q_n of every simulation for steps [c0, c1), one Philox block (four steps
// of one simulation) per thread, stored [n - c0][rep].
__global__ void od1d_noise_kernel(const Od1dArgs a, long long *q)
{
    const long long nb = (a.c1 - a.c0 + 3) >> 2;  // c0 is a multiple of 4
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= nb * a.n_rep) return;
    const int rep = (int)(i % a.n_rep);
    const long long blk = i / a.n_rep;
    const long long n0 = a.c0 + 4 * blk;
    const Normal4<double> z =
        philox_normals<double>(a.seed, 0u, a.uid_base + (uint32_t)rep, (uint32_t)(n0 >> 2), kTagOStep);
    const double v[4] = {z.n0, z.n1, z.n2, z.n3};
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        const long long n = n0 + l;
        if (n < a.c1) {
            const double qn = fma(a.amp, v[l], a.ck * trap_centre(a, rep, n));
            q[(n - a.c0) * a.n_rep + rep] = a.fixed ? __double2ll_rn(qn) + q_offset(a.q_off, n) : __double_as_longlong(qn);
        }
    }
}

// 32 simulations per CTA, steps [c0, c1): the parallel protocol (window rep /
// R throughout), the sequential protocol (window = step / tau, Sec. III (i))
// or constant-velocity pulling (the trap at lambda_1 + vdt (n - n_equil) from
// step n_equil on, the move before step n doing the work of Eq. (9) at the
// current x).  Warp 0 integrates, lane = simulation, a tile of kTile steps at
// a time from shared memory to shared memory; warps 1 - 3 meanwhile fetch the
// next tile's q_n and turn the previous tile's positions into samples and
// pulling work, so the dependent chain carries nothing else.  What bounds it is
// that chain: 118 cycles a step by itself (a product of limbs is four dependent
// 32 x 32 -> 64 multiplies of 9 - 12 cycles and a split), about 145 with the
// tile's barrier; one thread per simulation in FP64 with loads and samples in
// its loop took 403.  21 x 8 simulations x 2e4 steps, whole run with estimates:
// 4.62 -> 1.80 ms; 256 pulled simulations x 4400 steps: 2.27 -> 0.75 ms.
constexpr int kTile = 40;  // 41.5 KB of shared memory a CTA; 32 steps: 2.17 against 1.90 ms
static_assert(kTile % 8 == 0, "unrolled by 8");
constexpr int kOd1dThreads = 128;

__global__ void __launch_bounds__(kOd1dThreads) od1d_kernel(const Od1dArgs a)
{
    __shared__ long long Q[2][kTile][32];      // q_n
    __shared__ long long X[2][kTile + 1][32];  // positions before the tile's first step and after each
    __shared__ unsigned dbl_mask[2];           // lanes whose tile is in FP64 (bits of doubles)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rep = blockIdx.x * 32 + lane;
    const bool live = rep < a.n_rep;
    const int r = a.sequential ? rep : rep % a.replicas;
    const int w = a.sequential || !live ? 0 : rep / a.replicas;
    // this simulation's last step (its window's step count)
    long long end = a.c1;
    if (!a.sequential && live) end = end < a.nsteps_w[w] ? end : a.nsteps_w[w];
    if (!live || end < a.c0) end = a.c0;
    const double scale = scalbn(1.0, 62 - a.range_log2), unit = scalbn(1.0, a.range_log2 - 62);
    const double cA = a.cA, cB1 = a.cB1, cB = 1.0 + cB1;
    const long long tiles = (a.c1 - a.c0 + kTile - 1) / kTile;

    auto load_tile = [&](long long i, int row, int step) {
        const long long n0 = i * kTile;
        for (int s = row; s < kTile; s += step)
            if (live && n0 + s < a.c1 - a.c0) Q[i & 1][s][lane] = a.noise[(n0 + s) * a.n_rep + rep];
    };

    // warp 0: the position, in fixed point or (dbl) FP64
    FixedStep f{};
    long long Xi = 0;
    double x = 0.0;
    bool dbl = true;
    if (warp == 0 && live) {
        x = a.c0 == 0 ? (a.start ? a.start[rep] : a.x0) : a.state[2 * rep];
        if (a.fixed) {
            f = step_of(cA, cB1, a.range_log2);
            if (fabs(x) < scalbn(1.0, a.range_log2)) {
                Xi = __double2ll_rn(x * scale);
                dbl = false;
            }
        }
    }
    auto integrate = [&](long long i) {
        const long long n0 = a.c0 + i * kTile;
        const int b = (int)(i & 1);
        const int lim = end <= n0 ? 0 : (end - n0 < kTile ? (int)(end - n0) : kTile);
        const long long X0 = Xi;
        bool redo = dbl && lim > 0;
        if (!dbl) {
            X[b][0][lane] = Xi;
            unsigned guard = 0;  // top bit: a position outside [-2^62, 2^62)
            if (__all_sync(__activemask(), lim == kTile)) {
#pragma unroll 8
                for (int s = 0; s < kTile; ++s) {
                    Xi = fixed_step(f, Xi, Q[b][s][lane]);
                    X[b][s + 1][lane] = Xi;
                    guard |= range_guard(Xi);
                }
            } else {
                for (int s = 0; s < lim; ++s) {
                    Xi = fixed_step(f, Xi, Q[b][s][lane]);
                    X[b][s + 1][lane] = Xi;
                    guard |= range_guard(Xi);
                }
            }
            if (guard >> 31) {
                x = (double)X0 * unit;
                dbl = redo = true;
            }
        }
        if (redo) {
            X[b][0][lane] = __double_as_longlong(x);
#pragma unroll 4
            for (int s = 0; s < lim; ++s) {
                const long long qb = Q[b][s][lane];
                x = fma(x, fma(cA, x * x, cB), a.fixed ? (double)(qb - q_offset(a.q_off, n0 + s)) * unit : __longlong_as_double(qb));
                X[b][s + 1][lane] = __double_as_longlong(x);
            }
        }
        __syncwarp();
        const unsigned mask = __ballot_sync(0xffffffffu, dbl);
        if (lane == 0) dbl_mask[b] = mask;
    };

    // warps 1 - 3: the records of a finished tile; no division in the loop
    const int helper = warp - 1;
    static_assert(kOd1dHelpers == kOd1dThreads / 32 - 1, "every warp but the first records");
    int ww = w;
    RecordWalk walk;
    long long base = 0, wend = 0;
    auto enter_window = [&](int window, long long from) {
        ww = window;
        const long long origin = a.sequential ? (long long)ww * a.window_steps : 0;
        walk.enter(origin, a.nequil_w[ww], a.stride, from, helper);
        base = a.off_w[ww] + (long long)r * a.tw[ww];
        wend = a.sequential ? origin + a.window_steps : end;
    };
    // pulling work: W after the trap's first moves0 moves, and since then the
    // sum of X - lambda_1 in two 32-bit halves (every helper keeps it, each
    // converts for its own records)
    double W = 0.0;
    long long acc_h = 0, moves0 = 0, moves = 0;
    unsigned long long acc_l = 0;
    const double lam1 = a.lambda[0], kv = a.k * a.smd_vdt;
    const long long L1 = a.fixed ? __double2ll_rn(lam1 * scale) : 0;
    if (warp > 0 && live) {
        enter_window(a.sequential ? (int)(a.c0 / a.window_steps) : w, a.c0);
        if (a.wout) {
            W = a.c0 == 0 ? 0.0 : a.state[2 * rep + 1];
            moves = a.c0 - 1 - a.nequil_w[0];
            moves0 = moves = moves > 0 ? moves : 0;
        }
    }
    // sum over the moves m of k vdt (lambda_1 + vdt (m - 1/2) - x)
    auto fixed_work = [&] {
        const double m = (double)moves, m0 = (double)moves0;
        const double sum = ((double)acc_h * 4294967296.0 + (double)acc_l) * unit;
        return W + kv * (0.5 * a.smd_vdt * (m * m - m0 * m0) - sum);
    };
    auto records = [&](long long i) {
        if (!live) return;  // (such a lane has no window to record in)
        const int b = (int)(i & 1);
        const bool d = (dbl_mask[b] >> lane) & 1;
        const long long n0 = a.c0 + i * kTile, stop = end < n0 + kTile ? end : n0 + kTile;
        long long n = n0;  // positions before this step are in the work
        if (a.wout && d && moves != moves0) {  // FP64 from here on
            W = fixed_work();
            moves0 = moves;
            acc_h = 0;
            acc_l = 0;
        }
        const long long move1 = a.wout ? a.nequil_w[0] + 1 : 0;  // the step before which the trap first moves
        auto moves_to = [&](long long to) {                      // the trap's moves before steps [n, to)
            if (n < move1) n = move1;
            for (; n < to; ++n) {
                const long long v = X[b][n - n0][lane];
                moves = n - move1 + 1;
                if (d) {
                    const double lo = lam1 + a.smd_vdt * (double)(moves - 1), hi = lam1 + a.smd_vdt * (double)moves;
                    W += 0.5 * a.k * (hi - lo) * (hi + lo - 2.0 * __longlong_as_double(v));
                    moves0 = moves;
                } else {
                    const long long e = v - L1;
                    acc_h += e >> 32;
                    acc_l += (unsigned)e;
                }
            }
        };
        for (;;) {
            for (const long long seg = wend < stop ? wend : stop; walk.rec < seg; walk.next(a.stride)) {
                const long long v = X[b][walk.rec - n0 + 1][lane];
                a.xout[base + walk.at] = d ? (float)__longlong_as_double(v) : (float)v * (float)unit;
                if (a.wout) {
                    moves_to(walk.rec + 1);
                    a.wout[base + walk.at] = d ? W : fixed_work();
                }
            }
            if (!a.sequential || wend >= stop) break;
            enter_window(ww + 1, wend);
        }
        if (a.wout) moves_to(stop);
    };

    load_tile(0, warp, kOd1dThreads / 32);
    __syncthreads();
    for (long long i = 0; i <= tiles; ++i) {
        if (warp == 0) {
            if (i < tiles) integrate(i);
        } else {
            if (i + 1 < tiles) load_tile(i + 1, warp - 1, kOd1dThreads / 32 - 1);
            if (i > 0) records(i - 1);
        }
        __syncthreads();
    }
    if (!live || end <= a.c0) return;
    if (warp == 0) {
        if (!dbl) x = (double)Xi * unit;
        if (!isfinite(x)) atomicOr(a.err, kErrNonFinite);
        a.state[2 * rep] = x;
        if (!a.wout) a.state[2 * rep + 1] = 0.0;
    } else if (warp == 1 && a.wout) {
        a.state[2 * rep + 1] = moves != moves0 ? fixed_work() : W;
    }
}

long long od1d_noise_steps(int n_rep)
{
    // at most 2^23 normals (64 MB) per launch, between 64 and 8192 steps
    long long c = (1LL << 23) / (n_rep > 0 ? n_rep : 1);
    c = c < 64 ? 64 : (c > 8192 ? 8192 : c);
    return c & ~3LL;
}

cudaError_t od1d_launch(const Od1dParams &m, const RunLaunch &L, int n_rep, cudaStream_t st)
{
    if (L.noise == nullptr || L.noise_steps < 4 || (L.noise_steps & 3) != 0 || (L.step_begin & 3) != 0)
        return cudaErrorInvalidValue;
    if (L.sequential && L.window_steps < 1) return cudaErrorInvalidValue;
    Od1dArgs a{};
    a.x0 = m.x0;
    a.k = L.k;
    a.lambda = L.lambda;
    a.nsteps_w = L.nsteps_w;
    a.nequil_w = L.nequil_w;
    a.off_w = L.off_w;
    a.tw = L.tw;
    a.state = reinterpret_cast<double *>(L.state);
    a.start = L.start;
    a.xout = L.xout;
    a.err = L.err;
    a.replicas = L.replicas;
    a.stride = L.stride;
    a.n_rep = n_rep;
    a.uid_base = L.uid_base;
    a.seed = L.seed;
    a.sequential = L.sequential ? 1 : 0;
    a.window_steps = L.window_steps;
    a.wout = L.wout;
    a.smd_vdt = L.smd_vdt;
    a.noise = reinterpret_cast<long long *>(L.noise);
    // Fixed point where |x| < 2^b holds the traps, the start, the wells and six
    // widths of the trap, and where one step from inside cannot wrap a 64-bit
    // sum (which also bounds every coefficient): FP64 otherwise, for instance
    // for time steps near the scheme's stability limit.  Box-Muller's normals
    // stay below sqrt(66 ln 2) < 6.8.
    const double dtg = L.dt / L.gamma, reach = std::max({L.lambda_max, std::fabs(m.x0), m.a != 0.0 ? 1.0 : 0.0}) + 6.0 * std::sqrt(L.kT / L.k);
    const double cA = std::fabs(4.0 * m.a * dtg), cB1 = std::fabs((4.0 * m.a - L.k) * dtg);
    const double qmax = 6.8 * std::sqrt(2.0 * L.kT * dtg) + L.k * dtg * L.lambda_max;
    if (std::isfinite(reach) && reach > 0 && std::isfinite(cA) && std::isfinite(cB1) && std::isfinite(qmax)) {
        int b = 0;
        std::frexp(reach, &b);  // reach <= 2^b
        if (b >= -30 && b <= 30 && cB1 + std::ldexp(cA, 2 * b) + std::ldexp(qmax, -b) < 0.99) {
            a.fixed = 1;
            a.range_log2 = b;
        }
    }
    a.cA = -4.0 * m.a * dtg;
    a.cB1 = (4.0 * m.a - L.k) * dtg;
    a.q_off = a.fixed ? q_offset256(a.cA, a.cB1) : 0;
    const double scale = a.fixed ? std::ldexp(1.0, 62 - a.range_log2) : 1.0;
    a.amp = std::sqrt(2.0 * L.kT * dtg) * scale;
    a.ck = L.k * dtg * scale;
    for (long long c0 = L.step_begin; c0 < L.step_end; c0 += L.noise_steps) {
        const long long c1 = c0 + L.noise_steps < L.step_end ? c0 + L.noise_steps : L.step_end;
        const long long cells = ((c1 - c0 + 3) >> 2) * n_rep;
        a.c0 = c0;
        a.c1 = c1;
        od1d_noise_kernel<<<(unsigned)((cells + 255) / 256), 256, 0, st>>>(a, a.noise);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        od1d_kernel<<<(n_rep + 31) / 32, kOd1dThreads, 0, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Philox test hook: the same generator and FP32 Box-Muller as the integrator.
__global__ void philox_kernel(unsigned long long seed, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, int n,
                              uint32_t *raw, float *normals)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Ctr4 b = philox4x32_10(Ctr4{c0 + (uint32_t)i, c1, c2, c3}, (uint32_t)seed, (uint32_t)(seed >> 32));
    if (raw) {
        raw[4 * i + 0] = b.a;
        raw[4 * i + 1] = b.b;
        raw[4 * i + 2] = b.c;
        raw[4 * i + 3] = b.d;
    }
    if (normals) {
        const Normal4<float> z = box_muller(b, 0.0f);
        normals[4 * i + 0] = z.n0;
        normals[4 * i + 1] = z.n1;
        normals[4 * i + 2] = z.n2;
        normals[4 * i + 3] = z.n3;
    }
}

cudaError_t philox_launch(unsigned long long seed, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, int n,
                          uint32_t *raw, float *normals, cudaStream_t st)
{
    philox_kernel<<<(n + 255) / 256, 256, 0, st>>>(seed, c0, c1, c2, c3, n, raw, normals);
    return cudaGetLastError();
}

}  // namespace pmf
