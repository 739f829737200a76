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
// cycles.  Where a simulation's parameters bound its motion (fixed_range), its
// chain runs in 62-bit fixed point on the integer pipe instead (IMAD.WIDE: 5 cycles):
// X = x 2^S with |x| < 2^b, S = 62 - b, and
//   X' = X + Q + X w,  w = (cB - 1) + cA 4^b (X 2^-62)^2,
// products of 62-bit numbers within a few units of 2^(b-62) (9e-19 for the
// double well's b = 2), 1/128 of the FP64 rounding of a position near 1.  The
// products round down; left alone that drift adds up to 2 1/4 units /
// (k dt/gamma) where no well contracts the map faster (a = 0, k = 1, dt = 1e-3,
// b = 4: 7.5e-15 against FP64's 1.2e-15), so its mean is added to the terms
// that are there anyway, cB - 1 and q_n (the same case: 6e-17).  A simulation that leaves |x| < 2^b
// redoes the tile of steps it left in, and runs on, in FP64, until a tile ends within half the range.
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
    Od1dState *state;           // [n_rep]
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
    long long *noise;           // [c1 - c0][n_rep] q_n of this launch's steps (fixed point: q_n 2^S, else the double's bits)
    RangeRule rule;             // fixed point: range of a window,
    int range;                  //   or of the whole run (sequential, pulled)
    int q_off;                  //   mean of the last product's rounding (q_offset256)
    double cA, cB1;             // -4a dt/gamma, (4a - k) dt/gamma
    double amp, ck;             // sqrt(2 kT dt/gamma), k dt/gamma (set on the host: per thread
                                // they took a sixth of the pre-pass's FP64 operations)
};

// b of simulation rep, or kNoRange.
__device__ __forceinline__ int range_of(const Od1dArgs &a, int rep)
{
    if (a.sequential || a.wout) return a.range;
    const double l = fabs(a.lambda[rep / a.replicas]);
    return fixed_range(a.rule, l, l);
}
// v 2^s for a normal v (and result), or zero left alone, without the FP64 unit
__device__ __forceinline__ double scaled(double v, int s) { return __hiloint2double(__double2hiint(v) + (s << 20), __double2loint(v)); }

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
    const int b = range_of(a, rep), S = b == kNoRange ? 0 : 62 - b;
    const double amp = scaled(a.amp, S), ck = scaled(a.ck, S);
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        const long long n = n0 + l;
        if (n < a.c1) {
            const double qn = fma(amp, v[l], ck * trap_centre(a, rep, n));
            q[(n - a.c0) * a.n_rep + rep] = b != kNoRange ? __double2ll_rn(qn) + q_offset(a.q_off, n) : __double_as_longlong(qn);
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
// 32 x 32 -> 64 multiplies of 9 - 12 cycles and a split), about 130 with the
// tile's barrier; one thread per simulation in FP64 with loads and samples in
// its loop took 403.  21 x 8 simulations x 2e4 steps, whole run with estimates:
// 4.61 -> 1.72 ms; 256 pulled simulations x 4400 steps: 2.24 -> 0.68 ms.
constexpr int kTile = 40;  // 41.5 KB of shared memory a CTA; 32 steps: 2.17 against 1.90 ms
static_assert(kTile % 8 == 0, "unrolled by 8; a Philox block is four steps");
constexpr int kOd1dThreads = 128;

// Two tiles' buffers in shared memory.
struct Od1dTiles {
    long long (&Q)[2][kTile][32];      // q_n
    long long (&X)[2][kTile + 1][32];  // positions before the tile's first step and after each
    unsigned (&dbl_mask)[2];           // lanes whose tile is in FP64 (bits of doubles)
};
// What both roles know of a lane's simulation.
struct Od1dSim {
    int lane, rep, w, range;  // w: its window (0 in the sequential protocol)
    bool live, fixed;
    long long end, tiles;     // its last step (its window's step count), the launch's tiles
    double scale, unit;       // 2^S and 2^-S
};
// All four warps, from either role's loop.  The lanes of a warp, which run loops of
// their own lengths, come together first: the barrier wants whole warps.
__device__ __forceinline__ void tile_barrier()
{
    __syncwarp();
    asm volatile("bar.sync 0, %0;" ::"n"(kOd1dThreads) : "memory");
}
// Rows row, row + STEP, ... of tile i: all loads, then all stores.  A load and its
// store at a time are 14 latencies a helper, longer than the integrating
// warp's 40 steps (21 x 8 x 2e4 steps: 2350 us, now 1712).
template <int STEP>
__device__ __forceinline__ void load_tile(const Od1dArgs &a, const Od1dTiles &sh, const Od1dSim &m, long long i, int row)
{
    constexpr int kRows = (kTile + STEP - 1) / STEP;
    const long long n0 = i * kTile, left = a.c1 - a.c0 - n0;
    const int rows = !m.live ? 0 : (left < kTile ? (int)left : kTile);
    const long long *q = a.noise + (n0 + row) * a.n_rep + m.rep;
    long long v[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u)
        if (row + u * STEP < rows) v[u] = q[(long long)u * STEP * a.n_rep];
#pragma unroll
    for (int u = 0; u < kRows; ++u)
        if (row + u * STEP < rows) sh.Q[i & 1][row + u * STEP][m.lane] = v[u];
}

// Warp 0: the position, in fixed point or (dbl) FP64.
__device__ __forceinline__ void integrate_tiles(const Od1dArgs &a, const Od1dTiles &sh, const Od1dSim &m)
{
    const int lane = m.lane;
    const double cA = a.cA, cB = 1.0 + a.cB1;
    FixedStep f{};
    long long Xi = 0;
    double x = 0.0;
    bool dbl = true;
    if (m.live) {
        x = a.c0 == 0 ? (a.start ? a.start[m.rep] : a.x0) : a.state[m.rep].x;
        if (m.fixed) {
            f = step_of(cA, a.cB1, m.range);
            Xi = a.c0 == 0 ? (fabs(x) < scaled(1.0, m.range) ? __double2ll_rn(x * m.scale) : kNotFixed) : a.state[m.rep].fixed;
            dbl = Xi == kNotFixed;
        }
    }
    for (long long i = 0; i < m.tiles; ++i) {
        const long long n0 = a.c0 + i * kTile;
        const int b = (int)(i & 1);
        const int lim = m.end <= n0 ? 0 : (m.end - n0 < kTile ? (int)(m.end - n0) : kTile);
        const long long X0 = Xi;
        bool redo = dbl && lim > 0, tile_dbl = dbl;
        if (!dbl) {
            sh.X[b][0][lane] = Xi;
            unsigned guard = 0;  // top bit: a position outside [-2^62, 2^62)
            if (__all_sync(__activemask(), lim == kTile)) {
#pragma unroll 8
                for (int s = 0; s < kTile; ++s) {
                    Xi = fixed_step(f, Xi, sh.Q[b][s][lane]);
                    sh.X[b][s + 1][lane] = Xi;
                    guard |= range_guard(Xi);
                }
            } else {
                for (int s = 0; s < lim; ++s) {
                    Xi = fixed_step(f, Xi, sh.Q[b][s][lane]);
                    sh.X[b][s + 1][lane] = Xi;
                    guard |= range_guard(Xi);
                }
            }
            redo = guard >> 31;
        }
        if (redo) {
            if (!dbl) x = (double)X0 * m.unit;
            dbl = tile_dbl = true;
            sh.X[b][0][lane] = __double_as_longlong(x);
#pragma unroll 4
            for (int s = 0; s < lim; ++s) {
                const long long qb = sh.Q[b][s][lane];
                const double q = m.fixed ? (double)(qb - q_offset(a.q_off, n0 + s)) * m.unit : __longlong_as_double(qb);
                x = fma(x, fma(cA, x * x, cB), q);
                sh.X[b][s + 1][lane] = __double_as_longlong(x);
            }
            if (m.fixed && fabs(x) < scaled(0.5, m.range)) {  // well inside again
                Xi = __double2ll_rn(x * m.scale);
                dbl = false;
            }
        }
        __syncwarp();
        const unsigned mask = __ballot_sync(0xffffffffu, tile_dbl);
        if (lane == 0) sh.dbl_mask[b] = mask;
        tile_barrier();
    }
    tile_barrier();  // (the last tile's records)
    if (!m.live || m.end <= a.c0) return;
    if (!dbl) x = (double)Xi * m.unit;
    if (!isfinite(x)) atomicOr(a.err, kErrNonFinite);
    a.state[m.rep].x = x;
    a.state[m.rep].fixed = dbl ? kNotFixed : Xi;
}

// Warps 1 - 3: the next tile's q_n, and the records of the finished one; no
// division in the loop.
__device__ __forceinline__ void record_tiles(const Od1dArgs &a, const Od1dTiles &sh, const Od1dSim &m, int helper)
{
    const int lane = m.lane, r = a.sequential ? m.rep : m.rep % a.replicas;
    const float unit_f = __int_as_float(m.fixed ? (m.range - 62 + 127) << 23 : 0x3f800000);
    int ww = m.w;
    RecordWalk walk;
    long long base = 0, wend = 0;
    auto enter_window = [&](int window, long long from) {
        ww = window;
        const long long origin = a.sequential ? (long long)ww * a.window_steps : 0;
        walk.enter(origin, a.nequil_w[ww], a.stride, from, helper);
        base = a.off_w[ww] + (long long)r * a.tw[ww];
        wend = a.sequential ? origin + a.window_steps : m.end;
    };
    // pulling work: W after the trap's first moves0 moves, and since then the
    // sum of X - lambda_1 in two 32-bit halves (every helper keeps it, each
    // converts for its own records)
    double W = 0.0;
    long long acc_h = 0, moves0 = 0, moves = 0;
    unsigned long long acc_l = 0;
    const double lam1 = a.lambda[0], kv = a.k * a.smd_vdt;
    const long long L1 = m.fixed ? __double2ll_rn(lam1 * m.scale) : 0;
    if (m.live) {
        enter_window(a.sequential ? (int)(a.c0 / a.window_steps) : m.w, a.c0);
        if (a.wout) {
            moves = a.c0 - 1 - a.nequil_w[0];
            moves = moves > 0 ? moves : 0;
            if (a.c0 > 0) {
                const Od1dState &st = a.state[m.rep];
                W = st.work;
                moves0 = st.moves0;
                acc_h = st.acc_h;
                acc_l = st.acc_l;
            }
        }
    }
    // sum over the moves m of k vdt (lambda_1 + vdt (m - 1/2) - x)
    auto fixed_work = [&] {
        const double mm = (double)moves, m0 = (double)moves0;
        const double sum = ((double)acc_h * 4294967296.0 + (double)acc_l) * m.unit;
        return W + kv * (0.5 * a.smd_vdt * (mm * mm - m0 * m0) - sum);
    };
    auto records = [&](long long i) {
        if (!m.live) return;  // (such a lane has no window to record in)
        const int b = (int)(i & 1);
        const bool d = (sh.dbl_mask[b] >> lane) & 1;
        const long long n0 = a.c0 + i * kTile, stop = m.end < n0 + kTile ? m.end : n0 + kTile;
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
                const long long v = sh.X[b][n - n0][lane];
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
                const long long v = sh.X[b][walk.rec - n0 + 1][lane];
                a.xout[base + walk.at] = d ? (float)__longlong_as_double(v) : (float)v * unit_f;
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
    for (long long i = 0; i <= m.tiles; ++i) {
        if (i + 1 < m.tiles) load_tile<kOd1dHelpers>(a, sh, m, i + 1, helper);
        if (i > 0) records(i - 1);
        tile_barrier();
    }
    if (helper == 0 && a.wout && m.live && m.end > a.c0) {
        Od1dState &st = a.state[m.rep];
        st.work = W;
        st.moves0 = moves0;
        st.acc_h = acc_h;
        st.acc_l = acc_l;
    }
}

__global__ void __launch_bounds__(kOd1dThreads) od1d_kernel(const Od1dArgs a)
{
    static_assert(kOd1dHelpers == kOd1dThreads / 32 - 1, "every warp but the first records");
    __shared__ long long Q[2][kTile][32], X[2][kTile + 1][32];
    __shared__ unsigned dbl_mask[2];
    const Od1dTiles sh{Q, X, dbl_mask};
    const int warp = threadIdx.x >> 5;
    Od1dSim m;
    m.lane = threadIdx.x & 31;
    m.rep = blockIdx.x * 32 + m.lane;
    m.live = m.rep < a.n_rep;
    m.w = a.sequential || !m.live ? 0 : m.rep / a.replicas;
    m.end = a.c1;
    if (!a.sequential && m.live) m.end = m.end < a.nsteps_w[m.w] ? m.end : a.nsteps_w[m.w];
    if (!m.live || m.end < a.c0) m.end = a.c0;
    m.tiles = (a.c1 - a.c0 + kTile - 1) / kTile;
    m.range = m.live ? range_of(a, m.rep) : kNoRange;
    m.fixed = m.range != kNoRange;
    m.scale = scaled(1.0, m.fixed ? 62 - m.range : 0);
    m.unit = scaled(1.0, m.fixed ? m.range - 62 : 0);
    load_tile<kOd1dThreads / 32>(a, sh, m, 0, warp);
    tile_barrier();
    if (warp == 0) integrate_tiles(a, sh, m);
    else record_tiles(a, sh, m, warp - 1);
}

long long od1d_noise_steps(int n_rep)
{
    // at most 2^23 normals (64 MB) per launch, between 80 and 8160 steps, whole
    // tiles: a tile begins at the same steps in every launch
    long long c = (1LL << 23) / (n_rep > 0 ? n_rep : 1);
    c = c < 2 * kTile ? 2 * kTile : (c > 8192 ? 8192 : c);
    return c - c % kTile;
}

// The range holds the trap, the start, the wells and six widths of the trap, and
// one step from inside cannot wrap a 64-bit sum (which also bounds every
// coefficient): FP64 otherwise, for instance for time steps near the scheme's
// stability limit.  Box-Muller's normals stay below sqrt(66 ln 2) < 6.8.
RangeRule od1d_range_rule(const Od1dParams &m, double k, double kT, double dt, double gamma)
{
    RangeRule r;
    const double dtg = dt / gamma, amp = std::sqrt(2.0 * kT * dtg), ck = k * dtg;
    r.hold = std::max(std::fabs(m.x0), m.a != 0.0 ? 1.0 : 0.0);
    r.pad = 6.0 * std::sqrt(kT / k);
    r.width = std::sqrt(kT / (k + 4.0 * std::fabs(m.a)));
    // between the trap and the wells, which an inverted potential has not
    r.well = m.a == 0.0 ? INFINITY : (m.a > 0.0 ? 1.0 : 0.0);
    const double cA = std::fabs(4.0 * m.a * dtg), cB1 = std::fabs((4.0 * m.a - k) * dtg);
    if (!std::isnormal(amp) || !std::isnormal(ck)) return r;
    for (int b = -30; b <= 30; ++b)
        if (cB1 + std::ldexp(cA, 2 * b) + 6.8 * std::ldexp(amp, -b) + ck < 0.99) r.fits |= 1ull << (b + 30);
    return r;
}

cudaError_t od1d_launch(const Od1dParams &m, const RunLaunch &L, int n_rep, cudaStream_t st)
{
    if (L.noise == nullptr || L.noise_steps < kTile || L.noise_steps % kTile != 0 || L.step_begin % kTile != 0)
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
    a.state = reinterpret_cast<Od1dState *>(L.state);
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
    const double dtg = L.dt / L.gamma;
    a.cA = -4.0 * m.a * dtg;
    a.cB1 = (4.0 * m.a - L.k) * dtg;
    a.amp = std::sqrt(2.0 * L.kT * dtg);
    a.ck = L.k * dtg;
    a.rule = od1d_range_rule(m, L.k, L.kT, L.dt, L.gamma);
    a.range = fixed_range(a.rule, L.lambda_max, L.lambda_min);
    a.q_off = a.rule.fits ? q_offset256(a.cA, a.cB1) : 0;
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
