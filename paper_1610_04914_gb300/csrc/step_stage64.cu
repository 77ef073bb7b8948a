// FP64 step of the chain tableaus (RK4, RK2 midpoint, Heun): one kernel per
// Runge-Kutta stage, one thread per site (four lanes on the smallest lattices).
//
// What bounds it: GB300's FP64 pipe, about two lanes per SM and cycle, so a
// warp's FP64 instruction takes as long as some sixty other instructions and
// everything else (index arithmetic, neighbour loads from L1/L2, the stage
// arrays' DRAM traffic) hides behind it.  A halo, which recomputes stages at
// sites that another block owns, is then the worst trade: the z-marching tile
// with a halo of four that this path replaced computed 16 x 16 columns for
// 8 x 8 outputs, four times the FP64 work.  Here every stage of every site is
// computed exactly once, and the stage inputs X_j go through memory.  RK4,
// one interval: 128^3 (4 steps, one pulse) 16.08 -> 3.60 ms, 16^3 (10 steps,
// one pulse, observables) 2.09 -> 0.25 ms; with the sums below off the FP64
// pipe and the cheaper noise draw 1.97 and 0.23 ms, with the products
// folded into the update and a short reciprocal root 1.86 ms; the pipe is then
// 85% active at 128^3.  16^3 with four lanes per site: 0.175 ms.
//
// The accumulator of the tableau is not kept: with K_j = dt f(X_j) and
// X_{j+1} = s + a_{j+1,j} K_j, every K_j but the last is (X_{j+1} - s)/a_{j+1,j},
// so the last stage forms
//   y = s + sum_{j=2..S} g_j (X_j - s) + b_S K_S,  g_j = b_{j-1}/a_{j,j-1},
// from the stage inputs (own site only; RK4: (X_2 + 2 X_3 + X_4 - s)/3 + K_4/6), then renormalises and, on pulse
// steps, rotates.  For S = 4, X_2 lives in the step's output array (the last
// stage reads it at its own site before it writes there), X_3 and X_4 in
// scratch (6N doubles); for S = 2, X_2 in scratch (3N).
#include <cuda_runtime.h>

#include "pdl.cuh"
#include "spin_device.cuh"
#include "spin_internal.h"

namespace spin {

namespace {

struct Stage64Args {
    const double* x[3];    // stage input X_j (with neighbours)
    const double* s[3];    // state before the step (own site)
    const double* q[2][3]; // last stage of S = 4: X_2, X_3 (own site)
    const double* hs[3];
    double* out[3];        // X_{j+1}, or the new state
    int nx, ny, nz, N;
    // J, 2D, H and the factor of h_i times c = dt a_{j+1,j} (last stage: dt b_S,
    // of S = 4 thrice that), slow equation: times -c lambda
    double J, twoD, H[3], hc, lambda;
    double unscale;        // last stage without renormalisation: factor of the result
    double g0, gx;         // last stage of S = 2: weights of s and X_2
    int bc, renorm;
    int pdl;   // host: launch as a programmatic dependent
    uint64_t seed, replica;
    double sigma;
    const long long* interval;
};

// Fixed-point sums of doubles without the FP64 pipe: the mantissas, shifted to
// the largest exponent of the terms, add as 64-bit integers and the sum is rounded
// once to nearest.  A term loses what lies below 2^-59 of the largest one's power of
// two, 64 times less than the first rounding of the additions in a row may cost;
// only where the terms cancel to below that do the additions keep more ({1, -1,
// 2^-70} gives 0 here).  Those are 5 of a component's 12 FP64 instructions per
// stage, and the integer pipes are idle.  Magnitudes below 2^-923 count as zero; where a term is above
// 2^977, infinite or NaN (emax > kMaxExp) the caller takes the plain sum.
constexpr unsigned kMinExp = 100u, kMaxExp = 2000u;
__device__ __forceinline__ unsigned exponent(double v) { return ((unsigned)__double2hiint(v) >> 20) & 0x7FFu; }
// v in units of 2^(emax - 1082): 53 bits at bits 7 .. 59, shifted right
__device__ __forceinline__ long long fixed(double v, unsigned emax) {
    const unsigned h = (unsigned)__double2hiint(v);
    const unsigned long long m = (((unsigned long long)((h & 0xFFFFFu) | 0x100000u) << 32) |
                                  (unsigned)__double2loint(v)) << 7;
    const long long x = (long long)(m >> min(emax - ((h >> 20) & 0x7FFu), 63u));
    const long long sg = (long long)((int)h >> 31);
    return (x ^ sg) - sg;
}
// Kept out of line: inlined, the compiler would execute it for every site.
__device__ __noinline__ double plain_sum6(double a, double b, double c, double d, double e, double f) {
    return ((a + b) + (c + d)) + (e + f);
}
__device__ __forceinline__ double sum6(const double (&q)[6]) {
    unsigned emax = kMinExp;
#pragma unroll
    for (int k = 0; k < 6; ++k) emax = max(emax, exponent(q[k]));
    if (emax > kMaxExp) return plain_sum6(q[0], q[1], q[2], q[3], q[4], q[5]);
    long long S = 0;   // six terms below 2^60 each
#pragma unroll
    for (int k = 0; k < 6; ++k) S += fixed(q[k], emax);
    return from_fixed(S, emax);
}
// x2 + 2 x3 + x4 - s: the part of the RK4 result that its stage inputs hold,
// times three
__device__ __noinline__ double plain_rk4_sum(double x2, double x3, double x4, double s) {
    return (x2 + 2.0 * x3) + (x4 - s);
}
__device__ __forceinline__ double rk4_sum(double x2, double x3, double x4, double s) {
    const unsigned emax = max(max(exponent(x2), exponent(x3)), max(max(exponent(x4), exponent(s)), kMinExp));
    if (emax > kMaxExp) return plain_rk4_sum(x2, x3, x4, s);
    return from_fixed(fixed(x2, emax) + 2 * fixed(x3, emax) + fixed(x4, emax) - fixed(s, emax), emax);
}

enum StageRole { kFirst, kMiddle, kLast2, kLast4 };

// With h = c H_eff (c folded into the constants), c f = v x (h - lambda v x h),
// c f = v x (v x h) for the slow equation, and the second product is added to
// the state by its own multiply-adds: 15 FP64 instructions after the field, 18
// when the two products, their sum and the update are taken one by one.

// WIDE: neighbour sums through the integer pipes, for lattices that fill the FP64
// pipe (up to one warp per scheduler, 19456 sites, latencies count instead, of which
// the integer form has more: RK4 us per step, plain / integer sums, 23^3 15.8 / 16.0,
// 24^3 15.3 / 15.8, 26^3 16.3 / 16.2, 27x27x26 16.2 / 16.4).
template <int ROLE, bool PREC, bool HSITE, bool PULSE, bool WIDE>
__global__ void __launch_bounds__(128) k_stage64(const __grid_constant__ Stage64Args a) {
    pdl_go();
    const unsigned iu = blockIdx.x * blockDim.x + threadIdx.x;   // N < 2^31, the last block may pass it
    if (iu >= (unsigned)a.N) return;
    const int i = (int)iu;
    const int row = i / a.nx, x = i - row * a.nx;
    const int z = row / a.ny, y = row - z * a.ny;
    const int P = a.nx * a.ny;
    const int xm = x > 0 ? i - 1 : i + (a.nx - 1), xp = x < a.nx - 1 ? i + 1 : i - (a.nx - 1);
    const int ym = y > 0 ? i - a.nx : i + (a.ny - 1) * a.nx, yp = y < a.ny - 1 ? i + a.nx : i - (a.ny - 1) * a.nx;
    const int zm = z > 0 ? i - P : i + (a.nz - 1) * P, zp = z < a.nz - 1 ? i + P : i - (a.nz - 1) * P;
    // free boundaries: a neighbour across a face is a zero spin
    const bool fx0 = a.bc && x == 0, fx1 = a.bc && x == a.nx - 1;
    const bool fy0 = a.bc && y == 0, fy1 = a.bc && y == a.ny - 1;
    const bool fz0 = a.bc && z == 0, fz1 = a.bc && z == a.nz - 1;
    pdl_wait();
    double h[3], v[3], s[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double* q = a.x[c];
        v[c] = q[i];
        const double nb[6] = {fx0 ? 0.0 : q[xm], fx1 ? 0.0 : q[xp], fy0 ? 0.0 : q[ym],
                              fy1 ? 0.0 : q[yp], fz0 ? 0.0 : q[zm], fz1 ? 0.0 : q[zp]};
        s[c] = ROLE == kFirst ? v[c] : a.s[c][i];
        const double sum = WIDE ? sum6(nb) : ((nb[0] + nb[1]) + (nb[2] + nb[3])) + (nb[4] + nb[5]);
        h[c] = fma(a.J, sum, a.H[c]);
        if (HSITE) h[c] = fma(a.hc, a.hs[c][i], h[c]);
    }
    h[2] = fma(a.twoD, v[2], h[2]);
    double g[3] = {v[1] * h[2] - v[2] * h[1], v[2] * h[0] - v[0] * h[2], v[0] * h[1] - v[1] * h[0]};
    if (PREC) {
#pragma unroll
        for (int c = 0; c < 3; ++c) g[c] = fma(-a.lambda, g[c], h[c]);
    }
    double o[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double base = s[c];
        if (ROLE == kLast4) {   // three times the result
            const double x2 = a.q[0][c][i], x3 = a.q[1][c][i];
            base = rk4_sum(x2, x3, v[c], s[c]);
        } else if (ROLE == kLast2) {
            base = a.g0 * s[c] + a.gx * v[c];
        }
        const int d = (c + 1) % 3, e = (c + 2) % 3;
        o[c] = fma(v[d], g[e], fma(-v[e], g[d], base));
    }
    if (ROLE == kLast2 || ROLE == kLast4) {
        const double inv = a.renorm ? inv_root(o[0] * o[0] + o[1] * o[1] + o[2] * o[2]) : a.unscale;
#pragma unroll
        for (int c = 0; c < 3; ++c) o[c] *= inv;
        if (PULSE)
            pulse_site<double>(o[0], o[1], o[2], a.seed, (uint64_t)i, (uint64_t)*a.interval, a.replica, a.sigma);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) a.out[c][i] = o[c];
}

// The smallest lattices: four lanes per site, one component each (the fourth
// repeats the third).  A warp's FP64 instruction takes 64 cycles of its
// scheduler whatever its active lanes, and with a warp or two per scheduler a
// stage lasts as long as the FP64 instructions of one warp, 34 with plain sums;
// split by component a lane executes 12 (the pulse: half).  The other components' spins,
// fields and cross products come by shuffles, the arithmetic is that of
// k_stage64.  What is left is the launch and the loads: 2.5 us per stage.  Ten
// RK4 steps with a pulse and one launch graph, one thread per site against four
// lanes: 8^3 146 and 99 us, 16^3 150 and 107, 21^3 156 and 135, 22^3 162 and
// 137, 24^3 156 and 166; two stages: 21^3 88 and 80, 24^3 87 and 98.
constexpr int kLaneSites = 152 * 72;
__device__ __forceinline__ double lane_get(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }

template <int ROLE, bool PREC, bool HSITE, bool PULSE>
__global__ void __launch_bounds__(32) k_stage64_lanes(const __grid_constant__ Stage64Args a) {
    pdl_go();
    const int lane = (int)(threadIdx.x & 31), first = lane & ~3, c = min(lane & 3, 2);
    const int l1 = first + (c + 1) % 3, l2 = first + (c + 2) % 3;   // lanes of the next two components
    const int iu = (int)(blockIdx.x * 8 + (threadIdx.x >> 2));
    const bool mine = iu < a.N && (lane & 3) < 3;
    const int i = min(iu, a.N - 1);
    const int row = i / a.nx, x = i - row * a.nx;
    const int z = row / a.ny, y = row - z * a.ny;
    const int P = a.nx * a.ny;
    const int nb[6] = {x > 0 ? i - 1 : i + (a.nx - 1), x < a.nx - 1 ? i + 1 : i - (a.nx - 1),
                       y > 0 ? i - a.nx : i + (P - a.nx), y < a.ny - 1 ? i + a.nx : i - (P - a.nx),
                       z > 0 ? i - P : i + (a.nz - 1) * P, z < a.nz - 1 ? i + P : i - (a.nz - 1) * P};
    const bool cut[6] = {a.bc && x == 0, a.bc && x == a.nx - 1, a.bc && y == 0,
                         a.bc && y == a.ny - 1, a.bc && z == 0, a.bc && z == a.nz - 1};
    auto pick = [c](const auto& p) { return c == 0 ? p[0] : c == 1 ? p[1] : p[2]; };
    const double* q = pick(a.x);
    const double* sp = pick(a.s);
    const double Hc = pick(a.H);
    pdl_wait();
    double n[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) n[k] = cut[k] ? 0.0 : q[nb[k]];
    const double v = q[i], s = ROLE == kFirst ? v : sp[i];
    double x2 = 0, x3 = 0;
    if (ROLE == kLast4) {
        x2 = pick(a.q[0])[i];
        x3 = pick(a.q[1])[i];
    }
    const double hs = HSITE ? pick(a.hs)[i] : 0.0;
    double p = 0;
    if (PULSE) {
        // drawn while the loads above are in flight; components 0 and 1 of G
        // share a radius and an angle, 2 has its own
        const Words4 w = noise_words(a.seed, (uint64_t)i, (uint64_t)*a.interval, a.replica);
        const double r = Gauss<double>::root(Gauss<double>::neg2log(Gauss<double>::u01(c == 2 ? w.w[2] : w.w[0])));
        double cs, sn;
        Gauss<double>::angle(c == 2 ? w.w[3] : w.w[1], cs, sn);
        p = a.sigma * (r * (c == 1 ? sn : cs));
    }
    double h = fma(a.J, ((n[0] + n[1]) + (n[2] + n[3])) + (n[4] + n[5]), Hc);
    if (HSITE) h = fma(a.hc, hs, h);
    h = fma(a.twoD, c == 2 ? v : 0.0, h);
    const double v1 = lane_get(v, l1), v2 = lane_get(v, l2);
    double g = v1 * lane_get(h, l2) - v2 * lane_get(h, l1);
    if (PREC) g = fma(-a.lambda, g, h);
    double base = s;
    if (ROLE == kLast4) base = rk4_sum(x2, x3, v, s);
    if (ROLE == kLast2) base = a.g0 * s + a.gx * v;
    double o = fma(v1, lane_get(g, l2), fma(-v2, lane_get(g, l1), base));
    if (ROLE == kLast2 || ROLE == kLast4) {
        const double sq = o * o;
        const double n2 = (lane_get(sq, first) + lane_get(sq, first + 1)) + lane_get(sq, first + 2);
        o *= a.renorm ? inv_root(n2) : a.unscale;
        if (PULSE) {
            double s0 = lane_get(o, first), s1 = lane_get(o, first + 1), s2 = lane_get(o, first + 2);
            pulse_rotate<double>(s0, s1, s2, lane_get(p, first), lane_get(p, first + 1), lane_get(p, first + 2), a.sigma);
            o = c == 0 ? s0 : c == 1 ? s1 : s2;
        }
    }
    if (mine) pick(a.out)[i] = o;
}

template <int ROLE, bool PREC, bool HSITE, bool PULSE>
cudaError_t stage_launch(const Stage64Args& a, cudaStream_t st) {
    if (a.N <= kLaneSites)
        return launch_pdl(a.pdl != 0, k_stage64_lanes<ROLE, PREC, HSITE, PULSE>, dim3((unsigned)((a.N + 7) / 8)), dim3(32), 0,
                          st, a);
    // up to one warp per scheduler: one warp per block, spread over the SMs
    const bool wide = a.N > 152 * 4 * 32;
    const dim3 block(wide ? 128 : 32), grid((unsigned)(((unsigned)a.N + block.x - 1) / block.x));
    return wide ? launch_pdl(a.pdl != 0, k_stage64<ROLE, PREC, HSITE, PULSE, true>, grid, block, 0, st, a)
                : launch_pdl(a.pdl != 0, k_stage64<ROLE, PREC, HSITE, PULSE, false>, grid, block, 0, st, a);
}

template <int ROLE, bool PULSE>
cudaError_t stage_dispatch(const Stage64Args& a, cudaStream_t st, bool prec, bool hs) {
    if (prec) return hs ? stage_launch<ROLE, true, true, PULSE>(a, st) : stage_launch<ROLE, true, false, PULSE>(a, st);
    return hs ? stage_launch<ROLE, false, true, PULSE>(a, st) : stage_launch<ROLE, false, false, PULSE>(a, st);
}

// The four-stage tableau whose result the last stage forms with fixed weights.
bool rk4_weights(const Tableau& tb) {
    const double third[3] = {tb.b[0] / tb.a[1][0], tb.b[1] / tb.a[2][1] / 2.0, tb.b[2] / tb.a[3][2]};
    for (double g : third)
        if (!(g > 1.0 / 3.0 - 1e-15 && g < 1.0 / 3.0 + 1e-15)) return false;
    return true;
}

}  // namespace

// scratch doubles (in units of N) the step needs
int stage64_scratch(int stages) { return stages == 4 ? 6 : 3; }

cudaError_t launch_step_stage64(const StepLaunch<double>& L) {
    const Tableau& tb = *L.tab;
    const int S = tb.stages;
    const size_t N = (size_t)L.g.N();
    Stage64Args a{};
    a.nx = L.g.nx;
    a.ny = L.g.ny;
    a.nz = L.g.nz;
    a.N = (int)N;
    a.lambda = L.ph.lambda;
    a.bc = L.bc;
    a.renorm = L.renorm;
    a.pdl = L.into == kStream;
    a.seed = L.seed;
    a.replica = L.replica;
    a.sigma = L.sigma;
    a.interval = L.d_interval;
    for (int c = 0; c < 3; ++c) {
        a.hs[c] = L.hs[c];
        a.s[c] = L.in[c];
    }
    const bool prec = L.precession != 0, hs = L.hs[0] != nullptr;
    auto scale = [&](double c) {
        const double k = prec ? c : -c * L.ph.lambda;
        a.J = k * L.ph.J;
        a.twoD = k * L.ph.twoD;
        for (int q = 0; q < 3; ++q) a.H[q] = k * L.ph.H[q];
        a.hc = k;
    };
    if (S == 4 && !rk4_weights(tb)) return cudaErrorInvalidValue;
    // stage 1 .. S-1 write X_2 .. X_S, of S = 4 the first into the output array
    auto scratch = [&](int q, int c) { return L.tmp + ((size_t)q * 3 + c) * N; };
    const double* prev[3] = {L.in[0], L.in[1], L.in[2]};
    for (int j = 1; j <= S; ++j) {
        for (int c = 0; c < 3; ++c) {
            a.x[c] = prev[c];
            a.out[c] = (j == S || (j == 1 && S == 4)) ? L.out[c] : scratch(S == 4 ? j - 2 : 0, c);
        }
        cudaError_t e;
        if (j < S) {
            scale(tb.a[j][j - 1] * L.dt);
            e = j == 1 ? stage_dispatch<kFirst, false>(a, L.stream, prec, hs)
                       : stage_dispatch<kMiddle, false>(a, L.stream, prec, hs);
        } else {
            scale((S == 4 ? 3.0 : 1.0) * tb.b[S - 1] * L.dt);
            a.unscale = S == 4 ? 1.0 / 3.0 : 1.0;
            a.gx = tb.b[0] / tb.a[1][0];
            a.g0 = 1.0 - a.gx;
            if (S == 4) {
                for (int c = 0; c < 3; ++c) {
                    a.q[0][c] = L.out[c];
                    a.q[1][c] = scratch(0, c);
                }
                e = L.pulse ? stage_dispatch<kLast4, true>(a, L.stream, prec, hs)
                            : stage_dispatch<kLast4, false>(a, L.stream, prec, hs);
            } else {
                e = L.pulse ? stage_dispatch<kLast2, true>(a, L.stream, prec, hs)
                            : stage_dispatch<kLast2, false>(a, L.stream, prec, hs);
            }
        }
        if (e != cudaSuccess) return e;
        for (int c = 0; c < 3; ++c) prev[c] = a.out[c];
    }
    return cudaSuccess;
}

}  // namespace spin
