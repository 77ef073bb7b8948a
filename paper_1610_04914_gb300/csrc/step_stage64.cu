// FP64 step of the chain tableaus (RK4, RK2 midpoint, Heun): one kernel per
// Runge-Kutta stage, one thread per site.
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
// one pulse, observables) 2.09 -> 0.25 ms.
//
// The accumulator of the tableau is not kept: with K_j = dt f(X_j) and
// X_{j+1} = s + a_{j+1,j} K_j, every K_j but the last is (X_{j+1} - s)/a_{j+1,j},
// so the last stage forms
//   y = g_0 s + sum_{j=2..S} g_j X_j + b_S K_S,  g_j = b_{j-1}/a_{j,j-1},
//   g_0 = 1 - sum_j g_j
// from the stage inputs (own site only), then renormalises and, on pulse
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
    double J, twoD, H[3], lambda;
    double c;              // dt a_{j+1,j}; last stage: dt b_S
    double g0, gx, gq[2];  // last stage: weights of s, X_S, X_2, X_3
    int bc, renorm;
    uint64_t seed, replica;
    double sigma;
    const long long* interval;
};

enum StageRole { kFirst, kMiddle, kLast2, kLast4 };

template <int ROLE, bool PREC, bool HSITE, bool PULSE>
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
        const double l = fx0 ? 0.0 : q[xm], r = fx1 ? 0.0 : q[xp];
        const double u = fy0 ? 0.0 : q[ym], d = fy1 ? 0.0 : q[yp];
        const double b = fz0 ? 0.0 : q[zm], t = fz1 ? 0.0 : q[zp];
        s[c] = ROLE == kFirst ? v[c] : a.s[c][i];
        h[c] = a.J * (((l + r) + (u + d)) + (b + t)) + a.H[c];
        if (HSITE) h[c] += a.hs[c][i];
    }
    h[2] += a.twoD * v[2];
    double f[3];
    llg_rhs<double, PREC>(v[0], v[1], v[2], h[0], h[1], h[2], a.lambda, f[0], f[1], f[2]);
    double o[3];
    if (ROLE == kFirst || ROLE == kMiddle) {
#pragma unroll
        for (int c = 0; c < 3; ++c) o[c] = s[c] + a.c * f[c];
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double acc = a.g0 * s[c];
            if (ROLE == kLast4) {
                acc += a.gq[0] * a.q[0][c][i];
                acc += a.gq[1] * a.q[1][c][i];
            }
            acc += a.gx * v[c];
            o[c] = acc + a.c * f[c];
        }
        if (a.renorm) {
            const double inv = rsqrt(o[0] * o[0] + o[1] * o[1] + o[2] * o[2]);
#pragma unroll
            for (int c = 0; c < 3; ++c) o[c] *= inv;
        }
        if (PULSE)
            pulse_site<double>(o[0], o[1], o[2], a.seed, (uint64_t)i, (uint64_t)*a.interval, a.replica, a.sigma);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) a.out[c][i] = o[c];
}

template <int ROLE, bool PREC, bool HSITE, bool PULSE>
cudaError_t stage_launch(const Stage64Args& a, cudaStream_t st) {
    // small lattices are spread over the SMs one warp per block
    const int threads = a.N <= 152 * 4 * 32 ? 32 : 128;
    return launch_pdl(k_stage64<ROLE, PREC, HSITE, PULSE>, dim3((unsigned)((a.N + threads - 1) / threads)), dim3(threads),
                      0, st, a);
}

template <int ROLE, bool PULSE>
cudaError_t stage_dispatch(const Stage64Args& a, cudaStream_t st, bool prec, bool hs) {
    if (prec) return hs ? stage_launch<ROLE, true, true, PULSE>(a, st) : stage_launch<ROLE, true, false, PULSE>(a, st);
    return hs ? stage_launch<ROLE, false, true, PULSE>(a, st) : stage_launch<ROLE, false, false, PULSE>(a, st);
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
    a.J = L.ph.J;
    a.twoD = L.ph.twoD;
    a.lambda = L.ph.lambda;
    a.bc = L.bc;
    a.renorm = L.renorm;
    a.seed = L.seed;
    a.replica = L.replica;
    a.sigma = L.sigma;
    a.interval = L.d_interval;
    for (int c = 0; c < 3; ++c) {
        a.H[c] = L.ph.H[c];
        a.hs[c] = L.hs[c];
        a.s[c] = L.in[c];
    }
    const bool prec = L.precession != 0, hs = L.hs[0] != nullptr;
    // weights of the stage inputs X_2 .. X_S in the result
    double g[5] = {}, g0 = 1.0;
    for (int j = 2; j <= S; ++j) {
        g[j] = tb.b[j - 2] / tb.a[j - 1][j - 2];
        g0 -= g[j];
    }
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
            a.c = tb.a[j][j - 1] * L.dt;
            e = j == 1 ? stage_dispatch<kFirst, false>(a, L.stream, prec, hs)
                       : stage_dispatch<kMiddle, false>(a, L.stream, prec, hs);
        } else {
            a.c = tb.b[S - 1] * L.dt;
            a.g0 = g0;
            a.gx = g[S];
            if (S == 4) {
                a.gq[0] = g[2];
                a.gq[1] = g[3];
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
