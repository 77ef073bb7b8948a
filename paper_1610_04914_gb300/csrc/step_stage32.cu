// FP32 step of the chain tableaus on small lattices: one kernel per Runge-Kutta
// stage, one thread per site.
//
// What bounds a small lattice is latency: the z-marching tile (patch_tile.cuh)
// takes a chain of at least 2S-1 iterations of about a microsecond on the few
// SMs its tiles reach, while a stage kernel is one round of loads from L2, one
// right-hand side and one store on all SMs (45x37x27 with site fields, 10 RK4
// steps with two pulses and three observables: 250 -> 203 us).  The stage inputs and the
// accumulator go through memory (L2); every site is computed once.  The
// arithmetic of a site is the tile's, operation by operation, so the states are
// bitwise the same.
#include <cuda_runtime.h>

#include "pdl.cuh"
#include "spin_internal.h"

namespace spin {

namespace {

struct Stage32Args {
    const float* x[3];   // stage input X_j (with neighbours)
    const float* s[3];   // state before the step (own site)
    const float* hs[3];
    float* y[3];         // accumulator s + sum_l b_l K_l: read for j > 1, written for j < S (STORE: always)
    float* xn[3];        // X_{j+1}; j = S: the new state
    float* sn[3];        // STORE: sum_nn X_j
    int nx, ny, nz, N;
    float J, twoD, H[3], nlambda, c, b;   // c = dt a_{j+1,j}, b = dt b_j
    int bc, renorm;
    int pdl;   // host: launch as a programmatic dependent
};

// FIRST: j = 1 (x is s); LAST: j = S.
template <bool FIRST, bool LAST, bool PREC, bool HSITE, bool STORE>
__global__ void __launch_bounds__(128) k_stage32(const __grid_constant__ Stage32Args a) {
    const unsigned iu = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)iu;
    const int row = i / a.nx, x = i - row * a.nx;
    const int z = row / a.ny, y = row - z * a.ny;
    const int P = a.nx * a.ny;
    const int nb[6] = {x > 0 ? i - 1 : i + (a.nx - 1), x < a.nx - 1 ? i + 1 : i - (a.nx - 1),
                       y > 0 ? i - a.nx : i + (P - a.nx), y < a.ny - 1 ? i + a.nx : i - (P - a.nx),
                       z > 0 ? i - P : i + (a.nz - 1) * P, z < a.nz - 1 ? i + P : i - (a.nz - 1) * P};
    // free boundaries: a neighbour across a face is a zero spin
    const bool cut[6] = {a.bc && x == 0, a.bc && x == a.nx - 1, a.bc && y == 0,
                         a.bc && y == a.ny - 1, a.bc && z == 0, a.bc && z == a.nz - 1};
    pdl_wait();
    pdl_go();
    if (iu >= (unsigned)a.N) return;
    float v[3], s[3], h[3], acc[3], sum[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float* q = a.x[c];
        v[c] = q[i];
        s[c] = FIRST ? v[c] : a.s[c][i];
        acc[c] = FIRST ? v[c] : a.y[c][i];
        float n[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) n[k] = cut[k] ? 0.f : q[nb[k]];
        // ((x-1 + x+1) + (y-1 + y+1)) + z-1, then z+1
        sum[c] = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(n[0], n[1]), __fadd_rn(n[2], n[3])), n[4]), n[5]);
        h[c] = __fmaf_rn(a.J, sum[c], a.H[c]);
        if (HSITE) h[c] = __fadd_rn(h[c], a.hs[c][i]);
    }
    h[2] = __fmaf_rn(a.twoD, v[2], h[2]);
    const float ax = __fmaf_rn(-v[2], h[1], __fmul_rn(v[1], h[2]));
    const float ay = __fmaf_rn(-v[0], h[2], __fmul_rn(v[2], h[0]));
    const float az = __fmaf_rn(-v[1], h[0], __fmul_rn(v[0], h[1]));
    const float bx = __fmaf_rn(-v[2], ay, __fmul_rn(v[1], az));
    const float by = __fmaf_rn(-v[0], az, __fmul_rn(v[2], ax));
    const float bz = __fmaf_rn(-v[1], ax, __fmul_rn(v[0], ay));
    const float f[3] = {PREC ? __fmaf_rn(a.nlambda, bx, ax) : __fmul_rn(a.nlambda, bx),
                        PREC ? __fmaf_rn(a.nlambda, by, ay) : __fmul_rn(a.nlambda, by),
                        PREC ? __fmaf_rn(a.nlambda, bz, az) : __fmul_rn(a.nlambda, bz)};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        acc[c] = __fmaf_rn(a.b, f[c], acc[c]);
        if (STORE) a.sn[c][i] = sum[c];
        if (!LAST || STORE) a.y[c][i] = acc[c];
        if (!LAST) a.xn[c][i] = __fmaf_rn(a.c, f[c], s[c]);
    }
    if (LAST) {
        const float n2 = __fmaf_rn(acc[0], acc[0], __fmaf_rn(acc[1], acc[1], __fmul_rn(acc[2], acc[2])));
        const float inv = rsqrtf(n2);
#pragma unroll
        for (int c = 0; c < 3; ++c) a.xn[c][i] = a.renorm ? __fmul_rn(acc[c], inv) : acc[c];
    }
}

template <bool FIRST, bool LAST, bool STORE>
cudaError_t stage32(const Stage32Args& a, bool prec, bool hs, cudaStream_t st) {
    const int threads = a.N <= 152 * 128 ? 32 : 128;
    const dim3 grid((unsigned)((a.N + threads - 1) / threads)), block(threads);
    if (prec)
        return hs ? launch_pdl(a.pdl != 0, k_stage32<FIRST, LAST, true, true, STORE>, grid, block, 0, st, a)
                  : launch_pdl(a.pdl != 0, k_stage32<FIRST, LAST, true, false, STORE>, grid, block, 0, st, a);
    return hs ? launch_pdl(a.pdl != 0, k_stage32<FIRST, LAST, false, true, STORE>, grid, block, 0, st, a)
              : launch_pdl(a.pdl != 0, k_stage32<FIRST, LAST, false, false, STORE>, grid, block, 0, st, a);
}

template <bool STORE>
cudaError_t run_stages(const StepLaunch<float>& L) {
    const Tableau& tb = *L.tab;
    const int S = tb.stages;
    const size_t N = (size_t)L.g.N();
    Stage32Args a{};
    a.nx = L.g.nx;
    a.ny = L.g.ny;
    a.nz = L.g.nz;
    a.N = (int)N;
    a.J = L.ph.J;
    a.twoD = L.ph.twoD;
    a.nlambda = -L.ph.lambda;
    a.bc = L.bc;
    a.renorm = L.renorm;
    a.pdl = L.into == kStream;
    for (int c = 0; c < 3; ++c) {
        a.H[c] = L.ph.H[c];
        a.hs[c] = L.hs[c];
        a.s[c] = L.in[c];
        a.x[c] = L.in[c];
        // the accumulator lives in the output arrays until the last stage
        a.y[c] = STORE ? L.st_y[c] : L.out[c];
    }
    const bool prec = L.precession != 0, hs = L.hs[0] != nullptr;
    for (int j = 1; j <= S; ++j) {
        for (int c = 0; c < 3; ++c) {
            // X_2, X_3, X_4: scratch arrays 0, 1, 0
            a.xn[c] = j == S ? L.out[c] : STORE ? L.st_x[j - 1][c] : L.tmp + ((size_t)((j - 1) & 1) * 3 + c) * N;
            a.sn[c] = STORE ? L.st_n[j - 1][c] : nullptr;
        }
        a.c = j < S ? (float)(tb.a[j][j - 1] * L.dt) : 0.f;
        a.b = (float)(tb.b[j - 1] * L.dt);
        const cudaError_t e = j == 1   ? stage32<true, false, STORE>(a, prec, hs, L.stream)
                              : j == S ? stage32<false, true, STORE>(a, prec, hs, L.stream)
                                       : stage32<false, false, STORE>(a, prec, hs, L.stream);
        if (e != cudaSuccess) return e;
        for (int c = 0; c < 3; ++c) a.x[c] = a.xn[c];
    }
    return cudaSuccess;
}

}  // namespace

// Lattices that take the stage kernels.  In interval graphs, us per step, tile /
// stages: RK4 16^3 10.6 / 7.2, 32^3 10.3 / 7.7, 45x37x27 12.0 / 8.6, 48^3 10.7 /
// 10.3, 56^3 11.8 / 12.7; with site fields 56^3 14.3 / 13.1, 64^3 15.2 / 15.9;
// RK2 16^3 7.3 / 3.7, 48^3 8.1 / 5.2, 64^3 7.8 / 7.6, 72^3 9.4 / 9.7; with site
// fields 72^3 10.8 / 10.3, 80^3 10.7 / 12.7.  With the stage store, whose arrays
// both forms write, per backward pass of 20 steps: RK4 32^3 663 / 525, 64^3 1235
// / 1184, 96^3 3668 / 3655, 112^3 5994 / 6134.
bool stage32_small(const Geom& g, int stages, bool field, bool store) {
    const long long side = store ? 96 : stages == 4 ? (field ? 56 : 48) : (field ? 72 : 64);
    return g.N() <= side * side * side;
}
int stage32_scratch(int stages) { return stages == 2 ? 3 : 6; }

cudaError_t launch_step_stage32(const StepLaunch<float>& L) {
    return L.st_n[0][0] ? run_stages<true>(L) : run_stages<false>(L);
}

}  // namespace spin
