// One integration step delta t of the noiseless Landau-Lifshitz equation,
// Eq. (LLL), on the simple-cubic lattice, followed by renormalisation and, on
// pulse steps, the noise rotation of Eq. (s_rotation).  The paths:
//  * chain tableaus (RK4, RK2 midpoint, Heun: stage j needs only K_{j-1}) in
//    FP32: one fused kernel per step, all stages on chip (patch_tile.cuh); on
//    small lattices one kernel per stage (step_stage32.cu);
//  * chain tableaus in FP64: one kernel per stage (step_stage64.cu);
//  * Butcher RK5 in FP32 without a per-site field: two fused three-stage
//    segments (step_rk5.cu);
//  * any tableau, any precision: one stencil kernel per stage plus a combine
//    kernel, stage states in the workspace (below).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "spin_device.cuh"
#include "spin_internal.h"

namespace spin {

Tableau tableau_for(int integrator) {
    Tableau t{};
    switch (integrator) {
        case 0:  // classical RK4
            t.stages = 4;
            t.a[1][0] = 0.5;
            t.a[2][1] = 0.5;
            t.a[3][2] = 1.0;
            t.b[0] = 1.0 / 6.0;
            t.b[1] = 2.0 / 6.0;
            t.b[2] = 2.0 / 6.0;
            t.b[3] = 1.0 / 6.0;
            t.chain = true;
            break;
        case 1:  // Butcher's RK5 as listed in the paper's Appendix
            t.stages = 6;
            t.a[1][0] = 0.25;
            t.a[2][0] = 0.125;
            t.a[2][1] = 0.125;
            t.a[3][1] = -0.5;
            t.a[3][2] = 1.0;
            t.a[4][0] = 3.0 / 16.0;
            t.a[4][3] = 9.0 / 16.0;
            t.a[5][0] = -3.0 / 7.0;
            t.a[5][1] = 2.0 / 7.0;
            t.a[5][2] = 12.0 / 7.0;
            t.a[5][3] = -12.0 / 7.0;
            t.a[5][4] = 8.0 / 7.0;
            t.b[0] = 7.0 / 90.0;
            t.b[2] = 32.0 / 90.0;
            t.b[3] = 12.0 / 90.0;
            t.b[4] = 32.0 / 90.0;
            t.b[5] = 7.0 / 90.0;
            t.chain = false;
            break;
        case 2:  // RK2 midpoint
            t.stages = 2;
            t.a[1][0] = 0.5;
            t.b[1] = 1.0;
            t.chain = true;
            break;
        default:  // Heun
            t.stages = 2;
            t.a[1][0] = 1.0;
            t.b[0] = 0.5;
            t.b[1] = 0.5;
            t.chain = true;
            break;
    }
    return t;
}

template <typename real>
cudaError_t prepare_step_kernels() {
    if (sizeof(real) != 4) return cudaSuccess;   // the FP64 kernels use no dynamic shared memory
    const cudaError_t e = prepare_patch_kernels();
    return e == cudaSuccess ? prepare_rk5_kernels() : e;
}
template cudaError_t prepare_step_kernels<float>();
template cudaError_t prepare_step_kernels<double>();

// ---------------------------------------------------------------------------
// Generic tableau: stencil-per-stage kernels
// ---------------------------------------------------------------------------

template <typename real>
struct Vec3P {
    const real* p[3];
};

// K = dt f(x) over the lattice; neighbours read from global memory.  Blocks
// of kGX threads along x on a (x tile, row) grid: one integer division per row
// (y, z), none per site; periodic neighbours wrap by comparison.
constexpr int kGX = 128;

template <typename real, bool PREC, bool HSITE>
__global__ void __launch_bounds__(kGX) k_stage_rhs(Vec3P<real> x, Vec3P<real> hs, real* __restrict__ K0,
                                                   real* __restrict__ K1, real* __restrict__ K2, int nx, int ny,
                                                   int nz, Phys<real> ph, real dt, int bc) {
    const int xi = blockIdx.x * kGX + threadIdx.x;
    if (xi >= nx) return;
    const long long P = (long long)nx * ny;
    const long long N = P * nz;
    const int rows = ny * nz;
    for (int row = blockIdx.y; row < rows; row += gridDim.y) {
        const int zi = row / ny;
        const int yi = row - zi * ny;
        const long long i = (long long)row * nx + xi;
        const long long nb[6] = {xi > 0 ? i - 1 : i + (nx - 1),
                                 xi < nx - 1 ? i + 1 : i - (nx - 1),
                                 yi > 0 ? i - nx : i + (long long)(ny - 1) * nx,
                                 yi < ny - 1 ? i + nx : i - (long long)(ny - 1) * nx,
                                 zi > 0 ? i - P : i + (N - P),
                                 zi < nz - 1 ? i + P : i - (N - P)};
        // free boundaries: a neighbour across a face does not exist
        const real w[6] = {(bc && xi == 0) ? real(0) : real(1), (bc && xi == nx - 1) ? real(0) : real(1),
                           (bc && yi == 0) ? real(0) : real(1), (bc && yi == ny - 1) ? real(0) : real(1),
                           (bc && zi == 0) ? real(0) : real(1), (bc && zi == nz - 1) ? real(0) : real(1)};
        real h[3], s[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const real* q = x.p[c];
            const real sum = w[0] * q[nb[0]] + w[1] * q[nb[1]] + w[2] * q[nb[2]] + w[3] * q[nb[3]] + w[4] * q[nb[4]] +
                             w[5] * q[nb[5]];
            h[c] = ph.J * sum + ph.H[c];
            if (HSITE) h[c] += hs.p[c][i];
            s[c] = q[i];
        }
        h[2] += ph.twoD * s[2];
        real f[3];
        llg_rhs<real, PREC>(s[0], s[1], s[2], h[0], h[1], h[2], ph.lambda, f[0], f[1], f[2]);
        K0[i] = dt * f[0];
        K1[i] = dt * f[1];
        K2[i] = dt * f[2];
    }
}

template <typename real>
struct CombineArgs {
    const real* s[3];
    const real* K[6];  // each K[l] points at 3N: components at K[l] + c*N
    real coef[6];
    int nk;
    real* out[3];
    int renorm, pulse;
    uint64_t seed, replica;
    real sigma;
    const long long* interval;
};

// out = s + sum_l coef[l] K_l, optionally renormalised and pulsed.  The term
// count NK is a template argument (dispatched on the host), so the pointer
// table is indexed with constants and stays in the kernel parameters.
template <typename real, int NK>
__global__ void k_combine(CombineArgs<real> a, long long N) {
    const long long k = a.pulse ? *a.interval : 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
         i += (long long)gridDim.x * blockDim.x) {
        real v[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            real acc = a.s[c][i];
#pragma unroll
            for (int l = 0; l < NK; ++l)
                if (a.coef[l] != real(0)) acc += a.coef[l] * a.K[l][c * N + i];
            v[c] = acc;
        }
        if (a.renorm) {
            const real inv = Math<real>::rsqrt_(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
            v[0] *= inv;
            v[1] *= inv;
            v[2] *= inv;
        }
        if (a.pulse) pulse_site<real>(v[0], v[1], v[2], a.seed, (uint64_t)i, (uint64_t)k, a.replica, a.sigma);
        a.out[0][i] = v[0];
        a.out[1][i] = v[1];
        a.out[2][i] = v[2];
    }
}

template <typename real>
static void launch_combine(int nk, const CombineArgs<real>& c, long long N, int blocks, int threads, cudaStream_t st) {
    switch (nk) {
        case 1: k_combine<real, 1><<<blocks, threads, 0, st>>>(c, N); break;
        case 2: k_combine<real, 2><<<blocks, threads, 0, st>>>(c, N); break;
        case 3: k_combine<real, 3><<<blocks, threads, 0, st>>>(c, N); break;
        case 4: k_combine<real, 4><<<blocks, threads, 0, st>>>(c, N); break;
        case 5: k_combine<real, 5><<<blocks, threads, 0, st>>>(c, N); break;
        default: k_combine<real, 6><<<blocks, threads, 0, st>>>(c, N); break;
    }
}

template <typename real>
static cudaError_t launch_generic(const StepLaunch<real>& L) {
    const Tableau& tb = *L.tab;
    const long long N = L.g.N();
    const int threads = 256;
    const int blocks = (int)std::min<long long>((N + threads - 1) / threads, 152LL * 16);
    // tmp layout: K_1..K_S (3N each), then x (3N)
    real* K[6];
    for (int j = 0; j < tb.stages; ++j) K[j] = L.tmp + (size_t)j * 3 * N;
    real* xs = L.tmp + (size_t)tb.stages * 3 * N;
    const bool hs = L.hs[0] != nullptr;
    Vec3P<real> hv{{L.hs[0], L.hs[1], L.hs[2]}};
    const long long rows = (long long)L.g.ny * L.g.nz;
    const dim3 rgrid((L.g.nx + kGX - 1) / kGX, (unsigned)std::min<long long>(rows, 65535));
    for (int j = 0; j < tb.stages; ++j) {
        Vec3P<real> xv;
        if (j == 0) {
            xv = Vec3P<real>{{L.in[0], L.in[1], L.in[2]}};
        } else {
            CombineArgs<real> c{};
            for (int q = 0; q < 3; ++q) {
                c.s[q] = L.in[q];
                c.out[q] = xs + (size_t)q * N;
            }
            for (int l = 0; l < j; ++l) {
                c.K[l] = K[l];
                c.coef[l] = (real)tb.a[j][l];
            }
            c.nk = j;
            launch_combine<real>(j, c, N, blocks, threads, L.stream);
            xv = Vec3P<real>{{xs, xs + N, xs + 2 * N}};
        }
        real* k0 = K[j];
        if (L.precession) {
            if (hs)
                k_stage_rhs<real, true, true><<<rgrid, kGX, 0, L.stream>>>(xv, hv, k0, k0 + N, k0 + 2 * N, L.g.nx, L.g.ny, L.g.nz, L.ph, (real)L.dt, L.bc);
            else
                k_stage_rhs<real, true, false><<<rgrid, kGX, 0, L.stream>>>(xv, hv, k0, k0 + N, k0 + 2 * N, L.g.nx, L.g.ny, L.g.nz, L.ph, (real)L.dt, L.bc);
        } else {
            if (hs)
                k_stage_rhs<real, false, true><<<rgrid, kGX, 0, L.stream>>>(xv, hv, k0, k0 + N, k0 + 2 * N, L.g.nx, L.g.ny, L.g.nz, L.ph, (real)L.dt, L.bc);
            else
                k_stage_rhs<real, false, false><<<rgrid, kGX, 0, L.stream>>>(xv, hv, k0, k0 + N, k0 + 2 * N, L.g.nx, L.g.ny, L.g.nz, L.ph, (real)L.dt, L.bc);
        }
    }
    CombineArgs<real> c{};
    for (int q = 0; q < 3; ++q) {
        c.s[q] = L.in[q];
        c.out[q] = L.out[q];
    }
    for (int l = 0; l < tb.stages; ++l) {
        c.K[l] = K[l];
        c.coef[l] = (real)tb.b[l];
    }
    c.nk = tb.stages;
    c.renorm = L.renorm;
    c.pulse = L.pulse;
    c.seed = L.seed;
    c.replica = L.replica;
    c.sigma = L.sigma;
    c.interval = L.d_interval;
    launch_combine<real>(tb.stages, c, N, blocks, threads, L.stream);
    return cudaGetLastError();
}

// SPIN_TMA=1 and SPIN_TMEM=1 choose a form of the fused tile, at every size.
static bool tile_forced() {
    for (const char* name : {"SPIN_TMA", "SPIN_TMEM"}) {
        const char* env = std::getenv(name);
        if (env && env[0] == '1') return true;
    }
    return false;
}

template <typename real>
cudaError_t launch_step(const StepLaunch<real>& L) {
    if (L.tab->chain && !L.force_generic && (L.tab->stages == 4 || L.tab->stages == 2)) {
        if (sizeof(real) == 4) {
            const StepLaunch<float>& F = reinterpret_cast<const StepLaunch<float>&>(L);
            if (!stage32_small(L.g, L.tab->stages, F.hs[0] != nullptr, F.st_n[0][0] != nullptr) || tile_forced())
                return launch_step_patch(F);
            const cudaError_t e = launch_step_stage32(F);
            return e != cudaSuccess || !L.pulse ? e : launch_pulse_lattice(F);
        }
        return launch_step_stage64(reinterpret_cast<const StepLaunch<double>&>(L));
    }
    if (sizeof(real) == 4 && !L.force_generic && rk5_fused_supports(reinterpret_cast<const StepLaunch<float>&>(L)))
        return launch_step_rk5(reinterpret_cast<const StepLaunch<float>&>(L));
    return launch_generic<real>(L);
}

template cudaError_t launch_step<float>(const StepLaunch<float>&);
template cudaError_t launch_step<double>(const StepLaunch<double>&);

// ---------------------------------------------------------------------------
// Noise draw on its own (verification entry point)
// ---------------------------------------------------------------------------

template <typename real>
__global__ void k_noise_draw(uint64_t seed, long long k, long long replica, long long n, uint64_t* words,
                             real* gauss) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const Words4 w = noise_words(seed, (uint64_t)i, (uint64_t)k, (uint64_t)replica);
        if (words) {
#pragma unroll
            for (int q = 0; q < 4; ++q) words[4 * i + q] = w.w[q];
        }
        if (gauss) {
            real g0, g1, g2;
            Gauss<real>::draw(w, g0, g1, g2);
            gauss[3 * i + 0] = g0;
            gauss[3 * i + 1] = g1;
            gauss[3 * i + 2] = g2;
        }
    }
}

cudaError_t launch_noise_draw(uint64_t seed, long long k, long long replica, long long n, int precision,
                              uint64_t* words, void* gauss, cudaStream_t stream) {
    const int threads = 256;
    const int blocks = (int)std::max<long long>(1, std::min<long long>((n + threads - 1) / threads, 152LL * 8));
    if (precision == 64)
        k_noise_draw<double><<<blocks, threads, 0, stream>>>(seed, k, replica, n, words, (double*)gauss);
    else
        k_noise_draw<float><<<blocks, threads, 0, stream>>>(seed, k, replica, n, words, (float*)gauss);
    return cudaGetLastError();
}

__global__ void k_set_counter(long long* d, long long v) { *d = v; }

cudaError_t launch_set_counter(long long* d, long long value, cudaStream_t stream) {
    k_set_counter<<<1, 1, 0, stream>>>(d, value);
    return cudaGetLastError();
}

}  // namespace spin
