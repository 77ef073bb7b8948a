// Magnetisation and energy per spin, accumulated in FP64 (Sec. III.A samples
// at the end of every Delta t; Sec. IV's Heisenberg energy):
//   M = (1/N) sum_i s_i
//   E = (1/N) [ -J sum_<ij> s_i.s_j - D sum_i s_iz^2 - sum_i (H + h_i).s_i ]
// each bond counted once through the three forward neighbours of every site.
// Pass 1: one warp per lattice row, FP64 sums per lane, one 5-double record per
// block.  Pass 2: one block adds the block records in a fixed order, so the
// result is bitwise reproducible.
//
// What bounds it: GB300's FP64 pipe (a warp's FP64 instruction holds it for 16
// cycles of the SM) and, in pass 2, its latency.  So float terms convert to
// double by integer operations (to_f64), the block's sums are formed from
// shared memory with every lane busy (4 x 512 values by four warps: 80
// instructions; shuffle trees in every warp took 25 per warp, 400 per block),
// 1/N comes from the host, and both passes are programmatic dependents.  The two passes at 128^3, cold: FP32 25.5 + 9.7
// -> 16.0 + 7.3 us, FP64 121 -> 77 us for the first.
#include <cuda_runtime.h>

#include <algorithm>

#include "pdl.cuh"
#include "spin_device.cuh"
#include "spin_internal.h"

namespace spin {

namespace {

constexpr int kObsThreads = 512;
constexpr int kObsWarps = kObsThreads / 32;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of one lane over its share of rows: M and E in FP64, non-finite spins.
struct ObsLane {
    double m[3], e;
    int bad;
};

// Add one row's terms: row arrays at a, b, c (this row), their y+1 and z+1
// rows, weights wy, wz of those bonds and of the bond across the row's end.
// FP32: the terms are formed and summed over the lane's sites of the row in
// FP32, then added in FP64.  FP64: the sums of bonds and s_z^2 are kept apart
// and combined once per row, 13 FP64 operations a site.
template <typename real, bool HSITE>
__device__ __forceinline__ void obs_row(ObsLane& o, const real* sx, const real* sy, const real* sz, const real* hx,
                                        const real* hy, const real* hz, long long rb, long long rby,
                                        long long rbz, int nx, bool openx, bool openy, bool openz,
                                        double J, double D, double H0, double H1, double H2, int lane) {
    real m0 = 0, m1 = 0, m2 = 0, e = 0, sq = 0, hs = 0;
    const real Jr = (real)J, Dr = (real)D, H0r = (real)H0, H1r = (real)H1, H2r = (real)H2;
#pragma unroll 2
    for (int x = lane; x < nx; x += 32) {
        const long long i = rb + x;
        const bool last = x + 1 == nx;
        const long long ix = rb + (last ? 0 : x + 1), iy = rby + x, iz = rbz + x;
        const real a = sx[i], b = sy[i], c = sz[i];
        if (!finite_bits(a) || !finite_bits(b) || !finite_bits(c)) o.bad += 1;
        m0 += a;
        m1 += b;
        m2 += c;
        // forward bonds; with free boundaries none crosses the last face
        const bool ox = openx && last;
        const real x0 = ox ? real(0) : sx[ix], x1 = ox ? real(0) : sy[ix], x2 = ox ? real(0) : sz[ix];
        const real y0 = openy ? real(0) : sx[iy], y1 = openy ? real(0) : sy[iy], y2 = openy ? real(0) : sz[iy];
        const real z0 = openz ? real(0) : sx[iz], z1 = openz ? real(0) : sy[iz], z2 = openz ? real(0) : sz[iz];
        if (sizeof(real) == 8) {
            e += a * (x0 + y0 + z0);
            e += b * (x1 + y1 + z1);
            e += c * (x2 + y2 + z2);
            sq += c * c;
            if (HSITE) hs += hx[i] * a + hy[i] * b + hz[i] * c;
        } else {
            // contractions written out: the single-lattice and the batched
            // kernel then round alike
            const real bond = fma(a, x0 + y0 + z0, fma(b, x1 + y1 + z1, c * (x2 + y2 + z2)));
            real f0 = H0r, f1 = H1r, f2 = H2r;
            if (HSITE) {
                f0 += hx[i];
                f1 += hy[i];
                f2 += hz[i];
            }
            e += fma(-Jr, bond, fma(-Dr * c, c, -fma(f0, a, fma(f1, b, f2 * c))));
        }
    }
    o.m[0] += to_f64(m0);
    o.m[1] += to_f64(m1);
    o.m[2] += to_f64(m2);
    if (sizeof(real) == 8)
        o.e += -J * (double)e - D * (double)sq - (H0 * (double)m0 + H1 * (double)m1 + H2 * (double)m2) - (double)hs;
    else
        o.e += to_f64(e);
}

// The block's record (5 doubles) from its lanes' sums, in a fixed order.
__device__ __forceinline__ void obs_block(const ObsLane& o, double* __restrict__ rec) {
    __shared__ double red[4][kObsThreads];
    __shared__ int bad;
    const int t = threadIdx.x, w = t >> 5, l = t & 31;
    if (t == 0) bad = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) red[q][t] = o.m[q];
    red[3][t] = o.e;
    __syncthreads();
    const unsigned nb = __reduce_add_sync(0xffffffffu, (unsigned)o.bad);
    if (l == 0 && nb) atomicAdd(&bad, (int)nb);
    if (w < 4) {
        double v[kObsWarps];
#pragma unroll
        for (int q = 0; q < kObsWarps; ++q) v[q] = red[w][q * 32 + l];
#pragma unroll
        for (int s = kObsWarps / 2; s > 0; s >>= 1)
#pragma unroll
            for (int q = 0; q < s; ++q) v[q] += v[q + s];
        const double r = warp_sum(v[0]);
        if (l == 0) rec[w] = r;
    }
    __syncthreads();
    if (t == 0) rec[4] = (double)bad;
}

template <typename real, bool HSITE>
__global__ void __launch_bounds__(kObsThreads, 2)
    k_obs_partial(const real* sx, const real* sy, const real* sz, const real* hx, const real* hy, const real* hz,
                  int nx, int ny, int nz, double J, double D, double H0, double H1, double H2, double* __restrict__ partials,
                  int bc) {
    // one warp per lattice row (y, z); lanes stride along x, so no per-site
    // index division and the row's loads are coalesced
    pdl_wait();
    pdl_go();
    const long long P = (long long)nx * ny;
    const int rows = ny * nz;
    const int lane = threadIdx.x & 31;
    ObsLane o{};
    for (int row = blockIdx.x * kObsWarps + (threadIdx.x >> 5); row < rows; row += gridDim.x * kObsWarps) {
        const int z = row / ny, y = row - z * ny;
        obs_row<real, HSITE>(o, sx, sy, sz, hx, hy, hz, (long long)row * nx,
                             (long long)z * P + (long long)(y + 1 == ny ? 0 : y + 1) * nx,
                             (long long)(z + 1 == nz ? 0 : z + 1) * P + (long long)y * nx, nx, bc, bc && y + 1 == ny,
                             bc && z + 1 == nz, J, D, H0, H1, H2, lane);
    }
    obs_block(o, partials + (long long)blockIdx.x * 5);
}

__global__ void __launch_bounds__(kObsThreads) k_obs_final(const double* partials, int nblocks, double invN,
                                                           double* __restrict__ out5, double* __restrict__ ring, int ring_len,
                                                           long long* interval, long long* sample_count, int R) {
    __shared__ double tot[5];
    pdl_wait();
    long long m = 0, count = 0;
    if (ring && threadIdx.x == 0) {
        m = *interval;
        count = *sample_count;
    }
    // warp w < 5 adds value w over the blocks
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (w < 5) {
        double a0 = 0, a1 = 0, a2 = 0, a3 = 0;   // four chains: the additions' latency, not their number, counts here
        int b = l;
        for (; b + 96 < nblocks; b += 128) {
            a0 += partials[(long long)b * 5 + w];
            a1 += partials[(long long)(b + 32) * 5 + w];
            a2 += partials[(long long)(b + 64) * 5 + w];
            a3 += partials[(long long)(b + 96) * 5 + w];
        }
        for (; b < nblocks; b += 32) a0 += partials[(long long)b * 5 + w];
        const double r = warp_sum((a0 + a1) + (a2 + a3));
        if (l == 0) {
            tot[w] = w < 4 ? r * invN : r;
            out5[w] = tot[w];
        }
    }
    __syncthreads();
    if (ring && threadIdx.x == 0) {
        double* rec = ring + (count % ring_len) * 5;
        rec[0] = (double)((m + 1) * (long long)R);
        rec[1] = tot[0];
        rec[2] = tot[1];
        rec[3] = tot[2];
        rec[4] = tot[3];
        *interval = m + 1;
        *sample_count = count + 1;
    }
}

// Batched replicas: the same row-wise reduction, each block on a row range
// of one replica; the final pass gives one record per replica.
__global__ void __launch_bounds__(kObsThreads, 2)
    k_obs_batch_partial(const float* sx, const float* sy, const float* sz,
                        const BatchRep* __restrict__ reps, const ObsBlock* __restrict__ blocks, double J, double D,
                        double H0, double H1, double H2, double* __restrict__ partials) {
    pdl_wait();
    pdl_go();
    const ObsBlock ob = blocks[blockIdx.x];
    const BatchRep rp = reps[ob.rep];
    const int L = rp.L;
    const long long P = (long long)L * L;
    const int lane = threadIdx.x & 31;
    ObsLane o{};
    for (int row = ob.row0 + (threadIdx.x >> 5); row < ob.row0 + ob.nrows; row += kObsWarps) {
        const int z = row / L, y = row - z * L;
        obs_row<float, false>(o, sx + rp.off, sy + rp.off, sz + rp.off, nullptr, nullptr, nullptr, (long long)row * L,
                              (long long)z * P + (long long)(y + 1 == L ? 0 : y + 1) * L,
                              (long long)(z + 1 == L ? 0 : z + 1) * P + (long long)y * L, L, false, false, false, J, D,
                              H0, H1, H2, lane);
    }
    obs_block(o, partials + (long long)blockIdx.x * 5);
}

// one warp per replica at a time, 32 warps
constexpr int kObsFinalThreads = 1024;
__global__ void __launch_bounds__(kObsFinalThreads) k_obs_batch_final(const double* partials,
                                                                      const int* __restrict__ first_block,
                                                                      const BatchRep* __restrict__ reps, int nrep,
                                                                      double* __restrict__ out, double* __restrict__ ring,
                                                                      int ring_len, long long* interval,
                                                                      long long* sample_count, int R) {
    pdl_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long m = ring ? *interval : 0;
    const long long count = ring ? *sample_count : 0;
    const long long slot = ring ? count % ring_len : 0;
    for (int r = w; r < nrep; r += kObsFinalThreads >> 5) {
        const double L = (double)reps[r].L;
        const double invN = 1.0 / (L * L * L);
        double acc[5] = {0, 0, 0, 0, 0};
        for (int b = first_block[r] + lane; b < first_block[r + 1]; b += 32)
            for (int q = 0; q < 5; ++q) acc[q] += partials[(long long)b * 5 + q];
        for (int q = 0; q < 5; ++q) acc[q] = warp_sum(acc[q]);
        if (lane == 0) {
            double* o = out + (long long)r * 5;
            for (int q = 0; q < 4; ++q) o[q] = acc[q] * invN;
            o[4] = acc[4];
            if (ring) {
                double* rec = ring + (slot * nrep + r) * 5;
                rec[0] = (double)((m + 1) * (long long)R);
                for (int q = 0; q < 4; ++q) rec[1 + q] = acc[q] * invN;
            }
        }
    }
    __syncthreads();
    if (ring && threadIdx.x == 0) {
        *interval = m + 1;
        *sample_count = count + 1;
    }
}

}  // namespace

int observables_blocks(Geom g) {
    const long long rows = (long long)g.ny * g.nz;
    return (int)std::max<long long>(1, std::min<long long>((rows + kObsWarps - 1) / kObsWarps, 152LL * 2));
}

template <typename real>
cudaError_t launch_observables(const real* s[3], const real* hs[3], Geom g, Phys<double> ph, double* partials,
                               int nblocks, double* out5, double* sample_ring, int ring, long long* d_interval,
                               long long* d_sample_count, int R, cudaStream_t stream, int bc, int into) {
    const double D = 0.5 * ph.twoD;
    const dim3 grid(nblocks), block(kObsThreads);
    const bool pdl = pdl_after_step(into, (int)sizeof(real), g.N());
    const cudaError_t e =
        hs[0] ? launch_pdl(pdl, k_obs_partial<real, true>, grid, block, 0, stream, s[0], s[1], s[2], hs[0], hs[1], hs[2], g.nx,
                           g.ny, g.nz, ph.J, D, ph.H[0], ph.H[1], ph.H[2], partials, bc)
              : launch_pdl(pdl, k_obs_partial<real, false>, grid, block, 0, stream, s[0], s[1], s[2], hs[0], hs[1], hs[2], g.nx,
                           g.ny, g.nz, ph.J, D, ph.H[0], ph.H[1], ph.H[2], partials, bc);
    if (e != cudaSuccess) return e;
    return launch_pdl(pdl, k_obs_final, dim3(1), dim3(160), 0, stream, (const double*)partials, nblocks, 1.0 / (double)g.N(), out5,
                        sample_ring, ring, d_interval, d_sample_count, R);
}

cudaError_t launch_observables_batch(const float* s[3], const BatchRep* reps, const ObsBlock* blocks, int nblocks,
                                     const int* first_block, int nrep, Phys<double> ph, double* partials,
                                     double* out, double* ring, int ring_len, long long* d_interval,
                                     long long* d_sample_count, int R, cudaStream_t stream, int into) {
    const cudaError_t e = launch_pdl(into == kStream, k_obs_batch_partial, dim3(nblocks), dim3(kObsThreads), 0, stream, s[0], s[1], s[2], reps,
                                     blocks, ph.J, 0.5 * ph.twoD, ph.H[0], ph.H[1], ph.H[2], partials);
    if (e != cudaSuccess) return e;
    return launch_pdl(into == kStream, k_obs_batch_final, dim3(1), dim3(kObsFinalThreads), 0, stream, (const double*)partials, first_block, reps, nrep, out,
                        ring, ring_len, d_interval, d_sample_count, R);
}

template cudaError_t launch_observables<float>(const float* s[3], const float* hs[3], Geom, Phys<double>, double*, int,
                                               double*, double*, int, long long*, long long*, int, cudaStream_t, int, int);
template cudaError_t launch_observables<double>(const double* s[3], const double* hs[3], Geom, Phys<double>, double*,
                                                int, double*, double*, int, long long*, long long*, int, cudaStream_t,
                                                int, int);

}  // namespace spin

// ---------------------------------------------------------------------------
// Observables without any allocation by the library or the caller.
//
// Some callers cannot call cudaMalloc (or ask a framework to allocate) at the
// point where they want the magnetisation and energy: code running inside a
// strict memory budget, a host thread that must not take the allocator's
// lock, or a plug-in that only receives pointers to existing arrays.  For
// them this entry point keeps the reduction's scratch -- one 5-double record
// per block of the first pass -- in a fixed file-scope device array that is
// part of the loaded module, so nothing is allocated per call.
// ---------------------------------------------------------------------------

#include <mutex>

#include "../../include/spinpulse.h"

namespace spin {
namespace {

constexpr int kNoAllocMaxBlocks = SPIN_NOALLOC_MAX_BLOCKS;
// Block records of the first reduction pass, shared by every call on a device.
static __device__ __align__(256) double g_noalloc_partials[kNoAllocMaxBlocks * 5];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double* g_noalloc_addr[kMaxDevices] = {};

// Device address of the scratch array on the current device.  In host code
// the array's name is only a host-side stand-in, so its address must come
// from cudaGetSymbolAddress, called with the device current.  Outside stream
// capture it is looked up on every call (a cudaDeviceReset reloads the module
// and may move the array); a call on a capturing stream reuses the address
// the last uncaptured call found on this device.
cudaError_t noalloc_scratch(cudaStream_t st, double** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (cap == cudaStreamCaptureStatusNone) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_partials);
        if (e != cudaSuccess) return e;
        g_noalloc_addr[dev] = static_cast<double*>(p);
    } else if (!g_noalloc_addr[dev]) {
        return cudaErrorStreamCaptureUnsupported;
    }
    *out = g_noalloc_addr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace spin

extern "C" int spin_observables_noalloc(int32_t precision, const void* sx, const void* sy, const void* sz,
                                        const void* h_site, int32_t nx, int32_t ny, int32_t nz, double J, double D,
                                        const double H[3], int32_t bc, double* out5, void* cuda_stream) {
    using namespace spin;
    if (!sx || !sy || !sz || !out5 || !H) return SPIN_EINVAL;
    if (bc != 0 && bc != 1) return SPIN_EINVAL;
    if (precision != 32 && precision != 64) return SPIN_EINVAL;
    if (nx < 1 || ny < 1 || nz < 1) return SPIN_EINVAL;
    const Geom g{nx, ny, nz};
    if (g.N() > (long long)SPIN_NOALLOC_MAX_SITES) return SPIN_EINVAL;  // beyond the stated maximum
    const int nblocks = observables_blocks(g);
    if (nblocks > kNoAllocMaxBlocks) return SPIN_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    double* scratch = nullptr;
    const cudaError_t es = noalloc_scratch(st, &scratch);
    if (es == cudaErrorStreamCaptureUnsupported) return SPIN_EINVAL;
    if (es != cudaSuccess) return SPIN_ECUDA;
    Phys<double> ph{};
    ph.J = J;
    ph.twoD = 2.0 * D;
    ph.H[0] = H[0];
    ph.H[1] = H[1];
    ph.H[2] = H[2];
    const size_t comp = (size_t)(precision == 64 ? 8 : 4) * (size_t)g.N();
    const int into = launch_into(st) == kStream ? kIntervalGraph : kCallersGraph;   // large lattices: ordinary launches
    cudaError_t e;
    if (precision == 32) {
        const float* s[3] = {(const float*)sx, (const float*)sy, (const float*)sz};
        const float* hs[3] = {nullptr, nullptr, nullptr};
        if (h_site)
            for (int c = 0; c < 3; ++c) hs[c] = (const float*)((const char*)h_site + c * comp);
        e = launch_observables<float>(s, hs, g, ph, scratch, nblocks, out5, nullptr, 0, nullptr, nullptr, 1, st, bc, into);
    } else {
        const double* s[3] = {(const double*)sx, (const double*)sy, (const double*)sz};
        const double* hs[3] = {nullptr, nullptr, nullptr};
        if (h_site)
            for (int c = 0; c < 3; ++c) hs[c] = (const double*)((const char*)h_site + c * comp);
        e = launch_observables<double>(s, hs, g, ph, scratch, nblocks, out5, nullptr, 0, nullptr, nullptr, 1, st, bc, into);
    }
    return e == cudaSuccess ? SPIN_OK : SPIN_ECUDA;
}
