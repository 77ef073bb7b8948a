// Device-side building blocks of the pulse-noise step (arXiv:1610.04914):
// the counter-based noise generator, Box-Muller, the pulse rotation and the
// right-hand side of the noiseless Landau-Lifshitz equation.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "noise_tables.cuh"

namespace spin {

// Key word 1 of the noise stream ("noise" in ASCII).
constexpr uint64_t kStreamNoise = 0x6E6F697365ULL;

// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds, each
// multiplying counter words 0 and 2 by the two round constants, crossing the
// high halves with words 1 and 3 and the key, then bumping the key by the
// two Weyl increments.
struct Words4 {
    uint64_t w[4];
};

// 64x64 -> 128-bit product: low word by the wrapping multiply, high word by
// the compiler's multiply-high intrinsic.
__device__ __forceinline__ void mul64_wide(uint64_t a, uint64_t m, uint64_t& hi, uint64_t& lo) {
    lo = a * m;
    hi = __umul64hi(a, m);
}

__device__ __forceinline__ Words4 philox4x64_10(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                                                uint64_t k0, uint64_t k1) {
    constexpr uint64_t kMulA = 0xD2E7470EE14C6C93ULL;
    constexpr uint64_t kMulB = 0xCA5A826395121157ULL;
    constexpr uint64_t kWeylA = 0x9E3779B97F4A7C15ULL;
    constexpr uint64_t kWeylB = 0xBB67AE8584CAA73BULL;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint64_t hiA, loA, hiB, loB;
        mul64_wide(c0, kMulA, hiA, loA);
        mul64_wide(c2, kMulB, hiB, loB);
        const uint64_t n0 = hiB ^ c1 ^ k0;
        const uint64_t n2 = hiA ^ c3 ^ k1;
        c0 = n0;
        c1 = loB;
        c2 = n2;
        c3 = loA;
        k0 += kWeylA;
        k1 += kWeylB;
    }
    return Words4{{c0, c1, c2, c3}};
}

__device__ __forceinline__ Words4 noise_words(uint64_t seed, uint64_t site, uint64_t k, uint64_t replica) {
    return philox4x64_10(site, k, replica, 0ULL, seed, kStreamNoise);
}

// Exact float -> double for FP64 accumulation of FP32 terms, with 32-bit integer
// operations only: the hardware conversion uses this GPU's FP64 pipe, which
// runs at ~1/64 of the FP32 rate and is needed for the FP64 additions
// themselves.  The exponent is rebased from 127 to 1023; subnormals are first
// scaled by 2^24; zeros, infinities and NaNs keep their sign and payload.
// (Every case is selected, none branched to: a conversion instruction in a
// rare branch would be executed always, with its result discarded.)
__device__ __forceinline__ double to_f64(float f) {
    const unsigned b = __float_as_uint(f);
    const bool sub = (b & 0x7F800000u) == 0u;
    const unsigned m = sub ? __float_as_uint(f * 16777216.0f) : b;
    const unsigned e = (m >> 23) & 0xFFu;
    const unsigned x = e == 0u ? 0u : e == 0xFFu ? 2047u : e + (sub ? 872u : 896u);
    return __hiloint2double((int)((b & 0x80000000u) | (x << 20) | ((m & 0x7FFFFFu) >> 3)), (int)(m << 29));
}
__device__ __forceinline__ double to_f64(double d) { return d; }

// Box-Muller.  Uniforms are u = ((w >> 11) + 1/2) 2^-53 in (0, 1); G0, G1 from
// (u0, u1) and G2 from (u2, u3).
template <typename real>
struct Gauss;

template <>
struct Gauss<double> {
    // (k + 1/2) 2^-53, k = w >> 11, correctly rounded: k + 1/2 = m/2 with the
    // 54-bit odd integer m, exact in a double unless its top bit is set, when
    // the dropped last bit is a tie (to even).  Integer operations only: the
    // conversion, the addition and the scaling would take three instructions
    // of the FP64 pipe, which bounds the FP64 kernels.
    __device__ __forceinline__ static double u01(uint64_t w) {
        uint64_t m = (w >> 10) | 1ULL;
        if (m >> 53) m = ((m >> 1) + ((m >> 1) & 1ULL)) << 1;
        const int lz = __clzll((long long)m);
        // value m 2^-54: exponent 63 - lz - 54, mantissa below the leading bit
        return __longlong_as_double((long long)(((uint64_t)(1023 + 9 - lz) << 52) + ((m << lz) << 1 >> 12)));
    }
    // -2 ln u for u in (0, 1), table-driven (P. T. P. Tang, ACM TOMS 16, 1990):
    // u = 2^e m, m in [sqrt(1/2), sqrt(2)), ln m = -ln c + ln(1 + r) with c from
    // the table, r = m c - 1, |r| <= 2^-8, and the series of ln(1 + r) to r^7.
    // Ten FP64 instructions (log: about 35; the pulse of an FP64 128^3 lattice
    // 657 -> 414 us with root and angle below).  Near u = 1, c = 1 and e = 0: no
    // cancellation.  Error up to 1.9 units in the last place (the library's about
    // one), 0.45 rms; with the angles below, which take the 54-bit uniform where a
    // library call takes its 53-bit rounding, the Gaussians of 2^19 draws are off
    // by 1.5e-16 rms against 113-bit arithmetic, 2.9e-16 with the library's calls.
    __device__ __forceinline__ static double neg2log(double u) {
        const int h = __double2hiint(u);
        const int e = (h - 0x3FE6A09E) >> 20;
        const int mh = h - (e << 20);
        const double m = __hiloint2double(mh, __double2loint(u));
        const double2 t = __ldg(&kLogTable[((mh - 0x3FE00000 + (1 << 12)) >> 13) - kLogFirst]);
        const double r = fma(m, t.x, -1.0);
        double q = fma(1.0 / 7.0, r, -1.0 / 6.0);
        q = fma(q, r, 1.0 / 5.0);
        q = fma(q, r, -1.0 / 4.0);
        q = fma(q, r, 1.0 / 3.0);
        q = fma(q, r, -1.0 / 2.0);
        const double l = fma(r * r, q, r);
        return fma(-2.0, l, fma(to_f64((float)e), -1.3862943611198906188, t.y));   // -2 ln 2
    }
    // sqrt of a normal x: the FP32 reciprocal root of x with its mantissa cut to
    // 24 bits, then one third-order step; five FP64 instructions, error below one
    // unit in the last place.
    __device__ __forceinline__ static double root(double x) {
        const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
        const float xf = __uint_as_float(((h - 0x38000000u) << 3) | (l >> 29));
        const double g = to_f64(rsqrtf(xf));
        const double t = x * g;
        const double d = fma(-t, g, 1.0);
        return fma(t * d, fma(0.375, d, 0.5), t);
    }
    // cos and sin of 2 pi u, u = (2k+1) 2^-54 the uniform of word w: the nearest
    // multiple of 2 pi/64 from the table, the rest (|phi| <= pi/64) by series.
    __device__ __forceinline__ static void angle(uint64_t w, double& c, double& s) {
        const uint64_t m = (w >> 10) | 1ULL;
        const unsigned k = (unsigned)((m + (1ULL << 47)) >> 48);
        const long long d = (long long)(m - ((uint64_t)k << 48));   // |d| <= 2^47
        const double2 t = __ldg(&kTrigTable[k & 63u]);
        // d as a double: added to the bits of 1.5 2^52, which is then subtracted
        const double x = __longlong_as_double(0x4338000000000000LL + d) - 6755399441055744.0;
        const double phi = x * 3.4878684980086318e-16;               // 2 pi 2^-54
        const double z = phi * phi;
        double p = fma(-1.0 / 5040.0, z, 1.0 / 120.0);
        p = fma(p, z, -1.0 / 6.0);
        const double sn = fma(phi * z, p, phi);
        double q = fma(1.0 / 40320.0, z, -1.0 / 720.0);
        q = fma(q, z, 1.0 / 24.0);
        q = fma(q, z, -0.5);
        const double cm = z * q;                                     // cos(phi) - 1
        c = fma(t.x, cm, fma(-t.y, sn, t.x));
        s = fma(t.y, cm, fma(t.x, sn, t.y));
    }
    __device__ __forceinline__ static void draw(const Words4& w, double& g0, double& g1, double& g2) {
        const double r0 = root(neg2log(u01(w.w[0])));
        const double r2 = root(neg2log(u01(w.w[2])));
        double s1, c1, s3, c3;
        angle(w.w[1], c1, s1);
        angle(w.w[3], c3, s3);
        g0 = r0 * c1;
        g1 = r0 * s1;
        g2 = r2 * c3;
    }
};

template <>
struct Gauss<float> {
    // Same real numbers as the double path, each rounded once to float: the
    // 54-bit odd integer m = 2(w>>11)+1 to 24 bits.  From 2^34 on, m's bits
    // above 2^32 (hi) and the 23 below them with the last one set (sticky: m is
    // odd, and the rounding boundary lies at least one bit higher) convert
    // exactly by exponent tricks, so one addition rounds like m itself.  Below
    // (one word in 2^20), m shifted to 32 bits with the same sticky bit goes
    // through the 32-bit conversion.  The 64-bit conversion instruction is
    // avoided: it runs on GB300's narrow FP64 pipe.
    __device__ __forceinline__ static float u01(uint64_t w) {
        const unsigned wh = (unsigned)(w >> 32);
        const unsigned hi = wh >> 10;
        const unsigned b = __funnelshift_r((unsigned)w, wh, 19) & 0x7FFFFFu;
        const float h = __fmaf_rn(__uint_as_float(0x4B000000u | hi), 2.384185791015625e-07f, -2.0f);   // hi 2^-22
        const float l = __fmaf_rn(__uint_as_float(0x4B000001u | b), 2.8421709430404007e-14f,
                                  -2.384185791015625e-07f);                                            // b 2^-45
        float u = __fadd_rn(h, l);
        if (hi < 4u) {
            const unsigned lo = __funnelshift_r((unsigned)w, wh, 10) | 1u;   // m's low 32 bits
            u = hi ? __uint2float_rn((hi << 30) | (lo >> 2) | 1u) * 2.2204460492503131e-16f   // 2^-52
                   : __uint2float_rn(lo) * 5.5511151231257827e-17f;                           // 2^-54
        }
        return u;
    }
    __device__ __forceinline__ static void draw(const Words4& w, float& g0, float& g1, float& g2) {
        const float r0 = sqrtf(-2.0f * logf(u01(w.w[0])));
        const float r2 = sqrtf(-2.0f * logf(u01(w.w[2])));
        float s1, c1;
        sincospif(2.0f * u01(w.w[1]), &s1, &c1);
        g0 = r0 * c1;
        g1 = r0 * s1;
        g2 = r2 * cospif(2.0f * u01(w.w[3]));
    }
};

template <typename real>
struct Math;
template <>
struct Math<float> {
    __device__ __forceinline__ static float rsqrt_(float x) { return rsqrtf(x); }
    __device__ __forceinline__ static float sqrt_(float x) { return sqrtf(x); }
    __device__ __forceinline__ static void sincos_(float x, float* s, float* c) { sincosf(x, s, c); }
};
template <>
struct Math<double> {
    __device__ __forceinline__ static double rsqrt_(double x) { return 1.0 / sqrt(x); }
    __device__ __forceinline__ static double sqrt_(double x) { return sqrt(x); }
    __device__ __forceinline__ static void sincos_(double x, double* s, double* c) { sincos(x, s, c); }
};

// 1/sqrt(x) from the FP32 reciprocal root of x cut to 24 bits and one
// third-order step, as in Gauss<double>::root: five FP64 instructions.  Outside
// the normal floats' range (zero, infinite and NaN arguments among it) the
// library's, out of line so that it is not executed for every site.
static __device__ __noinline__ double plain_rsqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ double inv_root(double x) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    if (h - 0x38100000u >= 0x0FE00000u) return plain_rsqrt(x);
    const double g = to_f64(rsqrtf(__uint_as_float(((h - 0x38000000u) << 3) | (l >> 29))));
    const double d = fma(-(x * g), g, 1.0);
    return fma(g * d, fma(0.375, d, 0.5), g);
}

// S 2^(emax - 1082) rounded once to nearest, with integer operations (an FP64
// instruction or conversion takes as long as some sixty of them); emax is such
// that the result is a normal number.
__device__ __forceinline__ double from_fixed(long long S, unsigned emax) {
    const long long sg = S >> 63;
    const unsigned long long a = (unsigned long long)((S ^ sg) - sg);
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << lz;      // leading bit at 63
    unsigned long long r = n >> 11;
    const unsigned rem = (unsigned)n & 0x7FFu;
    r += (rem > 0x400u || (rem == 0x400u && (r & 1ULL))) ? 1ULL : 0ULL;
    // leading bit of a at bit 63 - lz: biased exponent emax + 4 - lz, of which
    // the mantissa's leading bit adds one
    r += (unsigned long long)(emax + 3u - (unsigned)lz) << 52;
    r |= (unsigned long long)sg & 0x8000000000000000ULL;
    return a == 0ULL ? 0.0 : __longlong_as_double((long long)r);
}

// sin(phi)/phi and (1 - cos(phi))/phi^2 for p = phi^2 <= kSmallPhi2: the Taylor
// series in p, truncated below the type's rounding (the first omitted terms are
// p^7/15! = 1.3e-8 and p^11/23! = 1.6e-16 at p = 4).
constexpr float kSmallPhi2 = 4.0f;
__device__ __forceinline__ void rotation_series(float p, float& sinc, float& cosc) {
    sinc = 1.0f / 6227020800.0f;
    sinc = __fmaf_rn(sinc, p, -1.0f / 39916800.0f);
    sinc = __fmaf_rn(sinc, p, 1.0f / 362880.0f);
    sinc = __fmaf_rn(sinc, p, -1.0f / 5040.0f);
    sinc = __fmaf_rn(sinc, p, 1.0f / 120.0f);
    sinc = __fmaf_rn(sinc, p, -1.0f / 6.0f);
    sinc = __fmaf_rn(sinc, p, 1.0f);
    cosc = 1.0f / 87178291200.0f;
    cosc = __fmaf_rn(cosc, p, -1.0f / 479001600.0f);
    cosc = __fmaf_rn(cosc, p, 1.0f / 3628800.0f);
    cosc = __fmaf_rn(cosc, p, -1.0f / 40320.0f);
    cosc = __fmaf_rn(cosc, p, 1.0f / 720.0f);
    cosc = __fmaf_rn(cosc, p, -1.0f / 24.0f);
    cosc = __fmaf_rn(cosc, p, 0.5f);
}
__device__ __forceinline__ void rotation_series(double p, double& sinc, double& cosc) {
    sinc = 1.0 / 51090942171709440000.0;              // 21!
    sinc = fma(sinc, p, -1.0 / 121645100408832000.0);  // 19!
    sinc = fma(sinc, p, 1.0 / 355687428096000.0);      // 17!
    sinc = fma(sinc, p, -1.0 / 1307674368000.0);       // 15!
    sinc = fma(sinc, p, 1.0 / 6227020800.0);
    sinc = fma(sinc, p, -1.0 / 39916800.0);
    sinc = fma(sinc, p, 1.0 / 362880.0);
    sinc = fma(sinc, p, -1.0 / 5040.0);
    sinc = fma(sinc, p, 1.0 / 120.0);
    sinc = fma(sinc, p, -1.0 / 6.0);
    sinc = fma(sinc, p, 1.0);
    cosc = 1.0 / 1124000727777607680000.0;             // 22!
    cosc = fma(cosc, p, -1.0 / 2432902008176640000.0);  // 20!
    cosc = fma(cosc, p, 1.0 / 6402373705728000.0);      // 18!
    cosc = fma(cosc, p, -1.0 / 20922789888000.0);       // 16!
    cosc = fma(cosc, p, 1.0 / 87178291200.0);
    cosc = fma(cosc, p, -1.0 / 479001600.0);
    cosc = fma(cosc, p, 1.0 / 3628800.0);
    cosc = fma(cosc, p, -1.0 / 40320.0);
    cosc = fma(cosc, p, 1.0 / 720.0);
    cosc = fma(cosc, p, -1.0 / 24.0);
    cosc = fma(cosc, p, 0.5);
}

// Rotation of s by the angle vector phi = sigma G, Eq. (s_rotation):
//   s' = s cos(phi) + (n x s) sin(phi) + n (n.s)(1 - cos(phi)),  n = phi/|phi|.
// Small angles (almost every pulse within the method's applicability
// condition sigma^2 <= 0.2) need no n: with the two even functions of phi
// above, s' = s (1 - phi^2 B) + (phi x s) A + phi (phi.s) B, which saves the
// square root, the division and the sine and cosine.
// kSeriesSigma: sigma up to which the series is tried.  There phi^2 passes
// kSmallPhi2 with probability below 1e-6 (chi-squared, three degrees), so the
// warp does not diverge; for larger sigma every site takes the general form.
constexpr float kSeriesSigma = 0.35f;
// Contractions are written out, so that every kernel that rotates rounds alike.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
template <typename real>
__device__ __forceinline__ real dot_rn(real ax, real ay, real az, real bx, real by, real bz) {
    return fma(az, bz, fma(ay, by, mul_rn(ax, bx)));
}
template <typename real>
__device__ __forceinline__ void pulse_rotate(real& sx, real& sy, real& sz, real px, real py, real pz, real sigma) {
    const real phi2 = dot_rn(px, py, pz, px, py, pz);
    real nx = px, ny = py, nz = pz, A, C, B;   // s' = s C + (n x s) A + n (n.s) B
    if (sigma <= real(kSeriesSigma) && phi2 <= real(kSmallPhi2)) {
        rotation_series(phi2, A, B);
        C = fma(-phi2, B, real(1));
    } else {
        if (!(phi2 > real(0))) return;
        const real phi = Math<real>::sqrt_(phi2);
        const real inv = real(1) / phi;
        nx = mul_rn(px, inv);
        ny = mul_rn(py, inv);
        nz = mul_rn(pz, inv);
        Math<real>::sincos_(phi, &A, &C);
        B = real(1) - C;
    }
    const real om = mul_rn(dot_rn(nx, ny, nz, sx, sy, sz), B);
    const real cx = fma(ny, sz, -mul_rn(nz, sy));
    const real cy = fma(nz, sx, -mul_rn(nx, sz));
    const real cz = fma(nx, sy, -mul_rn(ny, sx));
    sx = fma(nx, om, fma(cx, A, mul_rn(sx, C)));
    sy = fma(ny, om, fma(cy, A, mul_rn(sy, C)));
    sz = fma(nz, om, fma(cz, A, mul_rn(sz, C)));
}

// One pulse on one site: draw G_i for pulse k, rotate by sigma G_i.
template <typename real>
__device__ __forceinline__ void pulse_site(real& sx, real& sy, real& sz, uint64_t seed, uint64_t site,
                                           uint64_t k, uint64_t replica, real sigma) {
    const Words4 w = noise_words(seed, site, k, replica);
    real g0, g1, g2;
    Gauss<real>::draw(w, g0, g1, g2);
    pulse_rotate<real>(sx, sy, sz, mul_rn(sigma, g0), mul_rn(sigma, g1), mul_rn(sigma, g2), sigma);
}

// isfinite without the FP64 pipe (its comparison would run there)
__device__ __forceinline__ bool finite_bits(float f) { return (__float_as_uint(f) & 0x7F800000u) != 0x7F800000u; }
__device__ __forceinline__ bool finite_bits(double d) {
    return ((unsigned)__double2hiint(d) & 0x7FF00000u) != 0x7FF00000u;
}

// Right-hand side of Eq. (LLL) with a rectangular-noise field zeta, which
// enters the precession term only:  f = s x (H + zeta) - lambda s x (s x H).
template <typename real>
__device__ __forceinline__ void llg_rhs_noise(real sx, real sy, real sz, real hx, real hy, real hz, real zx,
                                              real zy, real zz, real lambda, real& fx, real& fy, real& fz) {
    const real cx = sy * hz - sz * hy;
    const real cy = sz * hx - sx * hz;
    const real cz = sx * hy - sy * hx;
    const real bx = sy * cz - sz * cy;
    const real by = sz * cx - sx * cz;
    const real bz = sx * cy - sy * cx;
    const real px = hx + zx, py = hy + zy, pz = hz + zz;
    fx = (sy * pz - sz * py) - lambda * bx;
    fy = (sz * px - sx * pz) - lambda * by;
    fz = (sx * py - sy * px) - lambda * bz;
}

// Right-hand side of Eq. (LLL) without noise, given H_eff = (hx, hy, hz):
//   a = s x H,  b = s x a
//   precessional: f = a - lambda b;   slow (precession dropped): f = -lambda b
template <typename real, bool PREC>
__device__ __forceinline__ void llg_rhs(real sx, real sy, real sz, real hx, real hy, real hz, real lambda,
                                        real& fx, real& fy, real& fz) {
    const real ax = sy * hz - sz * hy;
    const real ay = sz * hx - sx * hz;
    const real az = sx * hy - sy * hx;
    const real bx = sy * az - sz * ay;
    const real by = sz * ax - sx * az;
    const real bz = sx * ay - sy * ax;
    if (PREC) {
        fx = ax - lambda * bx;
        fy = ay - lambda * by;
        fz = az - lambda * bz;
    } else {
        fx = -lambda * bx;
        fy = -lambda * by;
        fz = -lambda * bz;
    }
}

}  // namespace spin
