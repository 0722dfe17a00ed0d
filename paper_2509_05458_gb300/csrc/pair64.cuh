// FP64 building blocks of the pair kernels (near field, direct sum, gradient).
//
// What bounds them: this chip issues one FP64 warp instruction per 16 SM
// cycles, i.e. per 64 issue slots, so a pair costs its FP64 instructions and
// nothing else. Each function takes its starting value from FP32 and integer
// instructions (almost free beside that) and spends FP64 instructions only on
// the correction or on a short polynomial about a table entry; conversions
// between FP32 and FP64, which also run on the FP64 pipe, are done on the bits.
//   crsqrt64  17 FP64 instructions: FP32 root, one third-order Newton step
//   crcp64    12: likewise
//   wave64    28: table of e^{2 pi i k/256} and 2^{k/256}, short Taylor series
//   clog64    28: table reciprocal, log(1 + d) for |d| < 0.0037
//   hankel_factor 32 a function: Taylor cells of the smooth factor of H_0, H_1
// The library calls they replace (hypot, sqrt, division with scaling, sincos,
// exp, log, atan2, the 24-point quadrature of H_nu) cost about 35 (3D Laplace)
// to 6000 (2D Helmholtz beyond |z| = 6) FP64 instructions per pair more.
// Arguments outside the range that the bit operations cover (and 0, NaN, Inf)
// take the general functions of cfmm_special.cuh.
#pragma once

#include "cfmm_special.cuh"

namespace cfmm {

constexpr int kAngTab = 256;      // directions of wave64
constexpr int kExpTab = 256;      // 2^(k/256)
constexpr int kLogRad = 256;      // radial cells per octave of clog64
constexpr int kLogAng = 1024;     // angular cells of clog64
// cells of hankel_factor in s = 1/z, nested grids l = 0, 1, 2 of step 2^(l-6):
// Re s = 0 .. 2^(l-1), Im s = -2^(l-1) .. 0.75 2^(l-1)
constexpr int kHkDeg = 8;
constexpr int kHkNx = 33, kHkNeg = 32, kHkNy = 57, kHkGrids = 3;

struct PairTab {
    double2 ang[kAngTab];         // (cos, sin)(2 pi k/256)
    double ex[kExpTab];           // 2^(k/256)
    double2 lrad[kLogRad];        // reciprocal radius with 20 bits, -log of it
    double2 ldir[kLogAng];        // conjugate direction, 27 bits a component
    double2 llog[kLogAng];        // -log of it (length and angle)
    double2 hk[kHkGrids * kHkNx * kHkNy][2][kHkDeg + 1];   // Taylor coefficients of the H_0 and H_1 factors
};

// double -> float by truncation of the bits, for |v| < 2^127 (below 2^-126: 0 of v's sign,
// which tells the side of the branch cut)
__device__ __forceinline__ float seed_f32(double v) {
    unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    unsigned f = __funnelshift_l(lo, hi, 3) + 0x40000000u;
    f = (f & 0x7fffffffu) | (hi & 0x80000000u);
    return __uint_as_float((hi & 0x7fffffffu) < 0x38100000u ? hi & 0x80000000u : f);
}
// float -> double on the bits (normal values; 0 becomes 2^-127)
__device__ __forceinline__ double widen_f32(float v) {
    unsigned u = __float_as_uint(v);
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ float rsqrt_ap(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_ap(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// the larger component in [2^-60, 2^60): squares stay inside the FP32 range
__device__ __forceinline__ bool seed_range(cd z) {
    unsigned a = (unsigned)__double2hiint(z.x) & 0x7fffffffu, b = (unsigned)__double2hiint(z.y) & 0x7fffffffu;
    return max(a, b) - 0x3c300000u < 0x07800000u;
}

static __device__ __noinline__ cd crsqrt_general(cd z) { return cinv(csqrt_p(z)); }
static __device__ __noinline__ cd crcp_general(cd z) { return cinv(z); }
static __device__ __noinline__ cd expi_general(cd z) { return cexp_i(z); }
static __device__ __noinline__ cd clog_general(cd z) {
    return cd{0.5 * log(cabs2(z)), atan2(z.y, z.x)};
}

// 1/sqrt(z), principal branch. FP32 value y (relative error below 2^-20), then
// with h = 1 - z y^2: y + y h (1/2 + 3h/8), error O(h^3) < 2^-58.
__device__ __forceinline__ cd crsqrt64(cd z) {
    if (!seed_range(z)) return crsqrt_general(z);
    float a = seed_f32(z.x), b = seed_f32(z.y);
    float m2 = fmaf(a, a, b * b);
    float im = rsqrt_ap(m2);
    float t2 = 0.5f * fmaf(m2, im, fabsf(a));
    float rt = rsqrt_ap(t2);
    float t = t2 * rt, u = 0.5f * b * rt;
    bool pos = a >= 0.f;
    double yr = widen_f32(im * (pos ? t : fabsf(u)));
    double yi = widen_f32(-im * (pos ? u : copysignf(t, b)));
    double sr = fma(-yi, yi, yr * yr), si = (yr + yr) * yi;
    double hr = fma(z.y, si, fma(-z.x, sr, 1.0));
    double hi = fma(-z.y, sr, -(z.x * si));
    double pr = fma(0.375, hr, 0.5), pi = 0.375 * hi;
    double qr = fma(-hi, pi, hr * pr), qi = fma(hi, pr, hr * pi);
    return cd{fma(-yi, qi, fma(yr, qr, yr)), fma(yi, qr, fma(yr, qi, yi))};
}

// 1/z: FP32 value y, then with e = 1 - z y: y + y (e + e^2), error O(e^3).
__device__ __forceinline__ cd crcp64(cd z) {
    if (!seed_range(z)) return crcp_general(z);
    float a = seed_f32(z.x), b = seed_f32(z.y);
    float im = rcp_ap(fmaf(a, a, b * b));
    double yr = widen_f32(a * im), yi = widen_f32(-b * im);
    double er = fma(z.y, yi, fma(-z.x, yr, 1.0)), ei = fma(-z.y, yr, -(z.x * yi));
    double pr = fma(-ei, ei, fma(er, er, er)), pi = fma(er + er, ei, ei);
    return cd{fma(-yi, pi, fma(yr, pr, yr)), fma(yi, pr, fma(yr, pi, yi))};
}

// wavenumber k, 1/k, k^{-1/2} and k 256/(2 pi), k 256/log 2
struct Wave {
    double k, ik, isk, ka, kb;
};

// e^{i k r} for r = r2 y, y = 1/r: k Re r = a 2 pi/256 + t and -k Im r =
// b log(2)/256 + v with a, b whole and the constants in two parts, the first of
// 31 bits, so that its product with a (b) is exact and t, v see k r unrounded.
// Beyond |k Re r| = 8, where the rounding of r itself shows in the phase, the
// residual r2 - r^2 corrects it (an FP32 product). sin t and cos t - 1 by their
// Taylor series to t^5 and t^6, e^v to v^4 (|t| < 0.0123, |v| < 0.00136; remainders below
// 1e-17, that of e^v below 4e-17).
__device__ __forceinline__ cd wave64(const PairTab* __restrict__ T, const Wave& w, cd r2, cd y, cd& r) {
    r = y * r2;
    const double kMagic = 6755399441055744.0;                            // 1.5 2^52
    double ka = fma(r.x, w.ka, kMagic), kb = fma(-r.y, w.kb, kMagic);
    int ia = __double2loint(ka), ib = __double2loint(kb);
    // |k Re r| < 2^16, |k Im r| < 700 (the high words tell larger values, NaN and Inf)
    if (__double2hiint(ka) - 0x43380000 + 1 > 1u || __double2hiint(kb) - 0x43380000 + 1 > 1u ||
        abs(ia) > (1 << 21) || abs(ib) > 258531)
        return expi_general(w.k * r);
    ka -= kMagic;
    kb -= kMagic;
    double2 cs = __ldg(&T->ang[ia & (kAngTab - 1)]);
    double ex = __ldg(&T->ex[ib & (kExpTab - 1)]);
    ex = __hiloint2double(__double2hiint(ex) + ((ib >> 8) << 20), __double2loint(ex));
    double t = fma(-ka, 9.495469541415925e-13, fma(w.k, r.x, -(ka * 0.024543692605220713)));
    double v = fma(-kb, 1.6548911585192516e-12, fma(-w.k, r.y, -(kb * 0.002707606172407395)));
    if (abs(ia) > 326 && seed_range(r2)) {
        float er = seed_f32(fma(r.y, r.y, fma(-r.x, r.x, r2.x))), ei = seed_f32(fma(-2.0 * r.x, r.y, r2.y));
        float yr = seed_f32(y.x), yi = seed_f32(y.y), k = 0.5f * seed_f32(w.k);
        t += widen_f32(k * fmaf(-ei, yi, er * yr));
        v -= widen_f32(k * fmaf(ei, yr, er * yi));
    }
    double t2 = t * t;
    double sn = fma(t * t2, fma(t2, 1.0 / 120.0, -1.0 / 6.0), t);
    double cm = t2 * fma(t2, fma(t2, -1.0 / 720.0, 1.0 / 24.0), -0.5);
    double c = fma(-cs.y, sn, fma(cs.x, cm, cs.x)), s = fma(cs.x, sn, fma(cs.y, cm, cs.y));
    double e = v * fma(v, fma(v, fma(v, 1.0 / 24.0, 1.0 / 6.0), 0.5), 1.0);
    e = fma(ex, e, ex);
    return cd{e * c, e * s};
}

// (log |z|, arg z): c = 2^-e rad_j dir_k close to 1/z with log c tabulated (the
// products of the short table values are exact), d = z c - 1, |d| < 0.0037, and
// log(1 + d) = d (1 - d/2 + .. - d^5/6) (remainder below 2e-18), the polynomial
// with real coefficients by the two-term recurrence in 2 Re d and |d|^2.
__device__ __forceinline__ cd clog64(const PairTab* __restrict__ T, cd z) {
    if (!seed_range(z)) return clog_general(z);
    float a = seed_f32(z.x), b = seed_f32(z.y);
    float m2 = fmaf(a, a, b * b);
    unsigned mb = __float_as_uint(m2 * rsqrt_ap(m2));                     // |z|
    int e = (int)(mb >> 23) - 127, j = (mb >> 15) & (kLogRad - 1);
    int k = __float2int_rn(atan2f(b, a) * (kLogAng / 6.2831853f)) & (kLogAng - 1);
    double2 rad = __ldg(&T->lrad[j]), dir = __ldg(&T->ldir[k]), lg = __ldg(&T->llog[k]);
    double rs = __hiloint2double(__double2hiint(rad.x) - (e << 20), __double2loint(rad.x));
    double cr = rs * dir.x, ci = rs * dir.y;
    double dr = fma(-z.y, ci, fma(z.x, cr, -1.0)), di = fma(z.y, cr, z.x * ci);
    double s = dr + dr, v = fma(dr, dr, di * di);
    double b5 = -1.0 / 6.0, b4 = fma(s, b5, 1.0 / 5.0);
    double b3 = fma(-v, b5, fma(s, b4, -1.0 / 4.0)), b2 = fma(-v, b4, fma(s, b3, 1.0 / 3.0));
    double b1 = fma(-v, b3, fma(s, b2, -1.0 / 2.0));
    double qr = fma(-v, b2, fma(dr, b1, 1.0)), qi = di * b1;
    // e as a double: the bits of 2^52 + 2^31 + e
    double ed = __hiloint2double(0x43300000, (int)((unsigned)e ^ 0x80000000u)) - 4503601774854144.0;
    double ang = lg.y;
    // the angle table holds (-pi, pi]; cells around the cut keep the sign of Im z
    if (k == kLogAng / 2 && __double2hiint(z.y) < 0) ang -= 6.283185307179586476925;
    return cd{fma(ed, 0.69314718055994530942, (rad.y + lg.x) + fma(-di, qi, dr * qr)), ang + fma(di, qr, dr * qi)};
}

// H_nu(z) = e^{iz} z^{-1/2} g_nu(1/z), nu = 0, 1: g is smooth in s = 1/z away
// from the negative imaginary z axis, so its Taylor polynomial of degree 8 about
// the nearest grid point (step 1/64 up to |Re s|, |Im s| < 1/2, then 1/32 up to
// 1 and 1/16 up to 2: |z| > 1/2) leaves at most 4.8e-16 of g where -pi/4 <= arg z <=
// pi/2 (in 40 digits: 4.7e-16 at s = 0.0547 (1 + i), the sector's edge; 7e-17 at s =
// (1 + i)/128, 3e-18 at s = 1/128). Returns the cell of s and the offset from its centre,
// -1 outside.
__device__ __forceinline__ int hankel_cell(cd s, cd& ds) {
    int hx = __double2hiint(s.x), hy = __double2hiint(s.y);
    int m = max(hx & 0x7fffffff, hy & 0x7fffffff);
    int l = m < 0x3fe00000 ? 0 : m < 0x3ff00000 ? 1 : 2;
    // nearest grid point from the low bits of s + 1.5 2^(46 - l)
    const double magic = __hiloint2double(0x42d80000 + (l << 20), 0);
    double kx = s.x + magic, ky = s.y + magic;
    int ix = __double2loint(kx), iy = __double2loint(ky) + kHkNeg;
    ds.x = s.x - (kx - magic);
    ds.y = s.y - (ky - magic);
    bool in = m < 0x40000000 && (unsigned)ix < (unsigned)kHkNx && (unsigned)iy < (unsigned)kHkNy && hy <= hx;
    return in ? (l * kHkNy + iy) * kHkNx + ix : -1;
}
__device__ __forceinline__ cd hankel_factor(const double2* __restrict__ c, cd d) {
    double2 t = __ldg(c + kHkDeg);
    cd p = {t.x, t.y};
#pragma unroll
    for (int k = kHkDeg - 1; k >= 0; --k) {
        t = __ldg(c + k);
        p = cmac(cd{t.x, t.y}, p, d);
    }
    return p;
}

// Device pointer of the current device's tables (p2p.cu), constants of a wavenumber
const PairTab* pair_tab_device();
Wave make_wave(double kappa);

// Tables of the current device: the host part (make_pair_tab, p2p.cu) and the
// Hankel cells (k_pair_hankel).
void make_pair_tab(PairTab* T);

// Taylor coefficients of g_nu at the grid points from the Laplace-type integral
// (Watson, Treatise, Sec. 7.2; see cfmm_special.cuh)
//   g_nu(s) = c_nu int_0^inf e^{-u} u^{nu-1/2} (1 + i s u/2)^{nu-1/2} du,
//   c_0 = sqrt(2)/pi e^{-i pi/4}, c_1 = 2 sqrt(2)/pi e^{-3 i pi/4},
// differentiated under the integral; u = exp(x - e^{-x}) and the trapezoidal rule
// in x (Takahasi and Mori's double exponential rule), step 1/10: the branch point
// u = 2i/s is at least pi/4 from the real axis in log u, an error below 1e-20.
static __global__ void k_pair_hankel(PairTab* T) {
    int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= 2 * kHkGrids * kHkNx * kHkNy) return;
    int nu = id & 1, cell = id >> 1;
    int ix = cell % kHkNx, iy = cell / kHkNx % kHkNy, l = cell / (kHkNx * kHkNy);
    double h = ldexp(1.0, l - 6);
    cd s = {ix * h, (iy - kHkNeg) * h};
    cd sum[kHkDeg + 1], low[kHkDeg + 1];
    for (int k = 0; k <= kHkDeg; ++k) sum[k] = low[k] = cd{0, 0};
    for (int j = -42; j <= 46; ++j) {
        double x = 0.1 * j, em = exp(-x), u = exp(x - em);
        double w = 0.1 * (1.0 + em) * exp(-u) * sqrt(u) * (nu ? u : 1.0);
        cd p = {1.0 - 0.5 * s.y * u, 0.5 * s.x * u};
        if (p.x == 0.0 && p.y == 0.0) continue;    // a cell on the cut: never used
        cd r = csqrt_p(p), ip = cinv(p);
        cd f = w * (nu ? r : cinv(r));
        cd step = cd{0.0, 0.5 * u} * ip;
        for (int k = 0; k <= kHkDeg; ++k) {
            // two-sum: the coefficients come out correctly rounded but for the terms' own rounding
            double a = sum[k].x + f.x, bb = a - sum[k].x;
            low[k].x += (sum[k].x - (a - bb)) + (f.x - bb);
            sum[k].x = a;
            a = sum[k].y + f.y;
            bb = a - sum[k].y;
            low[k].y += (sum[k].y - (a - bb)) + (f.y - bb);
            sum[k].y = a;
            f = ((nu - 0.5 - k) / (k + 1.0)) * (f * step);
        }
    }
    // sqrt(2)/pi (1 -+ i)/sqrt(2) etc.: c_0 = (1 - i)/pi, c_1 = -2 (1 + i)/pi
    const double ipi = 0.31830988618379067154;
    for (int k = 0; k <= kHkDeg; ++k) {
        cd v = sum[k] + low[k];
        v = nu ? (-2.0 * ipi) * (v * cd{1.0, 1.0}) : ipi * (v * cd{1.0, -1.0});
        T->hk[cell][nu][k] = make_double2(v.x, v.y);
    }
}

}  // namespace cfmm
