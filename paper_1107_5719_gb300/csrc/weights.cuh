// Segment weights of the linear-in-tau source integral, FP64 and FP32 forms,
// shared by the formal-solution kernels (device code only).
//
// Over a segment of optical depth x the intensity gains
//   w_cur S(downstream) + w_up S(upstream),
//   w_cur = 1 - (1-e)/x,  w_up = (1-e)/x - e,  e = exp(-x),
// the exact integral of S(t) e^{-t} for S linear in t.  With
// phi2(z) = (e^z - 1 - z)/z^2 = sum_{n>=0} z^n/(n+2)!  these are
//   w_cur = x phi2(-x),  w_up = e x phi2(x),  e = 1 - x + x w_cur,
// and phi2(+-x) = E +- O with E = sum_j x^{2j}/(2j+2)!,
// O = x sum_j x^{2j}/(2j+3)!: a cancellation-free form for small x.
#pragma once

#include <cuda_runtime.h>

#include "exptable.cuh"

namespace rt3d {
namespace {

// ---- FP64 -----------------------------------------------------------------
//
// The FP64 pipe of GB300 issues about 2 DFMA per SM per clock, so the FP64
// weights are written to use few FP64 instructions; FP32 and integer ones
// are nearly free beside them.  A segment is taken together with the
// transmission T at its near end: b = T w_cur, g = T w_up, Tn = T e.
//
//  x < 1/2: the series phi2(-x) = sum_k (-x)^k/(k+2)! by Horner, its terms
//    below 2^-32 of the sum in FP32 (their rounding, 2^-22 of them, is below
//    the last bit of the FP64 result): from k = 3, 5, 6 or 9 on for x <
//    2^-9, 2^-5, 2^-3 or 1/2, so 3, 5, 6 or 9 FP64 operations (two series of
//    five in x^2 before).  Then, a = T x:  b = a phi2(-x),
//    Tn = (T - a) + x b,  g = (a - b) - x b: six more.  No exp call; against
//    50 digits, T = 1: 1.6e-16, 1.4e-16 and 2.6e-16 relative at most.
//  x >= 1/2: e^-x by a two-level form of Tang's table-driven method (ACM TOMS
//    15, 1989): -x = k ln2/65536 + r, |r| <= 5.3e-6, k = 65536 n + 256 j1 + j2,
//    e^-x = 2^n 2^{j1/256} 2^{j2/65536} (1 + r + r^2/2), the quadratic term
//    (1.4e-11) and the low part of k ln2/65536 in FP32; then q = (T - Tn)/x
//    from the reciprocal seed r0, x r0 = 1 - d, as (T - Tn) r0 (1 + d + d^2);
//    b = T - q, g = q - Tn: 14 operations for the three products.
//    Above x = 700 e is taken as 0 (it would scale I by < 1e-304).
//  Branch tests compare the high word of x (x >= 0) as an integer, so they
//    take no FP64 compare.

constexpr int kExpTable = 512;

// tab[j] = 2^{j/256}, tab[256 + j] = 2^{j/65536} (call from every thread, then
// __syncthreads())
__device__ const exptable::Table64 g_exp_table = exptable::table64();

__device__ __forceinline__ void fill_exp_table(double* tab)
{
    for (int j = threadIdx.x; j < kExpTable; j += blockDim.x) tab[j] = __ldg(&g_exp_table.v[j]);
}

// The leading 24 bits of x >= 0, x < 2^127 (below 2^-126: 2^-126 or a little
// more), and a positive normal float as a double, both on the integer pipe.
__device__ __forceinline__ float lead_float(double x)
{
    const int hi = max(__double2hiint(x), 0x38100000) - 0x38000000;
    return __int_as_float((int)__funnelshift_l((unsigned)__double2loint(x), (unsigned)hi, 3));
}

__device__ __forceinline__ double pos_double(float f)
{
    const unsigned u = __float_as_uint(f);
    return __hiloint2double((int)(u >> 3) + 0x38000000, (int)(u << 29));
}

// T e^{-x}, 1e-3 < x <= 700
__device__ __forceinline__ double exp_neg_times(double T, double x, const double* __restrict__ tab)
{
    constexpr double kMagic = 6755399441055744.0;        // 1.5 * 2^52: round to integer
    constexpr double kInvL = 94548.4621996991;            // 65536 / ln 2
    constexpr double kL1 = 1.0576586617430806e-05;        // ln2/65536, leading part
    constexpr float kL2 = 3.345677e-17f;                  // (ln2/65536 - kL1) 65536/ln2
    const double t = fma(-x, kInvL, kMagic);
    const int k = __double2loint(t);                      // round(-65536 x / ln2)
    const double r = fma(-(t - kMagic), kL1, -x);
    const float rf = lead_float(fabs(r));
    const double u = r + pos_double(fmaf(0.5f * rf, rf, kL2 * lead_float(x)));
    // 2^n into the exponent field of the first factor (normal for x <= 700)
    const double t1 = tab[(k >> 8) & 255];
    const double m = T * __hiloint2double(__double2hiint(t1) + (k >> 16) * (1 << 20), __double2loint(t1)) *
                     tab[256 + (k & 255)];
    return fma(m, u, m);
}

// n / x from the hardware reciprocal seed (20 bits), x > 0 normal
__device__ __forceinline__ double div_seed(double n, double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double d = fma(-x, r, 1.0);
    const double q = n * r;
    return fma(q, fma(d, d, d), q);
}

constexpr int kHi2m9 = 0x3F600000;       // high words of 2^-9,
constexpr int kHi2m5 = 0x3FA00000;       // 2^-5,
constexpr int kHi2m3 = 0x3FC00000;       // 2^-3,
constexpr int kHiQuarter = 0x3FD00000;   // 1/4,
constexpr int kHiHalf = 0x3FE00000;      // 1/2
constexpr int kHi700 = 0x4085E000;       // and 700

// phi2(-x), x < 1/2; hx the high word of x
__device__ __forceinline__ double phi2_neg64(double x, int hx)
{
    const float xf = lead_float(x);
    double r;
    if (hx < kHi2m9) {
        r = pos_double(fmaf(-xf, fmaf(-xf, 1.0f / 5040, 1.0f / 720), 1.0f / 120));
    } else {
        if (hx < kHi2m5) {
            r = pos_double(fmaf(-xf, fmaf(-xf, 1.0f / 362880, 1.0f / 40320), 1.0f / 5040));
        } else {
            if (hx < kHi2m3) {
                r = pos_double(fmaf(-xf, fmaf(-xf, 1.0f / 3628800, 1.0f / 362880), 1.0f / 40320));
            } else {
                r = pos_double(fmaf(-xf, fmaf(-xf, fmaf(-xf, fmaf(-xf, 1.0f / 1307674368000.0f,
                                                                   1.0f / 87178291200.0f),
                                                        1.0f / 6227020800.0f),
                                              1.0f / 479001600), 1.0f / 39916800));
                r = fma(-x, r, 1.0 / 3628800);
                r = fma(-x, r, 1.0 / 362880);
                r = fma(-x, r, 1.0 / 40320);
            }
            r = fma(-x, r, 1.0 / 5040);
        }
        r = fma(-x, r, 1.0 / 720);
        r = fma(-x, r, 1.0 / 120);
    }
    r = fma(-x, r, 1.0 / 24);
    r = fma(-x, r, 1.0 / 6);
    return fma(-x, r, 0.5);
}

// b = T w_cur, g = T w_up, Tn = T e of a segment of optical depth x
__device__ __forceinline__ void seg_step64(double T, double x, const double* __restrict__ tab, double& b,
                                           double& g, double& Tn)
{
    const int hx = __double2hiint(x);
    if (hx < kHiHalf) {
        const double a = T * x;
        b = a * phi2_neg64(x, hx);
        Tn = fma(x, b, T - a);
        g = fma(-x, b, a - b);
    } else {
        Tn = hx < kHi700 ? exp_neg_times(T, x, tab) : 0.0;
        const double q = div_seed(T - Tn, x);
        b = T - q;
        g = q - Tn;
    }
}

__device__ __forceinline__ void seg_weights64(double x, const double* __restrict__ tab, double& wc,
                                              double& wu, double& e)
{
    seg_step64(1.0, x, tab, wc, wu, e);
}

// Cutoff test on exponent fields only (integer pipe).  With T < 2^(eT+1),
// smax < 2^(es+1), |I| >= 2^eI and cut >= 2^-lc (lc = ceil(-log2 cut)),
// eI - eT >= es + lc + 2 guarantees T * smax <= cut * |I|, i.e. the rest of
// the characteristic changes I by at most cut * |I|.  `need` = es + lc + 2.
__device__ __forceinline__ bool cut_now(double T, double I, int need)
{
    const int eT = (__double2hiint(T) >> 20) & 0x7ff;
    const int eI = (__double2hiint(I) >> 20) & 0x7ff;
    return eI - eT >= need;
}

__device__ __forceinline__ int cut_need(double smax, double cut)
{
    // cut <= 0 disables the test (need larger than any exponent gap)
    if (!(cut > 0.0)) return 4096;       // never cut
    if (!(smax > 0.0)) return -4096;     // S = 0 and no boundary intensity: I = 0 exactly
    const int es = ((__double2hiint(smax) >> 20) & 0x7ff) - 1023;
    const int lc = (int)ceil(-log2(cut));
    return es + lc + 2;
}

// ---- FP32 -----------------------------------------------------------------
//
//  x < 2: phi2(+-x) = E(z) +- x Q(z) with E, Q degree-4 polynomials in
//  z = x^2 fitted on z in [0, 4] for the least maximum relative error
//  (fit_weights32.py: 1.9e-8 for E, 3.0e-8 for Q with the coefficients
//  rounded to FP32, against 2e-9 truncation for seven Taylor terms each);
//  x >= 2: closed form (1-e loses nothing there).  e from the MUFU ex2.
__device__ __forceinline__ float ex2_approx(float y)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
    return r;
}

__device__ __forceinline__ float rcp_approx(float y)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
    return r;
}

// E(z) and Q(z), z = x^2 < 4: phi2(+-x) = E +- x Q
__device__ __forceinline__ void phi2_eq32(float z, float& E, float& Q)
{
    E = fmaf(fmaf(fmaf(2.968770900e-07f, z, 2.472764936e-05f), z, 1.388992299e-03f), z,
             4.166661575e-02f);
    E = fmaf(E, z, 0.5f);
    Q = fmaf(fmaf(fmaf(2.669341548e-08f, z, 2.749998430e-06f), z, 1.984207920e-04f), z,
             8.333329111e-03f);
    Q = fmaf(Q, z, 1.666666716e-01f);
}

// E = phi2 even part, O = odd part at x < 2 (phi2(+-x) = E +- O)
__device__ __forceinline__ void phi2_parts32(float x, float& E, float& O)
{
    float Q;
    phi2_eq32(x * x, E, Q);
    O = Q * x;
}

__device__ __forceinline__ void seg_weights32(float x, float& wc, float& wu, float& e)
{
    constexpr float kLog2e = 1.4426950408889634f;
    e = ex2_approx(-x * kLog2e);
    if (x < 2.0f) {
        float E, O;
        phi2_parts32(x, E, O);
        wc = x * (E - O);
        wu = (x * e) * (E + O);
    } else {
        const float q = (1.0f - e) * rcp_approx(x);
        wc = 1.0f - q;
        wu = q - e;
    }
}

}  // namespace
}  // namespace rt3d
