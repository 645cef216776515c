// Segment weights and bilinear interpolation in double-float (df.cuh), shared
// by the double-float kernels (device code only).
#pragma once

#include "df.cuh"
#include "exptable.cuh"

namespace rt3d {
namespace {

constexpr int kExpTableDF = 256;

// tab[j] = 2^{-j/256} and tab[256 + j] = 1 - 2^{-j/256} (accurate relative to
// itself), as double-float pairs (call from all threads, then sync)
__device__ const exptable::TableDF g_exp_table_df = exptable::table_df();

__device__ __forceinline__ void fill_exp_table_df(dfl* tab)
{
    for (int j = threadIdx.x; j < 2 * kExpTableDF; j += blockDim.x)
        tab[j] = dfl{__ldg(&g_exp_table_df.v[j][0]), __ldg(&g_exp_table_df.v[j][1])};
}

// e^{-x} and 1 - e^{-x} for 0.05 <= x <= 80 (Tang's table-driven method in
// double-float): k = round(256 x / ln2), m = k >> 8, j = k & 255,
// r = x - k ln2/256 (|r| <= 1.4e-3, ln2/256 split into three floats as in
// Cody & Waite, the products formed exactly), p = e^{-r} - 1 =
// -r + r^2/2 - r^3 (1/6 - r/24) (the cubic and quartic terms in FP32,
// < 5e-10), and with t = 2^{-m} 2^{-j/256}:
//   e = t + t p,   1 - e = (1 - t) - t p.
// For m = 0 the factor 1 - t comes from its own table (1 - e would
// otherwise inherit the table's rounding relative to e, which cancels);
// for m >= 1, t <= 1/2 and 1 - t loses nothing.
__device__ __forceinline__ void exp_neg_df(dfl x, const dfl* __restrict__ tab, dfl& e, dfl& om)
{
    constexpr float kInvL = 369.3299255371094f;          // 256 / ln 2 (rounding only)
    constexpr float kL1 = 0.0027076061815023422f;         // ln2/256 = kL1 + kL2 + kL3
    constexpr float kL2 = -7.440055516116928e-12f;
    constexpr float kL3 = -3.4309311478864607e-19f;
    const float k = rintf(x.h * kInvL);
    dfl r = df_add_s(x, df_neg(two_prod(k, kL1)));
    r = df_add_s(r, df_neg(two_prod(k, kL2)));
    r = df_add_f(r, -k * kL3);
    const dfl r2 = df_mul(r, r);
    const float tail = r2.h * r.h * fmaf(-r.h, 1.0f / 24.0f, 1.0f / 6.0f);
    const dfl p = df_add_s(df_neg(r), df_add_f(df_scale(r2, 0.5f), -tail));
    const int ki = (int)k;
    const int m = ki >> 8, j = ki & (kExpTableDF - 1);
    const float sc = __int_as_float((127 - m) << 23);   // 2^-m, normal for x <= 80
    const dfl t = df_scale(tab[j], sc);
    const dfl tp = df_mul(t, p);
    const dfl c = m == 0 ? tab[kExpTableDF + j] : df_add_f(df_neg(t), 1.0f);
    e = df_add_s(t, tp);
    om = df_sub_s(c, tp);
}

// c - x r, |x r| < |c|, r and the result unnormalised pairs (the low part a
// few units of 2^-24 of the high one)
__device__ __forceinline__ dfl horner_df(dfl x, dfl r, float ch, float cl)
{
    const dfl p = two_prod(x.h, r.h);
    const float pl = fmaf(x.l, r.h, fmaf(x.h, r.l, p.l));
    const float s = ch - p.h;
    return dfl{s, ((ch - s) - p.h) + (cl - pl)};
}

// phi2(-x) = sum_k (-x)^k/(k+2)!, x < 1/2, by Horner; the terms below 2^-28 of
// the sum in FP32 (their rounding is below 2^-52): from k = 3, 4 or 8 on.
__device__ __forceinline__ dfl phi2_neg_df(dfl x)
{
    const float f = -x.h;
    dfl r;
    if (x.h < 0.03125f) {
        if (x.h < 0.001953125f) {
            r = dfl{fmaf(f, fmaf(f, 1.0f / 5040, 1.0f / 720), 1.0f / 120), 0.f};
        } else {
            r = dfl{fmaf(f, fmaf(f, fmaf(f, 1.0f / 362880, 1.0f / 40320), 1.0f / 5040), 1.0f / 720), 0.f};
            r = horner_df(x, r, 0.00833333377f, -4.34617203e-10f);
        }
    } else {
        r = dfl{fmaf(f, fmaf(f, fmaf(f, fmaf(f, 1.0f / 87178291200.0f, 1.0f / 6227020800.0f),
                                     1.0f / 479001600), 1.0f / 39916800), 1.0f / 3628800), 0.f};
        r = horner_df(x, r, 2.75573188e-06f, 3.79357122e-14f);
        r = horner_df(x, r, 2.48015876e-05f, -3.40699609e-13f);
        r = horner_df(x, r, 0.000198412701f, -2.72559687e-12f);
        r = horner_df(x, r, 0.00138888892f, -3.36310944e-11f);
        r = horner_df(x, r, 0.00833333377f, -4.34617203e-10f);
    }
    r = horner_df(x, r, 0.0416666679f, -1.24176347e-09f);
    r = horner_df(x, r, 0.166666672f, -4.96705388e-09f);
    r = horner_df(x, r, 0.5f, 0.f);
    return quick_two_sum(r.h, r.l);
}

// (a - b) + c with |a| >= |b|, |a - b| >= |c|
__device__ __forceinline__ dfl sub_add_df(dfl a, dfl b, dfl c)
{
    const dfl s = quick_two_sum(a.h, -b.h);
    const dfl u = quick_two_sum(s.h, c.h);
    return quick_two_sum(u.h, ((a.l - b.l) + s.l) + (c.l + u.l));
}

// A segment of optical depth x with the transmission T at its near end:
// b = T w_cur, g = T w_up, Tn = T e (definitions as weights.cuh).  Below
// x = 1/2 from the series, a = T x: b = a phi2(-x), Tn = (T - a) + x b,
// g = (a - b) - x b, about 100 FP32 operations and half of what the
// exponential and the division of the closed form take.
__device__ __forceinline__ void seg_step_df(dfl T, dfl x, const dfl* __restrict__ tab, dfl& b, dfl& g,
                                            dfl& Tn)
{
    if (x.h < 0.5f) {
        const dfl a = df_mul(T, x);
        b = df_mul(a, phi2_neg_df(x));
        dfl xb = two_prod(x.h, b.h);
        xb.l = fmaf(x.l, b.h, fmaf(x.h, b.l, xb.l));
        Tn = sub_add_df(T, a, xb);
        g = sub_add_df(a, b, df_neg(xb));
    } else {
        dfl e, om;
        if (x.h <= 80.0f) {
            exp_neg_df(x, tab, e, om);
        } else {
            e = df_make(0.f, 0.f);
            om = df_make(1.f, 0.f);
        }
        // q = om / x: FP32 quotient and two corrections from the residual
        // (one leaves a relative error near 2^-44, amplified in 1 - q)
        const dfl q = df_div_s(om, x);
        b = df_mul(T, df_add_f(df_neg(q), 1.0f));
        g = df_mul(T, df_sub_s(q, e));
        Tn = df_mul(T, e);
    }
}

// The same for T = 1: w_cur, w_up, e.
__device__ __forceinline__ void seg_weights_df(dfl x, const dfl* __restrict__ tab, dfl& wc, dfl& wu,
                                               dfl& e)
{
    seg_step_df(df_make(1.f, 0.f), x, tab, wc, wu, e);
}

// Bilinear interpolation of a double-float field: sum of four df products
// with the TwoProduct errors and cross terms gathered in one FP32 term.
__device__ __forceinline__ dfl bilin_df(float4 wh, float4 wl, float ah, float al, float bh, float bl,
                                        float ch, float cl, float dh, float dl)
{
    const dfl p0 = two_prod(wh.x, ah), p1 = two_prod(wh.y, bh), p2 = two_prod(wh.z, ch),
              p3 = two_prod(wh.w, dh);
    float err = p0.l + p1.l + p2.l + p3.l;
    err = fmaf(wh.x, al, err); err = fmaf(wh.y, bl, err); err = fmaf(wh.z, cl, err);
    err = fmaf(wh.w, dl, err);
    err = fmaf(wl.x, ah, err); err = fmaf(wl.y, bh, err); err = fmaf(wl.z, ch, err);
    err = fmaf(wl.w, dh, err);
    dfl s = two_sum(p0.h, p1.h);
    dfl t = two_sum(p2.h, p3.h);
    dfl u = two_sum(s.h, t.h);
    err += s.l + t.l + u.l;
    return quick_two_sum(u.h, err);
}

}  // namespace
}  // namespace rt3d
