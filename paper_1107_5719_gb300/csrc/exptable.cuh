// Powers of two with fractional exponents, for the tables of the segment
// weights: formed at compile time in pairs of doubles (the error-free sums and
// products of Knuth and Dekker), so correct to the last bit of the double they
// are rounded to.  A block copies its table from here: formed with exp2 and
// expm1 in every block, the tables took most of the time of a kernel whose
// blocks have few rays (k_sc_rec of 40 x 30 x 26 voxels x 234 directions,
// three or four rays a block: 373 us, 70 from here).
#pragma once

namespace rt3d {
namespace exptable {

struct dd {
    double h, l;
};

constexpr dd two_sum(double a, double b)
{
    const double s = a + b, bb = s - a;
    return dd{s, (a - (s - bb)) + (b - bb)};
}

constexpr dd halves(double a)
{
    const double t = 134217729.0 * a, h = t - (t - a);      // 2^27 + 1
    return dd{h, a - h};
}

constexpr dd mul(dd a, dd b)
{
    const double p = a.h * b.h;
    const dd x = halves(a.h), y = halves(b.h);
    const double e = ((x.h * y.h - p) + x.h * y.l + x.l * y.h) + x.l * y.l;
    return two_sum(p, e + (a.h * b.l + a.l * b.h));
}

constexpr dd add(dd a, dd b)
{
    const dd s = two_sum(a.h, b.h);
    return two_sum(s.h, s.l + (a.l + b.l));
}

// a / n
constexpr dd over(dd a, double n)
{
    const double q = a.h / n;
    const dd p = mul(dd{q, 0.0}, dd{n, 0.0});
    return two_sum(q, (((a.h - p.h) - p.l) + a.l) / n);
}

// 2^x, 0 <= x <= 1/2: sum of (x ln 2)^k / k!
constexpr dd pow2(double x)
{
    const dd y = mul(dd{0.69314718055994530942, 2.3190468138462995584e-17}, dd{x, 0.0});
    dd r{1.0, 0.0};
    for (int k = 24; k > 0; --k) r = add(dd{1.0, 0.0}, over(mul(y, r), k));
    return r;
}

// v[j] = 2^{j / scale}, j < 256, from the powers of the eight bits of j
struct Powers {
    dd v[256];
};
constexpr Powers powers(double scale)
{
    Powers p{};
    p.v[0] = dd{1.0, 0.0};
    for (int bit = 0; bit < 8; ++bit) {
        const int n = 1 << bit;
        const dd f = pow2(n / scale);
        for (int j = 0; j < n; ++j) p.v[n + j] = mul(p.v[j], f);
    }
    return p;
}

// FP64: 2^{j/256}, then 2^{j/65536}
struct Table64 {
    double v[512];
};
constexpr Table64 table64()
{
    const Powers a = powers(256.0), b = powers(65536.0);
    Table64 t{};
    for (int j = 0; j < 256; ++j) {
        t.v[j] = a.v[j].h;
        t.v[256 + j] = b.v[j].h;
    }
    return t;
}

// Double-float: 2^{-j/256}, then 1 - 2^{-j/256}, as pairs of floats
struct TableDF {
    float v[512][2];
};
constexpr TableDF table_df()
{
    const Powers a = powers(256.0);
    TableDF t{};
    for (int j = 0; j < 256; ++j) {
        const dd e = j == 0 ? dd{1.0, 0.0} : dd{0.5 * a.v[256 - j].h, 0.5 * a.v[256 - j].l};
        const dd c = add(dd{1.0, 0.0}, dd{-e.h, -e.l});
        t.v[j][0] = (float)e.h;
        t.v[j][1] = (float)((e.h - (double)t.v[j][0]) + e.l);
        t.v[256 + j][0] = (float)c.h;
        t.v[256 + j][1] = (float)((c.h - (double)t.v[256 + j][0]) + c.l);
    }
    return t;
}

}  // namespace exptable
}  // namespace rt3d
