// Taylor coefficients of w(z) = exp(-z^2) erfc(-i z) at the nodes of a grid
// over 0 <= x, y <= 10, computed on the host in double-double arithmetic so
// that the rounded coefficients are correct to the last place or so.
//
// From w' = -2 z w + 2 i / sqrt(pi) the coefficients c_n = w^(n) / n! obey
// c_{n+1} = -2 (z c_n + c_{n-1}) / (n + 1), n >= 1.  The first node is z = 10 i,
// by the Laplace continued fraction; the others follow by Taylor steps, down
// the imaginary axis and then outward along x.  In both directions an error,
// which evolves like exp(-z^2), shrinks against w, so the steps are stable.
#pragma once

#include <cmath>
#include <vector>

namespace genesis {

constexpr int kNodeGrid = 129;            // nodes per axis
constexpr double kNodeStep = 0.078125;    // 10 / 128, exact
constexpr int kNodeCoef = 11;             // coefficients kept per node

namespace nodes {

// Double-double: the unevaluated sum hi + lo (Dekker 1971).  No FMA and no
// wider type, so every host gives the same bits.
struct DD {
    double hi, lo;
};
inline DD quick(double a, double b)
{
    const double s = a + b;
    return {s, b - (s - a)};
}
inline DD add(DD a, DD b)
{
    const double s = a.hi + b.hi, v = s - a.hi;
    return quick(s, (a.hi - (s - v)) + (b.hi - v) + a.lo + b.lo);
}
inline DD mul(DD a, DD b)
{
    const double p = a.hi * b.hi;
    const double ca = 134217729.0 * a.hi, cb = 134217729.0 * b.hi;
    const double ah = ca - (ca - a.hi), bh = cb - (cb - b.hi), al = a.hi - ah, bl = b.hi - bh;
    const double e = ((ah * bh - p) + ah * bl + al * bh) + al * bl;
    return quick(p, e + (a.hi * b.lo + a.lo * b.hi));
}
inline DD neg(DD a) { return {-a.hi, -a.lo}; }
inline DD scale(DD a, double f) { return mul(a, {f, 0.0}); }
inline DD div(DD a, DD b)
{
    const double q1 = a.hi / b.hi;
    DD r = add(a, neg(scale(b, q1)));
    const double q2 = r.hi / b.hi;
    r = add(r, neg(scale(b, q2)));
    return add(quick(q1, q2), {r.hi / b.hi, 0.0});
}

struct CDD {
    DD re, im;
};
constexpr int kTerms = 24;  // terms of a step: the first omitted is below 1e-34

// c_0 .. c_{kTerms-1} at z = x + i y from w = w(z).
inline void taylor(double x, double y, CDD w, CDD c[kTerms])
{
    const DD two_isp = {0x1.20dd750429b6dp+0, 0x1.1ae3a914fed80p-56};  // 2 / sqrt(pi)
    auto zmul = [&](CDD a) {
        return CDD{add(scale(a.re, x), scale(a.im, -y)), add(scale(a.re, y), scale(a.im, x))};
    };
    c[0] = w;
    CDD t = zmul(w);
    c[1] = {scale(t.re, -2.0), add(scale(t.im, -2.0), two_isp)};
    for (int n = 1; n + 1 < kTerms; ++n) {
        t = zmul(c[n]);
        const DD d = {n + 1.0, 0.0};
        c[n + 1] = {div(scale(add(t.re, c[n - 1].re), -2.0), d), div(scale(add(t.im, c[n - 1].im), -2.0), d)};
    }
}

}  // namespace nodes

// Row (iy, ix) holds (re, im) of c_0 .. c_10 at z = ix step + i iy step.  At
// most half a step away on each axis the first omitted term is below 5e-17.
inline std::vector<double> faddeeva_nodes()
{
    using namespace nodes;
    std::vector<double> out((size_t)kNodeGrid * kNodeGrid * kNodeCoef * 2);
    CDD c[kTerms], axis;
    {
        const double y = (kNodeGrid - 1) * kNodeStep;
        DD t = {y, 0.0};
        for (int m = 300; m >= 1; --m) t = add({y, 0.0}, div({0.5 * m, 0.0}, t));
        axis = {div({0x1.20dd750429b6dp-1, 0x1.1ae3a914fed80p-57}, t), {0.0, 0.0}};  // 1 / sqrt(pi) / t
    }
    for (int iy = kNodeGrid - 1; iy >= 0; --iy) {
        CDD w = axis;
        for (int ix = 0; ix < kNodeGrid; ++ix) {
            taylor(ix * kNodeStep, iy * kNodeStep, w, c);
            double *o = &out[((size_t)iy * kNodeGrid + ix) * kNodeCoef * 2];
            for (int n = 0; n < kNodeCoef; ++n) {
                o[2 * n] = c[n].re.hi;
                o[2 * n + 1] = c[n].im.hi;
            }
            if (ix == 0 && iy > 0) {  // the axis node one row down: step -i h
                axis = c[kTerms - 1];
                for (int n = kTerms - 2; n >= 0; --n)
                    axis = {add(c[n].re, scale(axis.im, kNodeStep)), add(c[n].im, scale(axis.re, -kNodeStep))};
            }
            w = c[kTerms - 1];  // the next node of the row: step h
            for (int n = kTerms - 2; n >= 0; --n)
                w = {add(c[n].re, scale(w.re, kNodeStep)), add(c[n].im, scale(w.im, kNodeStep))};
        }
    }
    return out;
}

}  // namespace genesis
