// Taylor coefficients of w(z) = exp(-z^2) erfc(-i z) at the nodes of a grid
// over 0 <= x <= 10, -1.48 <= y <= 10, computed on the host in double-double
// arithmetic so that the rounded coefficients are correct to the last place or
// so.  (No physical damping lies below 0, but callers' own parameters and
// per-pixel bounds may.  Weideman's series, which FP64 takes elsewhere, is 5e-7
// from w at y = -1.5 and 4e-4 at -2, no better than the expansions of the last
// row.)
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

constexpr int kNodeGrid = 129;            // nodes per axis from 0 on
constexpr int kNodeBelow = 19;            // rows below y = 0
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

namespace nodes {

// w at the top node of the imaginary axis.
inline CDD axis_top()
{
    const double y = (kNodeGrid - 1) * kNodeStep;
    DD t = {y, 0.0};
    for (int m = 300; m >= 1; --m) t = add({y, 0.0}, div({0.5 * m, 0.0}, t));
    return {div({0x1.20dd750429b6dp-1, 0x1.1ae3a914fed80p-57}, t), {0.0, 0.0}};  // 1 / sqrt(pi) / t
}

// w at the axis node one row down from its expansion c: step -i h.
inline CDD axis_down(const CDD c[kTerms])
{
    CDD w = c[kTerms - 1];
    for (int n = kTerms - 2; n >= 0; --n)
        w = {add(c[n].re, scale(w.im, kNodeStep)), add(c[n].im, scale(w.re, -kNodeStep))};
    return w;
}

// The nodes of row iy from w on the axis, which moves one row down.
inline void row(int iy, CDD &axis, double *o)
{
    CDD c[kTerms], w = axis;
    for (int ix = 0; ix < kNodeGrid; ++ix, o += kNodeCoef * 2) {
        taylor(ix * kNodeStep, iy * kNodeStep, w, c);
        for (int n = 0; n < kNodeCoef; ++n) {
            o[2 * n] = c[n].re.hi;
            o[2 * n + 1] = c[n].im.hi;
        }
        if (ix == 0) axis = axis_down(c);
        w = c[kTerms - 1];  // the next node of the row: step h
        for (int n = kTerms - 2; n >= 0; --n)
            w = {add(c[n].re, scale(w.re, kNodeStep)), add(c[n].im, scale(w.im, kNodeStep))};
    }
}

}  // namespace nodes

constexpr int kNodeRow = kNodeGrid * kNodeCoef * 2;  // doubles in a row of nodes

// Row (iy, ix) holds (re, im) of c_0 .. c_10 at z = ix step + i iy step.  At
// most half a step away on each axis the first omitted term is below 5e-17.
inline std::vector<double> faddeeva_nodes()
{
    std::vector<double> out((size_t)kNodeGrid * kNodeRow);
    nodes::CDD axis = nodes::axis_top();
    for (int iy = kNodeGrid - 1; iy >= 0; --iy) nodes::row(iy, axis, &out[(size_t)iy * kNodeRow]);
    return out;
}

// The kNodeBelow rows below, y = -kNodeBelow step first.  w grows like 2
// exp(-z^2) there, and so does an error, so the relative accuracy stays; the
// expansions stay within 1e-13 |w|, 1e-14 down to y = -1.
inline std::vector<double> faddeeva_nodes_below()
{
    std::vector<double> out((size_t)kNodeBelow * kNodeRow);
    nodes::CDD axis = nodes::axis_top(), c[nodes::kTerms];
    for (int iy = kNodeGrid - 1; iy >= 0; --iy) {
        nodes::taylor(0.0, iy * kNodeStep, axis, c);
        axis = nodes::axis_down(c);
    }
    for (int iy = -1; iy >= -kNodeBelow; --iy) nodes::row(iy, axis, &out[(size_t)(iy + kNodeBelow) * kNodeRow]);
    return out;
}

}  // namespace genesis
