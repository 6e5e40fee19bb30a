// FP64 Voigt and Faraday-Voigt profiles of one model at all its wavelength
// points and Zeeman components, evaluated by a whole block (sm_103a).
//
// FP64 work is bound by the FP64 pipe, which takes 16 clocks of an SM per
// warp instruction, however many lanes are active.  What counts is the number
// of FP64 warp instructions per profile value, so:
//  * The damping a is the same at every point of a model, so near the line
//    cores w(x + i a) is a function of x alone.  For |x| < 10 it comes from
//    Taylor polynomials of degree 14 about 32 cell centres (cells of width
//    0.3125 in |x|; w(-x + i a) is the conjugate): 29 operations instead of
//    the 105 of Weideman's series.  The 32 lanes of one warp build the table,
//    a cell each: w at the centre from the Taylor coefficients of the nearest
//    node of a fixed grid (faddeeva_nodes.h; a step along i of at most 0.04)
//    and the further coefficients by c_{n+1} = -2 (z c_n + c_{n-1}) / (n + 1)
//    (from w' = -2 z w + 2 i / sqrt(pi)).  The first omitted term is below
//    6e-17.  Measured against 40-digit values the table is within 2e-16 of w;
//    Weideman's series with N = 36, used for |z| <= 8 elsewhere in FP64, is
//    within 1.5e-15 (the rounding of its long recurrence).
//  * Beyond |z|^2 = 100 the convergents of the Laplace continued fraction are
//    written in s = |z|^2 for real x (w = y P(s) / D(s) + i x Q(s) / D(s) up to
//    1 / sqrt(pi), real polynomials whose coefficients depend on a^2 alone and
//    are formed once per model): the 9th to |z|^2 = 170, the 7th to 500, the
//    5th beyond, 23 to 35 operations where the 9th in complex arithmetic
//    takes 56.  Each is within 4e-17 of w in its region.
//  * Points of one region are gathered into lists, block-wide, so that every
//    warp runs one branch with (nearly) all its lanes.
#pragma once

#include "faddeeva_nodes.h"
#include "fp64_util.cuh"
#include "kernels.h"

namespace genesis {

constexpr int kProfBlock = 128;   // threads per block, one wavelength each per pass
constexpr int kProfComps = 16;    // Zeeman components per pass
constexpr int kProfMaxComp = ME_MAX_LINES * (3 * ME_MAX_COMP + 1);  // field-free profiles included
constexpr int kCells = 32;
constexpr double kCellWidth = 0.3125;
constexpr int kTaylor = 14;  // degree

// Polynomials in s and Y = y^2 for the K-th convergent: with a(u), b(u) of
// CfPoly (u = z^2), i z b(u) conj(a(u)) = y P + i x Q and |a(u)|^2 = D, from
// u = p + i q, p = s - 2 Y, q = 2 x y and the recurrences of Re u^k and
// Im u^k / q in p and u conj(u) = s^2.
struct Poly2 {
    double c[12][7];  // c[i][j] s^i Y^j
    constexpr Poly2() : c() {}
    constexpr void add(const Poly2 &o, double f)
    {
        for (int i = 0; i < 12; ++i)
            for (int j = 0; j < 7; ++j) c[i][j] += f * o.c[i][j];
    }
    // this += f s^ds Y^dY o
    constexpr void add_shifted(const Poly2 &o, double f, int ds, int dY)
    {
        for (int i = 0; i + ds < 12; ++i)
            for (int j = 0; j + dY < 7; ++j) c[i + ds][j + dY] += f * o.c[i][j];
    }
};
template <int K> struct CfReal {
    Poly2 P, Q, D;
    constexpr CfReal() : P(), Q(), D()
    {
        constexpr CfPoly<K> cf{};
        constexpr int NA = (K + 1) / 2, NB = (K - 1) / 2;
        Poly2 re[NA + 1], im[NA + 1];  // Re u^k, Im u^k / q
        re[0].c[0][0] = 1.0;
        re[1].c[1][0] = 1.0;
        re[1].c[0][1] = -2.0;
        im[1].c[0][0] = 1.0;
        for (int k = 1; k < NA; ++k) {
            re[k + 1].add_shifted(re[k], 2.0, 1, 0);
            re[k + 1].add_shifted(re[k], -4.0, 0, 1);
            re[k + 1].add_shifted(re[k - 1], -1.0, 2, 0);
            im[k + 1].add_shifted(im[k], 2.0, 1, 0);
            im[k + 1].add_shifted(im[k], -4.0, 0, 1);
            im[k + 1].add_shifted(im[k - 1], -1.0, 2, 0);
        }
        Poly2 E, F;  // b conj(a) = E + i q F
        for (int m = 0; m <= NB; ++m)
            for (int n = 0; n <= NA; ++n) {
                const int lo = m < n ? m : n, d = m < n ? n - m : m - n;
                E.add_shifted(re[d], cf.b[m] * cf.a[n], 2 * lo, 0);
                F.add_shifted(im[d], (m > n ? 1.0 : -1.0) * cf.b[m] * cf.a[n], 2 * lo, 0);
            }
        for (int m = 0; m <= NA; ++m)
            for (int n = 0; n <= NA; ++n) {
                const int lo = m < n ? m : n, d = m < n ? n - m : m - n;
                D.add_shifted(re[d], cf.a[m] * cf.a[n], 2 * lo, 0);
            }
        P.add(E, -1.0);                  // P = -(2 (s - Y) F + E)
        P.add_shifted(F, -2.0, 1, 0);
        P.add_shifted(F, 2.0, 0, 1);
        Q.add(E, 1.0);                   // Q = E - 2 Y F
        Q.add_shifted(F, -2.0, 0, 1);
    }
};

// Rows of the coefficients of 5th, 7th and 9th: P_0..P_K, Q_0..Q_K, D_0..D_K
// (D's leading coefficient is 1), each a polynomial in Y of degree <= 5.
constexpr int kExtRows = 3 * (6 + 8 + 10);
struct ExtTable {
    double c[kExtRows][6];
    template <int K> constexpr int fill(int row)
    {
        constexpr CfReal<K> r{};
        for (int part = 0; part < 3; ++part)
            for (int i = 0; i <= K; ++i, ++row)
                for (int j = 0; j < 6; ++j) c[row][j] = (part == 0 ? r.P : part == 1 ? r.Q : r.D).c[i][j];
        return row;
    }
    constexpr ExtTable() : c() { fill<9>(fill<7>(fill<5>(0))); }
};
static __device__ const ExtTable d_ext{};

// First row and first coefficient of the K-th convergent in ExtTable's order.
template <int K> constexpr int kExtFirst = K == 5 ? 0 : K == 7 ? 18 : 42;

// Everything a block holds for one model.
struct ProfShared {
    double2 cell[kCells * (kTaylor + 1)];  // Taylor coefficients (re, im) of a cell, ascending
    double2 ext[kExtRows / 2];             // the convergents' coefficients, P scaled by y / sqrt(pi), Q by 1 / sqrt(pi)
    Geo<double> g;
    double thr[3];                         // |x| from which |z|^2 exceeds 100, 170, 500
    double inv[kProfMaxComp], off[kProfMaxComp];  // x = (lambda - lambda0) inv + off
    double q[kProfMaxComp];                // strength times eta_ratio / 2
    unsigned char line[kProfMaxComp], group[kProfMaxComp];  // 0 sigma_b, 1 pi, 2 sigma_r, 3 field-free; + 4: also field-free
    const double2 *row;  // without cells: the nodes of the damping's nearest row (NULL: the cells are built)
    double dy;           // and the damping's offset from it
    int ncomp;
    int count[4];                          // list lengths by region: table, 9th, 7th, 5th
};

__host__ __device__ inline int prof_components(const KProblem &pb)
{
    int n = 0;
    for (int l = 0; l < pb.n_lines; ++l)
        n += pb.line[l].ncomp[0] ? pb.line[l].ncomp[0] + pb.line[l].ncomp[1] + pb.line[l].ncomp[2] + (pb.fill ? 1 : 0) : 3;
    return n;
}
// Dynamic shared memory: ProfShared, the slots (x in, w out) of one pass and
// two lists that are filled from both ends.
inline size_t prof_smem(const KProblem &pb)
{
    const int n = prof_components(pb), c = n < kProfComps ? n : kProfComps;
    return sizeof(ProfShared) + (size_t)c * kProfBlock * (sizeof(double2) + 2 * sizeof(unsigned short));
}

// The row of nodes nearest to damping y and y's offset from it.  Dampings
// beyond the grid's ends get its first or last row.
__device__ __forceinline__ const double2 *node_row(const double2 *nodes, double y, double &dy)
{
    const double t = y + kNodeBelow * kNodeStep;  // also takes -0, whose bits are not those of 0
    const int n = __double2hiint(t) < 0 ? 0 : (int)(narrow(t) * (float)(1.0 / kNodeStep) + 0.5f);
    const int iy = min(n, kNodeBelow + kNodeGrid - 1) - kNodeBelow;
    dy = y - widen((float)iy * (float)kNodeStep);
    return nodes + iy * (kNodeGrid * kNodeCoef);
}

// One warp: the Taylor table of damping y, a cell per lane.
__device__ __forceinline__ void build_cells(ProfShared &S, const double2 *nodes, double y)
{
    const int lane = threadIdx.x & 31;
    const double x = (lane + 0.5) * kCellWidth;
    C2<double> m;
    if (y >= -kNodeBelow * kNodeStep) {  // from the node at x and the nearest y: a step along i
        double dy;
        const double2 *c = node_row(nodes, y, dy) + (4 * lane + 2) * kNodeCoef;
        const double2 top = __ldg(c + kNodeCoef - 1);
        m = {top.x, top.y};
#pragma unroll
        for (int n = kNodeCoef - 2; n >= 0; --n) {
            const double2 v = __ldg(c + n);
            m = {fma(-dy, m.y, v.x), fma(dy, m.x, v.y)};
        }
    } else {
        m = faddeeva_interior<double>(x, y);
    }
    C2<double> c = {-2.0 * (x * m.x - y * m.y), fma(-2.0, x * m.y + y * m.x, 1.12837916709551257390)};
    double2 *t = S.cell + lane * (kTaylor + 1);
    t[0] = make_double2(m.x, m.y);
    t[1] = make_double2(c.x, c.y);
#pragma unroll
    for (int n = 1; n < kTaylor; ++n) {
        const double f = -2.0 / (n + 1);
        const C2<double> d = {f * (x * c.x - y * c.y + m.x), f * (x * c.y + y * c.x + m.y)};
        t[n + 1] = make_double2(d.x, d.y);
        m = c;
        c = d;
    }
}

// One warp: the convergents' coefficients and the region thresholds.
__device__ __forceinline__ void build_exterior(ProfShared &S, double y)
{
    const int lane = threadIdx.x & 31;
    const double Y = y * y, isp = 0.56418958354775628695;
    if (lane < 3) {
        const double r2 = (lane == 0 ? 100.0 : lane == 1 ? 170.0 : 500.0) - Y;
        S.thr[lane] = r2 > 0.0 ? sqrt(r2) : 0.0;
    }
    for (int row = lane; row < kExtRows; row += 32) {
        const double *c = d_ext.c[row];
        double v = c[5];
#pragma unroll
        for (int j = 4; j >= 0; --j) v = fma(v, Y, c[j]);
        const int k = row < 18 ? 6 : row < 42 ? 8 : 10, part = (row - (row < 18 ? 0 : row < 42 ? 18 : 42)) / k;
        ((double *)S.ext)[row] = part == 0 ? v * (y * isp) : part == 1 ? v * isp : v;
    }
}

// One warp: the model's geometry (make_geo's formulas, the two sincos and the
// lines each on lanes of their own) and its Zeeman components.  p holds the
// parameters on every lane.
template <bool FILL>
__device__ __forceinline__ void build_geometry(ProfShared &S, const KProblem &pb, const double *p, double mu)
{
    const int lane = threadIdx.x & 31;
    double sn, cs;
    sincos_deg(lane == 0 ? p[1] : 2.0 * p[2], &sn, &cs);
    const double s2c = __shfl_sync(0xffffffffu, sn, 1), c2c = __shfl_sync(0xffffffffu, cs, 1);
    if (lane == 0) {
        Geo<double> &g = S.g;
        const double s2 = sn * sn, eta0 = p[6];
        g.a = p[5];
        g.a2 = p[5] * p[5];
        g.kIp = eta0 * s2;
        g.kIs = eta0 * 0.5 * fma(cs, cs, 1.0);
        g.kQ = g.kIp * c2c;
        g.kU = g.kIp * s2c;
        g.kV = eta0 * cs;
        g.kIp2 = g.kIp * g.kIp;
        g.kV2 = g.kV * g.kV;
        g.kUV = g.kU * g.kV;
        g.kQV = g.kQ * g.kV;
        g.S0 = p[7];
        g.muS1 = mu * p[8];
        g.eta0 = eta0;
        g.alpha = FILL ? p[9] : 1.0;
        S.ncomp = prof_components(pb);
    }
    if (lane < pb.n_lines) {
        const KLine &ln = pb.line[lane];
        int at = 0;  // the line's first component
        for (int l = 0; l < lane; ++l)
            at += pb.line[l].ncomp[0] ? pb.line[l].ncomp[0] + pb.line[l].ncomp[1] + pb.line[l].ncomp[2] + (FILL ? 1 : 0) : 3;
        const double inv = 1.0 / (p[4] * ln.dscale);
        const double cp = -(ln.lam0_c * p[3]) * inv;
        auto put = [&](int g, double off, double q) {
            S.inv[at] = inv;
            S.off[at] = off;
            S.q[at] = q;
            S.line[at] = (unsigned char)lane;
            S.group[at] = (unsigned char)g;
            ++at;
        };
        if (ln.ncomp[0] == 0) {
            const double vB = ln.zfac * p[0] * inv;
            put(0, cp + vB, ln.half_eta);
            put(FILL ? 5 : 1, cp, ln.half_eta);
            put(2, cp - vB, ln.half_eta);
        } else {
            const double vL = ln.zfacL * p[0] * inv;
            for (int g = 0; g < 3; ++g)
                for (int i = 0; i < ln.ncomp[g]; ++i) put(g, cp - vL * ln.cshift[g][i], ln.half_eta * ln.cstr[g][i]);
            if (FILL) put(3, cp, ln.half_eta);
        }
    }
}

// Building the cells costs one warp about 108 FP64 operations and saves each
// round of 32 interior points 16 of the 45 that an expansion from the grid's
// own nodes takes; about two fifths of the points are interior.  So the cells
// pay from some 540 points on; one-line models of 64 wavelengths (192 points)
// go without: a call for one 14.3 -> 12.5 us, 65 536 of them 2.28 -> 1.94 ms.
__device__ __forceinline__ bool use_cells(const KProblem &pb, double y)
{
    return prof_components(pb) * pb.n_lambda > 540 || !(y >= -kNodeBelow * kNodeStep);
}

// The model's tables in S: the cells, the geometry and the convergents'
// coefficients on a warp each, side by side (p as above).  Nothing in S may be
// read before a barrier (profile_sums begins with one).
template <bool FILL>
__device__ __forceinline__ void build_model(ProfShared &S, const KProblem &pb, const double *p, double mu)
{
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        const double y = p[5];
        const bool cells = use_cells(pb, y);
        if (cells) build_cells(S, pb.nodes, y);
        if ((threadIdx.x & 31) == 0) {
            double dy;
            const double2 *row = node_row(pb.nodes, y, dy);
            S.row = cells ? nullptr : row;
            S.dy = dy;
        }
    }
    if (warp == 1) build_geometry<FILL>(S, pb, p, mu);
    else if (warp == 2) build_exterior(S, p[5]);
}

// Profile sums of one wavelength: sum q w over each group's components.
struct ProfSums {
    double P, Pi, Sb, Sbi, Sr, Sri, P0;
};

// The K-th convergent at x (ext: its block of coefficients).
template <int K> __device__ __forceinline__ double2 convergent(const double2 *ext, double x, double Y)
{
    constexpr int H = (K + 1) / 2;
    const double s = fma(x, x, Y);
    double2 cp = ext[H - 1], cq = ext[2 * H - 1], cd = ext[3 * H - 1];
    double p = fma(cp.y, s, cp.x), q = fma(cq.y, s, cq.x), d = fma(s + cd.y, s, cd.x);
#pragma unroll
    for (int i = H - 2; i >= 0; --i) {
        cp = ext[i];
        cq = ext[H + i];
        cd = ext[2 * H + i];
        p = fma(fma(p, s, cp.y), s, cp.x);
        q = fma(fma(q, s, cq.y), s, cq.x);
        d = fma(fma(d, s, cd.y), s, cd.x);
    }
    const double r = rcp_newton(d);
    return make_double2(p * r, x * q * r);
}

// The Taylor polynomial of |x|'s cell.
__device__ __forceinline__ double2 from_cells(const ProfShared &S, double x)
{
    const double ax = fabs(x);
    const int c = min((int)(narrow(ax) * (float)(1.0 / kCellWidth)), kCells - 1);
    const double t = ax - widen(((float)c + 0.5f) * (float)kCellWidth);  // the centre is exact in FP32
    const double2 *k = S.cell + c * (kTaylor + 1);
    double2 w = k[kTaylor];
#pragma unroll
    for (int n = kTaylor - 1; n >= 0; --n) {
        const double2 v = k[n];
        w.x = fma(w.x, t, v.x);
        w.y = fma(w.y, t, v.y);
    }
    w.y = __hiloint2double(__double2hiint(w.y) ^ (__double2hiint(x) & (int)0x80000000), __double2loint(w.y));
    return w;
}

// w from the node nearest to (|x|, y): row = the nodes of y's nearest row, dy
// = y's offset from it.
__device__ __forceinline__ C2<double> from_node(const double2 *row, double x, double dy)
{
    const double ax = fabs(x);
    const int ix = min((int)(narrow(ax) * (float)(1.0 / kNodeStep) + 0.5f), kNodeGrid - 1);
    const double dx = ax - widen((float)ix * (float)kNodeStep);
    const double2 *c = row + ix * kNodeCoef;
    const double2 top = __ldg(c + kNodeCoef - 1);
    double re = top.x, im = top.y;
#pragma unroll
    for (int n = kNodeCoef - 2; n >= 0; --n) {
        const double2 v = __ldg(c + n);
        const double t = fma(re, dx, fma(-im, dy, v.x));
        im = fma(re, dy, fma(im, dx, v.y));
        re = t;
    }
    return {re, __hiloint2double(__double2hiint(im) ^ (__double2hiint(x) & (int)0x80000000), __double2loint(im))};
}

// Profile sums of one wavelength by one thread: doff(l) = lambda - lambda0_l,
// profile(x) = w(x + i a) for the model of geometry g.
template <bool FILL, class Offset, class Profile>
__device__ __forceinline__ ProfSums point_sums(const KProblem &pb, const Geo<double> &g, Offset doff, Profile profile)
{
    ProfSums S = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int l = 0; l < pb.n_lines; ++l) {
        const KLine &ln = pb.line[l];
        const double x0 = fma(doff(l), g.invD[l], g.cp[l]);
        const double q = ln.half_eta;
        if (ln.ncomp[0] == 0) {
#pragma unroll 1
            for (int c = 0; c < 3; ++c) {
                const double x = c == 0 ? x0 + g.vB[l] : c == 1 ? x0 : x0 - g.vB[l];
                const C2<double> w = profile(x);
                if (c == 0) {
                    S.Sb = fma(q, w.x, S.Sb);
                    S.Sbi = fma(q, w.y, S.Sbi);
                } else if (c == 1) {
                    S.P = fma(q, w.x, S.P);
                    S.Pi = fma(q, w.y, S.Pi);
                    if (FILL) S.P0 = fma(q, w.x, S.P0);
                } else {
                    S.Sr = fma(q, w.x, S.Sr);
                    S.Sri = fma(q, w.y, S.Sri);
                }
            }
        } else {
#pragma unroll 1
            for (int k = 0; k < 3; ++k)
#pragma unroll 1
                for (int i = 0; i < ln.ncomp[k]; ++i) {
                    const C2<double> w = profile(fma(-g.vL[l], ln.cshift[k][i], x0));
                    const double qc = q * ln.cstr[k][i];
                    if (k == 0) {
                        S.Sb = fma(qc, w.x, S.Sb);
                        S.Sbi = fma(qc, w.y, S.Sbi);
                    } else if (k == 1) {
                        S.P = fma(qc, w.x, S.P);
                        S.Pi = fma(qc, w.y, S.Pi);
                    } else {
                        S.Sr = fma(qc, w.x, S.Sr);
                        S.Sri = fma(qc, w.y, S.Sri);
                    }
                }
            if (FILL) S.P0 = fma(q, profile(x0).x, S.P0);
        }
    }
    return S;
}

// w(x + i a) for a thread on its own: the nearest node's expansion for |z|^2 <
// 100 and the 9th convergent in complex arithmetic beyond (row and dy as in
// from_node).
__device__ __forceinline__ C2<double> profile_alone(const double2 *row, double dy, double x, double a, double a2)
{
    if (__double_as_longlong(fma(x, x, a2)) < 0x4059000000000000ll) return from_node(row, x, dy);  // 100, as bits
    return faddeeva_exterior<double>(x, a, a2);
}

// Profile sums of wavelength j0 + threadIdx.x for the model in S, by all
// kProfBlock threads (those beyond nl help and get zeros).  Every thread of
// the block calls it (barriers inside, the first before anything in S is
// read).
template <bool FILL>
__device__ __forceinline__ ProfSums profile_sums(ProfShared &S, const KProblem &pb, int j0, int nl)
{
    __syncthreads();  // the model's tables are complete; an earlier call's slots have been read
    double2 *slot = (double2 *)(&S + 1);
    const int total = S.ncomp, npass = total < kProfComps ? total : kProfComps;
    const int cap = npass * kProfBlock;
    unsigned short *la = (unsigned short *)(slot + cap), *lb = la + cap;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned below = (1u << lane) - 1u;
    const double Y = S.g.a2;
    const long long t0 = __double_as_longlong(S.thr[0]), t1 = __double_as_longlong(S.thr[1]),
                    t2 = __double_as_longlong(S.thr[2]);
    const bool real = j0 + tid < nl;
    const double lam = pb.lam[real ? j0 + tid : 0];
    ProfSums r = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int c0 = 0; c0 < total; c0 += kProfComps) {
        const int nc = min(kProfComps, total - c0);
        if (c0 > 0) __syncthreads();  // the last pass's slots have been read
        if (tid < 4) S.count[tid] = 0;
        __syncthreads();
        // arguments, and the lists of their regions (|x| and the thresholds
        // compared as integers, off the FP64 pipe)
        int l = -1;
        double doff = 0.0;
        for (int c = 0; c < nc; ++c) {
            if (S.line[c0 + c] != l) {
                l = S.line[c0 + c];
                doff = lam - pb.line[l].lam0;
            }
            const double x = fma(doff, S.inv[c0 + c], S.off[c0 + c]);
            const long long ax = __double_as_longlong(x) & 0x7fffffffffffffffll;
            const int reg = ax < t0 ? 0 : ax < t1 ? 1 : ax < t2 ? 2 : 3;
            const int item = c * kProfBlock + tid;
            slot[item].x = x;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned m = __ballot_sync(0xffffffffu, real && reg == k);
                if (m == 0u) continue;
                int base = 0;
                if (lane == 0) base = atomicAdd(&S.count[k], __popc(m));
                base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & below);
                if (real && reg == k) {
                    unsigned short *list = k < 2 ? la : lb;
                    list[(k & 1) ? cap - 1 - base : base] = (unsigned short)item;
                }
            }
        }
        __syncthreads();
        // rounds of 32 items of one region, dealt to the warps
        const int n0 = S.count[0], n1 = S.count[1], n2 = S.count[2], n3 = S.count[3];
        const int r0 = (n0 + 31) >> 5, r1 = r0 + ((n1 + 31) >> 5), r2 = r1 + ((n2 + 31) >> 5),
                  r3 = r2 + ((n3 + 31) >> 5);
        for (int k = warp; k < r3; k += kProfBlock / 32) {
            if (k < r0) {
                const int i = k * 32 + lane;
                if (i < n0) {
                    double2 &s = slot[la[i]];
                    if (S.row) {
                        const C2<double> w = from_node(S.row, s.x, S.dy);
                        s = make_double2(w.x, w.y);
                    } else {
                        s = from_cells(S, s.x);
                    }
                }
            } else if (k < r1) {
                const int i = (k - r0) * 32 + lane;
                if (i < n1) {
                    double2 &s = slot[la[cap - 1 - i]];
                    s = convergent<9>(S.ext + 21, s.x, Y);
                }
            } else if (k < r2) {
                const int i = (k - r1) * 32 + lane;
                if (i < n2) {
                    double2 &s = slot[lb[i]];
                    s = convergent<7>(S.ext + 9, s.x, Y);
                }
            } else {
                const int i = (k - r2) * 32 + lane;
                if (i < n3) {
                    double2 &s = slot[lb[cap - 1 - i]];
                    s = convergent<5>(S.ext, s.x, Y);
                }
            }
        }
        __syncthreads();
        if (real) {
            for (int c = 0; c < nc; ++c) {
                const double2 w = slot[c * kProfBlock + tid];
                const double q = S.q[c0 + c];
                const int g = S.group[c0 + c];
                if (g == 0) {
                    r.Sb = fma(q, w.x, r.Sb);
                    r.Sbi = fma(q, w.y, r.Sbi);
                } else if (g == 2) {
                    r.Sr = fma(q, w.x, r.Sr);
                    r.Sri = fma(q, w.y, r.Sri);
                } else {
                    if (g != 3) {
                        r.P = fma(q, w.x, r.P);
                        r.Pi = fma(q, w.y, r.Pi);
                    }
                    if (FILL && g >= 3) r.P0 = fma(q, w.x, r.P0);
                }
            }
        }
    }
    return r;
}

// Closed form of K^-1 e (see me_point) from the profile sums.
template <bool FILL>
__device__ __forceinline__ Stokes4<double> stokes_of(const Geo<double> &g, const ProfSums &r)
{
    const double Sg = r.Sb + r.Sr, Sgi = r.Sbi + r.Sri, Dd = r.Sr - r.Sb, Di = r.Sri - r.Sbi;
    const double T = fma(-0.5, Sg, r.P), Ti = fma(-0.5, Sgi, r.Pi);
    const double eI = fma(g.kIs, Sg, fma(g.kIp, r.P, 1.0));
    const double pT = g.kIp2 * T, pTi = g.kIp2 * Ti, vD = g.kV2 * Dd, vDi = g.kV2 * Di;
    const double E2 = fma(pT, T, vD * Dd), rho2 = fma(pTi, Ti, vDi * Di), Pi = fma(pT, Ti, vD * Di);
    const double eI2 = eI * eI, G = eI2 + rho2;
    const double Delta = fma(eI2, G - E2, -(Pi * Pi));
    const double f = g.muS1 * (1.0 / Delta);
    const double A = f * fma(eI2, T, Ti * Pi), feI = f * eI, C = feI * fma(Dd, Ti, -(T * Di));
    Stokes4<double> s;
    s.I = fma(feI, G, g.S0);
    s.Q = -fma(g.kQ, A, g.kUV * C);
    s.U = fma(g.kQV, C, -(g.kU * A));
    s.V = -(f * g.kV) * fma(eI2, Dd, Di * Pi);
    if (FILL) fill_mix(s, g, r.P0);
    return s;
}

}  // namespace genesis
