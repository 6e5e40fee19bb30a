// FP64 fitness of one individual per thread (sm_103a): Eq. chisq of the
// Section 5 synthesis over the pixel's wavelengths.
//
// Bound by the FP64 pipe, as the profiles of profiles64.cuh, but here the
// lanes of a warp hold different dampings at one wavelength, so w(x + i a)
// comes
//  * for |z|^2 < 100 from the nearest node of the grid of faddeeva_nodes.h, a
//    Taylor polynomial of degree 10 in the complex offset (40 operations
//    where Weideman's series with N = 36 takes 105; within 2e-16 of w);
//  * to |z|^2 = 500 from the 9th convergent and beyond from the 5th, as real
//    polynomials in |z|^2 whose coefficients each individual forms once per
//    evaluation and keeps in shared memory (36 and 24 operations where the
//    9th in complex arithmetic takes 56).
// The weighted squared residuals are summed with Kahan's compensation in
// kShares sums of wavelengths j = r (mod kShares), added in the order of r:
// threads that share an individual take whole sums, so the value does not
// depend on how many there are.
#pragma once

#include "profiles64.cuh"

namespace genesis {

constexpr int kShares = 8;
constexpr int kF64Rows = 18 + 30;  // the 5th convergent's coefficients, then the 9th's

// Shared memory of npop individuals, all [row][individual].
struct Fit64Shared {
    double *coef;  // kF64Rows
    double *part;  // kShares
    int npop;
};
__host__ __device__ inline int fit64_doubles(int npop) { return (kF64Rows + kShares) * npop; }

// The convergents' coefficients of damping y, rows seg, seg + nseg, ...
__device__ __forceinline__ void fit64_coefficients(const Fit64Shared &S, int k, double y, int seg, int nseg)
{
    const double Y = y * y, isp = 0.56418958354775628695;
#pragma unroll 2
    for (int row = seg; row < kF64Rows; row += nseg) {
        const double *c = d_ext.c[row < 18 ? row : row - 18 + kExtFirst<9>];
        double v = c[5];
#pragma unroll
        for (int j = 4; j >= 0; --j) v = fma(v, Y, c[j]);
        const int part = row < 18 ? row / 6 : (row - 18) / 10;
        S.coef[row * S.npop + k] = part == 0 ? v * (y * isp) : part == 1 ? v * isp : v;
    }
}

// The K-th convergent from an individual's coefficients c (stride n).
template <int K> __device__ __forceinline__ C2<double> convergent_of(const double *c, int n, double x, double s)
{
    constexpr int H = K + 1;
    double p = c[K * n], q = c[(H + K) * n], d = s + c[(2 * H + K) * n];
#pragma unroll
    for (int i = K - 1; i >= 0; --i) {
        p = fma(p, s, c[i * n]);
        q = fma(q, s, c[(H + i) * n]);
        d = fma(d, s, c[(2 * H + i) * n]);
    }
    const double r = rcp_newton(d);
    return {p * r, x * q * r};
}

// One individual's geometry and what its profiles need.
struct Fit64Model {
    Geo<double> g;
    const double2 *row;  // nodes of the damping's nearest row
    double dy;
};
template <bool FILL>
__device__ __forceinline__ Fit64Model fit64_model(const KProblem &pb, const double *p, double mu)
{
    Fit64Model m;
    m.g = make_geo<double, 0, FILL>(pb, pb.n_lines, p, mu);
    m.row = node_row(pb.nodes, m.g.a, m.dy);
    return m;
}

__device__ __forceinline__ C2<double> fit64_profile(const Fit64Model &m, const double *coef, int n, double x)
{
    const double s = fma(x, x, m.g.a2);
    // as bits (s >= 0), off the FP64 pipe; NaN counts as far
    const long long b = __double_as_longlong(s);
    if (b < 0x4059000000000000ll) return from_node(m.row, x, m.dy);                    // 100
    if (b < 0x407f400000000000ll) return convergent_of<9>(coef + 18 * n, n, x, s);     // 500
    return convergent_of<5>(coef, n, x, s);
}

// Kahan's sum of the weighted squared residuals of wavelengths r, r +
// kShares, ... of the individual.  s_obs rows are (I, Q, U, V), s_doff rows
// lambda_j - lambda0_l for l = 0..3.  res, when not NULL, receives the
// residuals O - S as [4][nl] (verification only).
template <bool FILL, bool STORE>
__device__ __forceinline__ double fit64_share(const KProblem &pb, int nl, const Fit64Model &m, const double *coef, int n,
                                              const double *s_obs, const double *s_doff, const double *s_w2, int r,
                                              double *res)
{
    double sum = 0.0, comp = 0.0;
    for (int j = r; j < nl; j += kShares) {
        const ProfSums S = point_sums<FILL>(pb, m.g, [&](int l) { return s_doff[4 * j + l]; },
                                            [&](double x) { return fit64_profile(m, coef, n, x); });
        const Stokes4<double> s = stokes_of<FILL>(m.g, S);
        const double r0 = s_obs[4 * j] - s.I, r1 = s_obs[4 * j + 1] - s.Q, r2 = s_obs[4 * j + 2] - s.U,
                     r3 = s_obs[4 * j + 3] - s.V;
        if (STORE && res) {
            res[j] = r0;
            res[nl + j] = r1;
            res[2 * nl + j] = r2;
            res[3 * nl + j] = r3;
        }
        const double t = fma(s_w2[3] * r3, r3, fma(s_w2[2] * r2, r2, fma(s_w2[1] * r1, r1, (s_w2[0] * r0) * r0)));
        const double y = t - comp, u = sum + y;
        comp = (u - sum) - y;
        sum = u;
    }
    return sum - comp;
}

// The shares of one individual added in order.
__device__ __forceinline__ double fit64_total(const double *part, int n, int k, double inv_nu)
{
    double sum = 0.0, comp = 0.0;
#pragma unroll
    for (int r = 0; r < kShares; ++r) {
        const double y = part[r * n + k] - comp, u = sum + y;
        comp = (u - sum) - y;
        sum = u;
    }
    return (sum - comp) * inv_nu;
}

}  // namespace genesis
