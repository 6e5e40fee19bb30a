// Stokes synthesis, Jacobian, adjoint and FP64 chi-square kernels (sm_103a).
#include <algorithm>
#include <type_traits>

#include "async_copy.cuh"
#include "kernels.h"
#include "launch_rules.h"
#include "me_jac.cuh"
#include "profiles64.cuh"
#include "rng_device.cuh"

namespace genesis {

static __device__ double2 d_nodes[(kNodeBelow + kNodeGrid) * kNodeGrid * kNodeCoef];

cudaError_t upload_nodes(void **ptr)
{
    static const std::vector<double> below = faddeeva_nodes_below(), host = faddeeva_nodes();
    const size_t nb = below.size() * sizeof(double);
    cudaError_t e = cudaGetSymbolAddress(ptr, d_nodes);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(d_nodes, below.data(), nb);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(d_nodes, host.data(), host.size() * sizeof(double), nb);
    *ptr = (char *)*ptr + nb;  // row 0
    return e;
}

cudaError_t upload_tables_synth(const HostTables &t)
{
    return cudaMemcpyToSymbol(c_fad, &t.fad, sizeof(FaddeevaTables));
}

namespace {

constexpr int kSynthBlock = 128;

// Fill s_doff[l * nl + j] = lambda_j - lambda0_l for all lines (exact in FP64,
// rounded to R) and s_he[l] = eta_ratio_l / 2.
template <class R>
__device__ __forceinline__ void stage_offsets(const KProblem &pb, int nlines, R *s_doff, R *s_he)
{
    const int nl = pb.n_lambda;
    for (int i = threadIdx.x; i < nlines * nl; i += blockDim.x) {
        const int l = i / nl, j = i - l * nl;
        s_doff[i] = R(pb.lam[j] - pb.line[l].lam0);
    }
    if (threadIdx.x < ME_MAX_LINES)
        s_he[threadIdx.x] = threadIdx.x < nlines ? R(pb.line[threadIdx.x].half_eta) : R(0);
}

// A model's parameters (and mu) on every lane in the problem's precision: one
// lane loads and converts each (conversions take the FP64 pipe, a warp
// instruction in 16 clocks of an SM), shuffles spread them.
template <class R, int M>
__device__ __forceinline__ void load_model(const KProblem &pb, const double *params, const double *mu_px, int m, R (&p)[M],
                                           R &mu)
{
    const int lane = threadIdx.x & 31;
    const double v = lane < M ? params[(size_t)m * M + lane] : mu_px ? mu_px[m] : pb.mu;
    const R r = R(v);
#pragma unroll
    for (int d = 0; d < M; ++d) p[d] = __shfl_sync(0xffffffffu, r, d);
    mu = __shfl_sync(0xffffffffu, r, M);
}

// Blocks per SM that the FP32 Jacobian's registers have to allow: 20 011
// two-line models take 145, 128, 227 and 255 us at 3, 4, 5 and 6.
constexpr int kJacMinB = 4;

// Synthesis, and with JAC the Jacobian, a warp per model (or per `per` of its
// chunks of 32 wavelengths, where whole models would leave warps idle):
// lanes over wavelengths, the model's geometry formed once for the warp's
// chunks, the wavelength offsets once for all of a block's models.  A thread
// per (model, wavelength) formed both for every point: ten FP64 conversions
// per warp alone took longer than the synthesis.  A Jacobian row of Stokes s
// and 32 wavelengths leaves through shared memory as 32 M consecutive values,
// so that each store instruction writes whole sectors (lane by lane it wrote
// 4 of every 36 bytes).  20 011 two-line FP32 models, 128 wavelengths:
// syntheses 110 -> 55 us, Jacobians 267 -> 128 us.  chunks_per_warp says where
// k_points is the faster one.
template <int NL, bool FILL, bool JAC>
__global__ void __launch_bounds__(kSynthBlock, JAC ? kJacMinB : 8)
k_models(const __grid_constant__ KProblem pb, const double *__restrict__ params, const double *__restrict__ mu_px,
         int n, int per, float *__restrict__ stokes, float *__restrict__ jac)
{
    using R = float;
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int M = kNpar<FILL>;
    const int nl = pb.n_lambda, nlines = NL > 0 ? NL : pb.n_lines;
    R *s_he = (R *)smem;
    R *s_doff = s_he + ME_MAX_LINES;
    stage_offsets<R>(pb, nlines, s_doff, s_he);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    R *s_row = s_doff + nlines * nl + warp * 32 * M;
    R he[ME_MAX_LINES];
#pragma unroll
    for (int l = 0; l < ME_MAX_LINES; ++l) he[l] = s_he[l];
    const int chunks = (nl + 31) >> 5, groups = (chunks + per - 1) / per;
    const long long items = (long long)n * groups;
    for (long long it = (long long)blockIdx.x * (kSynthBlock / 32) + warp; it < items;
         it += (long long)gridDim.x * (kSynthBlock / 32)) {
        const int m = (int)(it / groups), c0 = (int)(it - (long long)m * groups) * per;
        R p[M], mu;
        load_model<R, M>(pb, params, mu_px, m, p, mu);
        std::conditional_t<JAC, GeoJ<R>, Geo<R>> G;
        if constexpr (JAC) G = make_geoj<R, NL, FILL>(pb, nlines, p, mu);
        else G = make_geo<R, NL, FILL>(pb, nlines, p, mu);
        for (int c = c0; c < min(c0 + per, chunks); ++c) {
            const int j = c * 32 + lane;
            const bool on = j < nl;
            R doff[ME_MAX_LINES];
#pragma unroll
            for (int l = 0; l < ME_MAX_LINES; ++l) doff[l] = l < nlines ? s_doff[l * nl + (on ? j : nl - 1)] : R(0);
            Stokes4<R> s;
            R J[4][M];
            if constexpr (JAC) me_point_jac<R, NL, FILL>(G, doff, he, nlines, pb.line, s, J);
            else s = me_point<R, NL, true, FILL>(G, doff, he, nlines, pb.line);
            if (stokes && on) {
                R *o = stokes + (size_t)m * 4 * nl + j;
                o[0] = s.I;
                o[nl] = s.Q;
                o[2 * nl] = s.U;
                o[3 * nl] = s.V;
            }
            if constexpr (JAC) {
                const int len = min(32, nl - c * 32) * M;
#pragma unroll
                for (int st = 0; st < 4; ++st) {
#pragma unroll
                    for (int k = 0; k < M; ++k) s_row[lane * M + k] = J[st][k];
                    __syncwarp();
                    R *o = jac + (((size_t)m * 4 + st) * nl + c * 32) * M;
#pragma unroll
                    for (int k = 0; k < M; ++k)
                        if (k * 32 + lane < len) o[k * 32 + lane] = s_row[k * 32 + lane];
                    __syncwarp();
                }
            }
        }
    }
}

// Synthesis, and with JAC the Jacobian, a thread per (model, wavelength): every
// lane works whatever the grid, but each forms its model's geometry.  FP32: see
// chunks_per_warp.  The FP64 Jacobian always runs here: it is bound by the FP64
// pipe, where a warp per model was 0 to 5 % slower (700 full-pattern models 556
// against 525 us).
template <class R, int NL, bool FILL, bool JAC>
__global__ void __launch_bounds__(kSynthBlock)
k_points(const __grid_constant__ KProblem pb, const double *__restrict__ params, const double *__restrict__ mu_px, int n,
         R *__restrict__ stokes, R *__restrict__ jac)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int nl = pb.n_lambda, nlines = NL > 0 ? NL : pb.n_lines;
    R *s_he = (R *)smem;
    R *s_doff = s_he + ME_MAX_LINES;
    stage_offsets<R>(pb, nlines, s_doff, s_he);
    __syncthreads();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)n * nl) return;
    const int m = (int)(i / nl), j = (int)(i - (long long)m * nl);
    constexpr int M = kNpar<FILL>;
    R p[M];
#pragma unroll
    for (int d = 0; d < M; ++d) p[d] = R(params[(size_t)m * M + d]);
    const R mu = mu_px ? R(mu_px[m]) : R(pb.mu);
    std::conditional_t<JAC, GeoJ<R>, Geo<R>> G;
    if constexpr (JAC) G = make_geoj<R, NL, FILL>(pb, nlines, p, mu);
    else G = make_geo<R, NL, FILL>(pb, nlines, p, mu);
    Stokes4<R> s;
    R J[4][M];
    if constexpr (!JAC && sizeof(R) == 8) {
        double dy;
        const double2 *row = node_row(pb.nodes, G.a, dy);
        s = stokes_of<FILL>(G, point_sums<FILL>(pb, G, [&](int l) { return s_doff[l * nl + j]; },
                                                [&](double x) { return profile_alone(row, dy, x, G.a, G.a2); }));
    } else {
        R doff[ME_MAX_LINES], he[ME_MAX_LINES];
#pragma unroll
        for (int l = 0; l < ME_MAX_LINES; ++l) {
            doff[l] = l < nlines ? s_doff[l * nl + j] : R(0);
            he[l] = s_he[l];
        }
        if constexpr (JAC) me_point_jac<R, NL, FILL>(G, doff, he, nlines, pb.line, s, J);
        else s = me_point<R, NL, true, FILL>(G, doff, he, nlines, pb.line);
    }
    if (stokes) {
        R *o = stokes + (size_t)m * 4 * nl;
        o[j] = s.I;
        o[nl + j] = s.Q;
        o[2 * nl + j] = s.U;
        o[3 * nl + j] = s.V;
    }
    if constexpr (JAC) {
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            R *o = jac + (((size_t)m * 4 + st) * nl + j) * M;
#pragma unroll
            for (int k = 0; k < M; ++k) o[k] = J[st][k];
        }
    }
}

// One warp per model: grad_params[m] = sum_{s, j} J[s][j][:] * grad_stokes[m][s][j].
template <class R, int NL, bool FILL = false>
__global__ void __launch_bounds__(kSynthBlock)
k_vjp(const __grid_constant__ KProblem pb, const double *__restrict__ params,
      const double *__restrict__ mu_px, int n, const R *__restrict__ gs, double *__restrict__ gp)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int nl = pb.n_lambda, nlines = NL > 0 ? NL : pb.n_lines;
    R *s_he = (R *)smem;
    R *s_doff = s_he + ME_MAX_LINES;
    stage_offsets<R>(pb, nlines, s_doff, s_he);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int m = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (m >= n) return;
    constexpr int M = kNpar<FILL>;
    R p[M];
#pragma unroll
    for (int d = 0; d < M; ++d) p[d] = R(params[(size_t)m * M + d]);
    const R mu = mu_px ? R(mu_px[m]) : R(pb.mu);
    const GeoJ<R> G = make_geoj<R, NL, FILL>(pb, nlines, p, mu);
    R he[ME_MAX_LINES];
#pragma unroll
    for (int l = 0; l < ME_MAX_LINES; ++l) he[l] = s_he[l];
    R acc[M];
#pragma unroll
    for (int k = 0; k < M; ++k) acc[k] = R(0);
    const R *g = gs + (size_t)m * 4 * nl;
    for (int j = lane; j < nl; j += 32) {
        R doff[ME_MAX_LINES];
#pragma unroll
        for (int l = 0; l < ME_MAX_LINES; ++l) doff[l] = l < nlines ? s_doff[l * nl + j] : R(0);
        Stokes4<R> s;
        R J[4][M];
        me_point_jac<R, NL, FILL>(G, doff, he, nlines, pb.line, s, J);
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            const R gv = g[st * nl + j];
#pragma unroll
            for (int k = 0; k < M; ++k) acc[k] += J[st][k] * gv;
        }
    }
#pragma unroll
    for (int k = 0; k < M; ++k) {
        double v = (double)acc[k];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) gp[(size_t)m * M + k] = v;
    }
}

// FP64 synthesis, one block per model (see profiles64.cuh), or one per pass over
// its wavelengths (blocks_per_model64): 65 536 two-line models 14.0 -> 4.8 ms
// against a thread per (model, wavelength) with Weideman's series, a call for
// one one-line model 27 -> 12.5 us; absolute error 1.5e-15 -> 7e-17 rms.
template <bool FILL>
__global__ void __launch_bounds__(kProfBlock)
k_synth64(const __grid_constant__ KProblem pb, const double *__restrict__ params, const double *__restrict__ mu_px,
          double *__restrict__ stokes)
{
    extern __shared__ __align__(16) unsigned char smem[];
    ProfShared &S = *(ProfShared *)smem;
    const int nl = pb.n_lambda, m = blockIdx.x;
    constexpr int M = kNpar<FILL>;
    double p[M];
#pragma unroll
    for (int d = 0; d < M; ++d) p[d] = params[(size_t)m * M + d];
    build_model<FILL>(S, pb, p, mu_px ? mu_px[m] : pb.mu);
    double *o = stokes + (size_t)m * 4 * nl;
    for (int j0 = blockIdx.y * kProfBlock; j0 < nl; j0 += gridDim.y * kProfBlock) {
        const ProfSums r = profile_sums<FILL>(S, pb, j0, nl);
        const int j = j0 + threadIdx.x;
        if (j < nl) {
            const Stokes4<double> s = stokes_of<FILL>(S.g, r);
            o[j] = s.I;
            o[nl + j] = s.Q;
            o[2 * nl + j] = s.U;
            o[3 * nl + j] = s.V;
        }
    }
}

// FP64 chi-square (Eq. chisq) of given parameters, one block per pixel,
// threads over wavelengths, on the profiles of profiles64.cuh.  Bound by the
// FP64 pipe: 65 536 two-line pixels took 13.5 ms with Weideman's series and
// the 9th convergent per thread (both branches in most warps, every division
// in full, the geometry on one thread), 5.1 ms now, and the relative error of
// chi2 against 64-bit references fell from 2.5e-13 to 8e-15 rms.
template <class RO, bool FILL>
__global__ void __launch_bounds__(kProfBlock)
k_chi2_f64(const __grid_constant__ KProblem pb, const RO *__restrict__ obs,
           const double *__restrict__ w_user, const double *__restrict__ mu_px, int npix,
           const double *__restrict__ params, double *__restrict__ chi2, const KSub sub)
{
    extern __shared__ __align__(16) unsigned char smem[];
    ProfShared &S = *(ProfShared *)smem;
    __shared__ double s_red[kProfBlock / 32][4];
    __shared__ double s_w2[4];
    const int nl = pb.n_lambda;
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (sub.count && b >= *sub.count) return;
    const int pix = sub.index ? sub.index[b] : b;
    if (pix < 0 || pix >= npix) return;
    const RO *o = obs + (size_t)pix * 4 * nl;
    constexpr int M = kNpar<FILL>;
    double p[M];
#pragma unroll
    for (int d = 0; d < M; ++d) p[d] = params[(size_t)pix * M + d];
    build_model<FILL>(S, pb, p, mu_px ? mu_px[pix] : pb.mu);
    if (warp == 3) weights64<RO>(o, nl, w_user, pix, s_w2);
    double ss[4] = {0, 0, 0, 0};
    for (int j0 = 0; j0 < nl; j0 += kProfBlock) {
        const ProfSums r = profile_sums<FILL>(S, pb, j0, nl);
        const int j = j0 + threadIdx.x;
        if (j < nl) {
            const Stokes4<double> s = stokes_of<FILL>(S.g, r);
            const double r0 = widen(o[j]) - s.I, r1 = widen(o[nl + j]) - s.Q;
            const double r2 = widen(o[2 * nl + j]) - s.U, r3 = widen(o[3 * nl + j]) - s.V;
            ss[0] += r0 * r0;
            ss[1] += r1 * r1;
            ss[2] += r2 * r2;
            ss[3] += r3 * r3;
        }
    }
    const double v = warp_sum4(ss[0], ss[1], ss[2], ss[3]);
    if ((lane & 7) == 0) s_red[warp][lane >> 3] = v;
    __syncthreads();
    if (warp == 0) {
        double a = 0.0;
        if (lane < 4) {
            for (int w = 0; w < kProfBlock / 32; ++w) a += s_red[w][lane];
            a *= s_w2[lane];
        }
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        if (lane == 0) chi2[pix] = a / (double)(4 * nl - M);
    }
}

// One pixel's search of k_line_centre on its staged row I (index 0 = grid
// point 0): T is the type its sums are exact or rounded in.
__device__ __forceinline__ double abs_add(double s, double a, double b) { return __dadd_rn(s, fabs(__dsub_rn(a, b))); }
__device__ __forceinline__ long long abs_add(long long s, long long a, long long b)
{
    const long long d = a - b;
    return s + (d < 0 ? -d : d);
}
constexpr long long kNoSum = 0x7fffffffffffffffll;  // above every sum
// Sums are >= 0, so an FP64 sum's bits order it; NaN is never the least.
__device__ __forceinline__ long long sum_order(double s) { return s == s ? __double_as_longlong(s) : kNoSum; }
__device__ __forceinline__ long long sum_order(long long s) { return s; }

// On return best = the least sum, bi its index (0x7fffffff: none) on every
// lane of the pixel, y0 and y2 the sums at bi - 1 and bi + 1 on its first lane
// where both are candidates.
template <int G, class T>
__device__ __forceinline__ void centre_search(const T *I, int W, int lo, int hi, int sub, T &best, int &bi, T &y0, T &y2)
{
    auto S = [&](int i) {
        T s = T(0);
        for (int j = 1; j <= W; ++j) s = abs_add(s, I[i + j], I[i - j]);
        return s;
    };
    long long key = kNoSum;
    best = T(0);
    bi = 0x7fffffff;
    for (int i = lo + sub; i <= hi; i += G) {
        const T s = S(i);
        if (sum_order(s) < key) {
            key = sum_order(s);
            best = s;
            bi = i;
        }
    }
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {
        const long long ok = __shfl_xor_sync(0xffffffffu, key, off);
        const T os = __shfl_xor_sync(0xffffffffu, best, off);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
        if (ok < key || (ok == key && oi < bi)) {
            key = ok;
            best = os;
            bi = oi;
        }
    }
    const bool inner = bi != 0x7fffffff && bi - 1 >= lo && bi + 1 <= hi;
    y0 = y2 = T(0);
    if (G == 1) {
        if (inner) {
            y0 = S(bi - 1);
            y2 = S(bi + 1);
        }
    } else {  // one on each of two lanes
        if (inner && sub < 2) y0 = S(bi + 2 * sub - 1);
        y2 = __shfl_down_sync(0xffffffffu, y0, 1);
    }
}

// Section 5.1 centre of symmetry, G lanes per pixel, 32 / G pixels per warp:
// S_i = sum_j |I(i+j) - I(i-j)| in FP64 in increasing j, candidates i dealt to
// the pixel's lanes, the argmin over i (ties to the lowest index) and the
// three-point parabola vertex, written without contraction.
// In FP64 the sums would bind the kernel: the FP64 pipe takes 16 clocks of an
// SM per warp instruction (whether one lane or 32 are active, so a warp per
// pixel wastes it on ragged rounds).  A float cube's samples are multiples of
// 2^(emin - 150), emin the row's least biased exponent, so where the row's
// exponents span few enough octaves that 24 bits, a sign, the span and the W
// terms fit 53 bits, every difference and sum is exact in FP64 and equals the
// same sum of 64-bit integers, which run on the integer pipe; other rows (and
// double cubes) are summed in FP64.  262 144 pixels, W = 10, 33 candidates:
// 2.40 ms with a warp per pixel in FP64, 0.47 ms with a lane each in FP64, 0.15
// ms with the integer sums, 0.12 ms with two lanes each (centre_lanes).
template <class RO, int G>
__global__ void __launch_bounds__(32)
k_line_centre(const __grid_constant__ KProblem pb, const RO *__restrict__ obs, int npix, int W, int lo,
              int hi, double *__restrict__ lam_c, int *__restrict__ idx)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int PIX = 32 / G;
    const int lane = threadIdx.x, nl = pb.n_lambda, sub = lane % G;
    const int pix0 = blockIdx.x * PIX, pix = pix0 + lane / G;
    double y0 = 0.0, y1 = 0.0, y2 = 0.0;
    int bi = 0x7fffffff;
    if (lo <= hi) {
        // I over [lo - W, hi + W], an odd row pitch (conflict-free column reads)
        const int j0 = lo - W, span = hi + W - j0 + 1, pitch = span | 1;
        bool exact = sizeof(RO) == 4;
        if constexpr (sizeof(RO) == 4) {
            long long *t = (long long *)smem;
            const unsigned room = 28 - (32 - __clz(W - 1));  // octaves left beside 25 bits and the terms' carry
            unsigned e_mine = 1u;
            float *raw = (float *)(t + PIX * pitch);  // the rows as they are
            for (int r = 0; r < PIX; ++r) {
                const float *o = obs + (size_t)min(pix0 + r, npix - 1) * 4 * nl + j0;
                for (int j = lane; j < span; j += 32) copy_async(raw + r * pitch + j, o + j);
            }
            copy_wait();
            for (int r = 0; r < PIX && exact; ++r) {
                const float *o = raw + r * pitch;
                unsigned emin = 255u, emax = 1u;
                for (int j = lane; j < span; j += 32) {
                    const unsigned m = __float_as_uint(o[j]) & 0x7fffffffu;
                    const unsigned e = max(m >> 23, 1u);
                    if (m) emin = min(emin, e);
                    emax = max(emax, e);
                }
                emin = __reduce_min_sync(0xffffffffu, emin);
                emax = __reduce_max_sync(0xffffffffu, emax);
                exact = emax < 255u && (emin == 255u || emax - emin <= room);
                emin = min(emin, 254u);  // an all-zero row
                if (r == lane / G) e_mine = emin;
                for (int j = lane; j < span; j += 32) {
                    const unsigned b = __float_as_uint(o[j]), e = (b >> 23) & 0xffu;
                    const unsigned mant = (b & 0x7fffffu) | (e ? 0x800000u : 0u);
                    const long long v = mant ? (long long)mant << min(max(e, 1u) - emin, 63u) : 0;
                    t[r * pitch + j] = (int)b < 0 ? -v : v;
                }
            }
            if (exact) {
                __syncwarp();
                long long s1, s0, s2;
                centre_search<G>(t + (lane / G) * pitch - j0, W, lo, hi, sub, s1, bi, s0, s2);
                const double unit = __hiloint2double((int)((e_mine + 873u) << 20), 0);  // 2^(emin - 150)
                y0 = (double)s0 * unit;
                y1 = (double)s1 * unit;
                y2 = (double)s2 * unit;
            }
        }
        if (!exact) {
            double *t = (double *)smem;
            __syncwarp();
#pragma unroll 8
            for (int r = 0; r < PIX; ++r) {
                const RO *o = obs + (size_t)min(pix0 + r, npix - 1) * 4 * nl + j0;
                for (int j = lane; j < span; j += 32) t[r * pitch + j] = (double)o[j];
            }
            __syncwarp();
            centre_search<G>(t + (lane / G) * pitch - j0, W, lo, hi, sub, y1, bi, y0, y2);
        }
    }
    if (pix >= npix || sub != 0) return;
    if (bi == 0x7fffffff) {
        lam_c[pix] = NAN;
        if (idx) idx[pix] = -1;
        return;
    }
    double xc = pb.lam[bi];
    if (bi - 1 >= lo && bi + 1 <= hi) {
        const double x0 = pb.lam[bi - 1], x1 = pb.lam[bi], x2 = pb.lam[bi + 1];
        const double d0 = __dsub_rn(x1, x0), d2 = __dsub_rn(x1, x2);
        const double e0 = __dsub_rn(y1, y0), e2 = __dsub_rn(y1, y2);
        const double num = __dsub_rn(__dmul_rn(__dmul_rn(d0, d0), e2), __dmul_rn(__dmul_rn(d2, d2), e0));
        const double den = __dsub_rn(__dmul_rn(d0, e2), __dmul_rn(d2, e0));
        if (den != 0.0) xc = __dsub_rn(x1, __dmul_rn(0.5, __ddiv_rn(num, den)));
    }
    lam_c[pix] = xc;
    if (idx) idx[pix] = bi;
}

template <class R> size_t offsets_smem(const KProblem &pb)
{
    return sizeof(R) * (ME_MAX_LINES + (size_t)pb.n_lines * pb.n_lambda);
}

template <class R, int NL, bool FILL, bool JAC>
cudaError_t points_t(const KProblem &pb, const double *params, const double *mu_px, int n, void *stokes, void *jac,
                     cudaStream_t st)
{
    const long long blocks = ((long long)n * pb.n_lambda + kSynthBlock - 1) / kSynthBlock;
    k_points<R, NL, FILL, JAC><<<(int)blocks, kSynthBlock, offsets_smem<R>(pb), st>>>(pb, params, mu_px, n, (R *)stokes,
                                                                                    (R *)jac);
    return cudaGetLastError();
}

template <int NL, bool FILL, bool JAC>
cudaError_t models_t(const KProblem &pb, const double *params, const double *mu_px, int n, void *stokes, void *jac,
                     cudaStream_t st)
{
    constexpr int kWarps = kSynthBlock / 32;
    constexpr int kBlocks = JAC ? kJacMinB : 8;  // resident per SM
    const int chunks = (pb.n_lambda + 31) / 32;
    const int per = chunks_per_warp(JAC, n, pb.n_lambda, pb.n_lines, prof_components(pb), NL > 0 && !has_pattern(pb),
                                    kBlocks);
    if (per == 0) return points_t<float, NL, FILL, JAC>(pb, params, mu_px, n, stokes, jac, st);
    const long long items = (long long)n * ((chunks + per - 1) / per);
    const long long blocks = std::min((items + kWarps - 1) / kWarps, (long long)kSMs * kBlocks);
    const size_t smem = offsets_smem<float>(pb) + (JAC ? sizeof(float) * kWarps * 32 * kNpar<FILL> : 0);
    auto kern = k_models<NL, FILL, JAC>;
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(int)blocks, kSynthBlock, smem, st>>>(pb, params, mu_px, n, per, (float *)stokes, (float *)jac);
    return cudaGetLastError();
}

template <bool FILL>
cudaError_t synth64_t(const KProblem &pb, const double *params, const double *mu_px, int n, void *stokes,
                      cudaStream_t st)
{
    const int blocks = blocks_per_model64(n, pb.n_lambda, prof_components(pb), kProfBlock);
    if (blocks == 0) return points_t<double, 0, FILL, false>(pb, params, mu_px, n, stokes, nullptr, st);
    auto kern = k_synth64<FILL>;
    const size_t smem = prof_smem(pb);
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(n, blocks), kProfBlock, smem, st>>>(pb, params, mu_px, (double *)stokes);
    return cudaGetLastError();
}

template <class R, int NL, bool FILL = false>
cudaError_t vjp_t(const KProblem &pb, const double *params, const double *mu_px, int n,
                  const void *gs, double *gp, cudaStream_t st)
{
    const int per = kSynthBlock / 32;
    k_vjp<R, NL, FILL><<<(n + per - 1) / per, kSynthBlock, offsets_smem<R>(pb), st>>>(pb, params, mu_px, n,
                                                                               (const R *)gs, gp);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_synth(const KProblem &pb, int dtype, const double *params, const double *mu_px,
                         int n, void *stokes, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    if (dtype != ME_F32)
        return pb.fill ? synth64_t<true>(pb, params, mu_px, n, stokes, st)
                       : synth64_t<false>(pb, params, mu_px, n, stokes, st);
    if (pb.fill) return models_t<0, true, false>(pb, params, mu_px, n, stokes, nullptr, st);
    if (pb.n_lines == 1) return models_t<1, false, false>(pb, params, mu_px, n, stokes, nullptr, st);
    if (pb.n_lines == 2) return models_t<2, false, false>(pb, params, mu_px, n, stokes, nullptr, st);
    return models_t<0, false, false>(pb, params, mu_px, n, stokes, nullptr, st);
}

cudaError_t launch_jac(const KProblem &pb, int dtype, const double *params, const double *mu_px,
                       int n, void *stokes, void *jac, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    if (dtype != ME_F32)
        return pb.fill ? points_t<double, 0, true, true>(pb, params, mu_px, n, stokes, jac, st)
                       : points_t<double, 0, false, true>(pb, params, mu_px, n, stokes, jac, st);
    if (pb.fill) return models_t<0, true, true>(pb, params, mu_px, n, stokes, jac, st);
    if (pb.n_lines == 1) return models_t<1, false, true>(pb, params, mu_px, n, stokes, jac, st);
    if (pb.n_lines == 2) return models_t<2, false, true>(pb, params, mu_px, n, stokes, jac, st);
    return models_t<0, false, true>(pb, params, mu_px, n, stokes, jac, st);
}

cudaError_t launch_vjp(const KProblem &pb, int dtype, const double *params, const double *mu_px,
                       int n, const void *gs, double *gp, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    if (pb.fill)
        return dtype == ME_F32 ? vjp_t<float, 0, true>(pb, params, mu_px, n, gs, gp, st)
                               : vjp_t<double, 0, true>(pb, params, mu_px, n, gs, gp, st);
    if (dtype == ME_F32) {
        if (pb.n_lines == 1) return vjp_t<float, 1>(pb, params, mu_px, n, gs, gp, st);
        if (pb.n_lines == 2) return vjp_t<float, 2>(pb, params, mu_px, n, gs, gp, st);
        return vjp_t<float, 0>(pb, params, mu_px, n, gs, gp, st);
    }
    return vjp_t<double, 0>(pb, params, mu_px, n, gs, gp, st);
}

namespace {

template <class RO, int G>
cudaError_t line_centre_t(const KProblem &pb, const void *obs, int npix, int W, int lo, int hi, double *lam_c,
                          int *idx, cudaStream_t st)
{
    constexpr int PIX = 32 / G;
    const int smem = lo <= hi ? PIX * ((hi - lo + 2 * W + 1) | 1) * (sizeof(RO) == 4 ? 12 : 8) : 0;
    auto kern = k_line_centre<RO, G>;
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(npix + PIX - 1) / PIX, 32, smem, st>>>(pb, (const RO *)obs, npix, W, lo, hi, lam_c, idx);
    return cudaGetLastError();
}

template <class RO>
cudaError_t line_centre_r(const KProblem &pb, const void *obs, int npix, int W, int lo, int hi, double *lam_c,
                          int *idx, cudaStream_t st)
{
    switch (lo <= hi ? centre_lanes(sizeof(RO) == 4, npix, hi - lo + 1, W, sizeof(RO) == 4 ? 12 : 8) : 1) {
    case 32: return line_centre_t<RO, 32>(pb, obs, npix, W, lo, hi, lam_c, idx, st);
    case 8: return line_centre_t<RO, 8>(pb, obs, npix, W, lo, hi, lam_c, idx, st);
    case 2: return line_centre_t<RO, 2>(pb, obs, npix, W, lo, hi, lam_c, idx, st);
    default: return line_centre_t<RO, 1>(pb, obs, npix, W, lo, hi, lam_c, idx, st);
    }
}

}  // namespace

cudaError_t launch_line_centre(const KProblem &pb, int dtype, const void *obs, int npix, int W, int lo,
                               int hi, double *lam_c, int *idx, cudaStream_t st)
{
    if (npix <= 0) return cudaSuccess;
    return dtype == ME_F32 ? line_centre_r<float>(pb, obs, npix, W, lo, hi, lam_c, idx, st)
                           : line_centre_r<double>(pb, obs, npix, W, lo, hi, lam_c, idx, st);
}

template <class RO, bool FILL>
static cudaError_t chi2_t(const KProblem &pb, const void *obs, const double *w, const double *mu_px, int npix,
                          const double *params, double *chi2, cudaStream_t st, KSub sub)
{
    auto kern = k_chi2_f64<RO, FILL>;
    const size_t smem = prof_smem(pb);
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<npix, kProfBlock, smem, st>>>(pb, (const RO *)obs, w, mu_px, npix, params, chi2, sub);
    return cudaGetLastError();
}

cudaError_t launch_chi2_f64(const KProblem &pb, int dtype, const void *obs, const double *w,
                            const double *mu_px, int npix, const double *params, double *chi2,
                            cudaStream_t st, KSub sub)
{
    if (npix <= 0) return cudaSuccess;
    if (dtype == ME_F32)
        return pb.fill ? chi2_t<float, true>(pb, obs, w, mu_px, npix, params, chi2, st, sub)
                       : chi2_t<float, false>(pb, obs, w, mu_px, npix, params, chi2, st, sub);
    return pb.fill ? chi2_t<double, true>(pb, obs, w, mu_px, npix, params, chi2, st, sub)
                   : chi2_t<double, false>(pb, obs, w, mu_px, npix, params, chi2, st, sub);
}

}  // namespace genesis
