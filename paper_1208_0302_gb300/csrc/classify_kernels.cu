// Section 2 pixel selection and weak-field fallback, Section 5.5 seeds and
// polarity, and the order-preserving selection of the pixels to invert.
#include "async_copy.cuh"
#include "fp64_util.cuh"
#include "kernels.h"
#include "launch_rules.h"

namespace genesis {

namespace {

constexpr int kSelectTile = 2048;    // flags per selection tile
constexpr int kSelectBlock = 256;    // threads per selection block, 8 flags each
constexpr double kPi = 3.14159265358979323846;

// Tile counts of me_select_static: a file-scope device array sized for
// ME_SELECT_STATIC_MAX_PIX flags (8192 tiles, 32 KiB).  Every slot a call uses
// is written by its count pass before the scan reads it, so nothing has to
// start at zero; concurrent calls share it and therefore race.
static __device__ __align__(256) int g_select_tiles[(ME_SELECT_STATIC_MAX_PIX + kSelectTile - 1) / kSelectTile];

// Three-point parabola vertex through (x0, y0), (x1, y1), (x2, y2), without
// contraction; x1 when the points are collinear.
__device__ __forceinline__ double vertex3(double x0, double x1, double x2, double y0, double y1, double y2)
{
    const double d0 = __dsub_rn(x1, x0), d2 = __dsub_rn(x1, x2);
    const double e0 = __dsub_rn(y1, y0), e2 = __dsub_rn(y1, y2);
    const double num = __dsub_rn(__dmul_rn(__dmul_rn(d0, d0), e2), __dmul_rn(__dmul_rn(d2, d2), e0));
    const double den = __dsub_rn(__dmul_rn(d0, e2), __dmul_rn(d2, e0));
    return den != 0.0 ? __dsub_rn(x1, __ddiv_rn(__dmul_rn(0.5, num), den)) : x1;
}

// Trapezoid weight of point j in the window [lo, hi].
__device__ __forceinline__ double trap_w(const double *lam, int lo, int hi, int j)
{
    if (lo == hi) return 0.0;
    const double a = j > lo ? __dsub_rn(lam[j], lam[j - 1]) : 0.0;
    const double b = j < hi ? __dsub_rn(lam[j + 1], lam[j]) : 0.0;
    return __dmul_rn(0.5, __dadd_rn(a, b));
}

__device__ __forceinline__ double degrees(double rad) { return __ddiv_rn(__dmul_rn(rad, 180.0), kPi); }

// A seed (B, psi, chi) from B_par and B_perp, psi reflected into the pixel's
// polarity half.
__device__ __forceinline__ void put_seed(double *sd, double bpar, double bperp, double psi, double chi, int pol)
{
    if ((pol > 0 && psi > 90.0) || (pol < 0 && psi < 90.0)) psi = __dsub_rn(180.0, psi);
    sd[0] = __dsqrt_rn(__dadd_rn(__dmul_rn(bpar, bpar), __dmul_rn(bperp, bperp)));
    sd[1] = psi;
    sd[2] = chi;
}

// An integer in the order of the finite doubles (-0 and +0 equal): FP64
// comparisons take the FP64 pipe, integer ones do not.
__device__ __forceinline__ long long order64(double x)
{
    const long long b = __double_as_longlong(x);
    return b == (long long)0x8000000000000000ull ? 0 : b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// The largest |x|, at least 0, NaN ignored.  FP64 ones compare as integers,
// off the FP64 pipe.
template <class RO> struct AbsMax {
    RO v = 0;
    __device__ __forceinline__ void add(RO x) { v = max_of(v, abs_of(x)); }
    __device__ __forceinline__ double get() const { return (double)v; }
};
template <> struct AbsMax<double> {
    long long b = 0;
    __device__ __forceinline__ void add(double x)
    {
        const long long m = __double_as_longlong(x) & 0x7fffffffffffffffll;
        if (m > b && m <= 0x7ff0000000000000ll) b = m;
    }
    __device__ __forceinline__ double get() const { return __longlong_as_double(b); }
};

constexpr int kChunk = 32;            // wavelengths staged at once
constexpr int kPitch = kChunk + 1;    // tile row pitch: a column read touches 32 banks

// Stage wavelengths [j0, j0 + kChunk) of the warp's 32 pixels: t[s][pixel]
// [j - j0], rows beyond the map repeating its last pixel.
template <class RO>
__device__ __forceinline__ void stage_chunk(RO *t, const RO *obs, int nl, int pix0, int npix, int j0)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();  // the tile's readers are done
    if (j0 + lane < nl) {
#pragma unroll 8
        for (int r = 0; r < 32; ++r) {
            const RO *o = obs + (size_t)min(pix0 + r, npix - 1) * 4 * nl + j0 + lane;
#pragma unroll
            for (int s = 0; s < 4; ++s) copy_async(t + (s * 32 + r) * kPitch + lane, o + (size_t)s * nl);
        }
    }
    copy_wait();
}

// Wavelength-only factors of the sums, the same for every pixel: h = lam[j+1]
// - lam[j], the second difference's denominator h1 h2 (h1 + h2) at j, their
// reciprocals (known_rcp), and the trapezoid weight of j in the line window.
struct GridTables {
    double h, rh, den, rden, wt;
};

// What the two warps of a ROLES = 2 block tell each other, per pixel.
struct ClassifyExchange {
    double qa, ub, dd, tvi, tvd;  // from the first
    int ip, im, pol;              // from the second
};

// Section 2 threshold, weak-field estimate, polarity and seeds in FP64, one
// pixel per lane.  Each running sum is taken in increasing index, so every
// result except the angles (atan2) repeats the plain sequential evaluation
// bit for bit.  Bound by the FP64 pipe, which takes 16 clocks of an SM per
// warp instruction whether one lane or all 32 are active: with a warp per
// pixel (its sums on 15 lanes, six divergent groups) an instruction served
// one pixel, here it serves 32.  The lanes read their pixels' columns of a
// tile that the warp stages 32 wavelengths at a time (rows of 128 bytes, so
// HBM reads stay coalesced; pitch 33, so the column reads are conflict-free).
// Extrema of the observed values are compared in their own type and those of
// I +- V as integers, off the FP64 pipe.  262 144 two-line pixels of a float
// cube: 48.5 ms with a warp per pixel, 1.29 ms
// with a lane.
// One warp per block, so that the blocks spread evenly over the SMs.  ROLES =
// 2 gives a block's 32 pixels a second warp that takes the sums of V, L and
// the centres of gravity: at one warp to an SM partition the chain of dependent
// FP64 operations is the time, and this shortens it (64 pixels: 104 -> 68 us).
template <class RO, int ROLES>
__global__ void __launch_bounds__(ROLES * 32)
k_classify(const __grid_constant__ KProblem pb, const RO *__restrict__ obs, int npix, const KClassify c)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int nl = pb.n_lambda, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool role_a = ROLES == 1 || warp == 0, role_b = ROLES == 1 || warp == 1;
    const double *lam = pb.lam;
    const int lo = c.c_lo, hi = c.c_hi;
    GridTables *tab = (GridTables *)smem;
    RO *t = (RO *)(tab + nl) + warp * 4 * 32 * kPitch;
    for (int j = max(lo - 1, 0) + threadIdx.x; j <= min(hi + 1, nl - 1); j += blockDim.x) {
        GridTables g = {};
        if (j + 1 < nl) {
            g.h = __dsub_rn(lam[j + 1], lam[j]);
            g.rh = known_rcp(g.h);
            if (j > 0) {
                const double h1 = __dsub_rn(lam[j], lam[j - 1]);
                g.den = __dmul_rn(__dmul_rn(h1, g.h), __dadd_rn(h1, g.h));
                g.rden = known_rcp(g.den);
            }
        }
        if (j >= lo && j <= hi) g.wt = trap_w(lam, lo, hi, j);
        tab[j] = g;
    }
    __syncthreads();
    const int pix0 = blockIdx.x * 32;
    const int pix = pix0 + lane;
    const RO *col = t + lane * kPitch;  // this lane's pixel, Stokes s at col[s * 32 * kPitch]
    constexpr int S = 32 * kPitch;
    int staged = -1;
    auto stage = [&](int j0) {
        if (staged != j0) stage_chunk(t, obs, nl, pix0, npix, j0);
        staged = j0;
    };

    // quiet-window means of I, Q, U, V and variances of Q, U, V
    const double nq = (double)(c.q_hi - c.q_lo);
    double mean[4] = {0.0, 0.0, 0.0, 0.0}, var[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j0 = c.q_lo / kChunk * kChunk; j0 < c.q_hi; j0 += kChunk) {
        stage(j0);
        for (int j = max(j0, c.q_lo); j < min(j0 + kChunk, c.q_hi); ++j)
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (role_a || s == 0) mean[s] = __dadd_rn(mean[s], widen(col[s * S + j - j0]));
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
        if (role_a || s == 0) mean[s] = __ddiv_rn(mean[s], nq);
    if (role_a) {
        for (int j0 = c.q_lo / kChunk * kChunk; j0 < c.q_hi; j0 += kChunk) {
            stage(j0);
            for (int j = max(j0, c.q_lo); j < min(j0 + kChunk, c.q_hi); ++j)
#pragma unroll
                for (int s = 1; s < 4; ++s) {
                    const double d = __dsub_rn(widen(col[s * S + j - j0]), mean[s]);
                    var[s] = __dadd_rn(var[s], __dmul_rn(d, d));
                }
        }
#pragma unroll
        for (int s = 1; s < 4; ++s) var[s] = __ddiv_rn(var[s], nq);
    }
    const double ic = mean[0];

    // one pass over the grid: extrema of |Q|, |U|, |V|; in the line window the
    // I+V, I-V cores, the V lobes and the sums
    AbsMax<RO> qx, ux, vx;
    RO vhi = 0, vlo = 0;
    long long vp = 0, vm = 0;
    int ip = hi + 1, im = hi + 1, jhi = hi + 1, jlo = hi + 1;
    double qa = 0.0, ub = 0.0, dd = 0.0;    // least-squares sums of Q I'', U I'', I''^2
    double av = 0.0, al = 0.0;              // trapezoid integrals of |V| and L
    double tvi = 0.0, tvd = 0.0;            // total variation of I and I'
    double np = 0.0, dp = 0.0, nm = 0.0, dm = 0.0;  // centre-of-gravity moments of I_c - (I +- V)
    double y1 = 0.0, q1 = 0.0, u1 = 0.0;  // I, Q, U at j-1
    double e1 = 0.0, sl1 = 0.0;           // I[j-1] - I[j-2] and its slope
    for (int j0 = 0; j0 < nl; j0 += kChunk) {
        const int j1 = min(j0 + kChunk, nl);
        if (!role_a && (j1 <= lo || j0 > hi)) continue;  // only the line window matters to the second role
        stage(j0);
        if (role_a) {  // on its own: inside the next loop 64 double pixels of 512 wavelengths took 195 us, now 110
#pragma unroll 8
            for (int j = 0; j < j1 - j0; ++j) {
                qx.add(col[S + j]);
                ux.add(col[2 * S + j]);
                vx.add(col[3 * S + j]);
            }
        }
        for (int j = max(j0, lo - 2); j < min(j1, hi + 2); ++j) {
            const RO qr = col[S + j - j0], ur = col[2 * S + j - j0], vr = col[3 * S + j - j0];
            const double I = widen(col[j - j0]), Q = widen(qr), U = widen(ur);
            if (role_a) {
                const double e = __dsub_rn(I, y1);
                const int m = j - 1;  // the point whose neighbours are now known
                if (m >= lo && m >= 1 && m <= hi) {
                    const double h1 = tab[m - 1].h, h2 = tab[m].h;
                    const double num = __dsub_rn(__dmul_rn(h1, e), __dmul_rn(h2, e1));
                    const double d2 = div_known(__dadd_rn(num, num), tab[m].den, tab[m].rden);
                    qa = __dadd_rn(qa, __dmul_rn(q1, d2));
                    ub = __dadd_rn(ub, __dmul_rn(u1, d2));
                    dd = __dadd_rn(dd, __dmul_rn(d2, d2));
                }
                if (m >= lo && j <= hi) {
                    tvi = __dadd_rn(tvi, fabs(e));
                    const double sl = div_known(e, tab[m].h, tab[m].rh);
                    if (m > lo) tvd = __dadd_rn(tvd, fabs(__dsub_rn(sl, sl1)));
                    sl1 = sl;
                }
                y1 = I;
                q1 = Q;
                u1 = U;
                e1 = e;
            }
            if (role_b && j >= lo && j <= hi) {
                const double V = widen(vr), wt = tab[j].wt, lj = lam[j];
                const double a = __dadd_rn(I, V), b = __dsub_rn(I, V);
                const long long ka = order64(a), kb = order64(b);
                if (j == lo || ka < vp) { vp = ka; ip = j; }
                if (j == lo || kb < vm) { vm = kb; im = j; }
                if (j == lo || vr > vhi) { vhi = vr; jhi = j; }
                if (j == lo || vr < vlo) { vlo = vr; jlo = j; }
                av = __dadd_rn(av, __dmul_rn(wt, fabs(V)));
                al = __dadd_rn(al, __dmul_rn(wt, __dsqrt_rn(__dadd_rn(__dmul_rn(Q, Q), __dmul_rn(U, U)))));
                const double ga = __dmul_rn(wt, __dsub_rn(ic, a)), gb = __dmul_rn(wt, __dsub_rn(ic, b));
                np = __dadd_rn(np, __dmul_rn(ga, lj));
                dp = __dadd_rn(dp, ga);
                nm = __dadd_rn(nm, __dmul_rn(gb, lj));
                dm = __dadd_rn(dm, gb);
            }
        }
    }
    int pol = jhi < jlo ? 1 : (jhi > jlo ? -1 : 0);
    if (ROLES == 2) {
        __shared__ ClassifyExchange s_x[32];
        ClassifyExchange &x = s_x[lane];
        if (role_a) {
            x.qa = qa;
            x.ub = ub;
            x.dd = dd;
            x.tvi = tvi;
            x.tvd = tvd;
        } else {
            x.ip = ip;
            x.im = im;
            x.pol = pol;
        }
        __syncthreads();
        qa = x.qa;
        ub = x.ub;
        dd = x.dd;
        tvi = x.tvi;
        tvd = x.tvd;
        ip = x.ip;
        im = x.im;
        pol = x.pol;
    }
    if (pix >= npix) return;
    const RO *o = obs + (size_t)pix * 4 * nl;

    // weak field
    const double two_kz = __dmul_rn(2.0, c.kz);
    double chi = degrees(__dmul_rn(0.5, atan2(-ub, -qa)));
    if (chi < 0.0) chi = __dadd_rn(chi, 180.0);
    const double amp = __dsqrt_rn(__dadd_rn(__dmul_rn(qa, qa), __dmul_rn(ub, ub)));
    const double bperp = dd > 0.0 ? __ddiv_rn(__dsqrt_rn(__ddiv_rn(__dmul_rn(4.0, amp), dd)), c.kz) : 0.0;
    double *sd = c.seeds ? c.seeds + (size_t)pix * 12 : nullptr;
    if (role_b && sd) {
        const double bpi = tvi > 0.0 ? __ddiv_rn(__dmul_rn(pol < 0 ? -1.0 : 1.0, av), __dmul_rn(c.kz, tvi)) : 0.0;
        const double bti = tvd > 0.0 ? __ddiv_rn(__dsqrt_rn(__ddiv_rn(__dmul_rn(4.0, al), tvd)), c.kz) : 0.0;
        put_seed(sd + 3, bpi, bti, degrees(atan2(bti, bpi)), chi, pol);
        const double bcog =
            (dp != 0.0 && dm != 0.0) ? __ddiv_rn(__dsub_rn(__ddiv_rn(np, dp), __ddiv_rn(nm, dm)), two_kz) : 0.0;
        put_seed(sd + 6, bcog, bperp, degrees(atan2(bperp, bcog)), chi, pol);
    }
    if (!role_a) return;

    // threshold
    const double qd = qx.get(), ud = ux.get(), vd = vx.get();
    const double p = __ddiv_rn(
        __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(qd, qd), __dmul_rn(ud, ud)), __dmul_rn(vd, vd))), ic);
    const double sp = __ddiv_rn(__dmul_rn(c.p_thresh, __dsqrt_rn(__dadd_rn(__dadd_rn(var[1], var[2]), var[3]))), ic);
    const int flag = p > sp ? 1 : 0;

    auto core = [&](int bi, bool plus) {
        if (bi - 1 < 0 || bi + 1 >= nl) return lam[bi];
        double y[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double I = (double)o[bi - 1 + k], V = (double)o[3 * nl + bi - 1 + k];
            y[k] = plus ? __dadd_rn(I, V) : __dsub_rn(I, V);
        }
        return vertex3(lam[bi - 1], lam[bi], lam[bi + 1], y[0], y[1], y[2]);
    };
    const double bpar = __ddiv_rn(__dsub_rn(core(ip, true), core(im, false)), two_kz);
    const double bmag = __dsqrt_rn(__dadd_rn(__dmul_rn(bpar, bpar), __dmul_rn(bperp, bperp)));
    const double theta = degrees(atan2(bperp, bpar));

    if (c.flag) c.flag[pix] = flag;
    if (c.polarity) c.polarity[pix] = pol;
    if (c.pol) {
        c.pol[(size_t)pix * 2] = p;
        c.pol[(size_t)pix * 2 + 1] = sp;
    }
    if (c.weak) {
        double *wo = c.weak + (size_t)pix * 5;
        wo[0] = bmag;
        wo[1] = theta;
        wo[2] = chi;
        wo[3] = bpar;
        wo[4] = bperp;
    }
    if (sd) {
        put_seed(sd, bpar, bperp, theta, chi, pol);
        put_seed(sd + 9, bpar, bperp, theta, chi, pol);
        sd[9] = 0.0;
    }
    if (c.best && !flag) {  // weak-field answer for the pixels below the threshold
        double *bo = c.best + (size_t)pix * c.npar;
        bo[0] = bmag;
        bo[1] = theta;
        bo[2] = chi;
        for (int d = 3; d < c.npar; ++d) bo[d] = __longlong_as_double(0x7ff8000000000000ll);
    }
}

// ------------------------------------------------------------- selection
// Three passes over tiles of kSelectTile flags: count per tile, exclusive
// scan of the tile counts (one block), and a scatter that re-counts inside
// each tile.  Each thread owns 8 consecutive flags, so indices come out in
// increasing order.

__device__ __forceinline__ int block_exclusive_scan(int x, int *s_warp, int &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int inc = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = lane < nw ? s_warp[lane] : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += y;
        }
        if (lane < nw) s_warp[lane] = w;  // inclusive prefix over warps
    }
    __syncthreads();
    total = s_warp[nw - 1];
    const int base = warp > 0 ? s_warp[warp - 1] : 0;
    __syncthreads();  // s_warp may be reused by the caller
    return base + inc - x;
}

__device__ __forceinline__ int tile_flags(const int *flag, int npix, int want, int first, unsigned &bits)
{
    int n = 0;
    bits = 0;
#pragma unroll
    for (int e = 0; e < kSelectTile / kSelectBlock; ++e) {
        const int i = first + e;
        if (i < npix && flag[i] == want) {
            bits |= 1u << e;
            ++n;
        }
    }
    return n;
}

__global__ void __launch_bounds__(kSelectBlock)
k_select_count(const int *__restrict__ flag, int npix, int want, int *__restrict__ tile_count)
{
    __shared__ int s_warp[32];
    unsigned bits;
    const int first = blockIdx.x * kSelectTile + threadIdx.x * (kSelectTile / kSelectBlock);
    int total;
    block_exclusive_scan(tile_flags(flag, npix, want, first, bits), s_warp, total);
    if (threadIdx.x == 0) tile_count[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_select_scan(int *__restrict__ tile, int ntiles, int *__restrict__ count)
{
    __shared__ int s_warp[32];
    const int per = (ntiles + blockDim.x - 1) / blockDim.x;
    const int t0 = threadIdx.x * per, t1 = min(t0 + per, ntiles);
    int sum = 0;
    for (int t = t0; t < t1; ++t) sum += tile[t];
    int total;
    int off = block_exclusive_scan(sum, s_warp, total);
    for (int t = t0; t < t1; ++t) {
        const int n = tile[t];
        tile[t] = off;
        off += n;
    }
    if (threadIdx.x == 0) *count = total;
}

__global__ void __launch_bounds__(kSelectBlock)
k_select_scatter(const int *__restrict__ flag, int npix, int want, const int *__restrict__ tile_off,
                 int *__restrict__ index)
{
    __shared__ int s_warp[32];
    unsigned bits;
    const int first = blockIdx.x * kSelectTile + threadIdx.x * (kSelectTile / kSelectBlock);
    int total;
    int pos = tile_off[blockIdx.x] + block_exclusive_scan(tile_flags(flag, npix, want, first, bits), s_warp, total);
#pragma unroll
    for (int e = 0; e < kSelectTile / kSelectBlock; ++e)
        if (bits & (1u << e)) index[pos++] = first + e;
}

// Section 5.3 bound rule, one thread per (pixel, parameter): [max(lo,
// p - lower), min(hi, p + upper)], the global interval where that is empty
// or the prefit is NaN.
__global__ void k_prefit_bounds(const double *__restrict__ p_hat, int npix, const KPrefitBounds r,
                                double *__restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int M = r.npar;
    if (i >= npix * M) return;
    const int pix = i / M, k = i - pix * M;
    const double p = p_hat[i];
    double a = __dsub_rn(p, r.lower[k]), b = __dadd_rn(p, r.upper[k]);
    if (!(a > r.lo[k])) a = r.lo[k];
    if (!(b < r.hi[k])) b = r.hi[k];
    if (!(a < b)) {
        a = r.lo[k];
        b = r.hi[k];
    }
    out[(size_t)pix * 2 * M + k] = a;
    out[(size_t)pix * 2 * M + M + k] = b;
}

}  // namespace

cudaError_t launch_prefit_bounds(const double *p_hat, int npix, const KPrefitBounds &r, double *out,
                                 cudaStream_t st)
{
    if (npix <= 0) return cudaSuccess;
    const int n = npix * r.npar;
    k_prefit_bounds<<<(n + 255) / 256, 256, 0, st>>>(p_hat, npix, r, out);
    return cudaGetLastError();
}

namespace {

template <class RO, int ROLES>
cudaError_t classify_t(const KProblem &pb, const void *obs, int npix, const KClassify &c, cudaStream_t st)
{
    const int smem = pb.n_lambda * (int)sizeof(GridTables) + ROLES * 4 * 32 * kPitch * (int)sizeof(RO);
    auto kern = k_classify<RO, ROLES>;
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(npix + 31) / 32, 32 * ROLES, smem, st>>>(pb, (const RO *)obs, npix, c);
    return cudaGetLastError();
}

}  // namespace

// The second role pays while two warps for every 32 pixels are at most one to
// each of the 608 SM partitions; beyond that the FP64 pipe is the limit.
cudaError_t launch_classify(const KProblem &pb, int dtype, const void *obs, int npix, const KClassify &c,
                            cudaStream_t st)
{
    if (npix <= 0) return cudaSuccess;
    const bool chain = npix <= kSMs * 4 / 2 * 32;
    if (dtype == ME_F32) return chain ? classify_t<float, 2>(pb, obs, npix, c, st) : classify_t<float, 1>(pb, obs, npix, c, st);
    return chain ? classify_t<double, 2>(pb, obs, npix, c, st) : classify_t<double, 1>(pb, obs, npix, c, st);
}

cudaError_t select_static_scratch(void **ptr, size_t *bytes)
{
    *bytes = sizeof(g_select_tiles);
    return cudaGetSymbolAddress(ptr, g_select_tiles);
}

size_t select_scratch_bytes(int npix)
{
    const size_t ntiles = npix > 0 ? ((size_t)npix + kSelectTile - 1) / kSelectTile : 0;
    return ntiles * sizeof(int);
}

cudaError_t launch_select(const int *flag, int npix, int want, int *index, int *count, void *scratch,
                          cudaStream_t st)
{
    if (npix <= 0) return cudaMemsetAsync(count, 0, sizeof(int), st);
    const int ntiles = (npix + kSelectTile - 1) / kSelectTile;
    int *tile = (int *)scratch;
    k_select_count<<<ntiles, kSelectBlock, 0, st>>>(flag, npix, want, tile);
    k_select_scan<<<1, 1024, 0, st>>>(tile, ntiles, count);
    k_select_scatter<<<ntiles, kSelectBlock, 0, st>>>(flag, npix, want, tile, index);
    return cudaGetLastError();
}

}  // namespace genesis
