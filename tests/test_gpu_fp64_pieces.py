"""The pieces of the FP64 profiles one by one, in a program of their own: the
reciprocal, the division by a known divisor and the conversions against CUDA's
own, and w(z) from the cells, the nodes and the convergents against 40-digit
values, on both sides of every region's edge."""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

mp = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1208_0302_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "profiles64.cuh"
using namespace genesis;
namespace genesis {
cudaError_t unused(const HostTables &t) { return cudaMemcpyToSymbol(c_fad, &t.fad, sizeof(FaddeevaTables)); }
}
static __device__ double2 d_table[(kNodeBelow + kNodeGrid) * kNodeGrid * kNodeCoef];

// out: 1/d, Newton and CUDA's; a/b known and CUDA's; f widened and converted; |d| narrowed and truncated
__global__ void k_scalar(const double *a, const double *b, const float *f, int n, double *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double *o = out + 8 * (size_t)i;
    o[0] = rcp_newton(b[i]);
    o[1] = __drcp_rn(b[i]);
    o[2] = div_known(a[i], b[i], known_rcp(b[i]));
    o[3] = __ddiv_rn(a[i], b[i]);
    o[4] = widen(f[i]);
    o[5] = (double)f[i];
    o[6] = narrow(fabs(b[i]));
    o[7] = __double2float_rz(fabs(b[i]));
}

// One warp per y: w(x + i y) by the cells, the nodes, the 9th, 7th and 5th
// convergents and by a thread on its own, for nx values of x each.
__global__ void __launch_bounds__(32) k_profiles(const double2 *nodes, const double *ys, const double *xs, int nx, double2 *out)
{
    __shared__ ProfShared S;
    const double y = ys[blockIdx.x];
    build_cells(S, nodes, y);
    build_exterior(S, y);
    __syncwarp();
    double dy;
    const double2 *row = node_row(nodes, y, dy);
    for (int i = threadIdx.x; i < nx; i += 32) {
        const double x = xs[(size_t)blockIdx.x * nx + i];
        double2 *o = out + ((size_t)blockIdx.x * nx + i) * 6;
        const C2<double> n = from_node(row, fabs(x) < 10.0 ? x : 10.0, dy), t = profile_alone(row, dy, x, y, y * y);
        o[0] = from_cells(S, fabs(x) < 10.0 ? x : 10.0);
        o[1] = make_double2(n.x, n.y);
        o[2] = convergent<9>(S.ext + 21, x, y * y);
        o[3] = convergent<7>(S.ext + 9, x, y * y);
        o[4] = convergent<5>(S.ext, x, y * y);
        o[5] = make_double2(t.x, t.y);
    }
}

template <class T> std::vector<T> get(FILE *f, size_t n)
{
    std::vector<T> v(n);
    if (fread(v.data(), sizeof(T), n, f) != n) v.clear();
    return v;
}
template <class T> T *up(const std::vector<T> &v)
{
    T *p = nullptr;
    cudaMalloc(&p, v.size() * sizeof(T));
    cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
    return p;
}
template <class T> void put(FILE *f, const T *d, size_t n)
{
    std::vector<T> v(n);
    cudaMemcpy(v.data(), d, n * sizeof(T), cudaMemcpyDeviceToHost);
    fwrite(v.data(), sizeof(T), n, f);
}
int main(int argc, char **argv)
{
    if (argc < 6) return 2;
    const int n = atoi(argv[3]), ny = atoi(argv[4]), nx = atoi(argv[5]);
    FILE *in = fopen(argv[1], "rb"), *to = fopen(argv[2], "wb");
    if (!in || !to) return 3;
    const auto a = get<double>(in, n), b = get<double>(in, n);
    const auto f = get<float>(in, n);
    const auto y = get<double>(in, ny), x = get<double>(in, (size_t)ny * nx);
    if (a.empty() || b.empty() || f.empty() || y.empty() || x.empty()) return 4;
    const auto low = faddeeva_nodes_below(), high = faddeeva_nodes();
    cudaMemcpyToSymbol(d_table, low.data(), low.size() * 8);
    cudaMemcpyToSymbol(d_table, high.data(), high.size() * 8, low.size() * 8);
    void *table = nullptr;
    cudaGetSymbolAddress(&table, d_table);
    double *o = up(std::vector<double>((size_t)n * 8));
    k_scalar<<<(n + 127) / 128, 128>>>(up(a), up(b), up(f), n, o);
    double2 *w = up(std::vector<double2>((size_t)ny * nx * 6));
    k_profiles<<<ny, 32>>>((const double2 *)((char *)table + low.size() * 8), up(y), up(x), nx, w);
    if (cudaDeviceSynchronize() != cudaSuccess) return 5;
    put(to, o, (size_t)n * 8);
    put(to, w, (size_t)ny * nx * 6);
    fclose(to);
    return 0;
}
"""


def _inputs():
    r = np.random.default_rng(11)
    n = 1 << 20
    sign = lambda: np.where(r.random(n) < 0.5, -1.0, 1.0)
    a = sign() * np.ldexp(1.0 + r.random(n), r.integers(-690, 690, n))
    b = sign() * np.ldexp(1.0 + r.random(n), r.integers(-1000, 1000, n))
    near = slice(0, n // 2)  # divisors near which quotients are hard to round, in the range of a known reciprocal
    b[near] = sign()[near] * np.ldexp(1.0 + r.integers(0, 64, n)[near] * 2.0 ** -52 * r.choice([1, -1], n)[near],
                                      r.integers(-190, 190, n)[near])
    b[:4] = [1.0, -1.0, 3.0, 1.5]
    a[:8] = [0.0, -0.0, 1.0, 1e-320, np.inf, np.nan, 1e300, -1e-300]
    f = np.frombuffer(r.integers(0, 1 << 32, n, dtype=np.uint32).tobytes(), dtype=np.float32).copy()
    f[:9] = [0.0, -0.0, 1e-45, -1e-40, np.inf, -np.inf, np.nan, 3.4e38, 1.1754944e-38]
    # dampings about the nodes, the cells and the ends of the grid; x about the regions' edges and the cells'
    ys = np.array([0.0, 1e-310, 1e-9, 0.039, 0.0390625, 0.0391, 0.3, 1.0, 3.3, 7.07, 9.9, 9.96, 10.0, 12.0, 22.0, -0.0, -1e-3, -0.9])
    xs = np.empty((len(ys), 128))
    for i, y in enumerate(ys):
        edges = [np.sqrt(max(e - y * y, 0.0)) for e in (100.0, 170.0, 500.0)]
        about = [e * s for e in edges for s in (1 - 1e-12, 1 + 1e-12, 0.97, 1.03)]
        cells = [0.3125, 0.3125 - 1e-9, 3.125, 9.84375, 0.0390625, 5.0390625]
        some = np.concatenate([about, cells, [0.0, 1e-300, 1e-8, 30.0, 300.0, 1e4]])
        xs[i] = np.concatenate([some, r.uniform(0, 10, 60), r.uniform(10, 26, 128 - 60 - len(some))])
        xs[i, ::3] *= -1.0
    return a, b, f, ys, xs


@pytest.fixture(scope="module")
def pieces(tmp_path_factory):
    from paper_1208_0302_gb300 import build
    d = tmp_path_factory.mktemp("pieces")
    (d / "p.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-o", str(d / "p"), str(d / "p.cu")], check=True)
    a, b, f, ys, xs = _inputs()
    (d / "in").write_bytes(a.tobytes() + b.tobytes() + f.tobytes() + ys.tobytes() + xs.tobytes())
    subprocess.run([str(d / "p"), str(d / "in"), str(d / "out"), str(len(a)), str(len(ys)), str(xs.shape[1])], check=True,
                   timeout=120)
    raw = np.fromfile(d / "out")
    n = len(a) * 8
    return a, b, f, ys, xs, raw[:n].reshape(-1, 8), raw[n:].reshape(len(ys), xs.shape[1], 6, 2)


def test_reciprocal_division_conversions(pieces):
    a, b, f, _, _, o, _ = pieces
    assert np.max(np.abs(o[:, 0] - o[:, 1]) / np.spacing(np.abs(o[:, 1]))) <= 1.0  # within an ulp
    assert np.array_equal(o[:, 2], o[:, 3], equal_nan=True)                        # correctly rounded
    assert np.array_equal(o[:, 4], o[:, 5], equal_nan=True)
    assert np.array_equal(np.signbit(o[:, 4]), np.signbit(o[:, 5]))
    big, small = np.abs(b) >= 2.0 ** 128, np.abs(b) < 2.0 ** -126
    inside = ~big & ~small
    assert np.array_equal(o[inside, 6], o[inside, 7])
    assert np.all(o[small, 6] == 0.0) and np.all(o[big, 6] == np.finfo(np.float32).max)


def test_profiles_against_forty_digits(pieces):
    ys, xs, got = pieces[3], pieces[4], pieces[6]
    mp.mp.dps = 40
    for i, y in enumerate(ys):
        for j, x in enumerate(xs[i]):
            z = mp.mpc(x, y)
            w = mp.exp(-z * z) * mp.erfc(-1j * z)
            err = [float(abs(mp.mpc(*map(float, g)) - w)) for g in got[i, j]]
            s, mag = x * x + y * y, float(abs(w))
            # Taylor polynomials: the coefficients' rounding and one per Horner step of ratio < 1/6, 3 2^-53 in all,
            # truncation below 1.2e-16 of w (1e-14 below the axis), and the cancellation in c_1 = -2 z w + 1.13,
            # whose rounding enters times a step of 0.16
            inner = (3 * 2.0 ** -53 + (1.2e-16 if y >= 0 else 1e-14)) * max(mag, 1.0 if y < 0 else mag) + 1e-16
            # convergents: polynomials of degree <= 9, two roundings a degree in numerator and denominator, the
            # reciprocal and two products; truncation below 3e-17
            outer = 40 * 2.0 ** -53 * mag + 3e-17
            if s < 100.0 and abs(x) < 10.0:
                assert err[0] <= inner and err[1] <= inner, (x, y, err, mag)
            if 100.0 <= s:
                assert err[2] <= outer, (x, y, err, mag)
            if 170.0 <= s:
                assert err[3] <= outer, (x, y, err, mag)
            if 500.0 <= s:
                assert err[4] <= outer, (x, y, err, mag)
            assert err[5] <= (inner if s < 100.0 else outer), (x, y, err, mag)
