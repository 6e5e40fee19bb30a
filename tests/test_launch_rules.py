"""The launch rules by sizes (csrc/launch_rules.h) against times measured on a
GB300: where one of two kernels took at least 1.2 times the other's time, the
rule has to pick the faster."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1208_0302_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include <cstring>
#include "launch_rules.h"
using namespace genesis;
int main()
{
    char rule[32];
    while (std::scanf("%31s", rule) == 1) {
        if (!std::strcmp(rule, "models")) {
            int jac, lines, ncomp, triplets, nl, n;
            if (std::scanf("%d %d %d %d %d %d", &jac, &lines, &ncomp, &triplets, &nl, &n) != 6) return 1;
            std::printf("%d\n", chunks_per_warp(jac, n, nl, lines, ncomp, triplets, jac ? 4 : 8));
        } else if (!std::strcmp(rule, "blocks64")) {
            int n, nl, ncomp;
            if (std::scanf("%d %d %d", &n, &nl, &ncomp) != 3) return 1;
            std::printf("%d\n", blocks_per_model64(n, nl, ncomp, 128));
        } else if (!std::strcmp(rule, "segments")) {
            int npix, npop, nl, regs, fp64, split, plain;
            long long others;
            if (std::scanf("%d %d %d %d %d %d %d %lld", &npix, &npop, &nl, &regs, &fp64, &split, &plain, &others) != 8) return 1;
            std::printf("%d\n", ga_segments(npix, npop, nl, regs, fp64, split, plain, others));
        } else if (!std::strcmp(rule, "warps")) {
            int regs;
            if (std::scanf("%d", &regs) != 1) return 1;
            std::printf("%d\n", resident_warps(regs));
        } else if (!std::strcmp(rule, "centre")) {
            int integers, n, candidates, W;
            if (std::scanf("%d %d %d %d", &integers, &n, &candidates, &W) != 4) return 1;
            std::printf("%d\n", centre_lanes(integers, n, candidates, W, integers ? 12 : 8));
        }
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src = d / "rules.cpp"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-o", str(d / "rules"), str(src)], check=True)

    def run(calls):
        text = "\n".join(" ".join(str(x) for x in c) for c in calls)
        out = subprocess.run([str(d / "rules")], input=text, capture_output=True, text=True, check=True).stdout
        return [[float(x) for x in line.split()] for line in out.splitlines()]

    return run


# (Jacobian, lines, components, triplets, wavelengths, models): us of k_points, us of k_models
MODELS = [((1, 1, 3, 1, 8, 30000), 38.7, 47.6), ((1, 1, 3, 1, 24, 8000), 32.8, 16.5), ((1, 1, 3, 1, 65, 8000), 59.9, 35.3),
          ((1, 1, 3, 1, 256, 600), 25.3, 14.9), ((1, 1, 3, 1, 257, 2500), 64.9, 33.3), ((1, 2, 6, 1, 8, 30000), 42.7, 62.3),
          ((1, 2, 6, 1, 20, 30000), 77.0, 62.9), ((1, 2, 6, 1, 128, 8000), 103.9, 56.1),
          ((1, 2, 6, 1, 129, 30000), 380.9, 223.9), ((1, 2, 15, 0, 6, 8000), 17.0, 30.4), ((1, 2, 15, 0, 32, 8000), 43.8, 31.2),
          ((1, 2, 15, 0, 32, 30000), 123.8, 102.2), ((1, 2, 15, 0, 257, 30000), 808.7, 616.3),
          ((1, 3, 9, 0, 65, 8000), 88.7, 66.0), ((1, 3, 9, 0, 192, 8000), 223.7, 127.2),
          ((1, 4, 69, 0, 16, 30000), 172.6, 378.3), ((1, 4, 69, 0, 64, 8000), 164.9, 205.0),
          ((1, 4, 69, 0, 128, 2500), 106.3, 128.9), ((0, 1, 3, 1, 97, 30000), 68.1, 51.8), ((0, 2, 6, 1, 8, 30000), 12.8, 35.2),
          ((0, 2, 6, 1, 96, 30000), 87.1, 68.2), ((0, 2, 6, 1, 129, 8000), 37.4, 29.6), ((0, 2, 6, 1, 512, 30000), 1025.7, 211.7),
          ((0, 2, 15, 0, 20, 30000), 39.4, 68.5), ((0, 2, 15, 0, 33, 30000), 62.4, 93.1), ((0, 2, 15, 0, 512, 8000), 295.4, 154.3),
          ((0, 3, 9, 0, 192, 30000), 288.2, 153.1), ((0, 4, 69, 0, 12, 2500), 19.0, 32.7), ((0, 4, 69, 0, 32, 30000), 220.1, 271.0),
          ((0, 4, 69, 0, 48, 8000), 90.9, 122.1)]


def test_models_or_points(rule):
    for (case, points, models), (per,) in zip(MODELS, rule([("models",) + m[0] for m in MODELS])):
        assert (per == 0) == (points < models), (case, per)
        assert per <= (case[4] + 31) // 32


# (models, wavelengths, components): us of k_points, of a block per model, of a block per pass
BLOCKS64 = [((20000, 3, 3), 66.2, 325.5, None), ((20000, 8, 6), 245.2, 424.6, None), ((20000, 8, 15), 539.6, 856.0, None),
            ((20000, 6, 69), 1797.0, 2801.9, None), ((20000, 24, 6), 675.8, 504.6, None), ((20000, 24, 69), 6346.8, 4116.0, None),
            ((600, 8, 3), 20.9, 16.5, None), ((2500, 32, 6), 138.7, 86.9, None), ((1, 257, 3), 18.9, 31.2, 17.7),
            ((1, 512, 6), 33.5, 64.3, 23.1), ((20, 512, 69), 203.6, 535.8, 145.4), ((150, 384, 15), 144.3, 99.6, 72.9),
            ((600, 512, 6), 319.6, 163.6, 183.7), ((20000, 257, 3), 3041.5, 1968.8, 2486.2), ((1, 64, 3), 19.0, 13.1, 13.1)]


def test_blocks_per_fp64_model(rule):
    for (case, points, one, passes), (got,) in zip(BLOCKS64, rule([("blocks64",) + b[0] for b in BLOCKS64])):
        best = min(t for t in (points, one, passes) if t is not None)
        took = {0: points, 1: one}.get(got, passes)
        assert took <= best * 1.06, (case, got)
        assert got <= (case[1] + 127) // 128


# (float cube, pixels, candidates, W): us by lanes per pixel
CENTRE = [((0, 700, 492, 10), {1: 434.1, 2: 224.4, 8: 60.3, 32: 23.3}), ((0, 1500, 257, 40), {1: 838.0, 2: 422.6, 8: 114.2, 32: 83.1}),
          ((0, 3000, 257, 10), {1: 237.6, 2: 124.7, 8: 43.9, 32: 48.0}), ((0, 6000, 48, 40), {1: 168.0, 2: 87.2, 8: 60.2, 32: 107.5}),
          ((0, 6000, 432, 40), {1: 2704.3, 2: 697.6, 8: 424.3, 32: 486.0}), ((0, 12000, 34, 1), {1: 23.0, 2: 15.2, 8: 15.1, 32: 27.1}),
          ((0, 12000, 34, 40), {1: 137.1, 2: 91.7, 8: 101.8, 32: 192.3}), ((0, 12000, 65, 1), {1: 27.3, 2: 18.6, 8: 15.1, 32: 29.3}),
          ((0, 70000, 126, 1), {1: 108.4, 2: 80.0, 8: 85.0, 32: 159.6}), ((0, 70000, 257, 1), {1: 392.7, 2: 225.7, 8: 152.4, 32: 228.3}),
          ((0, 70000, 492, 10), {1: 6610.1, 2: 2297.9, 8: 1473.5, 32: 1636.5}), ((0, 70000, 34, 10), {1: 124.4, 2: 135.5, 8: 165.9, 32: 361.6}),
          ((1, 3000, 24, 40), {1: 39.5, 2: 23.6, 8: 14.9, 32: 14.5}), ((1, 3000, 254, 1), {1: 52.1, 2: 30.4, 8: 15.2, 32: 15.3}),
          ((1, 12000, 34, 1), {1: 21.1, 2: 14.8, 8: 14.2, 32: 25.3}), ((1, 12000, 257, 1), {1: 110.6, 2: 62.5, 8: 25.1, 32: 28.7}),
          ((1, 25000, 48, 40), {1: 81.3, 2: 68.7, 8: 54.1, 32: 51.9}), ((1, 25000, 492, 10), {1: 799.9, 2: 457.3, 8: 145.5, 32: 87.9}),
          ((1, 70000, 65, 1), {1: 52.0, 2: 37.6, 8: 39.5, 32: 127.2}), ((1, 70000, 257, 1), {1: 435.2, 2: 239.5, 8: 85.4, 32: 131.2}),
          ((1, 70000, 510, 1), {1: 1347.7, 2: 732.0, 8: 202.1, 32: 133.7}), ((1, 70000, 34, 1), {1: 27.1, 2: 28.6, 8: 37.5, 32: 124.3})]


def test_lanes_per_line_centre(rule):
    for (case, us), (lanes,) in zip(CENTRE, rule([("centre",) + c[0] for c in CENTRE])):
        assert us[int(lanes)] <= 1.25 * min(us.values()), (case, lanes)


def ga_shared(nl, npop, split):
    """Bytes of an FP32 GA block with nine parameters (ga_smem_layout)."""
    pairs, total = (nl + 1) // 2, 0
    for n in (32 * pairs, 32 * pairs, 4 * npop, 128, 128, 32, 16, 240, 2048, 36 * npop, 64 * npop, 4 * pairs * npop * split):
        total = -(-total // 16) * 16 + n
    return -(-total // 16) * 16


# (pixels, population, wavelengths, registers): us split, us unsplit
SEGMENTS = [((456, 128, 384, 72), 2606, 2061), ((304, 128, 384, 80), 4475, 5505), ((456, 128, 512, 72), 3414, 2689),
            ((912, 64, 512, 72), 3448, 2867), ((1520, 32, 512, 72), 3500, 4335), ((608, 64, 128, 72), 536, 599),
            ((64, 64, 128, 72), 538, 1800), ((1, 128, 256, 72), 466, 930), ((304, 64, 256, 72), 508, 997)]


def test_ga_split(rule):
    calls = [("segments",) + c + (0, ga_shared(c[2], c[1], 1), ga_shared(c[2], c[1], 0), 0) for c, _, _ in SEGMENTS]
    for (case, split, plain), (n,) in zip(SEGMENTS, rule(calls)):
        assert (n > 1) == (split < plain), (case, n)
    # up to 144 wavelengths as many segments as the registers hold, but for a block or two to an SM
    (few,), (many,), (fp64,), (busy,) = rule([("segments", 64, 64, 128, 72, 0, ga_shared(128, 64, 1), ga_shared(128, 64, 0), 0),
                                              ("segments", 20000, 64, 128, 72, 0, ga_shared(128, 64, 1), ga_shared(128, 64, 0), 0),
                                              ("segments", 256, 64, 64, 128, 1, 60000, 60000, 0),
                                              ("segments", 64, 64, 128, 72, 0, ga_shared(128, 64, 1), ga_shared(128, 64, 0), 8512)])
    assert (few, many, fp64, busy) == (14, 1, 4, 1)


def test_split_blocks_fit_the_registers(rule):
    """A split block is launchable whatever cap the kernels are built with."""
    regs = list(range(24, 256))
    for r, (warps,) in zip(regs, rule([("warps", r) for r in regs])):
        assert 4 <= warps <= 32 and warps * 32 * -(-r // 8) * 8 <= 65536
    for npop in (32, 64, 96, 128, 256):
        calls = [("segments", n, npop, 128, r, fp64, 10000, 9000, 0) for n in (1, 152, 153, 500) for r in regs for fp64 in (0, 1)]
        for c, (s,) in zip(calls, rule(calls)):
            assert s == 1 or s * npop * -(-c[4] // 8) * 8 <= 65536, c
            assert s * npop <= 1024
