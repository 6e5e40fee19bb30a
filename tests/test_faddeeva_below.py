"""The rows of Taylor coefficients of w below the real axis (dampings below 0)
against scipy's wofz."""
import os
import subprocess

import numpy as np
import pytest

scipy_special = pytest.importorskip("scipy.special")
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1208_0302_gb300", "csrc")
N, BELOW, H, TERMS = 129, 19, 0.078125, 11


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("below")
    src = d / "below.cpp"
    src.write_text('#include <cstdio>\n#include "faddeeva_nodes.h"\n'
                   "int main() { auto v = genesis::faddeeva_nodes_below(); fwrite(v.data(), 8, v.size(), stdout); }\n")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "below"), str(src)], check=True)
    raw = subprocess.run([str(d / "below")], check=True, capture_output=True).stdout
    v = np.frombuffer(raw).reshape(BELOW, N, TERMS, 2)
    return v[..., 0] + 1j * v[..., 1]


@pytest.mark.parametrize("dx,dy", [(0.0, 0.0), (0.5, 0.5), (-0.5, 0.5), (0.5, -0.5), (-0.5, -0.5)])
def test_nodes_and_their_cells(rows, dx, dy):
    x, y = H * np.arange(1, N - 1)[None, :], H * np.arange(-BELOW, 0)[:, None]
    dz = H * (dx + 1j * dy)
    s = np.zeros((BELOW, N - 2), dtype=complex)
    for n in range(TERMS - 1, -1, -1):
        s = s * dz + rows[:, 1:N - 1, n]
    w = scipy_special.wofz(x + 1j * y + dz)
    # wofz's relative accuracy is 1e-13, that of its 2 exp(-z^2) term |z|^2 2^-52; the expansions are
    # within 1e-13 |w|; all relative to the larger of w's two terms where they cancel
    scale = np.maximum(np.abs(w), np.abs(2 * np.exp(-(x + 1j * y + dz) ** 2)))
    assert np.max(np.abs(s - w) / scale) < 2e-13
