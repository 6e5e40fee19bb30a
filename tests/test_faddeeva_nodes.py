"""The grid of Taylor coefficients behind the FP64 profiles: node values against
scipy's wofz, and expansions to the corners of a node's cell."""
import os
import subprocess

import numpy as np
import pytest

scipy_special = pytest.importorskip("scipy.special")
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1208_0302_gb300", "csrc")
N, H, TERMS = 129, 0.078125, 11


@pytest.fixture(scope="module")
def nodes(tmp_path_factory):
    d = tmp_path_factory.mktemp("nodes")
    src = d / "nodes.cpp"
    src.write_text('#include <cstdio>\n#include "faddeeva_nodes.h"\n'
                   "int main() { auto v = genesis::faddeeva_nodes(); fwrite(v.data(), 8, v.size(), stdout); }\n")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "nodes"), str(src)], check=True)
    raw = subprocess.run([str(d / "nodes")], check=True, capture_output=True).stdout
    v = np.frombuffer(raw).reshape(N, N, TERMS, 2)
    return v[..., 0] + 1j * v[..., 1]


def test_node_values(nodes):
    z = H * np.arange(N)[None, :] + 1j * H * np.arange(N)[:, None]
    w = scipy_special.wofz(z)  # relative accuracy 1e-13
    assert np.max(np.abs(nodes[..., 0] - w) / np.abs(w)) < 2e-13
    # c_1 = w' = -2 z w + 2 i / sqrt(pi), which cancels to about w / z at large z
    d = -2 * z * w + 2j / np.sqrt(np.pi)
    assert np.max(np.abs(nodes[..., 1] - d)) < 1e-12


@pytest.mark.parametrize("dx,dy", [(0.5, 0.5), (-0.5, 0.5), (0.5, -0.5), (0.0, 0.5)])
def test_expansions_reach_the_cell(nodes, dx, dy):
    # 11 terms: the first omitted is below (0.0553)^11 / Gamma(6.5) = 5e-17
    iy, ix = np.mgrid[1:N - 1, 1:N - 1]
    dz = H * (dx + 1j * dy)
    s = np.zeros(ix.shape, dtype=complex)
    for n in range(TERMS - 1, -1, -1):
        s = s * dz + nodes[1:N - 1, 1:N - 1, n]
    w = scipy_special.wofz(H * (ix + 1j * iy) + dz)
    assert np.max(np.abs(s - w) / np.abs(w)) < 2e-13
