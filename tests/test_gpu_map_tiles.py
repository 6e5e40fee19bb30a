"""Classification and line centres at the edges of their launch shapes: 32
pixels per warp, one- and two-warp blocks, 32, 8, 2 or 1 lanes per pixel, and
rows that the integer form of the centre sums cannot hold.  Bit for bit."""
import numpy as np
import pytest
import torch

import genesis_inputs as gi
from gpu_helpers import make_obs

pytestmark = pytest.mark.gpu


def _tile(a, n):
    return np.ascontiguousarray(a[np.arange(n) % len(a)])


@pytest.mark.parametrize("dtype,nl,npix", [("f32", 97, 31), ("f32", 128, 33), ("f64", 45, 64), ("f32", 128, 9728),
                                           ("f32", 131, 9729), ("f64", 96, 9761),
                                           ("f32", 340, 40)])
def test_classify_launch_shapes(gpu, orc, dtype, nl, npix):
    spec = gi.two_line_spec(nl)
    _, obs = make_obs(orc, spec, min(npix, 61), seed=nl)
    obs[0, :, :] = obs[0, :, :1]       # a flat pixel: every sum and difference is zero
    obs[1, 1:] = 0.0                   # unpolarised
    obs[2] *= 1e-30
    if dtype == "f32":
        obs = obs.astype(np.float32).astype(np.float64)
    quiet, core = (1, nl // 8), (nl // 2, nl - 2)
    ref = orc.classify(spec, obs, 3.0, quiet, 1, core)
    pb = gpu.Problem.from_spec(spec, dtype)
    got = gpu.classify(pb, torch.tensor(_tile(obs, npix), device="cuda", dtype=pb.torch_dtype), 3.0, quiet, 1, core)
    for k in ("flag", "polarity", "p", "sigma_p"):
        want = _tile(ref[k], npix)
        assert np.array_equal(got[k].cpu().numpy(), want.astype(got[k].cpu().numpy().dtype), equal_nan=True), k
    weak, seeds = got["weak"].cpu().numpy(), got["seeds"].cpu().numpy()
    for c, k in ((0, "B"), (3, "B_par"), (4, "B_perp")):
        assert np.array_equal(weak[:, c], _tile(ref[k], npix), equal_nan=True), k
    assert np.array_equal(seeds[:, :, 0], _tile(ref["seeds"], npix)[:, :, 0], equal_nan=True)
    # angles: atan2 of the same arguments, 1e-12 degree as in the small launches
    assert np.nanmax(np.abs(weak[:, 1] - _tile(ref["theta"], npix))) < 1e-12


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("npix", [1, 609, 2433, 9729])
def test_line_centre_launch_shapes(gpu, orc, dtype, npix):
    spec = gi.two_line_spec(101)
    _, obs = make_obs(orc, spec, min(npix, 83), seed=7)
    r = np.random.default_rng(npix)
    if len(obs) > 1:
        obs[1, 0] = 0.0                                  # every sum ties at zero
        obs[2, 0, 50] = 1e-25                            # too many octaves for the integer form
        obs[3, 0] = -obs[3, 0]
        obs[4, 0] = 2.0 ** r.integers(-11, 12, 101)      # 22 octaves: the integer form's last with W = 32
        obs[5, 0] = 2.0 ** r.integers(-12, 13, 101)      # one or two more
        obs[6, 0, ::3] = 0.0
        obs[7, 0] = 1e-40 * r.integers(0, 1000, 101)     # subnormal FP32 values
    if dtype == "f32":
        obs = obs.astype(np.float32).astype(np.float64)
    pb = gpu.Problem.from_spec(spec, dtype)
    ob = torch.tensor(_tile(obs, npix), device="cuda", dtype=pb.torch_dtype)
    for W, lo, hi in [(1, 0, 1 << 30), (10, 40, 90), (32, 0, 1 << 30), (50, 0, 100), (51, 0, 100)]:
        ref_c, ref_i = orc.line_centre(obs, spec.lambda_grid, W, lo, hi)
        lc, idx = gpu.line_centre(pb, ob, W, lo, hi)
        assert np.array_equal(idx.cpu().numpy(), _tile(ref_i, npix))
        assert np.array_equal(lc.cpu().numpy(), _tile(ref_c, npix), equal_nan=True)
