"""Line centres of large maps, where the number of lanes per pixel follows from
the window: one and two lanes per pixel, ragged last blocks, whole grids of 512
wavelengths.  Bit for bit."""
import numpy as np
import pytest
import torch

import genesis_inputs as gi
from gpu_helpers import make_obs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,nl,npix,W,lo,hi", [("f32", 27, 262147, 10, 0, 1 << 30), ("f64", 101, 41001, 50, 0, 100),
                                                   ("f64", 64, 41003, 10, 20, 50), ("f32", 96, 41001, 1, 40, 73),
                                                   ("f64", 512, 3001, 10, 0, 1 << 30), ("f32", 512, 12001, 40, 0, 1 << 30),
                                                   ("f64", 512, 701, 40, 0, 1 << 30)])
def test_large_maps(gpu, orc, dtype, nl, npix, W, lo, hi):
    spec = gi.two_line_spec(nl)
    _, obs = make_obs(orc, spec, 61, seed=nl)
    obs[1, 0] = 0.0         # every sum ties at zero
    obs[2, 0, nl // 2] = 1e-25  # too many octaves for the integer form
    obs[3, 0] = -obs[3, 0]
    if dtype == "f32":
        obs = obs.astype(np.float32).astype(np.float64)
    ref_c, ref_i = orc.line_centre(obs, spec.lambda_grid, W, lo, hi)
    rows = torch.arange(npix, device="cuda") % len(obs)
    pb = gpu.Problem.from_spec(spec, dtype)
    few = torch.tensor(obs, device="cuda", dtype=pb.torch_dtype)
    lc, idx = gpu.line_centre(pb, few[rows].contiguous(), W, lo, hi)
    assert torch.equal(idx, torch.tensor(ref_i, device="cuda", dtype=torch.int32)[rows])
    assert torch.allclose(lc, torch.tensor(ref_c, device="cuda")[rows], rtol=0.0, atol=0.0, equal_nan=True)
