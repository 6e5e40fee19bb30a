"""Classification with line windows at either end of a grid and within one
chunk of it, extrema (infinite ones too) and NaN beyond the windows: bit for
bit as the oracle."""
import numpy as np
import pytest
import torch

import genesis_inputs as gi
from gpu_helpers import make_obs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("nl,npix,core", [(512, 3, (300, 333)), (512, 70, (0, 3)), (200, 9731, (190, 199)), (97, 40, (32, 63)),
                                          (33, 40, (31, 32)), (130, 40, (64, 64))])
def test_windows_and_extrema(gpu, orc, dtype, nl, npix, core):
    spec = gi.two_line_spec(nl)
    _, obs = make_obs(orc, spec, min(npix, 47), seed=nl)
    quiet = (nl // 3, nl // 3 + 5)
    # a point in neither window, a chunk or more from the line's where there is one
    far = [j for j in range(nl) if not (quiet[0] <= j < quiet[1]) and not (core[0] - 1 <= j <= core[1] + 1)]
    obs[0, 1, far[0]], obs[0, 2, far[-1]] = -50.0, 70.0
    obs[1, 3, far[len(far) // 2]] = -np.inf
    obs[2, 1:, far[-1]] = np.nan
    if dtype == "f32":
        obs = obs.astype(np.float32).astype(np.float64)
    ref = orc.classify(spec, obs, 3.0, quiet, 1, core)
    assert np.isinf(ref["p"][1]) and np.isfinite(ref["p"][2])
    pb = gpu.Problem.from_spec(spec, dtype)
    rows = np.arange(npix) % len(obs)
    got = gpu.classify(pb, torch.tensor(obs[rows], device="cuda", dtype=pb.torch_dtype), 3.0, quiet, 1, core)
    for k in ("flag", "polarity", "p", "sigma_p"):
        out = got[k].cpu().numpy()
        assert np.array_equal(out, ref[k][rows].astype(out.dtype), equal_nan=True), k
    weak = got["weak"].cpu().numpy()
    for c, k in ((0, "B"), (3, "B_par"), (4, "B_perp")):
        assert np.array_equal(weak[:, c], ref[k][rows], equal_nan=True), k
