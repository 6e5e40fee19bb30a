"""FP64 synthesis and chi2 on the block-wide profiles, at the edges of their
regions and passes: |z|^2 = 100, 170, 500, dampings from 0 beyond the table,
grids of one to four passes over the wavelengths, more Zeeman components than
a pass holds."""
import numpy as np
import pytest
import torch

import genesis_inputs as gi

pytestmark = pytest.mark.gpu

MANY = [(6301.5091, 1.667, 3.5, 4, 1.5, 4, 1.2), (6302.5017, 2.5, 1.0, 3, 1.4, 4, 1.1), (6301.9, 1.0, 0.3),
        (6302.1, 1.2, 0.5, 2, 1.0, 1, 1.5)]  # 27 + 21 + 3 + 9 components


def _spec(kind, nl):
    lines = {"one": gi.one_line_spec().lines, "two": gi.two_line_spec().lines, "many": MANY}[kind]
    return gi.ProblemSpec(lines=lines, lambda_grid=np.linspace(6301.0, 6303.0, nl))


@pytest.mark.parametrize("kind,nl,fill", [("two", 128, False), ("one", 3, False), ("two", 129, True), ("one", 512, False),
                                          ("many", 97, False), ("many", 260, True)])
def test_synth_and_chi2(gpu, orc, kind, nl, fill):
    spec = _spec(kind, nl)
    spec.fill = fill
    lo, hi = (gi.PRIOR_LO_FILL, gi.PRIOR_HI_FILL) if fill else (gi.PRIOR_LO, gi.PRIOR_HI)
    P = gi.draw_params_uniform(40, nl, lo, hi)
    # dampings: none, subnormal, about the node and cell edges, the table's end, far beyond
    P[:12, 5] = [0.0, 1e-310, 1e-12, 0.078125, 0.15625, 1.0, 5.0, 9.95, 10.0, 10.05, 23.0, 400.0]
    P[12:16, 4] = [0.5, 2.0, 300.0, 2000.0]  # narrow lines (|x| to 4000) and lines wider than the grid
    P[16, 0] = 0.0
    P[17, 0] = 1e5                           # components far outside the grid
    ref = orc.synth(spec, P)
    pb = gpu.Problem.from_spec(spec, "f64")
    got = gpu.me_synth(pb, torch.tensor(P, device="cuda")).cpu().numpy()
    ic = (P[:, 7] + P[:, 8])[:, None, None]
    assert np.max(np.abs(got - ref) / np.maximum(np.abs(ref), ic)) <= 1e-12
    obs = ref + 1e-3 * ic * gi.draw_noise(len(P), nl, seed=3)
    w = np.repeat(1e3 / ic[:, :, 0], 4, axis=1)
    for dtype in ("f64", "f32"):
        o = obs.astype(np.float32).astype(np.float64) if dtype == "f32" else obs
        pd = gpu.Problem.from_spec(spec, dtype)
        ot = torch.tensor(o, device="cuda", dtype=pd.torch_dtype)
        for weights in (w, None):
            ww = orc.weights_invmax(o) if weights is None else weights
            want = np.einsum("ns,nsj->n", ww ** 2, (o - ref) ** 2) / (4 * nl - P.shape[1])
            c = gpu.me_chi2(pd, ot, torch.tensor(P, device="cuda"),
                            w=None if weights is None else torch.tensor(ww, device="cuda")).cpu().numpy()
            # the synthesis bar, 1e-12 I_c, against residuals of 1e-3 I_c
            assert np.max(np.abs(c - want) / want) <= 2e-9, (dtype, weights is None)
