"""FP64 synthesis, chi2 and GA fitness at dampings of -0 (which is 0) and a
little below 0 (which only callers' own values reach), on problems that build
the cells of profiles64.cuh and on problems that expand from its nodes, and the
node path at its edges: |z|^2 = 100, dampings about the grid's nodes and end."""
import numpy as np
import pytest
import torch

import genesis_inputs as gi

pytestmark = pytest.mark.gpu

BAR = 1e-12  # of max(|S|, I_c), as for the synthesis elsewhere
# the rows of nodes below 0 end at -1.48
BELOW = [-1e-310, -1e-12, -1e-3, -0.05, -0.1, -0.7]
EDGES = [0.0, 1e-310, 0.5 * 0.078125, 0.078125, 9.95, 9.9609375, 9.999999, 10.0, 10.05, 23.0]


def _spec(kind, nl, fill=False):
    # one line: 3 components; up to 180 wavelengths expand from the nodes, 181 build cells
    if kind == "one":
        return gi.ProblemSpec(lines=gi.one_line_spec().lines, lambda_grid=np.linspace(6302.0, 6303.0, nl), fill=fill)
    return gi.ProblemSpec(lines=gi.two_line_spec().lines, lambda_grid=np.linspace(6301.0, 6303.0, nl), fill=fill)


def _params(n, seed, fill):
    lo, hi = (gi.PRIOR_LO_FILL, gi.PRIOR_HI_FILL) if fill else (gi.PRIOR_LO, gi.PRIOR_HI)
    return gi.draw_params_uniform(n, seed, lo, hi)


def _scale(ref, P):
    return np.maximum(np.abs(ref), (P[:, 7] + P[:, 8])[:, None, None])


@pytest.mark.parametrize("kind,nl,fill", [("one", 64, False), ("one", 64, True), ("one", 180, False), ("one", 181, False),
                                          ("two", 3, False), ("two", 128, False), ("two", 140, True)])
def test_damping_zero_below_and_edges(gpu, orc, kind, nl, fill):
    spec = _spec(kind, nl, fill)
    P = _params(3 * (1 + len(BELOW) + len(EDGES)), nl, fill)
    a = np.array([-0.0] + BELOW + EDGES)
    P[:, 5] = np.tile(a, 3)
    P[len(a):2 * len(a), 4] = np.linspace(2.0, 60.0, len(a))  # |x| from inside 10 to far beyond on the grid
    minus0 = np.signbit(P[:, 5]) & (P[:, 5] == 0.0)
    assert minus0.sum() == 3
    ref = orc.synth(spec, P)
    pb = gpu.Problem.from_spec(spec, "f64")
    got = gpu.me_synth(pb, torch.tensor(P, device="cuda")).cpu().numpy()
    assert np.max(np.abs(got - ref) / _scale(ref, P)) <= BAR
    Z = P.copy()
    Z[minus0, 5] = 0.0
    zero = gpu.me_synth(pb, torch.tensor(Z, device="cuda")).cpu().numpy()
    assert np.array_equal(got[minus0], zero[minus0])
    ic = (P[:, 7] + P[:, 8])[:, None, None]
    for dtype in ("f64", "f32"):
        pd = gpu.Problem.from_spec(spec, dtype)
        obs = torch.tensor(ref + 1e-3 * ic * gi.draw_noise(len(P), nl, seed=5), device="cuda", dtype=pd.torch_dtype)
        o = obs.double().cpu().numpy()
        w = np.repeat(1e3 / ic[:, :, 0], 4, axis=1)
        want = np.einsum("ns,nsj->n", w ** 2, (o - ref) ** 2) / (4 * nl - P.shape[1])
        c = gpu.me_chi2(pd, obs, torch.tensor(P, device="cuda"), w=torch.tensor(w, device="cuda")).cpu().numpy()
        assert np.max(np.abs(c - want) / want) <= 2e-9, dtype  # 1e-12 I_c against residuals of 1e-3 I_c


def test_cells_and_nodes_agree(gpu):
    # 180 and 181 wavelengths of one line: the same models at the 180 they share
    lam = np.linspace(6302.0, 6303.0, 181)
    P = torch.tensor(_params(64, 9, False), device="cuda")
    out = []
    for grid in (lam[:180], lam):
        spec = gi.ProblemSpec(lines=gi.one_line_spec().lines, lambda_grid=grid)
        out.append(gpu.me_synth(gpu.Problem.from_spec(spec, "f64"), P)[:, :, :180])
    ic = (P[:, 7] + P[:, 8])[:, None, None]
    # each within 2e-16 of w per profile; eta0 <= 20 and the closed form carry it to at most 1e-13 I_c
    assert torch.max(torch.abs(out[0] - out[1]) / ic) < 1e-13


@pytest.mark.parametrize("kind,nl,npop,fill", [("one", 21, 32, False), ("two", 12, 64, True), ("two", 9, 288, False)])
def test_ga_fitness(gpu, orc, kind, nl, npop, fill):
    spec = _spec(kind, nl, fill)
    truth = _params(2, 3, fill)
    obs = orc.synth(spec, truth) + 1e-3 * gi.draw_noise(2, nl, seed=1)
    P = np.stack([_params(npop, 50 + i, fill) for i in range(2)])
    # populations above 256 take Weideman's series, within 4e-15 of w down to a damping of -0.1
    a = np.array([-0.0, 0.0] + (BELOW if npop <= 256 else BELOW[:-1]) + EDGES)
    P[:, :len(a), 5] = a
    pb = gpu.Problem.from_spec(spec, "f64")
    fit, res = gpu.ga_fitness(pb, torch.tensor(obs, device="cuda"), torch.tensor(P, device="cuda"), want_resid=True)
    flat = P.reshape(-1, P.shape[2])
    ref = orc.synth(spec, flat).reshape(res.shape)
    got = obs[:, None] - res.cpu().numpy()
    assert np.max(np.abs(got - ref) / _scale(ref.reshape(-1, 4, nl), flat).reshape(ref.shape)) <= BAR
    ww = orc.weights_invmax(obs)
    want = np.einsum("ns,npsj->np", ww ** 2, (obs[:, None] - ref) ** 2) / (4 * nl - P.shape[2])
    # residuals are of order I_c or more against 1e-12 of it
    assert np.max(np.abs(fit.cpu().numpy() - want) / want) <= 1e-9


def test_ga_below_zero_by_pixel_bounds(gpu, orc):
    """Per-pixel bounds that reach below 0 on both launch shapes: the same
    pixels split over threads (one pixel) and unsplit (many)."""
    spec = _spec("one", 16)
    truth = _params(4, 2, False)
    obs = torch.tensor(orc.synth(spec, truth), device="cuda")
    n = 152 * 8 + 1  # more than 16 warps per SM at population 64: unsplit
    cube = obs[torch.arange(n, device="cuda") % 4].contiguous()
    b = torch.empty((n, 2, 9), dtype=torch.float64, device="cuda")
    b[:, 0] = torch.tensor(gi.PRIOR_LO, dtype=torch.float64)
    b[:, 1] = torch.tensor(gi.PRIOR_HI, dtype=torch.float64)
    b[:, 0, 5] = -0.3
    ga = gpu.GaSettings(npop=64, ngen=4, nsamp=2, seed=4)
    pb = gpu.Problem.from_spec(spec, "f64")
    many = gpu.ga_invert_subset(pb, cube, gi.PRIOR_LO, gi.PRIOR_HI, ga, bounds_px=b, want_genes=True)
    few = gpu.ga_invert_subset(pb, cube[:3].contiguous(), gi.PRIOR_LO, gi.PRIOR_HI, ga, bounds_px=b[:3].contiguous(),
                               want_genes=True)
    for x, y in zip(few, many):
        assert torch.equal(x, y[:3])
    fit, _ = gpu.ga_fitness(pb, cube[:3].contiguous(), few[0][:, None, :].repeat(1, 32, 1).contiguous())
    assert torch.allclose(fit, few[1][:, None].expand(-1, 32), rtol=1e-9, atol=0.0)
