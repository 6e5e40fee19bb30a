"""The GA with its individuals' wavelengths split over threads (few pixels)
against the same pixels in a batch large enough to run unsplit: bit for bit."""
import numpy as np
import pytest
import torch

import genesis_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,nl,npop,fill", [("one", 5, 32, False), ("two", 128, 128, False), ("two", 97, 96, False),
                                               ("two", 64, 256, False), ("three", 33, 64, False),
                                               ("pattern", 41, 64, False), ("two", 31, 64, True),
                                               ("pattern", 24, 128, True)])
def test_split_equals_unsplit(gpu, kind, nl, npop, fill):
    lines = {"one": gi.one_line_spec().lines, "two": gi.two_line_spec().lines,
             "three": gi.two_line_spec().lines + [(6302.0, 1.3, 0.4)],
             "pattern": gi.two_line_pattern_spec().lines}[kind]
    spec = gi.ProblemSpec(lines=lines, lambda_grid=np.linspace(6301.2, 6302.9, nl), fill=fill)
    lo, hi = (gi.PRIOR_LO_FILL, gi.PRIOR_HI_FILL) if fill else (gi.PRIOR_LO, gi.PRIOR_HI)
    pb = gpu.Problem.from_spec(spec, "f32")
    whole = 152 * 28 // (npop // 32) + 152   # more blocks per SM than leave room for a second segment
    truth = torch.tensor(gi.draw_params_uniform(64, nl, lo, hi), device="cuda")
    rows = torch.arange(whole, device="cuda") % 64
    g = torch.Generator(device="cuda").manual_seed(nl)
    obs = gpu.me_synth(pb, truth)[rows]
    obs = (obs + 1e-3 * torch.randn(obs.shape, generator=g, device="cuda")).contiguous()
    pol = (torch.arange(whole, device="cuda", dtype=torch.int32) % 3) - 1
    seeds = torch.rand((whole, 2, 3), generator=g, device="cuda", dtype=torch.float64) * 100.0
    ga = gpu.GaSettings(npop=npop, ngen=7, nsamp=3, seed=5)

    def run(n):
        return gpu.ga_invert_subset(pb, obs[:n].contiguous(), lo, hi, ga, seeds=seeds[:n].contiguous(),
                                    polarity=pol[:n].contiguous(), want_genes=True)

    best, chi2, genes = run(whole)
    for n in (1, 3, 152, 153, 460, 1100):
        if n < whole:
            b, c, q = run(n)
            assert torch.equal(q, genes[:n]) and torch.equal(b, best[:n]) and torch.equal(c, chi2[:n]), n


@pytest.mark.parametrize("kind,nl,npop,fill", [("one", 5, 64, False), ("two", 43, 32, False), ("pattern", 9, 128, True),
                                               ("two", 16, 256, False)])
def test_split_equals_unsplit_fp64(gpu, kind, nl, npop, fill):
    lines = {"one": gi.one_line_spec().lines, "two": gi.two_line_spec().lines,
             "pattern": gi.two_line_pattern_spec().lines}[kind]
    spec = gi.ProblemSpec(lines=lines, lambda_grid=np.linspace(6301.2, 6302.9, nl), fill=fill)
    lo, hi = (gi.PRIOR_LO_FILL, gi.PRIOR_HI_FILL) if fill else (gi.PRIOR_LO, gi.PRIOR_HI)
    pb = gpu.Problem.from_spec(spec, "f64")
    whole = 152 * (8 // (npop // 32)) + 152   # one segment: two would exceed 16 warps per SM
    truth = torch.tensor(gi.draw_params_uniform(64, nl, lo, hi), device="cuda")
    obs = gpu.me_synth(pb, truth)[torch.arange(whole, device="cuda") % 64]
    g = torch.Generator(device="cuda").manual_seed(nl)
    obs = (obs + 1e-3 * torch.randn(obs.shape, generator=g, device="cuda", dtype=torch.float64)).contiguous()
    ga = gpu.GaSettings(npop=npop, ngen=5, nsamp=2, seed=5)

    def run(n):
        return gpu.ga_invert_batch(pb, obs[:n].contiguous(), lo, hi, ga, want_genes=True)

    best, chi2, genes = run(whole)
    for n in (1, 152, 153, 305):
        if n < whole:
            b, c, q = run(n)
            assert torch.equal(q, genes[:n]) and torch.equal(b, best[:n]) and torch.equal(c, chi2[:n]), n
    # the unsplit kernel's own evaluation of its answers, in FP64
    fit, _ = gpu.ga_fitness(pb, obs[:64].contiguous(), best[:64, None, :].repeat(1, npop, 1).contiguous())
    assert torch.allclose(fit, chi2[:64, None].expand(-1, npop), rtol=1e-11, atol=0.0)
