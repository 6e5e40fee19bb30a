"""Syntheses and Jacobians of many models on narrow and ragged grids, where a
thread takes one (model, wavelength): against the oracle and the general path,
and every copy of a model the same."""
import numpy as np
import pytest
import torch

import genesis_inputs as gi
from gpu_helpers import rel_err

pytestmark = pytest.mark.gpu

HEAVY = [(6301.5091, 1.667, 3.5, 4, 1.5, 4, 1.2), (6302.5017, 2.5, 1.0, 3, 1.4, 4, 1.1), (6302.0, 1.3, 0.4)]


def _spec(kind, nl, fill=False):
    lines = {"one": gi.one_line_spec().lines, "two": gi.two_line_spec().lines,
             "pattern": gi.two_line_pattern_spec().lines, "heavy": HEAVY}[kind]
    return gi.ProblemSpec(lines=lines, lambda_grid=np.linspace(6301.2, 6302.9, nl), fill=fill)


def _params(fill, seed):
    P = gi.draw_params_uniform(37, seed, *((gi.PRIOR_LO_FILL, gi.PRIOR_HI_FILL) if fill else (gi.PRIOR_LO, gi.PRIOR_HI)))
    P[:, 5] = np.maximum(P[:, 5], 0.02)
    return P


@pytest.mark.parametrize("kind,nl,n,fill", [("one", 3, 30001, False), ("two", 8, 30001, False), ("two", 33, 30001, False),
                                            ("pattern", 33, 12001, False), ("two", 17, 20001, True), ("heavy", 5, 77, False),
                                            ("heavy", 41, 3001, False)])
def test_fp32_points(gpu, orc, kind, nl, n, fill):
    spec, P = _spec(kind, nl, fill), _params(fill, nl)
    pb, pd = gpu.Problem.from_spec(spec, "f32"), gpu.Problem.from_spec(spec, "f64")
    few, rows = torch.tensor(P, device="cuda"), torch.arange(n, device="cuda") % len(P)
    many = few[rows].contiguous()
    ic = P[:, 7] + P[:, 8]
    st = gpu.me_synth(pb, many)
    assert torch.equal(st, st[:len(P)][rows])
    assert rel_err(st[:len(P)].double().cpu().numpy(), orc.synth(spec, P), ic) < 2e-5
    jac, st2 = gpu.me_synth_jac(pb, many, want_stokes=True)
    assert torch.equal(jac, jac[:len(P)][rows]) and torch.equal(st2, st2[:len(P)][rows])
    assert rel_err(st2[:len(P)].double().cpu().numpy(), orc.synth(spec, P), ic) < 2e-5
    # the general path (few models: a warp per model) evaluates the same expressions in the same precision, so
    # the two are no further from FP64 than twice one another, but for a few roundings of the largest entry
    want, general = gpu.me_synth_jac(pd, few), gpu.me_synth_jac(pb, few)
    scale = want.abs().amax(dim=(1, 2), keepdim=True) + 1e-30
    err, ref = (torch.max((j.double() - want).abs() / scale).item() for j in (jac[:len(P)], general))
    assert err < 2 * ref + 1e-6, (err, ref)


@pytest.mark.parametrize("kind,nl,n,fill", [("one", 3, 2001, False), ("two", 12, 2500, False), ("heavy", 6, 2000, False),
                                            ("two", 8, 3001, True),                       # a thread per point
                                            ("one", 129, 152, False), ("pattern", 300, 5, True),  # a block per pass
                                            ("two", 512, 1, False), ("two", 257, 153, False)])
def test_fp64_shapes(gpu, orc, kind, nl, n, fill):
    spec, P = _spec(kind, nl, fill), _params(fill, nl)
    P[:3, 5] = [0.0, 10.05, -0.0]  # none, beyond the node grid, none
    P[3, 4] = 0.5                  # narrow lines: |x| to thousands
    pb = gpu.Problem.from_spec(spec, "f64")
    rows = torch.arange(n, device="cuda") % len(P)
    got = gpu.me_synth(pb, torch.tensor(P, device="cuda")[rows].contiguous())
    m = min(n, len(P))
    assert torch.equal(got, got[:m][rows])
    ref = orc.synth(spec, P[:m])
    ic = (P[:m, 7] + P[:m, 8])[:, None, None]
    assert np.max(np.abs(got[:m].cpu().numpy() - ref) / np.maximum(np.abs(ref), ic)) <= 1e-12
