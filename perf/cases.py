"""Performance cases of the library: the calls that an inversion program makes.

Every case is a dict with a "kind" (which entry points run), the problem it
runs on (line list, wavelengths, precision, fill fraction) and its sizes:

    synth     me_synth of n parameter vectors
    grad      a gradient step's forward and backward pass (synth_autograd)
    jac       me_synth_jac: response functions of n models
    errors    me_chi2 and lm_uncertainty of a fitted map
    polish    lm_polish of a map from the answers of a coarser fit
    classify  pixel selection and line centres of a map (classify, select,
              line_centre)
    ga        ga_invert_batch
    serve     requests through the serving loop, host arrays in and out
    map       invert_map, the whole pipeline

Sizes come from the repository's workloads (one line over 64 wavelengths in
FP64 with population 64; two lines over 128 wavelengths with population 128
and 200 generations in FP32; serving requests of 64 to 4096 pixels with
populations 64 and 128 and 100 to 300 generations) and from ordinary slits
and map tiles.  Observed profiles are synthesised here in FP64 from seeded
truth with noise of 1e-3 of the continuum, so that they depend on the seed
alone.
"""
import math

import numpy as np
import torch

from paper_1208_0302_gb300 import api

LIGHT = 299792.458   # km/s
ZEEMAN = 4.6686e-13  # 1 / (A G)
RATIO = 10.0 ** (-0.718 + 1.235) * math.exp(-(3.654 - 3.686) / (8.617333262e-5 * 5000.0))
LINE1 = (6301.5091, 1.667, RATIO)
LINE1_FULL = LINE1 + (2, 11.0 / 6.0, 2, 1.5)  # Fe I 6301.5, J = 2 -> 2
LINE2 = (6302.5017, 2.5, 1.0)
LINES = {"one": [LINE2], "two": [LINE1, LINE2], "pattern": [LINE1_FULL, LINE2]}
GRID = {"one": (6302.0, 6303.0), "two": (6301.0, 6303.0), "pattern": (6301.0, 6303.0)}
LO = [0.0, 0.0, 0.0, -3.0, 20.0, 0.0, 1.0, 0.1, 0.1, 0.0]
HI = [3000.0, 180.0, 180.0, 3.0, 50.0, 0.5, 20.0, 1.0, 1.0, 1.0]
CHUNK = 2048  # pixels synthesised at once

MAP_GA = dict(npop=128, ngen=200)


def listed():
    return [
        # a single spectrum at the FP64 one-line setup, as a plot or an outer
        # optimiser asks for it: latency
        dict(name="synth_one", kind="synth", lines="one", nl=64, dtype="f64", fill=False, n=1),
        # forward and backward pass of a gradient-based fit over a batch
        dict(name="grad_batch", kind="grad", lines="two", nl=128, dtype="f32", fill=False, n=8192),
        # response functions of a slit's models, an odd number of them
        dict(name="jac_slit", kind="jac", lines="two", nl=128, dtype="f32", fill=False, n=20011),
        # chi2 and uncertainties of a fitted 256 x 256 map
        dict(name="errors_map", kind="errors", lines="two", nl=128, dtype="f32", fill=False, n=65536),
        # polish of a 256 x 256 map, ten iterations
        dict(name="polish_map", kind="polish", lines="two", nl=128, dtype="f32", fill=False, n=65536, iters=10),
        # a slit with the full Zeeman pattern, the fill fraction and an odd grid
        dict(name="polish_fill", kind="polish", lines="pattern", nl=111, dtype="f32", fill=True, n=1021, iters=10),
        # selection, weak-field answers and line centres of a 512 x 512 map
        dict(name="classify_map", kind="classify", lines="two", nl=128, dtype="f32", fill=False, n=262144),
        # the smallest serving request: latency of one GA run
        dict(name="ga_request", kind="ga", lines="two", nl=128, dtype="f32", fill=False, n=64, npop=64, ngen=100),
        # a 256 x 256 map at the headline budget: throughput
        dict(name="ga_map", kind="ga", lines="two", nl=128, dtype="f32", fill=False, n=65536, **MAP_GA),
        # the FP64 one-line workload, 16 x 16 pixels
        dict(name="ga_f64", kind="ga", lines="one", nl=64, dtype="f64", fill=False, n=256, npop=64, ngen=100),
        # four requests of mixed size through the serving loop, polished
        dict(name="serve_mix", kind="serve", lines="two", nl=128, dtype="f32", fill=False, n=900, parts=4),
        # the whole pipeline on a 96 x 96 tile
        dict(name="map_tile", kind="map", lines="two", nl=128, dtype="f32", fill=False, n=9216, **MAP_GA),
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["synth", "grad", "jac", "errors", "polish", "classify", "ga", "ga", "serve", "map"])
    lines = rng.choice(["one", "two", "two", "pattern"])
    c = dict(kind=kind, lines=lines, nl=rng.randint(48, 80) if lines == "one" else rng.randint(96, 144),
             dtype=rng.choice(["f32", "f32", "f64"]), fill=rng.random() < 0.25)
    if kind == "synth":
        c.update(n=logint(1, 8192))
    elif kind in ("grad", "jac"):
        c.update(n=logint(32, 8192))
    elif kind == "errors":
        c.update(n=logint(64, 16384), dtype="f32")
    elif kind == "polish":
        c.update(n=logint(64, 16384), dtype="f32", iters=rng.choice([10, 20]))
    elif kind == "classify":
        c.update(n=logint(64, 65536))
    elif kind == "ga":
        if c["dtype"] == "f64":  # FP64 maps of a few hundred pixels
            c.update(lines="one", nl=rng.randint(48, 80), n=logint(16, 300), npop=rng.choice([32, 64]), ngen=100)
        else:
            c.update(n=logint(1, 3000), npop=rng.choice([32, 64, 96, 128, 256]), ngen=rng.choice([100, 200, 300]))
    elif kind == "serve":
        c.update(n=logint(64, 1500), parts=rng.randint(1, 6), dtype="f32", fill=False)
    else:
        c.update(n=logint(64, 4096), npop=rng.choice([64, 128]), ngen=rng.choice([100, 200]), dtype="f32",
                 fill=False)
    return c


# ---------------------------------------------------------- plain FP64 model

class _Profile(torch.autograd.Function):
    """Re and Im of w(x + i a), a >= 0, by the trapezoidal rule with the pole's
    correction (Matta & Reichel 1971), with w' = -2 z w + 2 i / sqrt(pi)."""

    @staticmethod
    def forward(ctx, x, a):
        h, z = 0.5, torch.complex(x, a)
        frac = x / h - torch.floor(x / h)
        shifted = (frac < 0.25) | (frac > 0.75)  # nodes (k - 1/2) h there, k h elsewhere
        z2 = z * z
        # the node at 0 counts half; far from it in every shifted point
        s = torch.where(shifted, torch.zeros_like(z), 0.5 / torch.where(shifted, torch.ones_like(z), z2))
        for k in range(1, 14):
            t = (k - 0.5 * shifted.double()) * h
            s = s + torch.exp(-t * t) / (z2 - t * t)
        e = torch.exp(-2j * math.pi * z / h)
        pole = 2 * torch.exp(-z2) / torch.where(shifted, 1 + e, 1 - e)
        w = (2j * h / math.pi) * z * s + pole
        ctx.save_for_backward(z, w)
        return w.real.contiguous(), w.imag.contiguous()

    @staticmethod
    def backward(ctx, gh, gf):
        z, w = ctx.saved_tensors
        d = -2 * z * w + 2j / math.sqrt(math.pi)
        return gh * d.real + gf * d.imag, -gh * d.imag + gf * d.real


def _components(line):
    """(shifts [Larmor units, red positive], strengths) of sigma_b, pi, sigma_r."""
    if len(line) == 3:
        return [([(q * line[1])], [1.0]) for q in (-1, 0, 1)]
    jl, gl, ju, gu = line[3:]
    assert jl == ju
    out = []
    for q in (-1, 0, 1):
        rows = []
        for m in range(-ju, ju + 1):
            s = m * m if q == 0 else ((ju + m) * (ju - m + 1) if q < 0 else (ju - m) * (ju + m + 1))
            if -jl <= m + q <= jl and s > 0:
                rows.append((gl * (m + q) - gu * m, float(s)))
        tot = sum(s for _, s in rows)
        out.append(([r[0] for r in rows], [s / tot for _, s in rows]))
    return out


def _stokes(lines, lam, p, mu):
    """[..., 4] Stokes vectors in FP64: p's last axis holds the parameters, lam
    and mu broadcast against the axes before it."""
    deg = math.pi / 180.0
    b, th, ch, v, dw, a, eta0, s0, s1 = (p[..., k] for k in range(9))
    ct, s2 = torch.cos(th * deg), torch.sin(th * deg) ** 2
    P = Sb = Sr = Pi = Sbi = Sri = P0 = 0.0
    for line in lines:
        lam0, q = line[0], 0.5 * line[2]
        width = 1e-3 * lam0 / LINE2[0] * dw
        x = ((lam - lam0) - lam0 / LIGHT * v) / width
        larmor = ZEEMAN * lam0 * lam0 * b / width
        aa = a.expand(x.shape)
        sums = []
        for shifts, strengths in _components(line):
            h = f = 0.0
            for sh, st in zip(shifts, strengths):
                hh, ff = _Profile.apply(x - larmor * sh, aa)
                h, f = h + st * hh, f + st * ff
            sums.append((q * h, q * f))
        Sb, Sbi, P, Pi = Sb + sums[0][0], Sbi + sums[0][1], P + sums[1][0], Pi + sums[1][1]
        Sr, Sri = Sr + sums[2][0], Sri + sums[2][1]
        if p.shape[-1] == 10:
            P0 = P0 + q * _Profile.apply(x, aa)[0]
    T, Ti = P - 0.5 * (Sb + Sr), Pi - 0.5 * (Sbi + Sri)
    c2, sn2 = torch.cos(2 * ch * deg), torch.sin(2 * ch * deg)
    eI = 1 + eta0 * (s2 * P + 0.5 * (1 + ct * ct) * (Sb + Sr))
    eQ, eU, eV = eta0 * s2 * c2 * T, eta0 * s2 * sn2 * T, eta0 * ct * (Sr - Sb)
    rQ, rU, rV = eta0 * s2 * c2 * Ti, eta0 * s2 * sn2 * Ti, eta0 * ct * (Sri - Sbi)
    r2, e2, pi = rQ * rQ + rU * rU + rV * rV, eQ * eQ + eU * eU + eV * eV, eQ * rQ + eU * rU + eV * rV
    f = mu * s1 / (eI * eI * (eI * eI - e2 + r2) - pi * pi)
    I = s0 + f * eI * (eI * eI + r2)
    Q = -f * (eI * eI * eQ + eI * (eV * rU - eU * rV) + rQ * pi)
    U = -f * (eI * eI * eU + eI * (eQ * rV - eV * rQ) + rU * pi)
    V = -f * (eI * eI * eV + eI * (eU * rQ - eQ * rU) + rV * pi)
    if p.shape[-1] == 10:
        al = p[..., 9]
        quiet = s0 + mu * s1 / (1 + 2 * eta0 * P0)
        I, Q, U, V = al * I + (1 - al) * quiet, al * Q, al * U, al * V
    return torch.stack([I, Q, U, V], dim=-1)


# ------------------------------------------------------------------- inputs

def _lam(case):
    return np.linspace(*GRID[case["lines"]], case["nl"])


def _problem(case):
    return api.Problem(LINES[case["lines"]], _lam(case), LINE2[0], 1.0, case["dtype"], case["fill"])


def _npar(case):
    return 10 if case["fill"] else 9


def _torch_dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _uniform(case, g, n):
    m = _npar(case)
    lo, hi = (torch.tensor(v[:m], dtype=torch.float64, device="cuda") for v in (LO, HI))
    return lo + (hi - lo) * torch.rand((n, m), generator=g, dtype=torch.float64, device="cuda")


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 11)


def _near(case, g, truth, width):
    """Parameters about `width` of the prior range away from truth, inside it."""
    m = _npar(case)
    lo, hi = (torch.tensor(v[:m], dtype=torch.float64, device="cuda") for v in (LO, HI))
    step = width * (hi - lo) * torch.randn(truth.shape, generator=g, dtype=torch.float64, device="cuda")
    return torch.minimum(torch.maximum(truth + step, lo + 1e-3 * (hi - lo)), hi - 1e-3 * (hi - lo)).contiguous()


def _observe(case, g, truth, mu=None):
    """Profiles [n, 4, nl] of truth with noise of 1e-3 I_c, and I_c [n]."""
    n = truth.shape[0]
    lam = torch.tensor(_lam(case), dtype=torch.float64, device="cuda")
    ic = truth[:, 7] + (truth[:, 8] if mu is None else mu * truth[:, 8])
    obs = torch.empty((n, 4, case["nl"]), dtype=_torch_dtype(case), device="cuda")
    for i in range(0, n, CHUNK):
        p = truth[i:i + CHUNK, None, :]
        m = 1.0 if mu is None else mu[i:i + CHUNK, None]
        clean = _stokes(LINES[case["lines"]], lam, p, m).permute(0, 2, 1)
        noise = torch.randn(clean.shape, generator=g, dtype=torch.float32, device="cuda").double()
        obs[i:i + CHUNK] = (clean + 1e-3 * ic[i:i + CHUNK, None, None] * noise).to(obs.dtype)
    return obs, ic


def _weights(ic):
    return (1e3 / ic)[:, None].repeat(1, 4).contiguous()


def _sky(case, g, n):
    """Truth of a tile with 30 % strongly magnetised pixels, the rest quiet."""
    truth = _uniform(case, g, n)
    u = torch.rand((3, n), generator=g, dtype=torch.float64, device="cuda")
    truth[:, 0] = torch.where(u[0] < 0.3, 10.0 * 300.0 ** u[1], 50.0 * u[2])
    return truth


def _windows(case):
    """The quiet window [lo, hi) and the line window [lo, hi] about 6302.5 A."""
    nl = case["nl"]
    if case["lines"] == "one":
        return (0, nl // 8), 0, (nl // 4, 3 * nl // 4)
    return (0, nl // 16), len(LINES[case["lines"]]) - 1, (5 * nl // 8, 7 * nl // 8)


class _Serving:
    """A server and its requests' host arrays."""

    def __init__(self, pb, requests):
        self.requests = requests
        self.server = api.Server(pb, arena_bytes=64 << 20, max_inflight=16)

    def __del__(self):
        if hasattr(self, "server"):
            self.server.close()


def prepare(case, seed):
    kind, n, g = case["kind"], case["n"], _gen(seed)
    s = {"case": case, "pb": _problem(case), "seed": int(seed) & 0xFFFF}
    m = _npar(case)
    s["lo"], s["hi"] = LO[:m], HI[:m]
    if kind in ("synth", "jac"):
        s["params"] = _uniform(case, g, n)
    elif kind == "grad":
        s["params"] = _uniform(case, g, n).requires_grad_(True)
        s["up"] = torch.randn((n, 4, case["nl"]), generator=g, dtype=_torch_dtype(case), device="cuda")
    elif kind in ("errors", "polish"):
        truth = _uniform(case, g, n)
        s["obs"], ic = _observe(case, g, truth)
        s["w"] = _weights(ic)
        s["params"] = _near(case, g, truth, 0.002 if kind == "errors" else 0.02)
    elif kind == "classify":
        s["obs"], _ = _observe(case, g, _sky(case, g, n))
        s["pad"] = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        s["place"] = torch.arange(n, dtype=torch.int32, device="cuda")
    elif kind == "ga":
        s["obs"], _ = _observe(case, g, _uniform(case, g, n))
    elif kind == "serve":
        requests = []
        for k in range(case["parts"]):
            npix = max(1, case["n"] >> k)
            obs, ic = _observe(case, g, _sky(case, g, npix))
            ga = api.GaSettings(npop=(64, 128)[k % 2], ngen=(200, 100, 300)[k % 3], seed=s["seed"] + k)
            requests.append((obs.cpu().numpy(), _weights(ic).cpu().numpy(), ga))
        s["serving"] = _Serving(s["pb"], requests)
    else:
        mu = 0.2 + 0.8 * torch.rand(n, generator=g, dtype=torch.float64, device="cuda")
        s["obs"], ic = _observe(case, g, _sky(case, g, n), mu)
        s["w"], s["mu"] = _weights(ic), mu
    return s


def run(s):
    case, pb = s["case"], s["pb"]
    kind = case["kind"]
    if kind == "synth":
        return api.me_synth(pb, s["params"])
    if kind == "grad":
        stokes = api.synth_autograd(pb, s["params"])
        return {"stokes": stokes.detach(), "grad": torch.autograd.grad(stokes, s["params"], s["up"])[0]}
    if kind == "jac":
        jac, stokes = api.me_synth_jac(pb, s["params"], want_stokes=True)
        return {"jac": jac, "stokes": stokes}
    if kind == "errors":
        return {"chi2": api.me_chi2(pb, s["obs"], s["params"], w=s["w"]),
                "sigma": api.lm_uncertainty(pb, s["obs"], s["params"], w=s["w"])}
    if kind == "polish":
        p, chi2 = api.lm_polish(pb, s["obs"], s["params"], s["lo"], s["hi"], iters=case["iters"], w=s["w"])
        return {"params": p, "chi2": chi2}
    if kind == "classify":
        quiet, line, core = _windows(case)
        out = api.classify(pb, s["obs"], 10.0, quiet, line, core)
        index, count = api.select(out["flag"])
        out["index"] = torch.where(s["place"] < count, index, s["pad"])
        out["count"] = count
        out["centre"], out["centre_index"] = api.line_centre(pb, s["obs"], 10, *core)
        return out
    if kind == "ga":
        ga = api.GaSettings(npop=case["npop"], ngen=case["ngen"], seed=s["seed"])
        best, chi2, genes = api.ga_invert_batch(pb, s["obs"], s["lo"], s["hi"], ga, want_genes=True)
        return {"best": best, "chi2": chi2, "genes": genes}
    if kind == "serve":
        srv = s["serving"].server
        tickets = [srv.submit(obs, s["lo"], s["hi"], ga, polish_iters=10, polish_w=w)
                   for obs, w, ga in s["serving"].requests]
        done = [srv.poll(t) for t in tickets]
        return [{"best": r["best"], "chi2": r["chi2"]} for r in done]
    quiet, line, core = _windows(case)
    ga = api.GaSettings(npop=case["npop"], ngen=case["ngen"], seed=s["seed"])
    out = api.invert_map(pb, s["obs"], s["lo"], s["hi"], ga, 10.0, quiet, line, core, prefit=True,
                         polish_w=s["w"], mu_px=s["mu"])
    return {k: v for k, v in out.items() if k != "index"}  # written up to count only


# ------------------------------------------------------------ work and check

def work(case):
    """One reading of the inputs, one writing of the outputs; per wavelength
    point about 35 flops for each profile and 71 for the closed form, seven
    times the latter more for its derivatives."""
    kind, n, nl, m = case["kind"], case["n"], case["nl"], _npar(case)
    rs = 4 if case["dtype"] == "f32" else 8
    ncomp = sum(len(c[0]) for line in LINES[case["lines"]] for c in _components(line))
    point = nl * (35 * ncomp + 71)             # one synthesis
    deriv = nl * (55 * ncomp + 8 * 71)         # with its Jacobian
    normal = nl * 4 * (m * (m + 1) + 3 * m)    # J^T W^2 J and J^T W^2 r
    cube, par = 4 * nl * rs, 8 * m
    if kind == "synth":
        return {"bytes": n * (par + cube), "flops": n * point}
    if kind == "grad":
        return {"bytes": n * (2 * par + 2 * cube), "flops": n * (point + deriv + nl * 8 * m)}
    if kind == "jac":
        return {"bytes": n * (par + cube * (1 + m)), "flops": n * deriv}
    if kind == "errors":
        return {"bytes": n * (2 * par + cube + 32 + 8), "flops": n * (2 * point + deriv + normal)}
    if kind == "polish":
        return {"bytes": n * (2 * par + cube + 32 + 8),
                "flops": n * (2 * point + case["iters"] * (deriv + normal + point))}
    if kind == "classify":
        return {"bytes": n * (cube + 4 * 4 + 8 * (2 + 5 + 12 + 1) + 4), "flops": n * 60 * nl}
    if kind == "serve":
        total = {"bytes": 0, "flops": 0}
        for k in range(case["parts"]):
            npix, npop, ngen = max(1, n >> k), (64, 128)[k % 2], (200, 100, 300)[k % 3]
            total["bytes"] += npix * (par + cube + 32 + 8)
            total["flops"] += npix * ((npop * (ngen + 2.5) + 12) * point + 10 * (deriv + normal))
        return total
    syn = case["npop"] * (case["ngen"] + 2.5)  # three restarts of half the population
    if kind == "ga":
        return {"bytes": n * (par + cube + 8 + 2 * m), "flops": n * (syn + 1) * point}
    flagged = 0.25 * n
    return {"bytes": n * (6 * par + cube + 32 + 8 * 20),
            "flops": n * 60 * nl + flagged * ((syn + 53) * point + 50 * (deriv + normal))}


def _exact_rows(case, params, want_jac):
    """Stokes [n, 4, nl] and, if wanted, the Jacobian [n, 4, nl, m]."""
    lam = torch.tensor(_lam(case), dtype=torch.float64, device="cuda")
    lines, nl = LINES[case["lines"]], case["nl"]
    if not want_jac:
        return _stokes(lines, lam, params[:, None, :], 1.0).permute(0, 2, 1), None
    cols = []
    for k in range(4):  # each point's own copy of the parameters
        p = params[:, None, :].repeat(1, nl, 1).requires_grad_(True)
        st = _stokes(lines, lam, p, 1.0)
        cols.append(torch.autograd.grad(st[..., k].sum(), p)[0])
    return st.detach().permute(0, 2, 1), torch.stack(cols, dim=1)


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("synth", "grad", "jac", "errors"):
        return None  # searches and selections: no closed value
    s = prepare(case, seed)
    params = s["params"].detach()
    n, nl, m = case["n"], case["nl"], _npar(case)
    stokes, jacs, grads, chi2, sigma = [], [], [], [], []
    for i in range(0, n, CHUNK):
        st, jac = _exact_rows(case, params[i:i + CHUNK], kind != "synth")
        stokes.append(st)
        if kind == "jac":
            jacs.append(jac)
        elif kind == "grad":
            grads.append(torch.einsum("nsjk,nsj->nk", jac, s["up"][i:i + CHUNK].double()))
        elif kind == "errors":
            w, nu = s["w"][i:i + CHUNK], 4 * nl - m
            r = (s["obs"][i:i + CHUNK].double() - st) * w[:, :, None]
            chi2.append((r * r).sum((1, 2)) / nu)
            j = (jac * w[:, :, None, None]).reshape(-1, 4 * nl, m)
            h = (2.0 / nu) * torch.einsum("nrk,nrl->nkl", j, j)
            d = torch.diagonal(h, dim1=1, dim2=2).sqrt()
            inv = torch.linalg.inv(h / (d[:, :, None] * d[:, None, :]))
            sigma.append((torch.diagonal(inv, dim1=1, dim2=2) * chi2[-1][:, None] / m).sqrt() / d)
    if kind == "synth":
        return torch.cat(stokes)
    if kind == "jac":
        return {"jac": torch.cat(jacs), "stokes": torch.cat(stokes)}
    if kind == "grad":
        return {"stokes": torch.cat(stokes), "grad": torch.cat(grads)}
    return {"chi2": torch.cat(chi2), "sigma": torch.cat(sigma)}
