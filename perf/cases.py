"""The work that a program built on this library has it do, as measurable cases.

Each case names one public entry point and its sizes.  ``listed`` gives the
fixed ones, ``draw`` more of the same ranges, ``prepare`` the inputs and
handles that a program has in hand before the call, ``run`` one pass through
the entry point, ``work`` the bytes and operations the pass cannot do without,
and ``exact`` the same outputs in 64 bits from plain torch.

Inputs are seeded stand-ins with the statistics of ``workloads``: line lists
with centres and lower-state energies drawn uniformly, an opacity field with a
random walk and line spikes over wavenumber and trends in pressure and
temperature, proposals from the nine-parameter prior, Gaussian filters.
"""
import math

import numpy as np
import torch

import paper_2104_12522_gb300 as bart

H, C, KB, AMU = 6.62607015e-27, 2.99792458e10, 1.380649e-16, 1.66053906660e-24
C2, TREF, BAR = H * C / KB, 296.0, 1e6
R_SUN, R_JUP, AU = 6.957e10, 7.1492e9, 1.495978707e13
GRAV, MU, X0 = 2182.73, 2.3, 1e-4
THETA_LO = (-3.0, -1.5, -1.5, 0.0, 0.7, -3.0, -3.0, -3.0, -3.0)
THETA_HI = (0.0, 1.0, 1.0, 1.0, 1.3, 3.0, 3.0, 3.0, 3.0)
MASSES = (18.0, 28.0, 44.0, 16.0)
NU0 = 1000.0


# ------------------------------------------------------------------ the cases
def _emission(**kw):
    return dict(dict(kind="emission", n=1, S=4, L=100, M=20, N=100_000, dnu=0.02, angles=8, bands=10, spectra=False,
                     spans=False, profile=False, p_cloud=0.0, rayleigh=0.0, tau_max=0.0), **kw)


def _transit(**kw):
    return dict(dict(kind="transit", n=64, S=4, L=100, M=20, N=100_000, dnu=0.02, bands=12, level_lo=40, level_hi=150,
                     span_lo=10_000, span_hi=100_000, p_cloud=0.0, rayleigh=0.0), **kw)


def _opacity(**kw):
    return dict(dict(kind="opacity", entry="grid", S=1, lines=10_000, L=10, M=20, N=100_000, dnu=0.02), **kw)


def _surrogate(**kw):
    return dict(dict(kind="surrogate", B=2048, inputs=9, hidden=256, depth=3, bands=10), **kw)


def _training(**kw):
    return dict(dict(kind="training", B=1024, rows=20_000, steps=8, inputs=9, hidden=256, depth=3, bands=10), **kw)


def _retrieval(**kw):
    return dict(dict(kind="retrieval", chains=16, generations=64, S=4, L=100, M=20, N=100_000, dnu=0.02, bands=10,
                     screened=True), **kw)


def _contribution(**kw):
    return dict(dict(kind="contribution", n=4, S=4, L=100, M=20, N=100_000, dnu=0.02, angles=8, bands=10, rows=False),
                **kw)


def _statistics(**kw):
    return dict(dict(kind="statistics", n=20_000, chains=16, params=9, memory=150.0), **kw)


def listed():
    return [
        # the smallest call: one given temperature profile on a coarse grid (a plot, a check, a serial sampler)
        _emission(name="emission_one", n=1, S=2, L=60, M=1, N=2000, dnu=1.0, angles=4, bands=4, spectra=True,
                  profile=True),
        # one step of a 16-chain sampler on the full grid: what every retrieval iteration waits for
        _emission(name="emission_chains", n=16),
        # a population of 2,048 proposals on the full grid: prior draws, surrogate training sets
        _emission(name="emission_generation", n=2048),
        # odd sizes and options: packed spectra on spans, three species, a cloud deck and a Rayleigh haze
        _emission(name="emission_ragged", n=301, S=3, L=73, M=11, N=30_001, angles=4, bands=7, spectra=True,
                  spans=True, p_cloud=1.0, rayleigh=8.4e-45),
        # transit spectra of uneven instances
        _transit(name="transit_batch", n=1024),
        # opacities computed on the spot for one profile on a coarse grid
        _opacity(name="opacity_profile", entry="cells", S=2, lines=10_000, L=60, M=1, N=2000, dnu=1.0),
        # the opacity table: one species of the 5e6-line list, a tenth of its layers
        _opacity(name="opacity_table", S=1, lines=1_666_667, L=10, M=20, N=100_000),
        # the screening network over a population of proposals, and its training
        _surrogate(name="surrogate_forward", B=2048),
        _training(name="surrogate_training", B=1024),
        # the retrieval loop with the screening network
        _retrieval(name="retrieval_screened"),
        # the post-processing of a few spectra, and the convergence statistics of a chain
        _contribution(name="contribution_bands"),
        _statistics(name="chain_statistics"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["emission", "emission", "emission", "transit", "transit", "opacity", "opacity", "opacity",
                       "surrogate", "training", "retrieval", "contribution", "statistics"])
    grid = dict(S=rng.randint(1, 4), L=rng.randint(20, 120), M=rng.randint(2, 24), N=_log(rng, 500, 100_000),
                dnu=rng.choice([0.02, 0.025, 0.05]))
    if kind in ("emission", "contribution", "transit", "retrieval"):
        while grid["S"] * grid["L"] * grid["M"] * grid["N"] > 800_000_000:
            grid["N"] //= 2
    if kind == "emission":
        n = _log(rng, 1, 2048)
        while n * grid["N"] * grid["L"] > 1.5e10:
            n //= 2
        return _emission(n=n, angles=rng.choice([1, 2, 4, 8, 8, 16]) if n * grid["N"] * grid["L"] < 8e9 else 8,
                         bands=rng.randint(1, 16), spectra=n * grid["N"] < 2e8 and rng.random() < 0.5,
                         spans=rng.random() < 0.3, profile=rng.random() < 0.3, p_cloud=rng.choice([0.0, 0.0, 0.1]),
                         rayleigh=rng.choice([0.0, 0.0, 8.4e-45]), tau_max=rng.choice([0.0, 0.0, 0.0, 20.0]), **grid)
    if kind == "transit":
        n = _log(rng, 1, 1024)
        lo = rng.randint(5, 100)
        hi = rng.randint(lo, 150)
        span = _log(rng, 100, grid["N"]) if grid["N"] > 100 else grid["N"]
        return _transit(n=n, bands=rng.randint(1, 16), level_lo=lo, level_hi=hi, span_lo=max(1, span // 2),
                        span_hi=span, p_cloud=rng.choice([0.0, 0.0, 0.01]), rayleigh=rng.choice([0.0, 8.4e-45]), **grid)
    if kind == "opacity":
        c = _opacity(entry=rng.choice(["grid", "cells"]), S=rng.randint(1, 3), lines=_log(rng, 100, 400_000),
                     L=rng.randint(1, 30), M=rng.randint(1, 10), N=_log(rng, 500, 100_000),
                     dnu=rng.choice([0.02, 0.02, 0.05, 0.1, 0.25, 1.0]))
        while _evaluations(c) > 1.5e11:
            c["lines"] = max(1, c["lines"] // 2)
        return c
    net = dict(inputs=rng.choice([8, 9]), hidden=rng.choice([64, 128, 256, 256]), depth=rng.randint(2, 3),
               bands=rng.randint(4, 12))
    if kind == "surrogate":
        return _surrogate(B=_log(rng, 1, 4096), **net)
    if kind == "training":
        return _training(B=_log(rng, 32, 2048), steps=rng.randint(1, 8), **net)
    if kind == "retrieval":
        return _retrieval(chains=_log(rng, 6, 64), generations=rng.randint(4, 48), bands=rng.randint(4, 12),
                          screened=rng.random() < 0.5, **grid)
    if kind == "contribution":
        return _contribution(n=rng.randint(1, 4), angles=rng.choice([4, 8]), bands=rng.randint(1, 12),
                             rows=rng.random() < 0.3, **grid)
    return _statistics(n=_log(rng, 200, 20_000), chains=_log(rng, 2, 32), params=rng.randint(3, 9),
                       memory=float(_log(rng, 5, 150)))


# ------------------------------------------------------------------ inputs
_contexts = {}


def _context():
    """A program has one context for its whole life."""
    if "ctx" not in _contexts:
        _contexts["ctx"] = bart.Context(0)
    return _contexts["ctx"]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _axes(c):
    return (np.logspace(-8, 2, c["L"]) if c["L"] > 1 else np.array([0.1]),
            np.linspace(500.0, 3000.0, c["M"]) if c["M"] > 1 else np.array([1000.0]))


def _field(g, c):
    """Opacity field [S][L][M][N]: per species a base level, a detrended random walk over wavenumber, line spikes,
    a slope in log P per layer and a temperature trend per wavenumber."""
    S, L, M, N = c["S"], c["L"], c["M"], c["N"]
    p, t = _axes(c)
    lp = torch.tensor(np.log10(p) + 3.0, device="cuda", dtype=torch.float32)
    tt = torch.tensor((t - 1750.0) / 1250.0, device="cuda", dtype=torch.float32)[:, None]
    out = torch.empty((S, L, M, N), device="cuda", dtype=torch.float32)
    j = torch.arange(N, device="cuda", dtype=torch.float64)
    jc = j - j.mean()
    offs = torch.arange(-60, 61, device="cuda")
    for s in range(S):
        walk = torch.cumsum(0.2 * torch.randn(N, generator=g, device="cuda", dtype=torch.float64), 0)
        walk = walk - walk.mean() - jc * ((jc * walk).sum() / (jc * jc).sum().clamp_min(1e-30))
        walk *= 2.5 / walk.abs().max().clamp_min(1e-12)
        k = max(1, N // 50)
        at = torch.randint(0, N, (k, 1), generator=g, device="cuda")
        h, q = _uniform(g, 0.5, 3.0, k, 1), _uniform(g, 0.5, 0.9, k, 1)
        spikes = torch.zeros(N, device="cuda", dtype=torch.float64)
        where = (at + offs).clamp(0, N - 1)
        spikes.scatter_reduce_(0, where.reshape(-1), (h * q ** (where - at).abs()).reshape(-1), "amax")
        row = (_uniform(g, -23.5, -21.5, 1) + walk + spikes).float()
        pslope = _uniform(g, -0.3, 0.3, L).float()
        trend = _uniform(g, -1.0, 1.0, N).float() * tt
        for k in range(L):
            lg = row + pslope[k] * lp[k] + trend + 0.05 * torch.randn(M, N, generator=g, device="cuda")
            out[s, k] = torch.pow(10.0, lg.clamp(-30.0, -16.0))
    return out


def _filters(g, c):
    """[bands][N] Gaussian curves cut at three sigma, centres and widths spread over the grid."""
    width = c["N"] * c["dnu"]
    nu = NU0 + torch.arange(c["N"], device="cuda", dtype=torch.float64) * c["dnu"]
    cen = NU0 + width * _uniform(g, 0.05, 0.95, c["bands"], 1)
    sig = width * _uniform(g, 0.01, 0.1, c["bands"], 1) / 2.3548200450309493
    d = (nu - cen) / sig
    return torch.where(d.abs() <= 3.0, torch.exp(-0.5 * d * d), 0.0).float().contiguous()


def _theta(g, n, S):
    lo = torch.tensor(THETA_LO[: 5 + S], device="cuda", dtype=torch.float64)
    hi = torch.tensor(THETA_HI[: 5 + S], device="cuda", dtype=torch.float64)
    return (lo + (hi - lo) * torch.rand(n, 5 + S, generator=g, device="cuda", dtype=torch.float64)).float()


def _cfg(c, geometry=0):
    return dict(geometry=geometry, n_angles=c.get("angles", 8), g=GRAV, mu=MU, x0=[X0] * c["S"], t_int=100.0,
                t_star=5000.0, r_star_tp=0.756 * R_SUN, a_orbit=0.0312 * AU, t_min=500.0, t_max=3000.0, p_ref=0.1,
                p_top=1e-8, p_bot=100.0, tau_max=c.get("tau_max", 0.0), p_cloud=c.get("p_cloud", 0.0),
                rayleigh_coef=c.get("rayleigh", 0.0))


def _spans(g, c, lo, hi):
    # the lengths belong to the case (a packed output keeps its size from seed to seed), the places to the seed
    n, N = c["n"], c["N"]
    span = torch.tensor(np.random.RandomState(4000).randint(lo, hi + 1, n), device="cuda", dtype=torch.int64)
    start = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (N - span + 1)).long()
    start = torch.minimum(start, N - span)
    offs = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    offs[1:] = torch.cumsum(span, 0)
    return start, start + span, offs


def _lines(g, c, s):
    """Line list s on the grid's range, sorted by centre."""
    n = c["lines"]
    nu0 = torch.sort(NU0 + c["N"] * c["dnu"] * torch.rand(n, generator=g, device="cuda", dtype=torch.float64))[0]
    elow = _uniform(g, 0.0, 5000.0, n)
    logs = _uniform(g, -25.0, -19.0, n) - C2 * elow / (TREF * math.log(10.0))
    return nu0, logs.float(), elow.float(), _uniform(g, 0.05, 0.1, n).float(), MASSES[s]


def _inputs(c, seed):
    """Everything a case's entry point reads, from the seed alone."""
    g = _gen(seed)
    kind = c["kind"]
    d = {}
    if kind in ("emission", "transit", "contribution", "retrieval"):
        d["grid"], d["filters"] = _field(g, c), _filters(g, c)
        d["p"], d["t"] = _axes(c)
    if kind in ("emission", "contribution"):
        d["theta"] = _theta(g, c["n"], c["S"])
        if c.get("profile"):
            # an inversion near 1 mbar of random strength
            p = torch.tensor(d["p"], device="cuda")
            d["t_profile"] = (800.0 + _uniform(g, 100.0, 600.0, c["n"], 1) *
                              (1.0 - torch.tanh((torch.log10(p) + 3.0) / 0.5))).float().contiguous()
        if c.get("spans"):
            d["lo"], d["hi"], d["offs"] = _spans(g, c, max(1, c["N"] // 10), c["N"])
    elif kind == "transit":
        d["theta"] = _theta(g, c["n"], c["S"])
        d["levels"] = torch.randint(c["level_lo"], c["level_hi"] + 1, (c["n"],), generator=g, device="cuda",
                                    dtype=torch.int32)
        d["lo"], d["hi"], d["offs"] = _spans(g, c, min(c["span_lo"], c["N"]), min(c["span_hi"], c["N"]))
        d["r_planet"] = (_uniform(g, 1.0, 1.4, c["n"]) * R_JUP).float()
        d["r_star"] = (_uniform(g, 0.7, 1.2, c["n"]) * R_SUN).float()
    elif kind == "opacity":
        d["p"], d["t"] = _axes(c)
        if c["entry"] == "cells":
            lp = np.log10(d["p"])
            p, t = np.repeat(d["p"], c["M"]), np.tile(np.linspace(0.9, 1.1, c["M"]), c["L"])
            d["p"] = p
            d["t"] = t * np.repeat(800.0 + 350.0 * (1.0 - np.tanh((lp + 3.0) / 0.5)), c["M"])
        d["lines"] = [_lines(g, c, s) for s in range(c["S"])]
    elif kind in ("surrogate", "training"):
        widths = [c["inputs"]] + [c["hidden"]] * c["depth"] + [c["bands"]]
        parts = []
        for a, b in zip(widths[:-1], widths[1:]):
            parts += [torch.randn(b * a, generator=g, device="cuda") * math.sqrt(2.0 / a),
                      0.1 * torch.randn(b, generator=g, device="cuda")]
        d["widths"], d["params"] = widths, torch.cat(parts)
        rows = c["B"] if kind == "surrogate" else c["rows"]
        d["x"] = _theta(g, rows, c["inputs"] - 5)
        lo, hi = np.array(THETA_LO[: c["inputs"]]), np.array(THETA_HI[: c["inputs"]])
        d["scaling"] = ((0.5 * (lo + hi)).astype(np.float32), (2.0 / (hi - lo)).astype(np.float32),
                        np.full(c["bands"], 4.0, np.float32), np.full(c["bands"], 2.0, np.float32))
        if kind == "training":
            w = torch.randn(c["inputs"], c["bands"], generator=g, device="cuda") * 0.1
            d["y"] = torch.pow(10.0, 4.0 + torch.tanh(d["x"] @ w)).contiguous()
            d["rows"] = torch.randint(0, rows, (c["steps"], c["B"]), generator=g, device="cuda", dtype=torch.int32)
            # the end of a decaying schedule
            d["lr"] = [1e-5 * 0.5 * (1.0 + math.cos(math.pi * k / (c["steps"] + 1))) for k in range(c["steps"])]
    elif kind == "statistics":
        # series with an exponential memory, held where a step is rejected
        n, m = c["n"], c["chains"] * c["params"]
        f = torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64)[:, None]
        tau = c["memory"] * _uniform(g, 0.5, 1.5, 1, m)
        spec = torch.fft.rfft(torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64), dim=0)
        x = torch.fft.irfft(spec / torch.sqrt(1.0 + (2.0 * math.pi * f * tau) ** 2), n=n, dim=0)
        x = (x / x.std(dim=0)).reshape(n, c["chains"], c["params"])
        moved = torch.rand(n, c["chains"], generator=g, device="cuda") < 0.25
        moved[0] = True
        t = torch.arange(n, device="cuda")[:, None].expand(n, c["chains"])
        last = torch.cummax(torch.where(moved, t, torch.zeros_like(t)), dim=0)[0]
        d["chain"] = torch.gather(x, 0, last[:, :, None].expand_as(x)).float().contiguous()
    if kind == "retrieval":
        _retrieval_inputs(g, c, d)
    return d


def _retrieval_inputs(g, c, d):
    """Data at S/N 20 from a true state, chains scattered about it with their log-likelihoods, and a network that
    predicts the bands there: random hidden layers, the last layer fitted."""
    k = 5 + c["S"]
    lo = torch.tensor(THETA_LO[:k], device="cuda", dtype=torch.float64)
    hi = torch.tensor(THETA_HI[:k], device="cuda", dtype=torch.float64)
    true = lo + (hi - lo) * _uniform(g, 0.35, 0.65, 1, k)
    near = lambda n, r: torch.minimum(torch.maximum(true + r * (hi - lo) * torch.randn(  # noqa: E731
        n, k, generator=g, device="cuda", dtype=torch.float64), lo), hi).float()
    bands = lambda th, step: _emission_exact(dict(c, angles=8), dict(d, theta=th), step=step)[1]  # noqa: E731
    data = bands(true.float(), 1)[0]
    d["sigma"] = (data / 20.0).float()
    d["data"] = (data * (1.0 + 0.05 * torch.randn(c["bands"], generator=g, device="cuda", dtype=torch.float64))).float()
    d["x"] = near(c["chains"], 0.02).contiguous()
    chi2 = lambda b: -0.5 * (((b - d["data"].double()) / d["sigma"].double()) ** 2).sum(1)  # noqa: E731
    d["loglike"] = chi2(bands(d["x"], 1))
    if not c["screened"]:
        return
    widths = [k, 256, 256, 256, c["bands"]]
    th = near(400, 0.06)
    target = torch.log10(bands(th, max(1, c["N"] // 2000)).clamp_min(1e-30))
    h = (th.double() - true) / (0.1 * (hi - lo))
    parts = []
    for a, b in zip(widths[:-2], widths[1:-1]):
        w = torch.randn(b, a, generator=g, device="cuda") * math.sqrt(1.0 / a)
        bias = 0.3 * torch.randn(b, generator=g, device="cuda")
        parts += [w.reshape(-1), bias]
        h = torch.nn.functional.gelu(h @ w.bfloat16().double().T + bias.double())
    shift, scale = target.mean(0), 1.0 / target.std(0).clamp_min(1e-3)
    a = np.concatenate([h.cpu().numpy(), np.ones((len(h), 1))], 1)
    y = ((target - shift) * scale).cpu().numpy()
    sol = np.linalg.solve(a.T @ a + 1e-2 * np.eye(a.shape[1]), a.T @ y)
    parts += [torch.tensor(sol[:-1].T.copy(), device="cuda").float().reshape(-1),
              torch.tensor(sol[-1], device="cuda").float()]
    d["widths"], d["params"] = widths, torch.cat(parts)
    d["scaling"] = tuple(v.reshape(-1).cpu().numpy().astype(np.float32)
                         for v in (true, 10.0 / (hi - lo), shift, scale))
    d["loglike_s"] = chi2(_network(d, d["x"])[0])


# ------------------------------------------------------------------ one pass
def prepare(case, seed):
    c, ctx = case, _context()
    d = _inputs(c, seed)
    st = dict(d, case=c, ctx=ctx)
    kind = c["kind"]
    if "N" in c:
        st["nu"] = bart.NuGrid(NU0, c["dnu"], c["N"])
    if kind in ("emission", "transit"):
        st["cfg"] = _cfg(c, geometry=int(kind == "transit"))
        st["bands"] = torch.zeros((c["n"], c["bands"]), device="cuda")
        if kind == "transit" or c["spans"]:
            st["spectra"] = torch.zeros(int(d["offs"][-1]), device="cuda")
        else:
            st["spectra"] = torch.zeros((c["n"], c["N"]), device="cuda")
        if kind == "emission" and not c["spectra"]:
            st["spectra"] = None
    elif kind == "contribution":
        st["cfg"] = _cfg(c)
        st["bands"] = torch.zeros((c["n"], c["L"], c["bands"]), device="cuda")
        st["rows"] = torch.zeros((c["n"], c["L"], c["N"]), device="cuda") if c["rows"] else None
    elif kind == "opacity":
        st["lists"] = [bart.DeviceLines(*v) for v in d["lines"]]
        cells = (c["L"] * c["M"],) if c["entry"] == "cells" else (c["L"], c["M"])
        st["out"] = torch.zeros((c["S"], *cells, c["N"]), device="cuda")
    if "params" in d:
        most = c.get("B") or c["chains"]
        st["net"] = bart.Mlp(ctx, d["widths"], max_batch=most)
        st["net"].set_scaling(*d["scaling"])
        st["net"].set_params(d["params"])
        if kind == "surrogate":
            st["y"] = torch.zeros((c["B"], c["bands"]), device="cuda")
        elif kind == "training":
            st["loss"] = torch.zeros(c["steps"], device="cuda")
            st["trained"] = torch.zeros_like(d["params"])
    if kind == "retrieval":
        st["cfg"] = _cfg(dict(c, angles=8))
        k = 5 + c["S"]
        st["demc"] = bart.Demc(ctx, c["chains"], THETA_LO[:k], THETA_HI[:k])
        st["demc"].set_screen(1.0, 1.0)
        st["chain"] = torch.zeros((c["generations"], c["chains"], k), device="cuda")
    return st


def run(state):
    s, c, ctx = state, state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "emission":
        ctx.forward_spectra_batch(s["grid"], s["p"], s["t"], s["nu"], s["cfg"], theta=s["theta"],
                                  t_profile=s.get("t_profile"), nu_lo=s.get("lo"), nu_hi=s.get("hi"),
                                  spec_offsets=s.get("offs"), spectra=s["spectra"], filters=s["filters"],
                                  bands=s["bands"])
        return {"spectra": s["spectra"], "bands": s["bands"]}
    if kind == "transit":
        ctx.forward_spectra_batch(s["grid"], s["p"], s["t"], s["nu"], s["cfg"], theta=s["theta"],
                                  n_levels=s["levels"], nu_lo=s["lo"], nu_hi=s["hi"], spec_offsets=s["offs"],
                                  r_planet=s["r_planet"], r_star=s["r_star"], spectra=s["spectra"],
                                  filters=s["filters"], bands=s["bands"])
        return {"spectra": s["spectra"], "bands": s["bands"]}
    if kind == "opacity":
        f = ctx.opacity_cells if c["entry"] == "cells" else ctx.build_opacity_grid
        return f(s["lists"], s["p"], s["t"], s["nu"], 25.0, out=s["out"])
    if kind == "surrogate":
        return s["net"].forward(s["x"], out=s["y"])
    if kind == "training":
        # training restarts from the state's weights, so that every pass does the same
        s["net"].set_params(s["params"])
        s["net"].train_steps(s["x"], s["y"], s["rows"], s["lr"], loss=s["loss"])
        return {"params": s["net"].get_params(out=s["trained"]), "loss": s["loss"]}
    if kind == "retrieval":
        s["demc"].set_state(s["x"], s["loglike"], s.get("loglike_s"))
        got = ctx.retrieval_run(s["demc"], s.get("net"), s["grid"], s["p"], s["t"], s["nu"], s["cfg"], s["filters"],
                                s["data"], s["sigma"], c["generations"], chain=s["chain"])
        return {"chain": s["chain"], "counts": [got[k] for k in ("proposals", "screened_out", "exact_evals",
                                                                 "accepted")]}
    if kind == "contribution":
        ctx.contribution_functions(s["grid"], s["p"], s["t"], s["nu"], s["cfg"], theta=s["theta"], contrib=s["rows"],
                                   filters=s["filters"], bands=s["bands"])
        return {"rows": s["rows"], "bands": s["bands"]}
    speis, gr, ess = ctx.chain_stats(s["chain"])
    return {"speis": speis, "gr": gr, "ess": torch.tensor(ess, dtype=torch.float64)}


# ------------------------------------------------------------------ the least work
def _evaluations(c):
    return c["S"] * c["lines"] * c["L"] * c["M"] * min(2.0 * 25.0 / c["dnu"] + 1.0, c["N"])


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("emission", "contribution", "retrieval"):
        n = c["n"] if "n" in c else c["chains"] * c["generations"]
        points = n * c["N"] * (0.55 if c.get("spans") else 1.0)
        rows = 2.0 * c["S"] * c["L"] * points * 4.0 if c["M"] > 1 else c["S"] * c["L"] * points * 4.0
        table = c["S"] * c["L"] * c["M"] * c["N"] * 4.0
        outputs = points * 4.0 if c.get("spectra") else 0.0
        outputs += points * c["L"] * 4.0 if c.get("rows") else 0.0
        per = 4.0 * c["S"] + 4.0 * c.get("angles", 8) + 14.0
        return {"bytes": min(rows, table) + outputs + c["bands"] * c["N"] * 4.0, "flops": points * c["L"] * per}
    if kind == "transit":
        levels, span = 0.5 * (c["level_lo"] + c["level_hi"]), 0.5 * (c["span_lo"] + c["span_hi"])
        pairs = c["n"] * levels * span
        table = c["S"] * c["L"] * c["M"] * c["N"] * 4.0
        return {"bytes": min(16.0 * c["S"] * pairs, table) + c["n"] * span * 4.0,
                "flops": pairs * (8.0 * c["S"] + levels + 10.0)}
    if kind == "opacity":
        return {"bytes": c["S"] * (c["lines"] * 20.0 + c["L"] * c["M"] * c["N"] * 4.0),
                "flops": 10.0 * _evaluations(c)}
    if kind in ("surrogate", "training"):
        w = [c["inputs"]] + [c["hidden"]] * c["depth"] + [c["bands"]]
        params = sum(a * b + b for a, b in zip(w[:-1], w[1:]))
        if kind == "surrogate":
            return {"bytes": params * 2.0 + c["B"] * (w[0] + w[-1]) * 4.0, "flops": 2.0 * params * c["B"]}
        return {"bytes": params * 8.0 + c["steps"] * c["B"] * (w[0] + w[-1]) * 4.0,
                "flops": 6.0 * params * c["B"] * c["steps"]}
    series = c["chains"] * c["params"]
    return {"bytes": c["n"] * series * 4.0, "flops": 2.0 * c["n"] * series * 4.6 * c["memory"]}


# ------------------------------------------------------------------ 64 bits
def _e2(x):
    """Exponential integral E2 for x >= 0."""
    x = np.asarray(x, np.float64)
    small = np.clip(x, 1e-300, 1.0)
    term, total = np.ones_like(small), np.zeros_like(small)
    for k in range(1, 40):
        term = term * -small / k
        total = total + term / k
    low = np.exp(-small) - small * (-0.57721566490153286 - np.log(small) - total)
    big = np.clip(x, 1.0, 700.0)
    t = big + 2.0 * 400
    for k in range(399, -1, -1):   # the continued fraction of E_n, n = 2
        t = big + 2.0 + 2.0 * k - (k + 1.0) * (k + 2.0) / t
    return np.where(x <= 0, 1.0, np.where(x < 1.0, low, np.exp(-big) / t))


def _temperature(theta, p_bar):
    """T of theta [n][>=5] at pressures p_bar [..][L], clamped to the grid's range."""
    th = np.asarray(theta, np.float64)
    kappa, g1, g2 = (10.0 ** th[:, i : i + 1] for i in range(3))
    tau = kappa * np.asarray(p_bar, np.float64) * BAR / GRAV

    def xi(g):
        gt = g * tau
        return (2 / 3 + 2 / (3 * g) * (1 + (gt / 2 - 1) * np.exp(-gt)) + 2 * g / 3 * (1 - tau ** 2 / 2) * _e2(gt))

    irr = (th[:, 4:5] * math.sqrt(0.756 * R_SUN / (2 * 0.0312 * AU)) * 5000.0) ** 4
    t4 = 0.75 * 100.0 ** 4 * (2 / 3 + tau) + 0.75 * irr * ((1 - th[:, 3:4]) * xi(g1) + th[:, 3:4] * xi(g2))
    return np.clip(t4 ** 0.25, 500.0, 3000.0)


def _bracket(axis, v):
    """Lower node and upper weight of linear interpolation on an axis, as tensors."""
    axis, v = np.asarray(axis, np.float64), np.asarray(v, np.float64)
    if axis.size == 1:
        m, w = np.zeros(v.shape, np.int64), np.zeros(v.shape)
    else:
        m = np.clip(np.searchsorted(axis, v, side="right") - 1, 0, axis.size - 2)
        w = np.clip((v - axis[m]) / (axis[m + 1] - axis[m]), 0.0, 1.0)
    return torch.tensor(m, device="cuda"), torch.tensor(w, device="cuda")


def _band_means(spec, filters, lo=None, hi=None):
    """Trapezoid-weighted means of spec [n][N] (full grid) over the filters on each span."""
    n, N = spec.shape
    j = torch.arange(N, device="cuda")
    lo = torch.zeros(n, dtype=torch.int64, device="cuda") if lo is None else lo
    hi = torch.full((n,), N, dtype=torch.int64, device="cuda") if hi is None else hi
    w = ((j >= lo[:, None]) & (j < hi[:, None])).double()
    w[(j == lo[:, None]) | (j == hi[:, None] - 1)] *= 0.5
    f = filters.double()
    num, den = (w * spec) @ f.T, w @ f.T
    return torch.where(den > 0, num / den.clamp_min(1e-300), 0.0)


def _emission_exact(c, d, step=1, contributions=False):
    """Spectra [n][N] and band means of an emission batch (every step-th wavenumber), or the contribution rows
    [n][L][N] and their band means."""
    grid, p, n = d["grid"], d["p"], d["theta"].shape[0]
    S, L, M, N = grid.shape
    T = (d["t_profile"].double().cpu().numpy() if "t_profile" in d
         else _temperature(d["theta"].cpu().numpy(), p[None, :]))
    T = np.clip(T, 500.0, 3000.0)
    m, w = _bracket(d["t"], T)
    w = w[:, :, None]
    X = X0 * 10.0 ** d["theta"].double()[:, 5 : 5 + S] / (MU * AMU)
    mu, wt = np.polynomial.legendre.leggauss(c["angles"])
    mu, wt = 0.5 * (mu + 1.0), 0.5 * wt
    T = torch.tensor(T, device="cuda")
    deck = c.get("p_cloud", 0.0)
    last = L
    if deck > 0 and (p >= deck).any():
        last = max(int(np.argmax(p >= deck)) + 1, 2)
    index = torch.arange(0, N, step, device="cuda")
    spec = torch.zeros((n, len(index)), device="cuda", dtype=torch.float64)
    rows = torch.zeros((n, L, len(index)), device="cuda", dtype=torch.float64) if contributions else None
    chunk = max(64, int(1.5e7) // n)
    for a in range(0, len(index), chunk):
        idx = index[a : a + chunk]
        part = slice(a, a + len(idx))
        at = slice(int(idx[0]), int(idx[-1]) + 1, step)
        nu = NU0 + idx.double() * c["dnu"]
        ray = c.get("rayleigh", 0.0) * nu ** 4 / (MU * AMU)

        def level(k):
            chi = ray.expand(n, -1)
            for s in range(S):
                g = grid[s, k][:, at]
                low = g[m[:, k]].double()
                if M > 1:
                    low = low + w[:, k] * (g[m[:, k] + 1].double() - low)
                chi = chi + X[:, s : s + 1] * low
            return chi, 2 * H * C * C * nu ** 3 / torch.expm1(C2 * nu / T[:, k : k + 1])

        chi, B = level(0)
        tau = torch.zeros_like(chi)
        t_prev = [torch.ones_like(chi) for _ in mu]
        F, stop = torch.zeros_like(chi), torch.zeros_like(chi, dtype=torch.bool)
        for k in range(1, last):
            chi2, B2 = level(k)
            tau = tau + 0.5 * (chi + chi2) * ((p[k] - p[k - 1]) * BAR / GRAV)
            term = torch.zeros_like(F)
            for i in range(len(mu)):
                t = torch.exp(-tau / mu[i])
                if c.get("tau_max", 0.0) > 0:
                    t = torch.where(stop, t_prev[i], t)
                term += wt[i] * mu[i] * (t_prev[i] - t)
                t_prev[i] = t
            term *= 2 * math.pi * 0.5 * (B + B2)
            F += term
            if rows is not None:
                rows[:, k - 1, part] = term
            chi = chi2
            if c.get("tau_max", 0.0) > 0:
                B = torch.where(stop, B, B2)
                stop = stop | (tau > c["tau_max"])
            else:
                B = B2
        bottom = 2 * math.pi * B * sum(wt[i] * mu[i] * t_prev[i] for i in range(len(mu)))
        spec[:, part] = F + bottom
        if rows is not None:
            rows[:, last - 1, part] = bottom
    f = d["filters"][:, ::step]
    if rows is not None:
        return rows, torch.stack([_band_means(r, f) for r in rows])
    return spec, _band_means(spec, f, d.get("lo"), d.get("hi"))


def _transit_exact(c, d):
    grid = d["grid"]
    S, Lg, M, N = grid.shape
    out = torch.zeros(int(d["offs"][-1]), device="cuda", dtype=torch.float64)
    bands = torch.zeros((c["n"], c["bands"]), device="cuda", dtype=torch.float64)
    lp_axis = np.log10(d["p"])
    theta, levels = d["theta"].double().cpu().numpy(), d["levels"].cpu().numpy()
    lo_, hi_, offs = (d[k].cpu().numpy() for k in ("lo", "hi", "offs"))
    for i in range(c["n"]):
        L, lo, hi = int(levels[i]), int(lo_[i]), int(hi_[i])
        P = np.logspace(-8, 2, L)
        T = _temperature(theta[i : i + 1], P[None, :])[0]
        rp, rs = float(d["r_planet"][i]), float(d["r_star"][i])
        # hydrostatic radii with the reference pressure as a node
        lnp, ref = np.log(P), math.log(0.1)
        nodes, temps = np.append(lnp, ref), np.append(T, np.interp(ref, lnp, T))
        order = np.argsort(nodes, kind="stable")
        cum = np.append(0.0, np.cumsum(0.5 * (temps[order][1:] + temps[order][:-1]) * np.diff(nodes[order])))
        phi = np.empty(L + 1)
        phi[order] = cum
        phi = phi[:L] - phi[L]
        r = 1.0 / (1.0 / rp + KB / (MU * AMU * GRAV * rp * rp) * phi)
        deck = c.get("p_cloud", 0.0)
        E = max(int(np.argmax(P >= deck)) + 1, 2) if deck > 0 and (P >= deck).any() else L
        a, u = _bracket(lp_axis, np.log10(P[:E]))
        m, w = _bracket(d["t"], T[:E])
        u, w = u[:, None], w[:, None]
        a1, m1 = (a + 1 if Lg > 1 else a), (m + 1 if M > 1 else m)
        nu = NU0 + torch.arange(lo, hi, device="cuda", dtype=torch.float64) * c["dnu"]
        sig = c.get("rayleigh", 0.0) * nu ** 4 * torch.ones((E, 1), device="cuda", dtype=torch.float64)
        for s in range(S):
            g = grid[s][:, :, lo:hi]
            top = g[a, m].double() * (1 - w) + g[a, m1].double() * w
            low = g[a1, m].double() * (1 - w) + g[a1, m1].double() * w
            sig = sig + X0 * 10.0 ** theta[i, 5 + s] * (top * (1 - u) + low * u)
        alpha = sig * torch.tensor(P * BAR / (KB * T), device="cuda")[:E, None]
        mean = 0.5 * (alpha[:-1] + alpha[1:])
        b = r[:E, None]
        path = np.sqrt(np.maximum(r[None, :E] ** 2 - b * b, 0.0))
        ds = np.where(np.arange(E - 1)[None, :] < np.arange(E)[:, None], 2.0 * (path[:, :-1] - path[:, 1:]), 0.0)
        f = -torch.expm1(-(torch.tensor(ds, device="cuda") @ mean)) * torch.tensor(b, device="cuda")
        dr = torch.tensor(r[: E - 1] - r[1:E], device="cuda")[:, None]
        depth = (r[E - 1] ** 2 + 2.0 * (0.5 * (f[:-1] + f[1:]) * dr).sum(0)) / rs ** 2
        out[offs[i] : offs[i + 1]] = depth
        bands[i] = _band_means(depth[None, :], d["filters"][:, lo:hi])[0]
    return {"spectra": out, "bands": bands}


def _faddeeva_re(x, y):
    """Re w(x + i y), y > 0: the trapezoidal rule for w's integral with step 1/2, on nodes or midpoints (whichever
    are farther from x), plus the residue of the pole that lies between the rule's line and the real axis."""
    h = 0.5
    x = x.abs()
    f = x / h - torch.floor(x / h)
    mid = ((f < 0.25) | (f > 0.75)).double()
    total = torch.zeros_like(x)
    for k in range(-14, 15):
        t = (k + 0.5 * mid) * h
        total += torch.exp(-t * t) / ((x - t) ** 2 + y * y)
    v = total * (h * y / math.pi)
    # 2 exp(-z^2) / (1 -+ exp(-2 pi i z / h)) where y < pi / h
    near = (y < math.pi / h) & (x < 27.0)
    yc, xc = torch.where(near, y, 1.0), torch.where(near, x, 1.0)
    z = torch.complex(xc, yc)
    sign = torch.where(mid > 0, 1.0, -1.0)
    e = torch.exp(torch.complex(2 * math.pi * yc / h, -2 * math.pi * xc / h))
    return v + torch.where(near, (2.0 * torch.exp(-z * z) / (1.0 + sign * e)).real, 0.0)


def _opacity_exact(c, d):
    N, dnu = c["N"], c["dnu"]
    cells = [(p, t) for p in d["p"] for t in d["t"]] if c["entry"] == "grid" else list(zip(d["p"], d["t"]))
    shape = (c["S"], c["L"], c["M"], N) if c["entry"] == "grid" else (c["S"], len(cells), N)
    out = torch.zeros((c["S"], len(cells), N), device="cuda", dtype=torch.float64)
    half = min(int(math.ceil(25.0 / dnu)) + 1, N)
    off = torch.arange(-half, half + 1, device="cuda")
    for s, (nu0, logs, elow, gam, mass) in enumerate(d["lines"]):
        step = max(1, int(2e7) // len(off))
        for a in range(0, len(nu0), step):
            v0, lg, el, ga = (t[a : a + step].double() for t in (nu0, logs, elow, gam))
            j = torch.round((v0 - NU0) / dnu).long()[:, None] + off
            dist = (NU0 + j.double() * dnu) - v0[:, None]
            keep = (dist.abs() <= 25.0) & (j >= 0) & (j < N)
            j = j.clamp(0, N - 1)
            for q, (p, t) in enumerate(cells):
                S = (10.0 ** lg * (TREF / t) ** 1.5 * torch.exp(-C2 * el * (1 / t - 1 / TREF)) *
                     (-torch.expm1(-C2 * v0 / t)) / (-torch.expm1(-C2 * v0 / TREF)))
                inv = 1.0 / (v0 / C * math.sqrt(2 * KB * t / (mass * AMU)))
                y = ga * p * math.sqrt(TREF / t) * inv
                v = _faddeeva_re(dist * inv[:, None], y[:, None].expand_as(dist))
                v = torch.where(keep, v * (S * inv / math.sqrt(math.pi))[:, None], 0.0)
                out[s, q].index_add_(0, j.reshape(-1), v.reshape(-1))
    return out.reshape(shape)


def _network(d, x, params=None):
    """Physical outputs, standardised outputs and the layers' weights of the network in 64 bits: BF16 weights in the
    products, gradients passed to the master weights as they are."""
    w, at = d["widths"], 0
    params = d["params"].double() if params is None else params
    ish, isc, osh, osc = (torch.tensor(v, device="cuda").double() for v in d["scaling"])
    h = (x.double() - ish) * isc
    for i, (a, b) in enumerate(zip(w[:-1], w[1:])):
        W = params[at : at + a * b].reshape(b, a)
        W = W + (W.detach().float().bfloat16().double() - W.detach())
        h = h @ W.T + params[at + a * b : at + a * b + b]
        at += a * b + b
        if i + 2 < len(w):
            h = torch.nn.functional.gelu(h)
    return 10.0 ** (h / osc + osh), h


def _training_exact(c, d):
    """The losses of all steps; the weights themselves follow Adam's signs and have no value beyond them."""
    p = d["params"].double()
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    osh, osc = (torch.tensor(q, device="cuda").double() for q in d["scaling"][2:])
    for k, lr in enumerate(d["lr"]):
        r = d["rows"][k].long()
        q = p.clone().requires_grad_()
        loss = ((_network(d, d["x"][r], q)[1] - (torch.log10(d["y"][r].double()) - osh) * osc) ** 2).mean()
        loss.backward()
        losses.append(loss.detach())
        m, v = 0.9 * m + 0.1 * q.grad, 0.999 * v + 0.001 * q.grad ** 2
        p = p - lr * (m / (1 - 0.9 ** (k + 1))) / (torch.sqrt(v / (1 - 0.999 ** (k + 1))) + 1e-8)
    return {"params": None, "loss": torch.stack(losses)}


def _statistics_exact(c, d):
    x = d["chain"].double()
    n, C_, q = x.shape
    e = x - x.mean(0)
    var = (e * e).mean(0)
    f = torch.fft.rfft(e, n=2 * n, dim=0)
    rho = torch.fft.irfft(f.abs() ** 2, n=2 * n, dim=0)[: n // 2] / (n * var)
    below = rho[1:] < 0.01
    first = torch.where(below.any(0), below.int().argmax(0), torch.tensor(n // 2 - 1, device="cuda"))
    take = torch.arange(n // 2 - 1, device="cuda")[:, None, None] < first
    speis = 1.0 + 2.0 * (rho[1:] * take).sum(0)
    W = (e * e).sum(0).div(n - 1).mean(0)
    B = n * x.mean(0).var(0)
    gr = torch.sqrt(((n - 1) / n * W + B / n) / W)
    return {"speis": speis, "gr": gr, "ess": (n * C_ / speis.mean(0).max()).reshape(())}


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "retrieval":
        return None
    if kind in ("emission", "contribution") and c["n"] * c["L"] * c["N"] * c["angles"] > 3e10:
        return None
    if kind == "transit" and c["n"] * c["level_hi"] * c["span_hi"] * (c["level_hi"] + 64) > 6e12:
        return None
    if kind == "opacity" and _evaluations(c) > 3e9:
        return None
    d = _inputs(c, seed)
    if kind == "emission":
        spec, bands = _emission_exact(c, d)
        if not c["spectra"]:
            return {"spectra": None, "bands": bands}
        if c["spans"]:
            spec = torch.cat([spec[i, int(a) : int(b)] for i, (a, b) in enumerate(zip(d["lo"], d["hi"]))])
        return {"spectra": spec, "bands": bands}
    if kind == "contribution":
        rows, bands = _emission_exact(c, d, contributions=True)
        return {"rows": rows if c["rows"] else None, "bands": bands}
    if kind == "transit":
        return _transit_exact(c, d)
    if kind == "opacity":
        return _opacity_exact(c, d)
    if kind == "surrogate":
        return _network(d, d["x"])[0]
    if kind == "training":
        return _training_exact(c, d)
    return _statistics_exact(c, d)
