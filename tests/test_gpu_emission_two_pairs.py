"""Calls large enough for threads of four wavenumbers against the oracle, with the
options whose other tests are small: the optical-depth limit (neighbouring
wavenumbers stop at different levels), a cloud deck, Rayleigh scattering, spans
that start and end inside a thread's four, inactive entries, an invalid span, one
to four species, bands with and without spectra, and a captured graph."""
import numpy as np
import pytest

import workloads as W
from oracle import forward as Fw, radiation as R
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu

RTOL = 1e-4          # the spectra/band tolerance of the other forward-model tests
L, M, N, NB, DISTINCT = 45, 4, 1200, 5, 5
COUNT = -(-8 * 512 * 160 // N)


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


@pytest.mark.parametrize("S,angles,nu0,opts,spans,mask", [
    (1, 4, 1000.0, dict(tau_max=2.0), False, False), (2, 8, 1000.0, dict(tau_max=20.0), True, False),
    (3, 8, 1000.0, dict(p_cloud=0.7), False, False), (4, 4, 20_000.0, dict(rayleigh_coef=8.4e-45), False, False),
    (4, 8, 1000.0, dict(p_cloud=1e-3, tau_max=1.0), True, True), (2, 16, 9000.0, dict(rayleigh_coef=8.4e-45, tau_max=5.0), False, True),
    (4, 8, 1000.0, {}, False, False), (1, 1, 9000.0, {}, True, True)])
def test_against_the_oracle(ctx, S, angles, nu0, opts, spans, mask):
    import torch
    import paper_2104_12522_gb300 as bart
    p, t, dnu = W.log_pressures(L, 1e-8, 100.0), np.linspace(500.0, 3000.0, M), 0.05
    field = W.opacity_field(S, p, t, N, seed=50 + S)
    theta = W.proposals(DISTINCT, generation=S, n_species=S)
    rng = np.random.default_rng(S)
    which = np.arange(COUNT) % DISTINCT
    lo = (rng.integers(0, 40, DISTINCT) if spans else np.zeros(DISTINCT, int))[which].astype(np.int64)
    hi = N - (rng.integers(0, 40, DISTINCT) if spans else np.zeros(DISTINCT, int))[which].astype(np.int64)
    if spans:
        lo[:3], hi[:3] = [401, 402, 403], [402, 407, 409]       # within one thread's four, over two, over three
    offs = np.concatenate([[0], np.cumsum(hi - lo)]).astype(np.int64)
    bad = np.zeros(COUNT, bool)
    if spans:
        bad[6] = True
        lo_call, hi_call = lo.copy(), hi.copy()
        hi_call[6] = N + 1
    active = np.ones(COUNT, np.int32)
    if mask:
        active[3::4] = 0
    filt = W.gaussian_filters(W.nu_axis(nu0, dnu, N), NB, nu0 + 5.0, nu0 + 50.0, 2.0, 15.0)
    cfg = dict(geometry=0, n_angles=angles, g=W.HD189_GRAV_CGS, mu=W.MEAN_MOLECULAR_MASS_AMU, x0=[W.BASE_VMR] * S,
               t_int=W.T_INT_K, t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=500.0,
               t_max=3000.0, **opts)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    grid, th, fl, nu = dev(field), dev(theta[which]), dev(filt), bart.NuGrid(nu0, dnu, N)
    kw = dict(nu_lo=dev(lo_call), nu_hi=dev(hi_call), spec_offsets=dev(offs)) if spans else {}
    if mask:
        kw["active"] = dev(active)
    spec = torch.full((int(offs[-1]),), -1.0, device="cuda")
    bands, only = torch.full((COUNT, NB), -1.0, device="cuda"), torch.full((COUNT, NB), -1.0, device="cuda")

    def call(s, b):
        ctx.forward_spectra_batch(grid, p, t, nu, cfg, theta=th, spectra=s, filters=fl, bands=b, n=COUNT, **kw)

    def sync():
        if bad.any():
            with pytest.raises(Exception):        # the invalid span is reported
                ctx.sync()
        else:
            ctx.sync()

    call(spec, bands)
    sync()
    call(None, only)
    sync()
    assert any(" x4" in k for k in ctx.autotune_report())
    assert torch.equal(bands, only)
    graph = ctx.capture(lambda: call(spec, bands))
    first = spec.clone(), bands.clone()
    spec.fill_(-1.0)
    bands.fill_(-1.0)
    graph.launch()
    sync()
    assert torch.equal(spec, first[0]) and torch.equal(bands, first[1])
    spec, bands = spec.cpu().numpy(), bands.cpu().numpy()
    axis = W.nu_axis(nu0, dnu, N)
    ocfg = dict(cfg, tau_max=opts.get("tau_max"))
    full = [Fw.emission_spectrum(field.astype(np.float64), p, t, axis, theta[i], ocfg) for i in range(DISTINCT)]
    es = eb = 0.0
    for i in range(COUNT):
        got = spec[offs[i]:offs[i + 1]]
        if not active[i]:
            assert np.all(got == -1.0) and np.all(bands[i] == -1.0)
            continue
        if bad[i]:
            assert np.all(got == -1.0) and np.all(bands[i] == 0.0)
            continue
        F = full[which[i]][lo[i]:hi[i]]
        es = max(es, float(np.max(np.abs(got - F) / F)))
        bo = R.band_integrate(F, filt, int(lo[i]))
        assert np.all(bands[i][bo == 0] == 0)
        if np.any(bo > 0):
            eb = max(eb, float(np.max(np.abs(bands[i][bo > 0] - bo[bo > 0]) / bo[bo > 0])))
    print(f"S {S}, {angles} angles, {opts}: spectra {es:.2e}, bands {eb:.2e}")
    assert es < RTOL and eb < RTOL
