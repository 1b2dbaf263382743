"""Contribution functions and their band means at the kernels' edges against
the oracle: odd row lengths, spans that start on odd indices or hold one
point, one to four species, the optical-depth limit (each wavenumber of a pair
stopping on its own), filters that are empty or touch one point, layer counts
that leave a remainder of the band means' row groups, and a term that is not
finite outside a filter."""
import numpy as np
import pytest

import workloads as W
from oracle import forward as Fw, radiation as R
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


def _case(S, L, N, seed):
    p, t = W.log_pressures(L, 1e-8, 100.0), np.linspace(500.0, 3000.0, 6)
    cfg = dict(geometry=0, n_angles=4, g=W.HD189_GRAV_CGS, mu=2.3, x0=[W.BASE_VMR] * S, t_int=W.T_INT_K,
               t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=500.0, t_max=3000.0)
    filt = W.gaussian_filters(W.nu_axis(1000.0, 0.02, N), 4, 1000.0, 1000.0 + 0.02 * N, 0.1, 2.0, seed=seed)
    filt[2] = 0.0                               # empty
    filt[3] = 0.0
    filt[3, N // 2] = 0.7                       # one point
    return p, t, cfg, filt, W.opacity_field(S, p, t, N, seed=seed)


@pytest.mark.parametrize("S,L,N,tau_max", [(1, 2, 257, 0.0), (2, 9, 512, 0.0), (3, 16, 1001, 5.0), (4, 17, 766, 0.5)])
def test_contributions_at_edges(ctx, S, L, N, tau_max):
    import torch
    import paper_2104_12522_gb300 as bart
    p, t, cfg, filt, grid = _case(S, L, N, 41 + S)
    cfg["tau_max"] = tau_max
    n = 4
    theta = W.proposals(n, generation=S, n_species=S)
    lo = np.array([0, 1, 3, N - 1], np.int64)
    hi = np.array([N, N, N - 2, N], np.int64)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    rows = torch.full((n, L, N), -1.0, device="cuda")
    bands = torch.full((n, L, 4), -1.0, device="cuda")
    only = torch.full((n, L, 4), -1.0, device="cuda")
    nu = bart.NuGrid(1000.0, 0.02, N)
    args = (dev(grid), p, t, nu, cfg)
    ctx.contribution_functions(*args, theta=dev(theta), nu_lo=dev(lo), nu_hi=dev(hi), contrib=rows,
                               filters=dev(filt), bands=bands)
    ctx.contribution_functions(*args, theta=dev(theta), nu_lo=dev(lo), nu_hi=dev(hi), filters=dev(filt), bands=only)
    ctx.sync()
    assert torch.equal(bands, only)
    rows, bands = rows.cpu().numpy(), bands.cpu().numpy()
    ocfg = dict(cfg, tau_max=tau_max if tau_max > 0 else None)
    axis = W.nu_axis(1000.0, 0.02, N)
    for i in range(n):
        C = Fw.emission_contributions(grid[..., lo[i]:hi[i]].astype(np.float64), p, t, axis[lo[i]:hi[i]], theta[i],
                                      ocfg)
        got = rows[i][:, lo[i]:hi[i]]
        assert np.all(rows[i][:, :lo[i]] == -1.0) and np.all(rows[i][:, hi[i]:] == -1.0)
        if tau_max > 0:
            # FP32 and FP64 may pass the limit a level apart where a level's tau is within rounding of it
            T = Fw.tp_of(theta[i], p, ocfg)
            sub = grid[..., lo[i]:hi[i]].astype(np.float64)
            chi = Fw.mass_opacity(Fw.layer_opacity(sub, t, T), W.BASE_VMR * 10.0 ** theta[i, 5:5 + S], 2.3)
            tau = R.optical_depth(chi.T, p, cfg["g"])
            clear = np.all(np.abs(tau / tau_max - 1.0) > 1e-5, axis=1)
            assert clear.mean() > 0.9
            got, C = got[:, clear], C[:, clear]
        assert np.max(np.abs(got - C) / C.sum(axis=0)) < 1e-5
        # the band means of the rows the call itself returned: FP32 of a sum with 48 bits
        Bo = np.array([R.band_integrate(rows[i][k, lo[i]:hi[i]].astype(np.float64), filt, nu_lo=int(lo[i]))
                       for k in range(L)])
        assert np.allclose(bands[i], Bo, rtol=2.0 ** -23, atol=0.0)


def test_a_term_that_is_not_finite_reaches_every_band(ctx):
    import torch
    import paper_2104_12522_gb300 as bart
    S, L, N = 2, 9, 600
    p, t, cfg, filt, grid = _case(S, L, N, 77)
    grid[0, 4, :, 5] = np.nan                   # wavenumber 5 lies outside filter 3
    assert filt[3, 5] == 0.0
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    bands = torch.zeros((1, L, 4), device="cuda")
    ctx.contribution_functions(dev(grid), p, t, bart.NuGrid(1000.0, 0.02, N), cfg,
                               theta=dev(W.proposals(1, n_species=S)), filters=dev(filt), bands=bands)
    ctx.sync()
    b = bands.cpu().numpy()[0]
    assert np.all(np.isfinite(b[:3])) and np.all(np.isnan(b[4:, [0, 1, 3]])) and np.all(b[:, 2] == 0.0)
