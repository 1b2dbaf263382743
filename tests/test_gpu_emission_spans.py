"""What a grid holds outside an entry's span does not reach its bands, in calls
large enough for threads of four wavenumbers, with spans that start and end at
every place of a thread's four."""
import numpy as np
import pytest

import workloads as W
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_values_outside_a_span(bad):
    import torch
    import paper_2104_12522_gb300 as bart
    ctx = make_ctx()
    S, L, N, nb = 2, 12, 1024, 3
    p, t = W.log_pressures(L, 1e-8, 100.0), np.linspace(500.0, 3000.0, 3)
    cfg = dict(geometry=0, n_angles=4, g=W.HD189_GRAV_CGS, mu=2.3, x0=[W.BASE_VMR] * S, t_int=W.T_INT_K,
               t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=500.0, t_max=3000.0)
    nu, n = bart.NuGrid(1000.0, 0.02, N), -(-8 * 512 * 160 // N)
    field = W.opacity_field(S, p, t, N, seed=21)
    filt = torch.full((nb, N), 0.5, device="cuda")
    theta = torch.tensor(np.tile(W.proposals(4, n_species=S), (-(-n // 4), 1))[:n], device="cuda")
    # spans inside [400, 500), their ends up to a thread's four apart; nothing finite outside [lo, hi) of all of them
    got = []
    for lo0, hi0 in ((401, 502), (402, 501), (403, 503), (404, 500)):
        lo, hi = np.full(n, lo0), np.full(n, hi0)
        for fill in (None, bad):
            grid = field.copy()
            if fill is not None:
                grid[..., :lo0] = fill
                grid[..., hi0:] = fill
            bands = torch.full((n, nb), -1.0, device="cuda")
            spec = torch.full((n, hi0 - lo0), -1.0, device="cuda")
            dev = lambda v: torch.tensor(np.asarray(v, np.int64), device="cuda")
            ctx.forward_spectra_batch(torch.tensor(grid, device="cuda"), p, t, nu, cfg, theta=theta, nu_lo=dev(lo),
                                      nu_hi=dev(hi), spec_offsets=dev(np.arange(n + 1) * (hi0 - lo0)), spectra=spec,
                                      filters=filt, bands=bands)
            ctx.sync()
            got.append((spec, bands))
        assert torch.equal(got[-1][0], got[-2][0]) and torch.equal(got[-1][1], got[-2][1])
        assert torch.isfinite(got[-1][1]).all() and (got[-1][1] > 0).all()


def test_band_sums_of_wide_calls():
    """Band values against FP64 means of the same call's spectra: 16,384
    wavenumbers in 2 units or more of 8 tiles, sums in FP64 between tiles.
    With r = 2^-24 / sqrt 3 for one rounding (rms, at most), a tile's tree of
    sums rounds by sqrt(1 + 1/2 + 1/4 + ...) r, averaged over 16 tiles and more; a
    unit's sum once, averaged over the units; numerator and denominator alike;
    and the value once."""
    import torch
    import paper_2104_12522_gb300 as bart
    ctx = make_ctx()
    S, L, N, n, nb = 1, 6, 16_384, 1300, 8
    p, t = W.log_pressures(L, 1e-8, 100.0), np.linspace(500.0, 3000.0, 2)
    cfg = dict(geometry=0, n_angles=4, g=W.HD189_GRAV_CGS, mu=2.3, x0=[W.BASE_VMR] * S, t_int=W.T_INT_K,
               t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=500.0, t_max=3000.0)
    grid = torch.tensor(W.opacity_field(S, p, t, N, seed=22), device="cuda")
    theta = torch.tensor(W.proposals(n, n_species=S), device="cuda")
    filt = 0.5 + torch.rand((nb, N), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    spec, bands = torch.empty((n, N), device="cuda"), torch.empty((n, nb), device="cuda")
    ctx.forward_spectra_batch(grid, p, t, bart.NuGrid(1000.0, 0.02, N), cfg, theta=theta, spectra=spec, filters=filt,
                              bands=bands)
    ctx.sync()
    assert any(" x4" in k for k in ctx.autotune_report())
    w = filt.double()
    w[:, 0] *= 0.5
    w[:, -1] *= 0.5
    want = (spec.double() @ w.T) / w.sum(1)
    e = (bands.double() / want - 1.0).pow(2).mean().sqrt().item()
    print(f"band sums: {e:.2e}")
    assert e < (2.0 * (2.0 / 16.0 + 1.0 / 2.0) + 1.0) ** 0.5 * 2.0 ** -24 / 3.0 ** 0.5
