"""Columns that end early give the bits of those that take every layer, and only
where every opacity is finite and not negative: a NaN, an infinity or a negative
value below opaque levels does to a large call's spectra, and to a retrieval's
likelihoods, what it does to a single spectrum."""
import numpy as np
import pytest

import workloads as W
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu

S, L, N = 2, 60, 1024
P_BAR = W.log_pressures(L, 1e-8, 100.0)


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


def _field(scale, seed):
    rng = np.random.default_rng(seed)
    lg = scale + rng.uniform(-2.0, 2.0, (S, 1, 1, N)) + rng.uniform(-0.3, 0.3, (S, L, 1, N))
    return (10 ** lg).astype(np.float32)


def _cfg(**kw):
    return dict(dict(geometry=0, n_angles=4, g=W.HD189_GRAV_CGS, mu=2.3, x0=[1e-4, 3e-4], t_int=W.T_INT_K,
                     t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=1.0, t_max=1e5), **kw)


def _spectra(ctx, field, cfg, n):
    import torch
    import paper_2104_12522_gb300 as bart
    T = 500.0 + 2500.0 * np.linspace(0.0, 1.0, L) ** 4
    prof = torch.tensor(np.stack([T, T[::-1]]).astype(np.float32), device="cuda").repeat((n + 1) // 2, 1)[:n].contiguous()
    spec = torch.empty((n, N), device="cuda")
    ctx.forward_spectra_batch(torch.tensor(field, device="cuda"), P_BAR, [1000.0], bart.NuGrid(3000.0, 0.5, N), cfg,
                              t_profile=prof, spectra=spec, n=n)
    ctx.sync()
    return spec.cpu().numpy()


@pytest.mark.parametrize("tau_max", [0.0, 5.0])
@pytest.mark.parametrize("scale", [-24.0, -19.0, -15.0])
@pytest.mark.parametrize("value", [None, np.nan, np.inf, -np.inf, -1e-20])
def test_large_calls_match_single_spectra(ctx, value, scale, tau_max):
    field = _field(scale, 3)
    if value is not None:
        field[1, 55, 0, 100] = value
        field[0, 30, 0, 517] = value
    cfg = _cfg(tau_max=tau_max)
    large = _spectra(ctx, field, cfg, 1000)      # enough for threads of four wavenumbers, and for the check to pay
    assert any(" x4 ends" in k for k in ctx.autotune_report())
    few = _spectra(ctx, field, cfg, 2)
    want = np.tile(few, (-(-len(large) // 2), 1))[:len(large)]
    assert np.array_equal(large, want, equal_nan=True)
    if value is not None and np.isnan(value) and tau_max == 0.0:
        assert np.isnan(large[:, [100, 517]]).all() and np.isfinite(np.delete(large, [100, 517], 1)).all()


def test_retrieval_sees_a_nan_below_opaque_levels(ctx):
    import torch
    import paper_2104_12522_gb300 as bart
    C, nb = -(-8 * 512 * 160 // N), 3
    field = _field(-15.0, 4)
    cfg = _cfg(t_min=500.0, t_max=3000.0, n_angles=8)
    nu = bart.NuGrid(3000.0, 0.5, N)
    filt = torch.full((nb, N), 1.0, device="cuda")
    lo, hi = np.array(W.THETA_LO[:5 + S], np.float32), np.array(W.THETA_HI[:5 + S], np.float32)
    x = torch.tensor(W.proposals(C, n_species=S), device="cuda")
    accepted = []
    for value in (None, np.nan):
        if value is not None:
            field[0, 55, 0, 700] = value
        s = bart.Demc(ctx, C, lo, hi)
        s.set_state(x, torch.full((C,), -1e30, dtype=torch.float64, device="cuda"))
        got = ctx.retrieval_run(s, None, torch.tensor(field, device="cuda"), P_BAR, [1000.0], nu, cfg, filt,
                                torch.full((nb,), 1e4, device="cuda"), torch.full((nb,), 1e3, device="cuda"), 2)
        assert got["exact_evals"] > 0
        accepted.append(got["accepted"])
    assert accepted[0] > 0 and accepted[1] == 0
