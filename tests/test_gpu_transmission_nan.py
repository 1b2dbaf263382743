"""A NaN above opaque shells reaches a transit spectrum at its wavenumber, though
the shells above an opaque ray block are not summed: every shell is among the
lowest of some block.  No other wavenumber changes."""
import numpy as np
import pytest

import workloads as W
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,N", [(1, 259), (4, 300)])
def test_nan_above_opaque_shells(S, N):
    import torch
    import paper_2104_12522_gb300 as bart
    ctx = make_ctx()
    Lg, n = 60, 5
    p = W.log_pressures(Lg, 1e-8, 100.0)
    rng = np.random.default_rng(S)
    field = (10 ** rng.uniform(-17.0, -15.0, (S, Lg, 1, N))).astype(np.float32)
    inst = W.instances(n, N, lmin=30, lmax=150, span_lo=N, span_hi=N, seed=31)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    cfg = dict(geometry=1, g=W.HD189_GRAV_CGS, mu=W.MEAN_MOLECULAR_MASS_AMU, x0=[W.BASE_VMR] * S, t_int=W.T_INT_K,
               t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=500.0, t_max=3000.0,
               p_ref=W.HD189_PREF_BAR, p_top=1e-8, p_bot=100.0)
    filt = torch.ones((1, N), device="cuda")
    got = []
    at = [0, 77, N - 1]
    for bad in (False, True):
        if bad:
            field[S - 1, 12, 0, at] = np.nan
        spec, bands = torch.empty((n, N), device="cuda"), torch.empty((n, 1), device="cuda")
        ctx.forward_spectra_batch(dev(field), p, [1000.0], bart.NuGrid(1000.0, 0.05, N), cfg, theta=dev(inst.theta[:, :5 + S]),
                                  n_levels=dev(inst.n_levels), r_planet=dev(inst.r_planet), r_star=dev(inst.r_star),
                                  spectra=spec, filters=filt, bands=bands)
        ctx.sync()
        got.append((spec.cpu().numpy(), bands.cpu().numpy()))
    (clean, cb), (spec, bands) = got
    assert np.isfinite(clean).all() and np.isfinite(cb).all()
    assert np.isnan(spec[:, at]).all() and np.isnan(bands).all()
    assert np.array_equal(np.delete(spec, at, 1), np.delete(clean, at, 1))
