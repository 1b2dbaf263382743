"""Transit spectra where whole ray blocks are opaque over a warp (their outer
shells are not summed), transparent, and mixed, and where neighbouring levels
share all, two or none of their grid corners, against the oracle in 64 bits:
fewer and more levels than grid layers, level counts around the ray blocks of
4, the blocks' first 8 shells and the eighths, two grid layers, one temperature."""
import dataclasses

import numpy as np
import pytest

import workloads as W
from oracle import forward as Fw
from gpu_common import make_ctx, max_rel

pytestmark = pytest.mark.gpu

# every rounding of a sum over up to 192 shells and of a level's 40 operations at its worst
RTOL = (192 + 40) * 2.0 ** -24


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


@pytest.mark.parametrize("scale", [-10.0, 0.0, 3.0, 9.0])
@pytest.mark.parametrize("S,Lg,M,N", [(1, 30, 6, 259), (4, 60, 20, 128), (2, 8, 1, 131), (3, 2, 5, 64)])
def test_depths(ctx, S, Lg, M, N, scale):
    import torch
    import paper_2104_12522_gb300 as bart
    dnu = 0.05
    p = W.log_pressures(Lg, 1e-8, 100.0)
    t = np.linspace(500.0, 3000.0, M) if M > 1 else np.array([1000.0])
    rng = np.random.default_rng(Lg * 100 + M)
    field = W.opacity_field(S, p, np.linspace(500.0, 3000.0, max(M, 2)), N,
                            seed=3900 + S)[:, :, :M]
    field = (field.astype(np.float64) * 10 ** (scale + rng.uniform(-1.5, 1.5, (S, 1, 1, N)))).clip(1e-36, 1e-5)
    field = np.ascontiguousarray(field.astype(np.float32))
    levels = [2, 3, 5, 6, 9, 10, 12, 13, 17, 33, 40, 63, 97, 129, 191, 192]
    n = len(levels)
    inst = W.instances(n, N, lmin=2, lmax=192, span_lo=1, span_hi=N, seed=4200 + S)
    inst = dataclasses.replace(inst, theta=np.ascontiguousarray(inst.theta[:, :5 + S]))
    inst.n_levels[:] = levels
    inst.nu_lo[3:], inst.nu_hi[3:] = 0, N
    offs = np.concatenate([[0], np.cumsum(inst.nu_hi - inst.nu_lo)]).astype(np.int64)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    cfg = dict(geometry=1, g=W.HD189_GRAV_CGS, mu=W.MEAN_MOLECULAR_MASS_AMU, x0=[W.BASE_VMR] * S, t_int=W.T_INT_K,
               t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=500.0, t_max=3000.0,
               p_ref=W.HD189_PREF_BAR, p_top=1e-8, p_bot=100.0)
    spec = torch.empty(int(offs[-1]), dtype=torch.float32, device="cuda")
    ctx.forward_spectra_batch(dev(field), p, t, bart.NuGrid(1000.0, dnu, N), cfg, theta=dev(inst.theta),
                              n_levels=dev(inst.n_levels), nu_lo=dev(inst.nu_lo), nu_hi=dev(inst.nu_hi),
                              spec_offsets=dev(offs), r_planet=dev(inst.r_planet), r_star=dev(inst.r_star),
                              spectra=spec)
    ctx.sync()
    spec = spec.cpu().numpy()
    ocfg = {k: cfg[k] for k in ("g", "t_int", "t_star", "r_star_tp", "a_orbit", "t_min", "t_max", "x0", "mu", "p_ref",
                                "p_top", "p_bot")}
    e = 0.0
    for i in range(n):
        ref = Fw.transmission_spectrum(field.astype(np.float64), p, t, 1000.0, dnu, inst, i, ocfg)
        e = max(e, max_rel(spec[offs[i]:offs[i + 1]], ref))
    print(f"S {S}, grid {Lg} x {M} x {N}, x 1e{scale:.0f}: {e:.2e}")
    assert e < RTOL
