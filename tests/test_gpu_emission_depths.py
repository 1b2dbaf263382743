"""Columns whose warps lie wholly in transparent, wholly in opaque levels (where
a column ends early) and across both, against the oracle in 64 bits.
Interiors hotter than the top by factors that let the flux come from optical
depths of twenty and more, inversions, odd and even grid lengths, lengths
around a thread's two and four wavenumbers and a tile, few and many rows."""
import numpy as np
import pytest

import workloads as W
from oracle import forward as Fw, radiation as R
from gpu_common import make_ctx, max_rel

pytestmark = pytest.mark.gpu

# FP32 against FP64: the Planck exponent c2 nu / T (up to 29) rounds to 2^-24
# of itself, as does an optical depth of up to 25 that the flux comes from,
# with as many roundings as it has terms in its running sum (60, random)
RTOL = (29 + 25 * 60 ** 0.5) * 2.0 ** -24 + 8 * 2.0 ** -22


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


def _case(N, scale, seed, profile):
    rng = np.random.default_rng(seed)
    L, S = 60, 2
    p = W.log_pressures(L, 1e-8, 100.0)
    # neighbouring wavenumbers up to four decades apart, so that a warp holds opaque and transparent ones
    sig = 10 ** (scale + rng.uniform(-2.0, 2.0, (S, 1, 1, N)) + rng.uniform(-0.3, 0.3, (S, L, 1, N)))
    sig = sig.astype(np.float32)
    x = np.linspace(0.0, 1.0, L)
    T = {"hot_interior": 500.0 + 2500.0 * x ** 4, "inversion": 2500.0 - 1800.0 * x}[profile]
    return p, sig, T.astype(np.float32)


@pytest.mark.parametrize("n_angles", [2, 4, 8, 16])
@pytest.mark.parametrize("N,nu0,profile", [(1, 10000.0, "hot_interior"), (5, 1000.0, "inversion"),
                                           (516, 10000.0, "hot_interior"), (1027, 1000.0, "hot_interior"),
                                           (1540, 2000.0, "inversion"), (259, 3000.0, "hot_interior")])
@pytest.mark.parametrize("scale", [-30.0, -24.0, -20.0, -15.0])
def test_depths(ctx, n_angles, N, nu0, profile, scale):
    import torch
    import paper_2104_12522_gb300 as bart
    p, sig, T = _case(N, scale, N + n_angles, profile)
    x0 = [1e-4, 3e-4]
    cfg = dict(geometry=0, n_angles=n_angles, g=W.HD189_GRAV_CGS, mu=2.3, x0=x0, t_min=1.0, t_max=1e5)
    # threads of four wavenumbers take calls that fill the SMs: as many rows as that needs, on spans that start
    # and end inside a thread's four
    n = 1 if N % 4 else -(-8 * 512 * 160 // N)
    lo = np.arange(n) % 7 if n > 1 else np.zeros(1, np.int64)
    hi = N - np.arange(n) % 5 if n > 1 else np.full(1, N)
    offs = np.concatenate([[0], np.cumsum(hi - lo)])
    dev = lambda v: torch.tensor(v.astype(np.int64), device="cuda")
    spec = torch.empty(int(offs[-1]), device="cuda")
    ctx.forward_spectra_batch(torch.tensor(sig, device="cuda"), p, [1000.0], bart.NuGrid(nu0, 0.05, N), cfg,
                              t_profile=torch.tensor(T, device="cuda")[None].repeat(n, 1).contiguous(),
                              nu_lo=dev(lo), nu_hi=dev(hi), spec_offsets=dev(offs), spectra=spec, n=n)
    ctx.sync()
    spec = spec.cpu().numpy()
    chi = Fw.mass_opacity(sig[:, :, 0].astype(np.float64), np.asarray(x0), 2.3)
    F = R.emission_flux(chi, p, T.astype(np.float64), W.nu_axis(nu0, 0.05, N), W.HD189_GRAV_CGS, n_angles)
    e = max(max_rel(spec[offs[i]:offs[i + 1]], F[lo[i]:hi[i]]) for i in range(n))
    print(f"{n_angles} angles, {n} x {N} wavenumbers, 1e{scale:.0f}: {e:.2e}")
    assert e < RTOL
