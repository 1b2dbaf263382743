"""A graph keeps its scratch: replays after calls of the same entry point that
need more of it (more bands, a longer cutoff) give what they gave before."""
import numpy as np
import pytest

import workloads as W
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu


def _replays(ctx, call, out, larger):
    import torch
    call()
    ctx.sync()
    want = out.clone()
    g = ctx.capture(call)
    for q in range(3):
        out.zero_()
        torch.cuda.synchronize()
        g.launch()
        ctx.sync()
        assert torch.equal(out, want)
        larger(q)


def test_contribution_bands_after_calls_with_more_bands():
    import torch
    import paper_2104_12522_gb300 as bart
    ctx = make_ctx()
    S, L, N = 2, 12, 700
    p, t = W.log_pressures(L, 1e-8, 100.0), np.linspace(500.0, 3000.0, 4)
    cfg = dict(geometry=0, n_angles=4, g=W.HD189_GRAV_CGS, mu=2.3, x0=[W.BASE_VMR] * S, t_int=W.T_INT_K,
               t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=500.0, t_max=3000.0)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    filt = lambda n: dev(W.gaussian_filters(W.nu_axis(1000.0, 0.02, N), n, 1000.0, 1014.0, 0.1, 2.0))
    grid, theta, nu = dev(W.opacity_field(S, p, t, N, seed=7)), dev(W.proposals(2, n_species=S)), bart.NuGrid(1000.0, 0.02, N)
    few, bands = filt(3), torch.zeros((2, L, 3), device="cuda")
    contrib = torch.zeros((2, L, N), device="cuda")
    call = lambda: ctx.contribution_functions(grid, p, t, nu, cfg, theta=theta, contrib=contrib, filters=few, bands=bands)

    def larger(q):
        n = 400 << q
        ctx.contribution_functions(grid, p, t, nu, cfg, theta=theta, contrib=torch.zeros_like(contrib), filters=filt(n),
                                   bands=torch.zeros((2, L, n), device="cuda"))
        ctx.sync()

    _replays(ctx, call, bands, larger)


def test_dense_opacity_after_calls_with_longer_cutoffs():
    import torch
    import paper_2104_12522_gb300 as bart
    ctx = make_ctx()
    lists = [bart.device_lines(W.line_list(0, 3000, 950.0, 1060.0))]
    p, t, nu = np.array([1e-4, 0.1]), np.array([1500.0, 900.0]), bart.NuGrid(1000.0, 0.02, 500)
    out, other = torch.zeros((1, 2, 500), device="cuda"), torch.zeros((1, 2, 500), device="cuda")

    def larger(q):
        ctx.opacity_cells(lists, p, t, nu, 25.0 * (q + 2), out=other)
        ctx.sync()

    _replays(ctx, lambda: ctx.opacity_cells(lists, p, t, nu, 5.0, out=out), out, larger)


def test_capture_after_an_eager_call_with_a_mask():
    """A masked call needs no check of the grid, the unmasked one of the same shape does: its capture needs no
    eager call of its own."""
    import torch
    import paper_2104_12522_gb300 as bart
    ctx = make_ctx()
    S, L, N, n = 2, 60, 1024, 1000
    p = W.log_pressures(L, 1e-8, 100.0)
    cfg = dict(geometry=0, n_angles=4, g=W.HD189_GRAV_CGS, mu=2.3, x0=[W.BASE_VMR] * S, t_int=W.T_INT_K,
               t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM, t_min=500.0, t_max=3000.0)
    grid = torch.tensor(W.opacity_field(S, p, np.array([500.0, 3000.0]), N, seed=9)[:, :, :1].copy(), device="cuda")
    theta = torch.tensor(W.proposals(n, n_species=S), device="cuda")
    spec, nu = torch.zeros((n, N), device="cuda"), bart.NuGrid(1000.0, 0.05, N)
    call = lambda **kw: ctx.forward_spectra_batch(grid, p, [1000.0], nu, cfg, theta=theta, spectra=spec, **kw)
    call(active=torch.ones(n, dtype=torch.int32, device="cuda"))
    ctx.sync()
    want = spec.clone()
    g = ctx.capture(call)
    spec.zero_()
    torch.cuda.synchronize()
    g.launch()
    ctx.sync()
    assert torch.equal(spec, want)
