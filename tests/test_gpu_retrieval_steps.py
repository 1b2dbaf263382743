"""A retrieval's half-steps against the same steps made one by one through the
sampler's public calls: chain counts that do not fill the last CTA, more bands
than a warp has lanes, with and without the screen, with and without an archive.
Decisions compare log-likelihoods with logarithms of 53-bit uniform numbers, so
the states must be the same; log-likelihoods of band values that agree to 1e-6
are compared to 1e-4."""
import numpy as np
import pytest

import workloads as W
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu

S, L, M, N, DNU, D = 2, 12, 3, 200, 0.05, 7


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


@pytest.mark.parametrize("C,nb,screened,archive", [(6, 1, True, False), (8, 10, False, False), (10, 32, True, True),
                                                   (14, 33, True, False), (5, 64, False, True), (130, 40, True, True)])
def test_retrieval_equals_its_steps(ctx, C, nb, screened, archive):
    import torch
    import paper_2104_12522_gb300 as bart
    rng = np.random.default_rng(7000 + C)
    dev = lambda a, dt=torch.float32: torch.tensor(a, device="cuda", dtype=dt)
    lo = np.concatenate([W.THETA_LO[:5], W.THETA_LO[5:5 + S]]).astype(np.float32)
    hi = np.concatenate([W.THETA_HI[:5], W.THETA_HI[5:5 + S]]).astype(np.float32)
    grid = dev(rng.uniform(1e-24, 1e-19, (S, L, M, N)))
    p, t, nu = W.log_pressures(L, 1e-6, 10.0), np.linspace(500.0, 3000.0, M), bart.NuGrid(1000.0, DNU, N)
    cfg = dict(geometry=0, n_angles=4, g=W.HD189_GRAV_CGS, mu=W.MEAN_MOLECULAR_MASS_AMU, x0=[W.BASE_VMR] * S,
               t_int=W.T_INT_K, t_star=W.HD189_TSTAR_K, r_star_tp=W.HD189_RSTAR_CM, a_orbit=W.HD189_A_CM,
               t_min=500.0, t_max=3000.0)
    filt = dev(W.gaussian_filters(W.nu_axis(1000.0, DNU, N), nb, 1000.5, 1009.0, 0.5, 3.0))
    x0 = dev(lo + rng.uniform(0.2, 0.8, (C, D)) * (hi - lo))

    def exact(th, active=None):
        out = torch.zeros((C, nb), device="cuda")
        ctx.forward_spectra_batch(grid, p, t, nu, cfg, theta=th, filters=filt, bands=out, active=active)
        return out

    b0 = exact(x0)
    data, sigma = b0[0].clone(), (0.5 * b0[0]).contiguous()
    net = None
    if screened:
        net = bart.Mlp(ctx, [D, 16, nb], bf16_weights=True, log_outputs=True, max_batch=C)
        net.set_scaling(0.5 * (lo + hi), 2.0 / (hi - lo), np.log10(b0[0].cpu().numpy()).astype(np.float32),
                        np.full(nb, 0.2, np.float32))
        net.set_params(dev(rng.normal(0.0, 0.2, D * 16 + 16 + 16 * nb + nb)))

    def loglike(bands, mask=None):
        out = torch.empty(C, dtype=torch.float64, device="cuda")
        return ctx.loglike_bands(bands, data, sigma, out, mask=mask)

    def sampler():
        s = bart.Demc(ctx, C, lo, hi, jump_every=3, eps=0.02, seed=7)
        s.set_screen(0.5, 0.5)
        s.set_state(x0.clone(), loglike(b0), loglike(net.forward(x0)) if screened else None)
        if archive:
            s.set_archive(dev(lo + np.random.default_rng(1).uniform(size=(20, D)) * (hi - lo)), 20 + 3 * C, thin=2,
                          p_snooker=0.3)
        return s

    n_gen = 5
    a, b = sampler(), sampler()
    st = ctx.retrieval_run(a, net, grid, p, t, nu, cfg, filt, data, sigma, n_gen, use_graph=True)
    y = torch.empty((C, D), device="cuda")
    inbox, passed, acc = (torch.empty(C, dtype=torch.int32, device="cuda") for _ in range(3))
    n_pass = n_in = n_acc = 0
    for h in range(2 * n_gen):
        b.propose(h, y, inbox)
        ls = loglike(net.forward(y), mask=inbox) if screened else None
        if screened:
            b.screen(h, inbox, ls, passed)
        else:
            passed.copy_(inbox)
        b.accept(h, y, passed, loglike(exact(y, passed), mask=passed), ls, acc)
        n_in, n_pass, n_acc = n_in + int(inbox.sum()), n_pass + int(passed.sum()), n_acc + int(acc.sum())
    get = lambda s: s.get_state(torch.empty_like(x0), *(torch.empty(C, dtype=torch.float64, device="cuda")
                                                        for _ in range(1 + screened)))
    ga, gb = get(a), get(b)
    ctx.sync()
    assert torch.equal(ga[0], gb[0]) and n_in > 0
    for u, v in zip(ga[1:1 + screened + 1], gb[1:1 + screened + 1]):
        if u is not None:
            assert torch.allclose(u, v, rtol=1e-4, atol=1e-4)
    assert (st["proposals"], st["exact_evals"], st["accepted"]) == (n_in, n_pass, n_acc)
    if archive:
        assert a.archive_size() == b.archive_size() > 20
