"""Chain statistics at the edges of the kernels' tiles against the oracle:
fewer rows than a warp, chunk and tile remainders, series counts that are not
a multiple of 32, more lag chunks than slots, no crossing of the threshold, a
series that never moved, and a chain captured without an eager call before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from tests.gpu_common import make_ctx
    return make_ctx()


def _chain(n, C, d, phi, seed):
    rng = np.random.default_rng(seed)
    x = np.zeros((n, C, d))
    x[0] = rng.normal(size=(C, d))
    for t in range(1, n):
        x[t] = phi * x[t - 1] + rng.normal(size=(C, d))
    return (x + 3.0).astype(np.float32)


@pytest.mark.parametrize("n,C,d,phi,threshold", [
    (4, 2, 1, 0.0, 0.01), (5, 3, 2, 0.5, 0.01), (31, 2, 17, 0.9, 0.01), (64, 33, 1, 0.5, 0.01),
    (65, 3, 11, 0.9, -2.0), (1000, 2, 1, 0.99, 0.01), (4097, 5, 7, 0.98, 0.01), (4160, 40, 9, 0.3, 0.05)])
def test_chain_stats_at_tile_edges(ctx, n, C, d, phi, threshold):
    import torch
    from oracle import demc as D
    x = _chain(n, C, d, phi, n + C)
    if d > 1:
        x[:, 0, 1] = 2.5                      # never moved: SPEIS 1
    sp, gr, _ = ctx.chain_stats(torch.tensor(x, device="cuda"), threshold=threshold)
    ctx.sync()
    ref = np.array([[D.speis(x[:, c, q].astype(np.float64), threshold) for q in range(d)] for c in range(C)])
    # FP64 sums of at most n terms per lag and n/2 lags, against a bound of 1
    assert np.allclose(sp.cpu().numpy(), ref, rtol=1e-11, atol=1e-11)
    assert np.allclose(gr.cpu().numpy(), D.gelman_rubin(x.astype(np.float64)), rtol=1e-11)


def test_chain_stats_in_a_capture_of_its_own():
    """The first call of a context may be a captured one: the graph brings its own scratch."""
    import torch
    from tests.gpu_common import make_ctx
    x = torch.tensor(_chain(700, 4, 3, 0.9, 1), device="cuda")
    c = make_ctx()
    sp = torch.zeros((4, 3), dtype=torch.float64, device="cuda")
    gr = torch.zeros(3, dtype=torch.float64, device="cuda")
    g = c.capture(lambda: c._check(c.lib.bart_chain_stats(c.h, x.data_ptr(), 700, 4, 3, 0.01, sp.data_ptr(),
                                                          gr.data_ptr())))
    for _ in range(2):
        sp.zero_()
        gr.zero_()
        g.launch()
        c.sync()
        want, wgr, _ = c.chain_stats(x)
        assert torch.equal(sp, want) and torch.equal(gr, wgr)
