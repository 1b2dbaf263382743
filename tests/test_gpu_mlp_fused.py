"""The fused network kernels at the edges of their tiles against the oracle:
batches around the row tiles (8, 16, 32 rows) and the 64-row blocks of the
weight gradients, more tiles than SMs, widths around 16, 64, 128 and 256 (the
K steps, K blocks, halves and the widest layer), one layer, and training on
gathered rows.  A width of 257 takes the layer-by-layer kernels."""
import numpy as np
import pytest

import workloads as W
from oracle import mlp as N
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


def _check(ctx, widths, B, most=None):
    import torch
    import paper_2104_12522_gb300 as bart
    rng = np.random.default_rng(B + sum(widths))
    p = W.mlp_init(widths, seed=B)
    p += (0.05 * rng.normal(size=p.size)).astype(np.float32) * (p == 0)     # biases
    ni, no = widths[0], widths[-1]
    sc = (rng.normal(size=ni).astype(np.float32), rng.uniform(0.5, 2.0, ni).astype(np.float32),
          rng.normal(size=no).astype(np.float32), rng.uniform(0.5, 2.0, no).astype(np.float32))
    x = rng.normal(size=(B, ni)).astype(np.float32)
    t = rng.normal(size=(B, no)).astype(np.float32)
    net = bart.Mlp(ctx, widths, log_outputs=False, max_batch=most or B)
    net.set_scaling(*sc)
    net.set_params(torch.tensor(p, device="cuda"))
    dx, dt = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
    y = net.forward(dx).cpu().numpy().astype(np.float64)
    g, loss = net.gradient(dx, dt)
    ctx.sync()
    pw = N.weights_bf16(p, widths)
    xs = (x.astype(np.float64) - sc[0]) * sc[1]
    ts = (t.astype(np.float64) - sc[2]) * sc[3]
    want, _ = N.forward(pw, widths, xs)
    lo, go = N.loss_and_grad(pw, widths, xs, ts)
    got = (y - sc[2]) * sc[3]
    # FP32 operands enter as BF16 hi + lo (2^-16 of each), FP32 accumulation,
    # at most four layers
    assert np.linalg.norm(got - want) < 1e-4 * np.linalg.norm(want)
    assert abs(float(loss.cpu()) - lo) < 2e-4 * lo
    g, at = g.cpu().numpy().astype(np.float64), 0
    for a, b in zip(widths[:-1], widths[1:]):
        for n in (a * b, b):
            assert np.linalg.norm(g[at:at + n] - go[at:at + n]) < 1e-3 * np.linalg.norm(go[at:at + n])
            at += n


@pytest.mark.parametrize("B", [1, 7, 8, 9, 33, 63, 64, 65, 1000, 1217, 2433, 5000])
def test_batches(ctx, B):
    _check(ctx, [9, 256, 256, 256, 10], B)


@pytest.mark.parametrize("widths", [[1, 1], [256, 256], [17, 3], [8, 64, 10], [9, 65, 129, 12], [16, 15, 128, 130, 5],
                                    [130, 250, 7, 256, 200], [9, 257, 10]])
def test_widths(ctx, widths):
    _check(ctx, widths, 77, most=200)


def test_gathered_rows_and_a_bad_index(ctx):
    """Rows of a larger table; an index outside it is row 0 and is reported."""
    import torch
    import paper_2104_12522_gb300 as bart
    widths = [9, 64, 256, 10]
    rng = np.random.default_rng(3)
    x = torch.tensor(rng.normal(size=(500, 9)).astype(np.float32), device="cuda")
    t = torch.tensor(rng.normal(size=(500, 10)).astype(np.float32), device="cuda")
    rows = torch.tensor(rng.integers(0, 500, (3, 100)).astype(np.int32), device="cuda")
    p = torch.tensor(W.mlp_init(widths), device="cuda")
    nets = [bart.Mlp(ctx, widths, log_outputs=False, max_batch=128) for _ in range(2)]
    for n in nets:
        n.set_params(p)
    nets[0].train_steps(x, t, rows, [1e-3] * 3)
    for k in range(3):
        r = rows[k].long()
        nets[1].train_step(x[r].contiguous(), t[r].contiguous(), 1e-3)
    ctx.sync()
    assert torch.equal(nets[0].get_params(), nets[1].get_params())
    for n in nets:
        n.set_params(p)
    bad = rows[:1].clone()
    bad[0, 5] = 500
    good = rows[:1].clone()
    good[0, 5] = 0
    nets[0].train_steps(x, t, bad, [1e-3])
    status = 0
    try:
        ctx.sync()
    except bart.BartError as err:
        status = err.status
    assert status == 5
    nets[1].train_steps(x, t, good, [1e-3])
    ctx.sync()
    assert torch.equal(nets[0].get_params(), nets[1].get_params())
