"""Chain statistics depend on the caller's arrays alone: a captured graph stays
good after calls with longer chains, calls on two streams of one context do not
meet, and a context keeps little memory behind a call."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _chain(n, C, d, seed):
    rng = np.random.default_rng(seed)
    x = np.cumsum(rng.normal(size=(n, C, d)), axis=0)
    return (x - 0.98 * np.concatenate([np.zeros((1, C, d)), x[:-1]])).astype(np.float32)


def _outputs(torch, C, d):
    return torch.zeros((C, d), dtype=torch.float64, device="cuda"), torch.zeros(d, dtype=torch.float64, device="cuda")


def _call(ctx, x, sp, gr):
    n, C, d = x.shape
    ctx._check(ctx.lib.bart_chain_stats(ctx.h, x.data_ptr(), n, C, d, 0.01, sp.data_ptr(), gr.data_ptr()))


def test_graph_after_calls_with_longer_chains():
    import torch
    from tests.gpu_common import make_ctx
    ctx = make_ctx()
    x = torch.tensor(_chain(600, 4, 3, 1), device="cuda")
    sp, gr = _outputs(torch, 4, 3)
    _call(ctx, x, sp, gr)
    ctx.sync()
    want = sp.clone(), gr.clone()
    g = ctx.capture(lambda: _call(ctx, x, sp, gr))
    for n, C in ((5000, 9), (20_000, 33)):
        y = torch.tensor(_chain(n, C, 3, n), device="cuda")
        ctx.chain_stats(y)
        sp.zero_()
        gr.zero_()
        g.launch()
        ctx.sync()
        assert torch.equal(sp, want[0]) and torch.equal(gr, want[1])


def test_two_streams_of_a_context():
    import torch
    from tests.gpu_common import make_ctx
    ctx = make_ctx()
    xs = [torch.tensor(_chain(n, 8, 5, n), device="cuda") for n in (15_000, 9_000)]
    outs = [_outputs(torch, 8, 5) for _ in xs]
    want = []
    for x, o in zip(xs, outs):
        _call(ctx, x, *o)
        ctx.sync()
        want.append([v.clone() for v in o])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in xs]
    for _ in range(5):
        for o in outs:
            for v in o:
                v.zero_()
        torch.cuda.synchronize()
        for _ in range(3):
            for s, x, o in zip(streams, xs, outs):
                ctx._check(ctx.lib.bart_set_stream(ctx.h, s.cuda_stream))
                _call(ctx, x, *o)
        torch.cuda.synchronize()
        for o, w in zip(outs, want):
            assert all(torch.equal(a, b) for a, b in zip(o, w))
    ctx._check(ctx.lib.bart_set_stream(ctx.h, None))


def test_memory_kept_behind_a_call():
    import torch
    from tests.gpu_common import make_ctx
    ctx = make_ctx()
    sp, gr = _outputs(torch, 32, 40)
    x = torch.randn((40_000, 32, 40), device="cuda")      # 1,280 series of 480 kB: more than one batch of 512 MB
    _call(ctx, x[:64].contiguous(), sp, gr)               # loads the kernels
    ctx.sync()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    _call(ctx, x, sp, gr)
    ctx.sync()
    torch.cuda.synchronize()
    kept = before - torch.cuda.mem_get_info()[0]
    print(f"kept: {kept / 2 ** 20:.0f} MB")
    assert kept <= 96 << 20
