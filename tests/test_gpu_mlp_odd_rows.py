"""Networks too wide for the fused kernels whose buffers start off 16-byte
boundaries: an odd number of rows behind an odd number of inputs, and weights
behind odd widths.  The same network with room for an even number of rows has
aligned activations and runs the same sums, so the results are the same."""
import numpy as np
import pytest

from gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


@pytest.mark.parametrize("widths,B", [([9, 320, 10], 33), ([9, 301, 304, 7], 65), ([7, 288, 288, 5], 1)])
def test_rows_off_16_byte_boundaries(ctx, widths, B):
    import torch
    import paper_2104_12522_gb300 as bart
    g = torch.Generator(device="cuda").manual_seed(3)
    n = sum(a * b + b for a, b in zip(widths, widths[1:]))
    p = 0.05 * torch.randn(n, device="cuda", generator=g)
    x = torch.randn((B, widths[0]), device="cuda", generator=g)
    t = torch.rand((B, widths[-1]), device="cuda", generator=g) + 0.5
    out = []
    for room in (B, (B + 3) // 4 * 4):
        net = bart.Mlp(ctx, widths, bf16_weights=True, log_outputs=True, max_batch=room)
        net.set_params(p)
        y = net.forward(x).clone()
        for _ in range(2):
            net.train_step(x, t, 1e-3)
        ctx.sync()
        out.append((y, net.get_params().clone()))
    assert np.isfinite(out[0][0].cpu().numpy()).all()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
