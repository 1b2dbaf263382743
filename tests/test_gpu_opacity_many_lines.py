"""However many lines a block holds, their sum keeps FP32 precision: a list with
every line 2,048 times over (a million lines in one block of points) gives 2,048
times the opacity of the list with each line once, to a few roundings, near the
block and far from it, about real and complex centres and line by line at the
cutoff."""
import numpy as np
import pytest

import workloads as W
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cutoff", [25.0, 3.0])
def test_repeated_lines(cutoff):
    import torch
    import paper_2104_12522_gb300 as bart
    ctx = make_ctx()
    N, dnu, K, n = 1000, 0.02, 2048, 512
    rng = np.random.default_rng(8)
    one = W.LineList(np.sort(1000.0 + dnu * rng.uniform(399.6, 407.4, n)), rng.uniform(-24.0, -20.0, n).astype(np.float32),
                     rng.uniform(0.0, 3000.0, n).astype(np.float32), rng.uniform(0.05, 0.1, n).astype(np.float32), 18.0)
    many = W.LineList(*[np.repeat(v, K) for v in (one.nu0, one.log10_s296, one.elow, one.gamma_ref)], 18.0)
    p = np.array([1e-6, 0.1, 1.5, 10.0, 60.0])
    t = np.array([1500.0, 900.0, 1500.0, 2000.0, 700.0])
    a, b = (ctx.opacity_cells([bart.device_lines(v)], p, t, bart.NuGrid(1000.0, dnu, N), cutoff)[0].double() for v in (one, many))
    ctx.sync()
    on = a > 1e-30 * a.max(dim=1, keepdim=True).values
    assert torch.equal(on, b > 1e-30 * b.max(dim=1, keepdim=True).values)
    for c in range(p.size):
        r = (b[c] / K / a[c] - 1.0)[on[c]].abs()
        print(f"cutoff {cutoff}, cell {c}: rms {r.pow(2).mean().sqrt():.1e}, max {r.max():.1e}")
        # the few tens of roundings of a chunk's and a point's plain FP32 sums, in the same direction at most
        assert r.max() < 32 * 2.0 ** -25
