"""Band means of contribution rows whose terms, times the weights, are near or
below the smallest FP32 numbers, or above the largest in a sum, against FP64
means of the same rows: one rounding of the value."""
import numpy as np
import pytest

import workloads as W
from gpu_common import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weight", [1e-37, 1e-20, 1e-6, 1.0, 1e30, 1e38])
@pytest.mark.parametrize("T", [128.0, 150.0, 1000.0])
def test_band_means_of_small_terms(T, weight):
    import torch
    import paper_2104_12522_gb300 as bart
    ctx = make_ctx()
    S, L, N, nb = 1, 20, 2000, 3
    p = W.log_pressures(L, 1e-8, 100.0)
    rng = np.random.default_rng(11)
    grid = torch.tensor((10 ** rng.uniform(-24.0, -22.0, (S, L, 1, N))).astype(np.float32), device="cuda")
    cfg = dict(geometry=0, n_angles=8, g=W.HD189_GRAV_CGS, mu=2.3, x0=[1e-3], t_min=50.0, t_max=3000.0)
    # B of 128 K at 9,000 cm^-1 is 1e-37
    w = rng.uniform(0.5, 1.0, (nb, N)) * weight
    w[1, : N // 3] = 0.0
    filt = torch.tensor(w.astype(np.float32), device="cuda")
    rows, bands = torch.empty((1, L, N), device="cuda"), torch.empty((1, L, nb), device="cuda")
    ctx.contribution_functions(grid, p, [1000.0], bart.NuGrid(9000.0, 0.001, N), cfg,
                               t_profile=torch.full((1, L), T, device="cuda"), contrib=rows, filters=filt, bands=bands)
    ctx.sync()
    r, f, b = rows.double().cpu().numpy()[0], filt.double().cpu().numpy(), bands.double().cpu().numpy()[0]
    f[:, [0, -1]] *= 0.5
    want = (r @ f.T) / f.sum(1)
    # half a unit in the last place of a normal or denormal value, and FP64's own roundings
    assert np.all(np.abs(b - want) <= np.maximum(np.abs(want) * (2.0 ** -24 + 2.0 ** -40), 2.0 ** -150 * 1.001))
    assert np.any(b > 0)
