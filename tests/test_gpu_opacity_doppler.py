"""Dense lists at Doppler widths of more than a grid point (high wavenumbers, fine
grids) against the oracle: a strong line on each edge of a block of 8 points, whose
mid and far points take the block's moments, at Lorentz widths on both sides of
the real and complex centres, with gamma_ref in one bin and over several."""
import numpy as np
import pytest

import workloads as W
from oracle import opacity as O
from gpu_common import make_ctx, opacity_errors

pytestmark = pytest.mark.gpu

# the forms of single lines within 2e-6 (dense) to 8e-6 (line by line), the moments within 1.4e-6 of a line, FP32
# strengths within 4e-6
MAX_REL, L2_REL = 2e-5, 1e-5


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


@pytest.mark.parametrize("ratio", [1.0, 1.4, 3.5])
@pytest.mark.parametrize("T", [2000.0, 1380.0, 960.0, 240.0])
def test_wide_doppler_profiles(ctx, T, ratio):
    """x of a grid interval 0.41, 0.5, 0.6 and 1.2."""
    import paper_2104_12522_gb300 as bart
    N, dnu, nu0, cutoff = 400, 0.02, 10_000.0, 5.0
    rng = np.random.default_rng(int(T))
    n = 700
    cen = np.sort(nu0 + dnu * np.concatenate([rng.uniform(-200.0, 600.0, n), [199.51, 215.49]]))
    strong = np.isin(cen, nu0 + dnu * np.array([199.51, 215.49]))
    gref = 0.08 * ratio ** -rng.uniform(0.0, 1.0, cen.size)
    gref[strong] = 0.08
    logs = np.where(strong, -18.0, -23.0 + rng.uniform(-1.0, 1.0, cen.size))
    ll = W.LineList(cen, logs.astype(np.float32), rng.uniform(0.0, 500.0, cen.size).astype(np.float32),
                    gref.astype(np.float32), 16.0)
    width = np.array([0.01, 1.0, 2.5, 3.3, 4.0, 4.6, 6.0, 8.0, 12.0, 25.0])       # of the widest lines, in points
    p = width * dnu / (0.08 * np.sqrt(296.0 / T))
    t = np.full(p.size, T)
    got = ctx.opacity_cells([bart.device_lines(ll)], p, t, bart.NuGrid(nu0, dnu, N), cutoff)
    ctx.sync()
    ref = O.opacity_cells([ll], p, t, nu0, dnu, N, cutoff)
    errors = [opacity_errors(got[:, c].cpu().numpy(), ref[:, c]) for c in range(p.size)]
    print(f"T {T}, ratio {ratio}: " + ", ".join(f"{w}: {e:.1e}" for w, (e, _) in zip(width, errors)))
    assert all(e < MAX_REL and l2 < L2_REL for e, l2 in errors)
