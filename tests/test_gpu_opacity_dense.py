"""Dense line lists (a line per two grid points and more) against the oracle
and against the line-by-line kernel: ragged grid lengths around the blocks of 8
and 32 points, cutoffs above and below the near window and the grid, cutoffs
that are and are not whole grid steps, lines outside the grid, on grid points
and on top of one another, pressures from Doppler to broad Lorentz profiles
(some cells line by line), the line-strength bound, and two species at once."""
import numpy as np
import pytest

import workloads as W
from oracle import opacity as O
from gpu_common import make_ctx, opacity_errors

pytestmark = pytest.mark.gpu

# the paths' forms are within 8e-6 of a line's term (one-pole, line by line)
# and 1.6e-6 + 1.3e-6 + 2e-6 (dense); FP32 strengths within 4e-6
MAX_REL, L2_REL = 2e-5, 1e-5


@pytest.fixture(scope="module")
def ctx():
    return make_ctx()


def _list(s, n, lo, hi, dnu, seed):
    """A seeded list; a tenth of the lines on grid points, a tenth doubled."""
    ll = W.line_list(s, n, lo, hi)
    rng = np.random.default_rng(seed)
    nu0 = ll.nu0.copy()
    k = rng.integers(0, n, n // 10)
    nu0[k] = 1000.0 + np.round((nu0[k] - 1000.0) / dnu) * dnu
    k = rng.integers(0, n - 1, n // 10)
    nu0[k] = nu0[k + 1]
    order = np.argsort(nu0, kind="stable")
    return W.LineList(nu0[order], ll.log10_s296[order], ll.elow[order], ll.gamma_ref[order], ll.mass_amu)


CELLS = [(1e-8, 500.0), (1e-4, 3000.0), (1e-2, 900.0), (0.2, 1500.0), (1.0, 2000.0), (30.0, 700.0)]


@pytest.mark.parametrize("N,dnu,cutoff,lines", [
    (37, 0.02, 25.0, 300), (256, 0.02, 1.0, 2000), (700, 0.02, 1.013, 5000), (1000, 0.02, 5.0, 1500),
    (513, 0.05, 25.0, 4000), (321, 0.25, 9.6, 700), (500, 1.0, 25.0, 2500), (400, 1.0, 25.3, 300),
    (333, 0.1, 2.45, 9000)])
def test_dense_lists_match_the_oracle(ctx, N, dnu, cutoff, lines):
    import paper_2104_12522_gb300 as bart
    lo, hi = 1000.0 - 1.5 * cutoff, 1000.0 + N * dnu + 1.5 * cutoff
    # so many lines in the grid's range and its surroundings
    species = [_list(s, int(lines * (hi - lo) / (N * dnu)) + 64, lo, hi, dnu, N + s) for s in range(2)]
    p, t = np.array(CELLS).T
    nu = bart.NuGrid(1000.0, dnu, N)
    got = ctx.opacity_cells([bart.device_lines(s) for s in species], p, t, nu, cutoff)
    ctx.sync()
    ref = O.opacity_cells(species, p, t, 1000.0, dnu, N, cutoff)
    e, l2 = opacity_errors(got.cpu().numpy(), ref)
    print(f"N {N} dnu {dnu} cutoff {cutoff}: max rel {e:.2e}, L2 {l2:.2e}")
    assert e < MAX_REL and l2 < L2_REL


@pytest.mark.parametrize("ratio", [1.0, 1.3, 3.9, 6.0])
def test_wide_lorentz_profiles(ctx, ratio):
    """Widths from a few grid points to a sixth of the cutoff and beyond, with
    gamma_ref over one bin, several, and more than the kernels have bins for."""
    import paper_2104_12522_gb300 as bart
    N, dnu = 200, 0.02
    species = [_list(0, 11_000, 970.0, 1034.0, dnu, 3)]
    rng = np.random.default_rng(4)
    g = 0.1 * ratio ** -rng.uniform(0.0, 1.0, species[0].n)
    species[0] = W.LineList(species[0].nu0, species[0].log10_s296, species[0].elow, g.astype(np.float32), 18.0)
    p, t = np.array([(1.2, 1500.0), (2.5, 3000.0), (5.0, 1500.0), (12.0, 900.0), (40.0, 1500.0), (100.0, 600.0)]).T
    got = ctx.opacity_cells([bart.device_lines(s) for s in species], p, t, bart.NuGrid(1000.0, dnu, N), 25.0)
    ctx.sync()
    ref = O.opacity_cells(species, p, t, 1000.0, dnu, N, 25.0)
    e, l2 = opacity_errors(got.cpu().numpy(), ref)
    print(f"gamma_ref ratio {ratio}: max rel {e:.2e}, L2 {l2:.2e}")
    assert e < MAX_REL and l2 < L2_REL


def test_dense_and_line_by_line_agree(ctx):
    """The same list whole (dense) and in parts too thin for the dense path,
    added up in FP64; with and without the line-strength bound."""
    import paper_2104_12522_gb300 as bart
    N, dnu, parts = 3000, 0.02, 20
    ll = _list(1, 30_000, 995.0, 1065.0, dnu, 5)
    p, t = np.array(CELLS).T
    nu = bart.NuGrid(1000.0, dnu, N)
    whole = ctx.opacity_cells([bart.device_lines(ll)], p, t, nu, 25.0).cpu().numpy().astype(np.float64)
    thin = np.zeros_like(whole)
    for k in range(parts * 2):
        part = W.LineList(ll.nu0[k::parts * 2], ll.log10_s296[k::parts * 2], ll.elow[k::parts * 2],
                          ll.gamma_ref[k::parts * 2], ll.mass_amu)
        assert part.n < 0.5 * N
        thin += ctx.opacity_cells([bart.device_lines(part)], p, t, nu, 25.0).cpu().numpy()
    e, l2 = opacity_errors(whole, thin)
    assert e < MAX_REL and l2 < L2_REL
    ctx.set_line_threshold(1e-3)
    bound = ctx.opacity_cells([bart.device_lines(ll)], p, t, nu, 25.0).cpu().numpy()
    ctx.set_line_threshold(0.0)
    ref = np.array([[O.opacity_cell(ll, P, T, 1000.0, dnu, N, 25.0, 1000, 1100, rel_threshold=1e-3)
                     for P, T in zip(p, t)]])
    e, l2 = opacity_errors(bound[..., 1000:1100], ref)
    assert e < MAX_REL and l2 < L2_REL


def test_a_strong_line_that_has_been_cut_off_leaves_nothing(ctx):
    """Beyond a strong line's cutoff only the weak ones count, to full accuracy."""
    import paper_2104_12522_gb300 as bart
    N, dnu = 800, 0.02
    n = 600
    rng = np.random.default_rng(9)
    nu0 = np.sort(rng.uniform(1000.0, 1016.0, n))
    logs = np.full(n, -35.0, np.float32)
    logs[n // 2] = -19.0
    ll = W.LineList(nu0, logs, np.zeros(n, np.float32), np.full(n, 0.07, np.float32), 18.0)
    p, t = np.array([1e-6, 0.1]), np.array([1000.0, 1000.0])
    nu = bart.NuGrid(1000.0, dnu, N)
    got = ctx.opacity_cells([bart.device_lines(ll)], p, t, nu, 2.5).cpu().numpy().astype(np.float64)
    # against the line-by-line kernel (two halves too thin for the dense one):
    # both take the same FP32 strengths, whose error at ln S = -80 (several
    # roundings at that size) is above this bound.  Values of 1e-41 are FP32
    # denormals: spacing 2^-149
    ref = np.zeros_like(got)
    for k in range(2):
        half = W.LineList(nu0[k::2], logs[k::2], np.zeros(n // 2, np.float32), np.full(n // 2, 0.07, np.float32), 18.0)
        assert half.n < 0.5 * N
        ref += ctx.opacity_cells([bart.device_lines(half)], p, t, nu, 2.5).cpu().numpy()
    assert np.all(np.abs(got - ref) <= MAX_REL * ref + 3.0 * 2.0 ** -149)


@pytest.mark.parametrize("dnu,cutoff,ratio", [(0.02, 25.0, 2.0), (0.02, 0.7, 1.0), (0.1, 25.0, 3.9), (1.0, 40.0, 1.3),
                                              (0.005, 2.0, 3.0)])
def test_profiles_wider_than_a_sixth_of_the_cutoff(ctx, dnu, cutoff, ratio):
    """The lines of a block that a cutoff edge divides count one by one there;
    strong lines, so that powers of the widths would leave the FP32 range."""
    import paper_2104_12522_gb300 as bart
    N = 300
    lo, hi = 1000.0 - 1.2 * cutoff, 1000.0 + N * dnu + 1.2 * cutoff
    ll = _list(0, int(1.5 * (hi - lo) / dnu), lo, hi, dnu, 11)
    rng = np.random.default_rng(12)
    ll = W.LineList(ll.nu0, ll.log10_s296 + 4.0, ll.elow, (0.1 * ratio ** -rng.uniform(0.0, 1.0, ll.n)).astype(np.float32),
                    18.0)
    g = np.array([0.2, 0.5, 3.0, 20.0]) * cutoff          # widths of the widest lines, cm^-1
    t = np.array([600.0, 2500.0, 600.0, 1500.0])
    p = g / 0.1 * np.sqrt(t / 296.0)
    got = ctx.opacity_cells([bart.device_lines(ll)], p, t, bart.NuGrid(1000.0, dnu, N), cutoff)
    ctx.sync()
    ref = O.opacity_cells([ll], p, t, 1000.0, dnu, N, cutoff)
    e, l2 = opacity_errors(got.cpu().numpy(), ref)
    print(f"dnu {dnu} cutoff {cutoff}: max rel {e:.2e}, L2 {l2:.2e}")
    assert e < MAX_REL and l2 < L2_REL
