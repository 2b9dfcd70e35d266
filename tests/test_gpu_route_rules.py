"""Rules that choose between two routes to one result, on both sides of each line, against the CPU FP64
oracle (tolerances of the parity tests: 1e-10 of peak in FP64, 1e-5 in FP32)."""
import numpy as np
import pytest

import synthetic as syn
from oracle import core, noise
from _helpers import TOL, qgrid_tuple, rel_err_of_peak, to_library

pytestmark = pytest.mark.gpu
PREC = [(0, "fp64"), (1, "fp32")]


@pytest.fixture(scope="module")
def ctx():
    import paper_1809_07088_gb300 as ds
    c = ds.Context(0)
    yield c
    c.close()


def _dw_model(spread, xmax, count=(17, 17, 17)):
    """Spins with displacements whose largest |Q.u| over the grid's corners is xmax: Gaussian ones, or
    every atom at +u or -u (no voxel's mean is then carried by small arguments)."""
    m = syn.small_case(syn.SPIN, cells=(6, 5, 4), nsite=3, nmodels=3, seed=241)
    m.qgrid = syn.QGrid(h0=tuple(-(c // 2) / n for c, n in zip(count, m.cells)), step=tuple(1.0 / n for n in m.cells),
                        count=count)
    rng = np.random.default_rng(29)
    if spread == "gauss":
        u = rng.standard_normal(m.spins.shape)
    else:
        u = np.array([1.0, 0.7, -0.4]) * rng.choice([-1.0, 1.0], m.spins.shape[:-1])[..., None]
    m.disp = u.astype(np.float32)
    m.disp = (u * (xmax / core.x_max(m, m.qgrid))).astype(np.float32)
    return m


@pytest.mark.parametrize("spread", ["gauss", "pair"])
@pytest.mark.parametrize("xmax", [1.9, 2.1, 3.1, 3.4, 5.0, 6.5, 6.7, 7.0, 10.0, 20.0])
def test_debye_waller_grid_below_and_above_the_order_cap(ctx, spread, xmax):
    """Grids of more voxels than the moments have monomials (4495 at order 28): |Q.u| below and above the
    arguments whose series ends by that order (3.27 in FP64, 6.61 in FP32), where the direct sum serves."""
    m = _dw_model(spread, xmax)
    G = m.qgrid.g_index(m.cells)
    want = core.magnetic_intensity_fft(m, G, 0, dw=True)
    scale = np.max(core.magnetic_intensity_fft(m, G, 0))
    lm = to_library(ctx, m)
    for prec, tag in PREC:
        got, _ = lm.intensity(qgrid_tuple(m.qgrid), disorder=1, mode=0, precision=prec, dw_coupling=1)
        assert np.max(np.abs(got.reshape(-1) - want)) / scale < TOL[tag], tag


@pytest.mark.parametrize("xmax", [2.1, 4.0, 6.5])
def test_debye_waller_moments_of_large_arguments_keep_fp32(ctx, xmax):
    """Equal spins on atoms at +u or -u: each Bragg intensity is its value at rest times cos^2(Q.u), which the
    polynomial forms from terms up to cosh(6.5) = 330 times as large.  With FP64 moments T_mu is right to
    an FP32 rounding; the FP32 transform of 64 equal moments (6 stages), phase, |F|^2 and the projection
    leave a few dozen roundings of 6e-8: 4e-6 of the peak."""
    m = syn.small_case(syn.SPIN, cells=(4, 4, 4), nsite=1, nmodels=1, seed=244)
    m.lattice = (4.0, 4.0, 4.0, 90.0, 90.0, 90.0)
    m.spins = (np.zeros_like(m.spins) + np.array([0.6, -0.8, 0.0])).astype(np.float32)
    m.qgrid = syn.QGrid(h0=(-2.0,) * 3, step=(0.25,) * 3, count=(17,) * 3)
    u = np.array([1.0, 0.7, -0.4]) * np.random.default_rng(33).choice([-1.0, 1.0], m.spins.shape[:-1])[..., None]
    m.disp = u.astype(np.float32)
    m.disp = (u * (xmax / core.x_max(m, m.qgrid))).astype(np.float32)
    G = m.qgrid.g_index(m.cells)
    want = core.magnetic_intensity_fft(m, G, 0, dw=True)
    got, _ = to_library(ctx, m).intensity(qgrid_tuple(m.qgrid), disorder=1, mode=0, precision=1, dw_coupling=1)
    assert np.max(np.abs(got.reshape(-1) - want)) / np.max(core.magnetic_intensity_fft(m, G, 0)) < 4e-6


@pytest.mark.parametrize("prec,tag", PREC)
def test_debye_waller_moments_stay_within_the_budget(ctx, prec, tag):
    """The scratch of the moments counts against the context's budget: with one byte too little for it the
    direct sum, which needs none, serves the request."""
    import paper_1809_07088_gb300 as ds
    m = _dw_model("gauss", 1.0)
    G = m.qgrid.g_index(m.cells)
    want = core.magnetic_intensity_fft(m, G, 0, dw=True)
    scale = np.max(core.magnetic_intensity_fft(m, G, 0))
    opts = dict(disorder=1, mode=0, precision=prec, dw_coupling=1)
    _, info = to_library(ctx, m).intensity(qgrid_tuple(m.qgrid), **opts)
    small = ds.Context(0, info["workspace_bytes"] - 1)
    try:
        got, info2 = to_library(small, m).intensity(qgrid_tuple(m.qgrid), **opts)
    finally:
        small.close()
    assert info2["workspace_bytes"] < info["workspace_bytes"]
    assert np.max(np.abs(got.reshape(-1) - want)) / scale < TOL[tag]


def _undisplaced(sites):
    m = syn.small_case(syn.DISP, cells=(6, 5, 4), nsite=len(sites), nmodels=1, seed=242)
    m.sites = np.array(sites, dtype=np.float64)
    m.scat_len = np.full(len(sites), 1.3)
    m.ff_kind = np.zeros(len(sites), np.int32)
    m.ff_coef = np.zeros((len(sites), 9))
    m.occ = None
    m.disp = np.zeros_like(m.disp)
    return m


@pytest.mark.parametrize("nsb", [3, 4])
def test_subbox_points_systematic_absences_are_zero(ctx, nsb):
    """Three equal sites a third of a cell apart cancel exactly in FP32 at h not divisible by three when the
    atoms are not displaced: their factors 1, -1/2 + is and -1/2 - is are formed in FP64 and rounded
    once, and every other factor is shared by overlapping boxes."""
    m = _undisplaced([[0.0, 0.0, 0.0], [1.0 / 3.0, 0.0, 0.0], [2.0 / 3.0, 0.0, 0.0]])
    m.scat_len = np.ones(3)
    rng = np.random.default_rng(31)
    hkl = np.stack([rng.choice([-5.0, -2.0, -1.0, 1.0, 2.0, 4.0], 200), *rng.uniform(-2.0, 2.0, (2, 200))], -1)
    org = syn.random_origins(rng, 1, m.cells, 360)
    got, _ = to_library(ctx, m).subbox_points(hkl, org, disorder=2, mode=0, precision=1, subbox_n=nsb)
    assert np.all(got == 0.0)


def test_subbox_points_mean_term_of_an_undisplaced_crystal(ctx):
    """DIFFUSE boxes of an undisplaced crystal at Bragg positions.  FP64: <cos(Q.u)> = 1, the box phases are 1
    and 2^3 cells add without rounding, so F = 8 phi and the mean term, rounded once, is the same number.
    FP32: the atoms' fast sine and cosine (2^-20.9 at most) and a few roundings in F and the mean leave
    |F - K B| below 2e-6 of |F|, an intensity below 4e-12 of the Bragg peak."""
    m = _undisplaced([[0.3, 0.17, 0.71]])
    lm = to_library(ctx, m)
    rng = np.random.default_rng(32)
    hkl = rng.integers(-6, 7, (200, 3)).astype(np.float64)
    org = syn.random_origins(rng, 1, m.cells, 360)
    got, _ = lm.subbox_points(hkl, org, disorder=2, mode=1, precision=0, subbox_n=2)
    assert np.all(got == 0.0)
    got, _ = lm.subbox_points(hkl, org, disorder=2, mode=1, precision=1, subbox_n=2)
    bragg, _ = lm.subbox_points(hkl, org, disorder=2, mode=0, precision=1, subbox_n=2)
    assert np.all(got < 4e-12 * bragg)


@pytest.mark.parametrize("prec,tag", PREC)
@pytest.mark.parametrize("kind", ["occ", "spin", "disp"])
@pytest.mark.parametrize("nsite,nsb", [(2, 2), (4, 9), (7, 8), (8, 3), (9, 2), (12, 9), (16, 4), (16, 9)])
def test_subbox_points_shared_amplitudes_of_every_site_count(ctx, prec, tag, kind, nsite, nsb):
    """Instances of exactly nsite sites, of more sites with the idle ones left out, and of boxes wider than the
    register ring, with four boxes per cell (shared amplitudes) and one (box by box for most)."""
    code = {"occ": syn.OCC, "spin": syn.SPIN, "disp": syn.DISP}[kind]
    cells = (9, 10, 9) if nsb == 9 else (8, 9, 10)
    m = syn.small_case(code, cells=cells, nsite=nsite, nmodels=1, seed=245)
    lm = to_library(ctx, m)
    rng = np.random.default_rng(34)
    hkl = rng.uniform(-1.5, 1.5, (37, 3))
    for ratio in (1, 4):
        org = syn.random_origins(rng, 1, cells, max(2, ratio * int(np.prod(cells)) // nsb ** 3))
        got, _ = lm.subbox_points(hkl, org, disorder=code, mode=1, precision=prec, subbox_n=nsb)
        assert rel_err_of_peak(got, noise.subbox_intensity(m, kind, 1, nsb, hkl, org)) < TOL[tag]


@pytest.mark.parametrize("prec,tag", PREC)
def test_subbox_points_boxes_wider_than_two_rings(ctx, prec, tag):
    """Boxes of 17 cells: three blocks of tabulated phase powers along each axis."""
    m = syn.small_case(syn.DISP, cells=(18, 20, 18), nsite=5, nmodels=1, seed=247)
    rng = np.random.default_rng(35)
    hkl = rng.uniform(-1.5, 1.5, (5, 3))
    org = syn.random_origins(rng, 1, m.cells, 40)
    got, _ = to_library(ctx, m).subbox_points(hkl, org, disorder=2, mode=1, precision=prec, subbox_n=17)
    assert rel_err_of_peak(got, noise.subbox_intensity(m, "disp", 1, 17, hkl, org)) < TOL[tag]


@pytest.mark.parametrize("prec,tag", PREC)
@pytest.mark.parametrize("kernel", [1, 2])
def test_blocked_taylor_spectra_with_a_last_block_of_less_than_32(ctx, prec, tag, kernel):
    """Monomial spectra above the size (300 MB a site) from which they are stored by blocks of 32 k, on unequal
    axes whose half spectrum (23,100 values) ends in a block of 28, for two supercells of three sites: both
    Taylor kernels, with and without the mean, against the direct sum.  The order is far above what |Q.u| needs."""
    m = syn.small_case(syn.DISP, cells=(35, 30, 42), nsite=3, nmodels=2, seed=246, sigma=0.04)
    m.qgrid = syn.QGrid(h0=(-1.0 / 35, 29.0 / 30, -2.0 / 42), step=(1.0 / 35, 1.0 / 30, 1.0 / 42), count=(3, 3, 4))
    lm = to_library(ctx, m)
    for mode in (0, 1):
        got, info = lm.intensity(qgrid_tuple(m.qgrid), disorder=2, mode=mode, precision=prec,
                                 taylor_order=17 if prec == 0 else 22, taylor_kernel=kernel)
        assert info["n_monomials"] * 23100 * (16 if prec == 0 else 8) > 300 << 20
        want = core.displacive_intensity_direct(m, m.qgrid.hkl(), mode)
        assert rel_err_of_peak(got, want) < TOL[tag]


def test_shared_memory_limit_of_a_kernel_is_not_lowered_by_another_request(ctx):
    """Two threads ask for sub-box volumes of the same box width whose planes take different amounts of
    shared memory, both above the default limit: neither request's launch fails for the other's."""
    import threading
    import torch
    lms, grids = [], []
    for n in (100, 120):
        m = syn.small_case(syn.OCC, cells=(4, n, n), nsite=1, nmodels=1, seed=243,
                           qgrid=syn.QGrid(h0=(0.0, 0.0, 0.0), step=(0.25, 1.0 / n, 1.0 / n), count=(2, 2, 2)))
        lms.append(to_library(ctx, m))
        grids.append(qgrid_tuple(m.qgrid))
    errors = []

    def loop(i):
        out = torch.empty((2, 2, 2), device="cuda")
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(1500):
                    lms[i].intensity(grids[i], out=out, disorder=0, mode=1, precision=1, smoothing=2, subbox_n=2)
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    ts = [threading.Thread(target=loop, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errors
