"""Kernel variants at the sizes where a tile, a remainder or a route changes, against the CPU FP64
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


@pytest.mark.parametrize("prec,tag", PREC)
@pytest.mark.parametrize("m_,mp", [(2, 2), (3, 3), (2, 5), (4, 8)])
def test_lanczos_point_weights_near_bragg_and_half_positions(ctx, prec, tag, m_, mp):
    """Points on, and 1e-12 to 1e-6 beside, Bragg positions and the half positions between them, where
    the weights switch between the limit, the nearest and the next Bragg position; tap counts of every
    register size (4, 10, 32), equal and different sine arguments."""
    m = syn.small_case(syn.OCC, cells=(6, 5, 4), nsite=2, nmodels=1, seed=231)
    lm = to_library(ctx, m)
    d = np.array([0.0, 1e-12, -1e-12, 3e-9, -3e-8, 1e-6, -1e-6, 0.5, 0.5 + 1e-9, 0.5 - 1e-9, 0.25])
    Q = np.stack(np.meshgrid(d + 2.0, d[::-1] - 3.0, d[::3], indexing="ij"), -1).reshape(-1, 3)
    hkl = Q / np.array(m.cells, dtype=np.float64)
    got, _ = lm.intensity_points(hkl, disorder=0, mode=1, precision=prec, lanczos_m=m_, lanczos_mprime=mp)
    sel = np.arange(0, Q.shape[0], 7)
    want = noise.lanczos_resample(lambda G: core.occupancy_intensity_fft(m, G, 1),
                                  (hkl * np.array(m.cells))[sel], m_, mp)
    assert rel_err_of_peak(got[sel], want) < TOL[tag]


@pytest.mark.parametrize("prec,tag", PREC)
@pytest.mark.parametrize("sigma", [0.0, 0.02, 0.2, 0.45, 3.0])
@pytest.mark.parametrize("count", [(1, 1, 1), (5, 37, 3), (9, 11, 13)])
def test_debye_waller_grid_routes(ctx, prec, tag, sigma, count):
    """T_mu(G) on grids by the moments of the displacements (polynomial in the working type, in FP64)
    and by the direct sum, chosen on the device from x_max and the voxel count: no displacement, small
    and large ones, one voxel, more rows than a tile, a grid away from the origin."""
    m = syn.small_case(syn.SPIN, cells=(6, 5, 4), nsite=3, nmodels=3, seed=232)
    rng = np.random.default_rng(5)
    m.disp = (sigma * rng.standard_normal(m.spins.shape)).astype(np.float32)
    g0 = (-3, 2, -1)
    m.qgrid = syn.QGrid(h0=tuple(g / n for g, n in zip(g0, m.cells)), step=tuple(1.0 / n for n in m.cells), count=count)
    lm = to_library(ctx, m)
    got, _ = lm.intensity(qgrid_tuple(m.qgrid), disorder=1, mode=0, precision=prec, dw_coupling=1)
    want = core.magnetic_intensity_fft(m, m.qgrid.g_index(m.cells), 0, dw=True)
    scale = np.max(core.magnetic_intensity_fft(m, m.qgrid.g_index(m.cells), 0))
    assert np.max(np.abs(got.reshape(-1) - want)) / scale < TOL[tag]


@pytest.mark.parametrize("prec,tag", PREC)
@pytest.mark.parametrize("kind", ["occ", "spin", "disp"])
@pytest.mark.parametrize("cells,nsb,nsite,npts,mode", [((6, 5, 4), 4, 3, 130, 1), ((6, 5, 4), 3, 5, 128, 0),
                                                       ((4, 7, 8), 4, 1, 1, 1), ((9, 10, 9), 9, 1, 9, 1)])
def test_subbox_points_shared_cell_amplitudes(ctx, prec, tag, kind, cells, nsb, nsite, npts, mode):
    """Overlapping boxes at many origins (cell amplitudes shared by the boxes, rows of cells that wrap,
    a remainder of points, boxes as wide as a row and wider than the register ring) against the
    brute-force sum over boxes; occupancy weights with the displacements."""
    code = {"occ": syn.OCC, "spin": syn.SPIN, "disp": syn.DISP}[kind]
    nm = 1 if nsb > 8 else 2
    m = syn.small_case(code, cells=cells, nsite=nsite, nmodels=nm, seed=233)
    lm = to_library(ctx, m)
    rng = np.random.default_rng(11)
    hkl = rng.uniform(-1.7, 1.7, (npts, 3))
    org = syn.random_origins(rng, nm, cells, 3 * nm * int(np.prod(cells)) // (8 if nsb > 8 else 1))
    got, _ = lm.subbox_points(hkl, org, disorder=code, mode=mode, precision=prec, subbox_n=nsb)
    want = noise.subbox_intensity(m, kind, mode, nsb, hkl, org)
    assert rel_err_of_peak(got, want) < TOL[tag]


@pytest.mark.parametrize("prec,tag", PREC)
@pytest.mark.parametrize("kind,cells,nsb,nm", [("occ", (2, 3, 2), 1, 2), ("spin", (5, 4, 7), 2, 2), ("occ", (16, 18, 21), 8, 1),
                                               ("occ", (18, 20, 18), 9, 1)])
def test_subbox_correlations_by_planes(ctx, prec, tag, kind, cells, nsb, nm):
    """Windowed pair correlations of every box width: one cell, rows that are not multiples of four, more
    rows than row lanes, the widest box of the plane kernel and one beyond it, against the brute-force
    sum over boxes."""
    code = {"occ": syn.OCC, "spin": syn.SPIN}[kind]
    count = (3, 2, 4) if max(cells) > 8 else (7, 5, 6)
    grid = syn.QGrid(h0=tuple(-2.0 / n for n in cells), step=tuple(1.0 / n for n in cells), count=count)
    m = syn.small_case(code, cells=cells, nsite=2, nmodels=nm, seed=234, qgrid=grid)
    lm = to_library(ctx, m)
    got, _ = lm.intensity(qgrid_tuple(grid), disorder=code, mode=1, precision=prec, smoothing=2, subbox_n=nsb)
    want = noise.subbox_intensity(m, kind, 1, nsb, grid.hkl())
    assert rel_err_of_peak(got, want) < TOL[tag]


@pytest.mark.parametrize("n,off", [(8, 0), (16, 0), (20, 0), (8, 1), (6, 0)])
def test_displacive_adjoint_hermitian_part_and_full(ctx, n, off):
    """FP32 gradient on grids symmetric about the origin (the Hermitian part of Z on the stored half of the
    k, half-spectrum transform) and on a shifted or otherwise sized one (every k), against the FP64
    gradient, with occupancy weights and a dL/dI that is not symmetric."""
    m = syn.small_case(syn.DISP, cells=(n, n, n), nsite=3, nmodels=2, seed=235, sigma=0.08)
    c = n + 3
    m.qgrid = syn.QGrid(h0=tuple((off - c) / n for _ in range(3)), step=(1.0 / n,) * 3, count=(2 * c + 1,) * 3)
    lm = to_library(ctx, m)
    rng = np.random.default_rng(17)
    d = rng.standard_normal(m.qgrid.count)
    g64 = lm.backward(qgrid_tuple(m.qgrid), d, disorder=2, mode=0, precision=0, taylor_order=7)
    g32 = lm.backward(qgrid_tuple(m.qgrid), d.astype(np.float32), disorder=2, mode=0, precision=1, taylor_order=7)
    assert rel_err_of_peak(g32, g64) < 2e-5
