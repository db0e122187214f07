"""The FP64 stage at every tile height its launch rule takes (8, 7, 5, 4, 2 rows;
launch_stage_n in csrc/dg_kernels.cuh), on meshes with ragged last tiles, the
FP32 stage at the short ones (5, 4 rows), the FP64 stage's
one-lane-per-point kernel (csrc/dg_stage_f64pt.cuh) on the meshes below its line
(every RK kind, the status bits, bands, the global alpha), and the planar
shallow-water problem on both.  Tolerances as in
test_parity_gpu.py (tendencies, 3e-14 or 1e-6 of the magnitude bound; FP32
states 1e-5) and
test_plane_gpu.py (1e-12)."""
import numpy as np
import pytest

import oracle as O
from paper_2303_11767_gb300 import dgswe
from test_bands_gpu import _run_bands, _whole
from test_parity_gpu import assert_within, case, state_err, tend_err

pytestmark = pytest.mark.gpu

SMS = 152


def tile_rows(nlon, nlat, n):
    """The launch rule."""
    rows, best = 8, None
    costs = {1: (1.0, 1.1, 1.08, 0.96, 1.2), 2: (1.0, 1.1, 1.04, 0.96, 1.2), 3: (1.0, 1.03, 1.2, 1.0, 1.2)}
    for c, cost in zip((8, 5, 4, 7, 2), costs.get(n, (1.0, 1.03, 1.04, 1.02, 1.2))):
        tiles = -(-nlon // (32 // n)) * -(-nlat // c)
        if n == 1 and c == 7 and tiles <= SMS:
            continue
        per_sm = -(-tiles // SMS) * c
        work = cost * (max(per_sm, 3.5 * (-(-per_sm // 4))) if n >= 3 else per_sm)
        if best is None or work < best:
            rows, best = c, work
    return rows


MESHES = [(0, 122, 34, 2), (0, 190, 122, 5), (0, 65, 101, 4), (0, 340, 167, 7), (0, 241, 139, 8), (0, 194, 85, 2), (0, 259, 137, 5), (1, 231, 79, 8), (1, 148, 137, 5), (1, 231, 103, 4), (1, 156, 100, 7), (1, 131, 133, 2), (2, 55, 87, 4), (2, 199, 40, 7), (2, 131, 89, 5), (2, 107, 100, 8), (2, 216, 25, 2), (3, 52, 138, 7), (3, 169, 67, 4), (3, 189, 92, 5), (3, 147, 123, 8), (3, 162, 113, 2), (4, 149, 59, 5), (4, 81, 58, 7), (4, 203, 29, 8), (4, 125, 113, 2), (4, 89, 25, 4)]


@pytest.mark.parametrize("p,nlon,nlat,rows", MESHES)
def test_rhs_matches_oracle(p, nlon, nlat, rows):
    assert tile_rows(nlon, nlat, p + 1) == rows
    o, u = case(nlon, nlat, p, 11)
    with dgswe.Solver(nlon, nlat, p, precision="fp64") as s:
        k = s.rhs(u)
    what = f"rhs p={p} {nlon}x{nlat} fp64, {rows} tile rows"
    assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u), what), 3e-14, what)


@pytest.mark.parametrize("p,nx,ny", [(3, 50, 50), (1, 129, 113), (3, 81, 66), (4, 79, 66), (2, 5, 1), (4, 1, 3), (1, 7, 3), (3, 5, 1)])
def test_plane_swe_matches_oracle(p, nx, ny):
    L = 1.0e6
    with dgswe.Solver.plane_swe(nx, ny, p, L=L) as s:
        lam, th = s.projection_nodes()
        X, Y = lam[None, :] * 2 * np.pi / L, th[:, None] * 2 * np.pi / L
        h = 1000.0 + 5.0 * np.sin(X) * np.cos(Y)
        u = s.project_grid(lambda a, b: [h, h * 0.3 * np.cos(Y + 0 * X), h * 0.2 * np.sin(X + Y)])
        k = s.rhs(u)
    o = O.Oracle.plane_swe(nx, ny, p, L, dgswe.GRAVITY, 1.0e-4)
    assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u)), 3e-14, f"plane p={p} {nx}x{ny}")


POINTS = [(1, 7, 5), (1, 33, 19), (2, 7, 5), (2, 31, 18), (3, 7, 5), (3, 25, 17), (4, 7, 5), (4, 19, 13), (1, 2, 2), (4, 1, 2)]


@pytest.mark.parametrize("p,nlon,nlat", POINTS)
def test_point_stage_rhs_matches_oracle(p, nlon, nlat):
    o, u = case(nlon, nlat, p, 11)
    with dgswe.Solver(nlon, nlat, p, precision="fp64") as s:
        k = s.rhs(u)
        what = f"rhs p={p} {nlon}x{nlat} fp64, lane per point"
        assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u), what), 3e-14, what)
        s.set_option(dgswe.OPT_ALPHA_MODE, 1)
        k = s.rhs(u)
    o2 = O.Oracle.sphere(nlon, nlat, p, dgswe.EARTH_RADIUS, dgswe.GRAVITY, dgswe.OMEGA)
    o2.set_alpha_mode(1)
    assert_within(tend_err(k, o2.rhs(u), o2.rhs_magnitude(u)), 3e-14, what + ", global alpha")


@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("p,nlon,nlat", [(1, 33, 19), (2, 31, 18), (3, 25, 17), (4, 19, 13)])
def test_point_stage_steps_and_bands(p, nlon, nlat, order):
    torch = pytest.importorskip("torch")
    o, u = case(nlon, nlat, p, 11)
    dt = o.max_dt(u, 0.1)
    whole = _whole(u, nlon, nlat, p, "fp64", 4, dt, order, torch)[0]
    assert_within(state_err(whole, o.step(u, 4, dt, order)), 1e-12, f"RK{order} p={p}")
    assert np.array_equal(_run_bands(u, nlon, nlat, p, "fp64", 3, 4, dt, order, torch)[0], whole)


@pytest.mark.parametrize("j,i", [(0, 0), (12, 18), (6, 9)])
@pytest.mark.parametrize("value,status", [(np.nan, dgswe.DG_ENONFINITE), (-3.0e4, dgswe.DG_ENONPHYSICAL), (np.inf, dgswe.DG_ENONFINITE)])
def test_point_stage_reports_bad_states(j, i, value, status):
    _, u = case(19, 13, 4, 11)
    bad = u.copy()
    bad[j, i, 0, 0] = value
    with dgswe.Solver(19, 13, 4, precision="fp64") as s:
        with pytest.raises(dgswe.DGError) as e:
            s.rhs(bad)
        assert e.value.status == status
        s.rhs(u)


@pytest.mark.parametrize("p,nlon,nlat,rows", [(1, 156, 100, 7), (2, 131, 89, 5), (3, 52, 138, 7)])
def test_tile_rows_bands_get_the_whole_mesh_bits(p, nlon, nlat, rows):
    torch = pytest.importorskip("torch")
    assert tile_rows(nlon, nlat, p + 1) == rows
    o, u = case(nlon, nlat, p, 11)
    dt = o.max_dt(u, 0.1)
    whole = _whole(u, nlon, nlat, p, "fp64", 2, dt, 3, torch)[0]
    assert np.array_equal(_run_bands(u, nlon, nlat, p, "fp64", 3, 2, dt, 3, torch)[0], whole)


def tile_rows_f32(nlon, nlat, n):
    """The launch rule."""
    rows, best = 8, None
    for c, cost in ((8, 1.0), (5, 0.95 if n == 5 else 1.0 if n == 3 else 1.08), (4, 0.97 if n in (3, 5) else 1.03))[:2 if n == 1 else 3]:
        per_sm = c * -(-(-(-nlon // (32 // n)) * -(-nlat // c)) // SMS)
        if c < 8 and (per_sm > (10 if n == 1 else 20) or n <= 2 and c == 5 and best <= 8):
            continue
        work = cost * per_sm
        if best is None or work < best:
            rows, best = c, work
    return rows


F32 = [(0, 162, 37, 8), (0, 206, 93, 8), (0, 299, 149, 5), (4, 196, 97, 8), (4, 206, 103, 8), (1, 7, 15, 4), (1, 141, 67, 8), (1, 196, 97, 5), (2, 16, 46, 4), (2, 157, 43, 5), (3, 23, 9, 4), (3, 217, 44, 5), (4, 85, 44, 5), (4, 133, 69, 4)]


@pytest.mark.parametrize("p,nlon,nlat,rows", F32)
def test_short_fp32_tiles(p, nlon, nlat, rows):
    torch = pytest.importorskip("torch")
    assert tile_rows_f32(nlon, nlat, p + 1) == rows
    o, u = case(nlon, nlat, p, 11)
    with dgswe.Solver(nlon, nlat, p, precision="fp32") as s:
        k = s.rhs(u)
    what = f"rhs p={p} {nlon}x{nlat} fp32, {rows} tile rows"
    assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u), what), 1e-6, what)
    dt = o.max_dt(u, 0.1)
    for order in (3, 4):
        whole = _whole(u, nlon, nlat, p, "fp32", 3, dt, order, torch)[0]
        assert_within(state_err(whole, o.step(u, 3, dt, order)), 1e-5, what)
    assert np.array_equal(_run_bands(u, nlon, nlat, p, "fp32", 2, 3, dt, 4, torch)[0], whole)


def _rough(ny, nx, p):
    rng = np.random.default_rng(3)
    u = np.zeros((ny, nx, 3, (p + 1) ** 2))
    u[..., 0, 0] = 2.0 * 5960.0 + rng.normal(size=(ny, nx))
    u[..., 1:, :] = 1000.0 * rng.normal(size=u[..., 1:, :].shape)
    return u


@pytest.mark.parametrize("p,nlon,nlat,prec", [(1, 2, 262150, "fp32"), (0, 1, 458800, "fp64")])
def test_more_tile_rows_than_a_grid_dimension(p, nlon, nlat, prec):
    """Over 65535 tiles of 4 rows (the thread-per-element stage's) and of 7 (FP64).
    FP64 tolerance: near a pole cos(theta) carries the rounding of theta, 2^-52 nlat / pi of its value."""
    u = _rough(nlat, nlon, p)
    o = O.Oracle.sphere(nlon, nlat, p)
    with dgswe.Solver(nlon, nlat, p, precision=prec) as s:
        k = s.rhs(u)
    assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u)), 2.0 ** -52 * nlat if prec == "fp64" else 1e-6, f"rhs p={p} {nlon}x{nlat} {prec}")


def test_plane_with_more_tile_rows_than_a_grid_dimension():
    """Tolerance as in test_plane_gpu.py."""
    u = _rough(524300, 2, 0)
    with dgswe.Solver.plane_swe(2, 524300, 0, L=1.0e6) as s:
        k = s.rhs(u)
    o = O.Oracle.plane_swe(2, 524300, 0, 1.0e6, dgswe.GRAVITY, 1.0e-4)
    assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u)), 1e-12, "plane p=0 2x524300")
