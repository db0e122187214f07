"""The FP64 stage at every tile height its launch rule takes (8, 4, 2 rows;
launch_stage_n in csrc/dg_kernels.cuh), on meshes with ragged last tiles, and
the planar shallow-water problem on the same kernels.  Tolerances as in
test_parity_gpu.py (tendencies, 3e-14 of the magnitude bound) and
test_plane_gpu.py (1e-12)."""
import numpy as np
import pytest

import oracle as O
from paper_2303_11767_gb300 import dgswe
from test_parity_gpu import assert_within, case, tend_err

pytestmark = pytest.mark.gpu

SMS = 152


def tile_rows(nlon, nlat, n):
    """The launch rule."""
    rows, best = 8, None
    for c, cost in ((8, 1.0), (4, 1.02), (2, 1.2)):
        tiles = -(-nlon // (32 // n)) * -(-nlat // c)
        work = -(-tiles // SMS) * c * cost
        if best is None or work < best:
            rows, best = c, work
    return rows


MESHES = [(0, 7, 9, 2), (0, 97, 77, 4), (1, 7, 9, 2), (1, 49, 78, 4), (2, 7, 9, 2), (2, 31, 77, 4), (2, 102, 83, 8), (3, 7, 9, 2), (3, 25, 78, 4), (3, 82, 83, 8), (4, 7, 9, 2), (4, 19, 77, 4), (4, 61, 83, 8)]


@pytest.mark.parametrize("p,nlon,nlat,rows", MESHES)
def test_rhs_matches_oracle(p, nlon, nlat, rows):
    assert tile_rows(nlon, nlat, p + 1) == rows
    o, u = case(nlon, nlat, p, 11)
    with dgswe.Solver(nlon, nlat, p, precision="fp64") as s:
        k = s.rhs(u)
    what = f"rhs p={p} {nlon}x{nlat} fp64, {rows} tile rows"
    assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u), what), 3e-14, what)


@pytest.mark.parametrize("p,nx,ny,rows", [(3, 50, 50, 4), (1, 33, 53, 2), (3, 49, 66, 4), (4, 79, 66, 8), (2, 5, 1, 2), (4, 1, 3, 2)])
def test_plane_swe_matches_oracle(p, nx, ny, rows):
    assert tile_rows(nx, ny, p + 1) == rows
    L = 1.0e6
    with dgswe.Solver.plane_swe(nx, ny, p, L=L) as s:
        lam, th = s.projection_nodes()
        X, Y = lam[None, :] * 2 * np.pi / L, th[:, None] * 2 * np.pi / L
        h = 1000.0 + 5.0 * np.sin(X) * np.cos(Y)
        u = s.project_grid(lambda a, b: [h, h * 0.3 * np.cos(Y + 0 * X), h * 0.2 * np.sin(X + Y)])
        k = s.rhs(u)
    o = O.Oracle.plane_swe(nx, ny, p, L, dgswe.GRAVITY, 1.0e-4)
    assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u)), 3e-14, f"plane p={p} {nx}x{ny}")
