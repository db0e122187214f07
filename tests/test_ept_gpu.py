"""The one-thread-per-element FP32 stage (csrc/dg_stage_ept.cuh), at meshes just
above the size from which it runs: ragged last tiles in both directions, rows
that start anywhere in a 16-byte block (odd element counts), whole tiles, every
RK kind, the status bits, and bands of such a mesh.  Tolerances as in
test_parity_gpu.py: tendencies 1e-6 of the oracle's magnitude bound, states
1e-5."""
import numpy as np
import pytest

from paper_2303_11767_gb300 import dgswe
from test_bands_gpu import _run_bands, _whole
from test_parity_gpu import assert_within, case, state_err, tend_err

pytestmark = pytest.mark.gpu

MESHES = [(4, 151, 141), (4, 160, 136), (3, 211, 190), (3, 208, 200), (2, 145, 125), (2, 160, 116), (1, 229, 221), (1, 97, 521)]
WIDE = (4, 355, 177)   # 16 x 8 tiles would need a little more than a round: 32 x 4 ones run


@pytest.mark.parametrize("p,nlon,nlat", MESHES + [WIDE])
def test_rhs_matches_oracle(p, nlon, nlat):
    o, u = case(nlon, nlat, p, 11)
    with dgswe.Solver(nlon, nlat, p, precision="fp32") as s:
        k = s.rhs(u)
    what = f"rhs p={p} {nlon}x{nlat} fp32, thread per element"
    assert_within(tend_err(k, o.rhs(u), o.rhs_magnitude(u), what), 1e-6, what)


@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("p,nlon,nlat", [MESHES[0], MESHES[4]])
def test_steps_match_oracle(p, nlon, nlat, order):
    o, u = case(nlon, nlat, p, 11)
    dt = o.max_dt(u, 0.1)
    with dgswe.Solver(nlon, nlat, p, precision="fp32", rk_order=order) as s:
        s.set_state(u)
        s.step(3, dt)
        got = s.get_state()
    assert_within(state_err(got, o.step(u, 3, dt, order)), 1e-5, f"RK{order} p={p} {nlon}x{nlat}")


@pytest.mark.parametrize("p,nlon,nlat,nb", [(4, 151, 141, 3), (2, 145, 125, 4), (3, 211, 190, 2), (4, 355, 177, 2)])
def test_bands_equal_whole_mesh(p, nlon, nlat, nb):
    torch = pytest.importorskip("torch")
    o, u = case(nlon, nlat, p, 11)
    dt = o.max_dt(u, 0.1)
    got, _, _ = _run_bands(u, nlon, nlat, p, "fp32", nb, 3, dt, 3, torch)
    assert np.array_equal(got, _whole(u, nlon, nlat, p, "fp32", 3, dt, 3, torch)[0])


@pytest.mark.parametrize("p,nlon,nlat,nb", [(4, 151, 141, 3), (2, 145, 249, 2), (3, 211, 190, 4), (1, 229, 221, 8)])
def test_bands_with_their_own_kernel(p, nlon, nlat, nb):
    """DG_OPT_BAND_KERNEL: bands below the line of a mesh above it (145x249: the bands of 124 and 125 rows
    lie on both sides of it); other order of sums, so equal to the oracle's states and not to the mesh's bits."""
    torch = pytest.importorskip("torch")
    o, u = case(nlon, nlat, p, 11)
    dt = o.max_dt(u, 0.1)
    with dgswe.Solver.band(nlon, nlat, 0, 9, p, precision="fp32") as b, dgswe.Solver(9, 5, 1) as s:
        for handle, value in ((b, 2), (b, -1), (s, 1)):
            with pytest.raises(dgswe.DGError) as e:
                handle.set_option(dgswe.OPT_BAND_KERNEL, value)
            assert e.value.status == dgswe.DG_EINVAL
    got, mass, _ = _run_bands(u, nlon, nlat, p, "fp32", nb, 3, dt, 3, torch, own=1)
    want, whole_mass, _ = _whole(u, nlon, nlat, p, "fp32", 3, dt, 3, torch)
    assert not np.array_equal(got, want)   # the other kernel ran
    assert_within(state_err(got, o.step(u, 3, dt, 3)), 1e-5, f"own kernel p={p} {nlon}x{nlat}")
    assert abs(mass / whole_mass - 1) < 1e-9   # FP32 increments of the mean depth


@pytest.mark.parametrize("j,i", [(0, 0), (140, 150), (57, 64)])
@pytest.mark.parametrize("value,status", [(np.nan, dgswe.DG_ENONFINITE), (-3.0e4, dgswe.DG_ENONPHYSICAL)])
def test_bad_state_is_reported(j, i, value, status):
    o, u = case(151, 141, 4, 11)
    bad = u.copy()
    bad[j, i, 0, 0] = value
    with dgswe.Solver(151, 141, 4, precision="fp32") as s:
        with pytest.raises(dgswe.DGError) as e:
            s.rhs(bad)
        assert e.value.status == status
        s.rhs(u)   # the status is cleared
