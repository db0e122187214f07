"""The CFL step's wave-speed maximum (csrc/dg_kernels.cuh, speed_bound_kernel and
max_speed_kernel) against the oracle on states where its FP32 bounds matter:
rough states whose modes cancel, a fluid at rest (every element ties), a single
fast element, large offsets between the fields, and bad points anywhere."""
import numpy as np
import pytest

import oracle as O
from paper_2303_11767_gb300 import dgswe

pytestmark = pytest.mark.gpu

R, G, OMEGA = 6.37122e6, 9.80616, 7.292e-5


def _state(kind, nlon, nlat, p, rng):
    n2 = (p + 1) ** 2
    u = np.zeros((nlat, nlon, 3, n2))
    u[..., 0, 0] = 2.0 * 5960.0
    if kind == "rest":
        return u
    if kind == "rough":      # modes as large as the depth allows
        u[..., 0, 1:] = rng.normal(size=u[..., 0, 1:].shape) * 500.0 / n2
        u[..., 1:, :] = rng.normal(size=u[..., 1:, :].shape) * 2.0e5
    elif kind == "one":
        u[..., 1:, :] = rng.normal(size=u[..., 1:, :].shape)
        u[rng.integers(nlat), rng.integers(nlon), 1, 0] = 3.0e6
    elif kind == "shallow":  # depths down to a millimetre, speeds dominated by u
        u[..., 0, 0] = 2.0 * 10.0 ** rng.uniform(-3, 3, size=u.shape[:2])
        u[..., 1:, :] = rng.normal(size=u[..., 1:, :].shape) * 0.1
    elif kind == "close":    # all elements within 1e-6 of each other
        u[..., 0, 0] *= 1 + 1e-6 * rng.random(u.shape[:2])
    return u


@pytest.mark.parametrize("kind", ["rest", "rough", "one", "shallow", "close"])
@pytest.mark.parametrize("nlon,nlat,p", [(37, 21, 0), (33, 19, 1), (29, 23, 2), (31, 18, 3), (27, 17, 4), (5, 3, 4), (401, 247, 0)])
def test_max_dt_matches_oracle(nlon, nlat, p, kind):
    u = _state(kind, nlon, nlat, p, np.random.default_rng(nlon + p))
    want = O.Oracle.sphere(nlon, nlat, p, R, G, OMEGA).max_dt(u, 0.1)
    with dgswe.Solver(nlon, nlat, p, precision="fp64") as s:
        s.set_state(u)
        if want < 0:         # the oracle's answer for a depth that is not positive
            with pytest.raises(dgswe.DGError) as e:
                s.max_dt(0.1)
            assert e.value.status == dgswe.DG_ENONPHYSICAL
        else:
            assert abs(s.max_dt(0.1) / want - 1) < 1e-12
    if kind not in ("shallow",) and want > 0:
        with dgswe.Solver(nlon, nlat, p, precision="fp32") as s:
            s.set_state(u)
            assert abs(s.max_dt(0.1) / want - 1) < 1e-5


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("j,i", [(0, 0), (16, 26), (9, 13)])
def test_bad_depth_is_reported(j, i, prec):
    u = _state("rough", 27, 17, 4, np.random.default_rng(1))
    u[j, i, 0, 0] = -1.0
    with dgswe.Solver(27, 17, 4, precision=prec) as s:
        s.set_state(u)
        with pytest.raises(dgswe.DGError) as e:
            s.max_dt(0.1)
        assert e.value.status == dgswe.DG_ENONPHYSICAL


@pytest.mark.parametrize("p", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("h,u,deep", [(1e-27, 500.0, 1000.0), (1e-27, 500.0, 1e-22), (1e-40, 300.0, 10.0), (1e-33, 4e-4, 1e-30)])
def test_thin_fast_element(p, h, u, deep):
    """One element whose depth and momentum, or the momentum's square, lie below
    FP32's range, faster than the others."""
    nlon, nlat = (401, 247) if p == 0 else (23, 17)
    s = np.zeros((nlat, nlon, 3, (p + 1) ** 2))
    s[..., 0, 0] = 2.0 * deep
    s[5, 7, 0, 0], s[5, 7, 1, 0] = 2.0 * h, 2.0 * h * u
    want = O.Oracle.sphere(nlon, nlat, p, R, G, OMEGA).max_dt(s, 0.1)
    with dgswe.Solver(nlon, nlat, p, precision="fp64") as solver:
        solver.set_state(s)
        assert abs(solver.max_dt(0.1) / want - 1) < 1e-12
