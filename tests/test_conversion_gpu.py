"""The API's FP64 state to and from the FP32 (base, low) pair (to_internal_kernel,
to_api_kernel): bit for bit what the definition gives, for magnitudes from
subnormal to large, zeros of both signs and several blocks with a ragged end."""
import numpy as np
import pytest

from paper_2303_11767_gb300 import dgswe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nlon,nlat,p", [(37, 21, 4), (61, 33, 1), (5, 3, 0), (16, 8, 3), (29, 17, 2)])
def test_round_trip_is_the_definition(nlon, nlat, p):
    rng = np.random.default_rng(p)
    n2 = (p + 1) ** 2
    u = rng.normal(size=(nlat, nlon, 3, n2)) * 10.0 ** rng.uniform(-44, 30, size=(nlat, nlon, 3, n2))
    u[rng.random(u.shape) < 0.1] = 0.0
    u[rng.random(u.shape) < 0.05] = -0.0
    u[..., 0, 0] = 2.0 * (5960.0 + rng.normal(size=(nlat, nlon)))
    href = 0.0
    for x in u[..., 0, 0].reshape(-1):   # the mean depth, summed in element order
        href += x
    href = 0.5 * href / (nlon * nlat)
    v = u.copy()
    v[..., 0, 0] -= 2.0 * href
    with np.errstate(over="ignore"):
        hi = v.astype(np.float32)
        lo = (v - hi.astype(np.float64)).astype(np.float32)
    want = hi.astype(np.float64) + lo.astype(np.float64)
    want[..., 0, 0] += 2.0 * href
    with dgswe.Solver(nlon, nlat, p, precision="fp32") as s:
        s.set_state(u)
        got = s.get_state()
    assert np.array_equal(got, want)
