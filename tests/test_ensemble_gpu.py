"""Batched ensemble (one persistent launch per RK stage and degree for meshes of uneven
sizes and degrees): every member must evolve exactly as it does alone, and
match the FP64 oracle within the FP32 tolerance."""
import numpy as np
import pytest

import oracle as O
from paper_2303_11767_gb300 import dgswe, synth

pytestmark = pytest.mark.gpu

R, G, OMEGA = synth.EARTH_RADIUS, 9.80616, 7.292e-5
# (5, 3, 2) holds an odd number of values (405), so the degree-3 member after
# it must still start on a vector boundary
MEMBERS = [(5, 3, 2), (16, 8, 3), (20, 10, 1), (12, 7, 4), (24, 12, 2), (8, 4, 0), (40, 20, 4), (7, 5, 1)]


def _setup():
    states, dts, oracles = [], [], []
    for k, (nlon, nlat, p) in enumerate(MEMBERS):
        o = O.Oracle.sphere(nlon, nlat, p, R, G, OMEGA)
        u = o.project_tensor(synth.SmoothField(synth.ensemble_member_seed(k)).fields_grid)
        states.append(u)
        dts.append(o.max_dt(u, 0.1))
        oracles.append(o)
    return states, dts, oracles


def _rel(x, y):
    return max(np.linalg.norm(x[..., f, :] - y[..., f, :]) / np.linalg.norm(y[..., f, :]) for f in range(3))


@pytest.mark.parametrize("tile_rows", [4, 8])
def test_members_match_single_mesh_solver_and_oracle(tile_rows):
    states, dts, oracles = _setup()
    nsteps = 20
    nlon, nlat, deg = zip(*MEMBERS)
    with dgswe.Ensemble(nlon, nlat, deg, R, G, OMEGA) as e:
        e.set_option(dgswe.OPT_TILE_ROWS, tile_rows)
        e.set_option(dgswe.OPT_STEPS_PER_GRAPH, 8)
        for k, u in enumerate(states):
            e.set_state(k, u)
        e.set_dt(dts)
        m0 = [e.total_mass(k) for k in range(len(MEMBERS))]
        e.step(nsteps)
        assert e.stage_launches() == 3 * nsteps          # RK stages of all members
        for k, (nlon_k, nlat_k, p) in enumerate(MEMBERS):
            got = e.get_state(k)
            want = oracles[k].step(states[k], nsteps, dts[k], 3)
            assert _rel(got, want) < 1e-5, (k, _rel(got, want))
            assert abs(e.total_mass(k) / m0[k] - 1) < 1e-9
            if tile_rows == 8:                            # same tiles as the single-mesh kernel
                with dgswe.Solver(nlon_k, nlat_k, p, R, G, OMEGA, precision="fp32") as s:
                    s.set_state(states[k])
                    s.step(nsteps, dts[k])
                    alone = s.get_state()
                assert _rel(got, alone) < 1e-6, (k, _rel(got, alone))


def test_autotune_picks_a_valid_shape_and_restores_the_state():
    states, dts, _ = _setup()
    nlon, nlat, deg = zip(*MEMBERS)
    with dgswe.Ensemble(nlon, nlat, deg, R, G, OMEGA) as e:
        for k, u in enumerate(states):
            e.set_state(k, u)
        e.set_dt(dts)
        before = [e.get_state(k) for k in range(len(MEMBERS))]
        w, b, ms = e.autotune(trials=2)
        assert w in (4, 8) and 1 <= b <= 4 and ms > 0
        for k in range(len(MEMBERS)):
            np.testing.assert_array_equal(e.get_state(k), before[k])
        e.step(4)                                         # the chosen shape runs
        assert all(np.isfinite(e.get_state(k)).all() for k in range(len(MEMBERS)))


@pytest.mark.parametrize("degrees", [(3,), (2, 2), (0, 4), (4, 3, 2, 1, 0, 4)])
@pytest.mark.parametrize("nsteps", [1, 7])
def test_one_chain_of_launches_per_degree(degrees, nsteps):
    """No fork, one, and all five degrees; steps in graphs of 4 and the rest, on the caller's stream."""
    torch = pytest.importorskip("torch")
    mesh = [(12 + 3 * k, 9 + k) for k in range(len(degrees))]
    members = [(a, b, p) for (a, b), p in zip(mesh, degrees)]
    stream = torch.cuda.Stream()
    with dgswe.Ensemble(*zip(*members), R, G, OMEGA) as e:
        e.set_option(dgswe.OPT_STREAM, stream.cuda_stream)
        e.set_option(dgswe.OPT_STEPS_PER_GRAPH, 4)
        states, dts = [], []
        for k, (a, b, p) in enumerate(members):
            o = O.Oracle.sphere(a, b, p, R, G, OMEGA)
            u = o.project_tensor(synth.SmoothField(synth.ensemble_member_seed(k)).fields_grid)
            states.append((o, u))
            dts.append(o.max_dt(u, 0.1))
            e.set_state(k, u)
        e.set_dt(dts)
        e.step(nsteps)
        e.step(nsteps)
        assert e.stage_launches() == 6 * nsteps
        for k, (o, u) in enumerate(states):
            assert _rel(e.get_state(k), o.step(u, 2 * nsteps, dts[k], 3)) < 1e-5
