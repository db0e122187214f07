"""dg_project_nodal on the GPU: more point values than one portion of its
workspace, ragged last blocks, bands, and the host path that it takes while the
solver's stream is being captured (in which dg_step stays refused).  Tolerance
1e-12 of the largest mode, as in test_parity_gpu.py."""
import numpy as np
import pytest

import oracle as O
from paper_2303_11767_gb300 import dgswe

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _values(nlon, nlat, p, seed=5):
    rng = np.random.default_rng(seed)
    v = rng.normal(size=(nlat, nlon, 3, p + 9, p + 9))
    v[:, :, 0] += 5960.0
    return v


@pytest.mark.parametrize("nlon,nlat,p", [(101, 91, 4), (7, 5, 0), (1, 3, 2), (13, 11, 1), (45, 33, 3)])
def test_projection_matches_oracle(nlon, nlat, p):
    v = _values(nlon, nlat, p)
    want = O.Oracle.sphere(nlon, nlat, p).project(v)
    with dgswe.Solver(nlon, nlat, p) as s:
        for _ in range(2):   # the workspace is kept
            got = s.project_nodal(v)
            assert np.abs(got - want.reshape(got.shape)).max() <= 1e-12 * np.abs(want).max()


def test_band_projection_equals_the_whole_meshs():
    v = _values(44, 14, 3)
    with dgswe.Solver(44, 14, 3) as s, dgswe.Solver.band(44, 14, 5, 11, 3) as b:
        assert np.array_equal(b.project_nodal(np.ascontiguousarray(v[5:11])), s.project_nodal(v)[5:11])


def test_while_the_stream_is_captured():
    v = _values(13, 11, 2)
    stream = torch.cuda.Stream()
    with dgswe.Solver(13, 11, 2) as s:
        s.set_option(dgswe.OPT_STREAM, stream.cuda_stream)
        want = s.project_nodal(v)
        s.set_state(want)
        x = torch.zeros(4, device="cuda")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            x += 1
            got = s.project_nodal(v)
            with pytest.raises(dgswe.DGError) as e:
                s.step(1, 1.0)
        assert e.value.status == dgswe.DG_ECUDA
        assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max()
        graph.replay()
        torch.cuda.synchronize()
        assert x.tolist() == [1.0] * 4
        s.step(1, 1.0)
