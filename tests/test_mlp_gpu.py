"""The network kernels at the edges of their ranges against the FP64 reference:
layer sizes that the fused kernels take (up to 64 - 128 - 128 - 16) and that the
layer-by-layer ones take, batches around the 32-sample blocks, and one Adam step
(first step: w - lr g / (|g| + eps)).  Tolerances as in test_learned_gpu.py: 1e-5
of the largest output, 1e-4 of the largest gradient; parameters 1e-4 of the step
where the gradient is 1000 eps or more, the step's size elsewhere."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_2303_11767_gb300 import dgswe

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nin,H,nout,batch", [(60, 128, 12, 1), (60, 128, 12, 31), (60, 128, 12, 33), (60, 128, 12, 4096),
                                              (60, 128, 12, 8192), (64, 128, 16, 97), (1, 128, 1, 64), (65, 128, 12, 40),
                                              (20, 48, 7, 300), (60, 128, 17, 64)])
def test_network_matches_fp64_reference(nin, H, nout, batch):
    rng = np.random.default_rng(nin + batch)
    mlp = dgswe.MLP(nin, H, nout, seed=3)
    norm = (rng.normal(size=nin).astype(np.float32), (1 + rng.random(nin)).astype(np.float32),
            rng.normal(size=nout).astype(np.float32), (1 + rng.random(nout)).astype(np.float32))
    mlp.set_normalization(*norm)
    p = mlp.get_params()
    p += rng.normal(scale=0.01, size=p.shape).astype(np.float32)   # biases too
    mlp.set_params(p)
    x = (rng.normal(size=(batch, nin)) * norm[1] + norm[0]).astype(np.float32)
    t = (rng.normal(size=(batch, nout)) * norm[3] + norm[2]).astype(np.float32)
    dx, dt = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    y = torch.empty(batch, nout, dtype=torch.float32, device="cuda")
    mlp.forward(dx, y)
    nrm = tuple(a.astype(np.float64) for a in norm)
    want_y, _ = M.forward(p.astype(np.float64), x, nrm, nin, H, nout)
    assert np.abs(y.cpu().numpy() - want_y).max() < 1e-5 * np.abs(want_y).max()
    g, loss = mlp.gradients(dx, dt)
    want_loss, want_g = M.loss_and_grad(p.astype(np.float64), x, t, nrm, nin, H, nout)
    assert abs(loss / want_loss - 1) < 1e-5
    assert np.abs(g - want_g).max() < 1e-4 * np.abs(want_g).max()
    assert abs(mlp.train_step(dx, dt, 1e-3) / want_loss - 1) < 1e-5
    step = mlp.get_params().astype(np.float64) - p
    want_step = -1e-3 * want_g / (np.abs(want_g) + 1e-8)
    # FP32 rounding of the parameter, and the gradient's error where it is comparable with eps
    err, ulp = np.abs(step - want_step), 2.0 ** -23 * np.maximum(np.abs(p), 1e-3)
    firm = np.abs(want_g) > 1e-5 + 1e-3 * np.abs(want_g).max()
    assert np.all(err[firm] <= 1e-4 * 1e-3 + ulp[firm])
    assert np.all(np.abs(step) <= 1e-3 * 1.0001 + ulp)
    mlp.forward(dx, y)   # the weights of the next pass are the new ones
    want_y, _ = M.forward(mlp.get_params().astype(np.float64), x, nrm, nin, H, nout)
    assert np.abs(y.cpu().numpy() - want_y).max() < 1e-5 * np.abs(want_y).max()
