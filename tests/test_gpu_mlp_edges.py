"""The network kernels at the edges of their tiles: 16 samples per warp, 64 per
training CTA, 128 per forward CTA.  Bars as in test_gpu_mlp.py: BF16 operands
(8 significant bits, ~4e-3 each, a few layers deep) against FP64 give outputs
within 3e-2 of their RMS and gradients within 3e-2 in relative L2."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo
from paper_2204_10871_gb300 import irs
from gpu_common import params_pair, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 64, 65, 127, 129, 1000])
def test_forward_and_gradient_at_tile_edges(n):
    torch = require_gpu()
    rng = np.random.default_rng(n)
    theta = (mo.init_params(5) + rng.normal(0, 0.02, mo.N_PARAMS)).astype(np.float32)
    B = rng.normal(0, 2.0, (32, 2)).astype(np.float32)
    x = rng.uniform(-1, 1, (n, 2)).astype(np.float32)
    t = rng.normal(0, 1, (n, 8)).astype(np.float32)
    _, pl = params_pair(0.4, 0.1, 0.35, (-2.0, 2.0, -2.0, 2.0), 64, 16.0, method=irs.IRS_MLP)
    with irs.Plan(pl) as plan:
        irs.irs_mlp_params(plan.handle, theta, B)
        dx, dt = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
        y = irs.irs_mlp_forward(plan.handle, dx).cpu().numpy()
        grad, lsum = irs.irs_mlp_grad(plan.handle, dx, dt)
        plan.sync()
        grad, lsum = grad.cpu().numpy().astype(np.float64), float(lsum.cpu()[0])
    th, B, x, t = (v.astype(np.float64) for v in (theta, B, x, t))
    yo, _ = mo.forward(th, B, x)
    assert np.abs(y - yo).max() <= 3e-2 * np.sqrt(np.mean(yo ** 2))
    lo = mo.loss(th, B, x, t)
    assert abs(lsum / (n * 8) - lo) <= 1e-2 * lo
    go = mo.backward(th, B, x, t)
    assert np.linalg.norm(grad - go) <= 3e-2 * np.linalg.norm(go)
