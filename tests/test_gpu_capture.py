"""Maps captured into a caller's CUDA graph: the kernels of a map are chained
with programmatic launches, which a capture has to take over; replays give the
counts of a plain call, also after the lens values changed in place."""
import numpy as np
import pytest

import oracle
from paper_2204_10871_gb300 import irs
from gpu_common import lenses_for, params_pair, require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method,n", [(irs.IRS_INTERP, 400), (irs.IRS_INTERP, 0), (irs.IRS_BRUTE, 300)])
def test_captured_map_equals_a_plain_call(method, n):
    torch = require_gpu()
    args = (0.3, 0.0, 0.3, (-2.0, 2.0, -2.0, 2.0), 64, 9.0)
    po, pl = params_pair(*args, method=method, n_star=max(n, 50))
    fields = [to_dev(torch, *lenses_for(oracle.size(po), n, shape="uniform", seed=k, kappa_star=args[0]))
              for k in (1, 2)]
    with irs.Plan(pl) as plan:
        want = []
        for xy, m in fields:
            counts, mag = plan.make_map(xy, m)
            plan.sync()
            want.append((counts.cpu().numpy().copy(), mag.cpu().numpy().copy()))
        xy, m = fields[0][0].clone(), fields[0][1].clone()
        counts = torch.empty((64, 64), dtype=torch.uint32, device="cuda")
        mag = torch.empty((64, 64), dtype=torch.float32, device="cuda")
        side = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=side):
            plan.make_map(xy, m, counts, mag, stream=side)
        for k in (0, 1, 0):
            xy.copy_(fields[k][0])
            m.copy_(fields[k][1])
            graph.replay()
            torch.cuda.synchronize()
            assert np.array_equal(counts.cpu().numpy(), want[k][0])
            assert np.array_equal(mag.cpu().numpy(), want[k][1])
        plan.sync()
