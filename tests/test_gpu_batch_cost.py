"""A batch of maps with few cells: the shared ray pass cuts their cells into
shares, as a single map's does."""
import numpy as np
import pytest

from paper_2204_10871_gb300 import irs
from gpu_common import lenses_for, params_pair, require_gpu, to_dev
import oracle

pytestmark = pytest.mark.gpu


def _ms(torch, call):
    call()
    torch.cuda.synchronize()
    best = np.inf
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(10):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 10)
    return best


# (kappa_*, kappa_s, gamma, source region, pixels, rays/px), lenses: 250, 160 and 960 cells
@pytest.mark.parametrize("args,n", [((0.3, 0.0, 0.3, (-2.5, 2.5, -2.5, 2.5), 128, 25.0), 150),
                                    ((0.05, 0.0, 0.2, (-8.0, 8.0, -8.0, 8.0), 700, 100.0), 60),
                                    ((0.55, 0.25, 0.15, (-1.5, 1.5, -1.5, 1.5), 64, 25.0), 900)])
def test_a_batch_of_one_costs_what_the_map_costs(args, n):
    """The same kernels in a graph: no more than 1.25 times the single call (a
    whole cell per work item took 1.3 to 1.7 times), and the same counts."""
    torch = require_gpu()
    po, pl = params_pair(*args, method=irs.IRS_INTERP, n_star=n)
    dxy, dm = to_dev(torch, *lenses_for(oracle.size(po), n, shape="uniform", seed=41, kappa_star=args[0]))
    with irs.Plan(pl) as plan:
        single, _ = plan.make_map(dxy, dm, with_mag=False)
        batch = torch.zeros_like(single)
        alone = _ms(torch, lambda: irs.irs_make_map(plan.handle, dxy, dm, single))
        graph = _ms(torch, lambda: irs.irs_make_maps_batched([plan.handle], [dxy], [dm], [batch]))
        plan.sync()
        assert torch.equal(single, batch)
    print(f"single {alone:.4f} ms, batch of one {graph:.4f} ms")
    assert graph <= 1.25 * alone
