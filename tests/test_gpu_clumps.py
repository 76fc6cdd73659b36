"""Blocks of more near lenses than the ray pass's shared buffer, which is sized for
a uniform field: the clump of a map with all its lenses in half of the plane."""
import numpy as np
import pytest

from paper_2204_10871_gb300 import irs
from gpu_common import lenses_for, params_pair, require_gpu, to_dev
from test_gpu_ray_routes import _check
import oracle

pytestmark = pytest.mark.gpu

# no border, so that every ray is near the map
ARGS = (0.3, 0.0, 0.0, (-5.0, 5.0, -5.0, 5.0), 500, 400.0)


def _ms(torch, plan, dxy, dm):
    counts, _ = plan.make_map(dxy, dm)
    plan.sync()
    best = np.inf
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(4):
            irs.irs_make_map(plan.handle, dxy, dm, counts)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 4)
    return best


def test_full_blocks_cost_what_their_pairs_cost():
    """The same pair terms, in blocks of 300 lenses that the buffer holds and, with
    every lens in the left half, in blocks of 600 that it does not.  A warp's
    turn through the buffer is about 50 instructions for at least 25 lenses of 45
    each, 4 %; a quarter is allowed (fetched by every thread, the pairs of full
    blocks took twice as long).  14,000 cells, so that the last wave of work
    items (912 at a time, half of them heavy) is a small part."""
    torch = require_gpu()
    n = 480000
    po, pl = params_pair(*ARGS, border=0.0, method=irs.IRS_INTERP, n_star=n, cell_mult=5.77, kernel_variant=16)
    qo = oracle.size(po)
    xy, m = lenses_for(qo, n, shape="equal", seed=4, kappa_star=ARGS[0])
    half = xy.copy()
    half[:, 0] = qo.a1 + 0.5 * (xy[:, 0] - qo.a1)
    with irs.Plan(pl) as plan:
        even = _ms(torch, plan, *to_dev(torch, xy, m))
        clumped = _ms(torch, plan, *to_dev(torch, half, m))
    print(f"even {even:.3f} ms, clumped {clumped:.3f} ms")
    assert clumped <= 1.25 * even


@pytest.mark.parametrize("variant,mult", [(16, 0.7), (2, 0.0), (9, 1.5)])
@pytest.mark.parametrize("clump", [15, 33, 130, 900])
@pytest.mark.parametrize("at", [(0.02, 0.01), (0.8, 0.75)])
def test_full_blocks_equal_their_rays(clump, at, variant, mult):
    """A clump on the map, and one in the border, where most of its units are
    left out by their bound: the map and bands of rows against the chosen rays,
    which walk the lists in memory."""
    torch = require_gpu()
    args = (0.4, 0.0, 0.2, (-0.8, 0.8, -0.7, 0.7), (48, 42), 9.0)
    n = 900 + clump
    po, pl = params_pair(*args, method=irs.IRS_INTERP, n_star=n, kernel_variant=variant, cell_mult=mult)
    qo = oracle.size(po)
    xy, m = lenses_for(qo, n, shape="uniform", seed=3, kappa_star=args[0])
    centre = np.array([at[0] * qo.ix / 2, at[1] * qo.iy / 2])
    xy[:clump] = centre + np.random.default_rng(1).uniform(-0.02, 0.02, (clump, 2))
    with irs.Plan(pl) as plan:
        _check(torch, pl, plan, *to_dev(torch, xy, m))
