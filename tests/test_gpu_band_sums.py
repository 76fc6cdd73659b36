"""Bands of lattice rows add up to the whole map for every kernel of the ray
pass, wherever the bands begin: a ray's rounding must not depend on the band it
is shot in.  About 1e9 rays, so that a difference in the last bit of a
deflection moves some of them over a pixel edge."""
import pytest

from paper_2204_10871_gb300 import irs
from gpu_common import lenses_for, params_pair, require_gpu, to_dev
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 2, 3, 6, 16])
def test_bands_of_any_start_add_up(variant):
    torch = require_gpu()
    args = (0.3, 0.0, 0.3, (-2.5, 2.5, -2.5, 2.5), 128, 2000.0)
    po, pl = params_pair(*args, method=irs.IRS_INTERP, kernel_variant=variant)
    qo = oracle.size(po)
    xy, m = lenses_for(qo, 150, shape="uniform", seed=8, kappa_star=args[0])
    dxy, dm = to_dev(torch, xy, m)
    with irs.Plan(pl) as plan:
        full, _ = plan.make_map(dxy, dm)
        acc = torch.zeros_like(full)
        ny = int(plan.info.n_rays_y)
        for r0 in range(0, ny, 61):
            irs.irs_make_map_rows(plan.handle, dxy, dm, r0, min(ny, r0 + 61), acc)
        plan.sync()
    diff = (full.view(torch.int32).long() - acc.view(torch.int32).long()).abs().sum()
    assert int(diff) == 0
