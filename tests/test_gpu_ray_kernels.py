"""Every kernel of the interpolated ray pass, alone and in a batch, against the
chosen rays (a kernel of their own, which the deflection tests compare with the
oracle): integers from identical roundings, so the tolerance is zero."""
import numpy as np
import pytest

from paper_2204_10871_gb300 import irs
from gpu_common import lenses_for, params_pair, require_gpu, to_dev
from test_gpu_ray_routes import _check, _counts_of
import oracle

pytestmark = pytest.mark.gpu

KERNELS = [0, 1, 2, 3, 5, 9, 11, 14, 15, 16]  # variants with a kernel of their own


@pytest.mark.parametrize("mult", [0.0, 0.7])
@pytest.mark.parametrize("variant", KERNELS)
def test_map_bands_and_batch_equal_the_rays(variant, mult):
    torch = require_gpu()
    args = (0.35, 0.05, 0.25, (-2.0, 2.5, -1.9, 2.3), (77, 71), 16.0)
    po, pl = params_pair(*args, method=irs.IRS_INTERP, n_star=600, kernel_variant=variant, cell_mult=mult)
    qo = oracle.size(po)
    dxy, dm = to_dev(torch, *lenses_for(qo, 600, shape="salpeter", seed=11, kappa_star=args[0]))
    with irs.Plan(pl) as plan:
        _check(torch, pl, plan, dxy, dm)
        single, _ = plan.make_map(dxy, dm)
        batch = torch.zeros_like(single)
        irs.irs_make_maps_batched([plan.handle], [dxy], [dm], [batch])
        torch.cuda.synchronize()
        plan.sync()
        assert torch.equal(single, batch)


def test_a_band_of_the_high_resolution_lattice():
    """Seven rows, begun off a pair of rows, of the 9.6e10-ray lattice (1e6
    lenses, 10000^2 pixels) at its tuned setting: 6.5e6 rays."""
    torch = require_gpu()
    args = (0.35, 0.15, 0.4, (-12.5, 12.5, -12.5, 12.5), 10000, 40.0)
    po, pl = params_pair(*args, method=irs.IRS_INTERP, n_star=1000000, cell_mult=0.72, kernel_variant=16)
    qo = oracle.size(po)
    dxy, dm = to_dev(torch, *lenses_for(qo, 1000000, shape="uniform", seed=3, kappa_star=args[0]))
    with irs.Plan(pl) as plan:
        nrx = int(plan.info.n_rays_x)
        r0 = int(plan.info.n_rays_y) // 2 | 1
        counts = torch.zeros((10000, 10000), dtype=torch.uint32, device="cuda")
        irs.irs_make_map_rows(plan.handle, dxy, dm, r0, r0 + 7, counts)
        _, pix = plan.shoot_rays(dxy, dm, torch.arange(r0 * nrx, (r0 + 7) * nrx, device="cuda"))
        plan.sync()
    want = _counts_of(pix.cpu().numpy(), (10000, 10000))
    assert want.sum() > 100000
    assert np.array_equal(counts.cpu().numpy().astype(np.int64), want)
