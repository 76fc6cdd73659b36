"""Chosen rays of the brute force in one call and in pieces: a call that asks for
many rays per tile may serve them tile by tile, calls that ask for a few ray by
ray.  The same bits either way, and the one call is not the slower."""
import numpy as np
import pytest

from paper_2204_10871_gb300 import irs
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _ms(torch, calls):
    best = np.inf
    for _ in range(3):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for c in calls:
            c()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


# pixels per side, lenses, rays per tile: a lattice of many tiles with few lenses,
# where passing the indices once per tile would cost more than the lenses, and few tiles
@pytest.mark.parametrize("npix,n,per_tile,variant", [(1024, 100, 64, 0), (512, 3, 24, 0), (128, 1000, 64, 0),
                                                     (128, 1000, 64, 14), (128, 0, 24, 0)])
def test_one_call_equals_its_pieces(npix, n, per_tile, variant):
    """A quarter is allowed for the spread of two timings and for the model's."""
    torch = require_gpu()
    p = irs.make_params(0.1, 0.0, 0.0, (-2.0, 2.0, -2.0, 2.0), npix, 16.0, border=0.5, method=irs.IRS_BRUTE, n_star=10,
                        kernel_variant=variant)
    with irs.Plan(p) as plan:
        i = plan.info
        tiles = -(-int(i.n_rays_x) // 32) * -(-int(i.n_rays_y) // 64)
        rng = np.random.default_rng(npix + n)
        xy = torch.from_numpy(np.stack([rng.uniform(i.lens_x0, i.lens_x1, n), rng.uniform(i.lens_y0, i.lens_y1, n)], 1)).cuda()
        m = torch.ones(n, dtype=torch.float64, device="cuda")
        k = per_tile * tiles
        idx = torch.from_numpy(rng.integers(0, i.n_rays, k)).cuda()
        out = [(torch.zeros((k, 2), dtype=torch.float64, device="cuda"),
                torch.full((k,), -7, dtype=torch.int64, device="cuda")) for _ in range(2)]

        def shoot(dst, a, b):
            irs.irs_shoot_rays(plan.handle, xy, m, idx[a:b], dst[0][a:b], dst[1][a:b])

        step = 8 * tiles - 1
        pieces = [lambda a=a: shoot(out[1], a, min(k, a + step)) for a in range(0, k, step)]
        whole = [lambda: shoot(out[0], 0, k)]
        _ms(torch, whole), _ms(torch, pieces)
        one, many = _ms(torch, whole), _ms(torch, pieces)
        plan.sync()
    print(f"{tiles} tiles, {k} rays, {n} lenses: one call {one:.3f} ms, {len(pieces)} pieces {many:.3f} ms")
    assert torch.equal(out[0][0].view(torch.int64), out[1][0].view(torch.int64)) and torch.equal(out[0][1], out[1][1])
    assert one <= 1.25 * many
