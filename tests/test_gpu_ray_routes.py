"""The interpolated ray pass against the chosen-ray path, ray by ray: both run
the same arithmetic, so the pixels that irs_shoot_rays reports for every ray of
the lattice must add up to the count map exactly, whatever route the ray pass
takes for a cell -- last strips of few columns, cells cut into several work
items or several binning boxes, rays outside the box, row bands that start and
end inside a row group, blocks of more lenses than the shared buffer holds.
Both sides are integers from identical roundings: the tolerance is zero."""
import numpy as np
import pytest

from paper_2204_10871_gb300 import irs
from gpu_common import lenses_for, params_pair, require_gpu, to_dev
import oracle

pytestmark = pytest.mark.gpu

# (kappa_*, kappa_s, gamma, source region, pixels, rays/px, lenses, plane, options)
ROUTES = {
    "one row of cells per part": ((0.3, 0.0, 0.3, (-2.5, 2.5, -2.5, 2.5), 64, 4.0), 40, 0, {}),
    "strips of 1 to 31 columns": ((0.3, 0.1, 0.25, (-2, 3, -2.5, 2.1), (101, 93), 4.0), 900, 0, {"cell_mult": 0.7}),
    "four rays per cell side": ((0.4, 0.0, 0.1, (-1, 1, -1, 1), 40, 1.0), 20000, 0, {"kernel_variant": 16}),
    "several boxes per cell": ((0.3, 0.0, 0.2, (-3, 3, -3, 3), (600, 580), 1.0), 150, 0, {"kernel_variant": 14}),
    "every ray its own pixel": ((0.2, 0.0, -0.2, (-1, 1, -1, 1), (700, 900), 0.25), 60, 0, {"kernel_variant": 1}),
    "shared reciprocals": ((0.3, 0.0, 0.3, (-2, 2, -2, 2), 64, 9.0), 200, 0, {"kernel_variant": 2}),
    "circle off the origin": ((0.35, 0.1, 0.25, (-1.5, 2.5, -2.7, 1.3), (61, 67), 6.0), 700, 1, {"kernel_variant": 9}),
    # most units of these planes cannot reach the map and are left out by bound
    "a wide border": ((0.6, 0.0, 0.1, (-0.5, 0.5, -0.4, 0.4), (40, 32), 9.0), 900, 0, {"cell_mult": 0.7}),
    "few heavy lenses": ((0.1, 0.0, 0.1, (-1.0, 1.0, -1.0, 1.0), 60, 16.0), 5, 0, {}),
    "over-focused": ((0.9, 0.5, 0.15, (-1.0, 1.0, -0.8, 0.8), (50, 40), 9.0), 800, 0, {"kernel_variant": 16}),
    "no lenses": ((0.2, 0.1, 0.2, (-1.5, 1.5, -1.5, 1.5), 48, 10.25), 0, 0, {"n_star": 60}),
}


def _counts_of(pix, shape):
    pix = pix[pix >= 0]
    return np.bincount(pix, minlength=shape[0] * shape[1]).reshape(shape)


def _check(torch, pl, plan, dxy, dm):
    info = plan.info
    counts, _ = plan.make_map(dxy, dm)
    _, pix = plan.shoot_rays(dxy, dm, torch.arange(int(info.n_rays), device="cuda"))
    plan.sync()
    pix = pix.cpu().numpy()
    shape = (pl.npix_y, pl.npix_x)
    assert np.array_equal(counts.cpu().numpy().astype(np.int64), _counts_of(pix, shape))
    nrx, nry = int(info.n_rays_x), int(info.n_rays_y)
    for r0, r1 in ((1, 2), (nry // 3, nry // 3 + 13), (nry - 9, nry)):
        counts.zero_()
        irs.irs_make_map_rows(plan.handle, dxy, dm, r0, r1, counts)
        plan.sync()
        assert np.array_equal(counts.cpu().numpy().astype(np.int64), _counts_of(pix[r0 * nrx:r1 * nrx], shape)), (r0, r1)


@pytest.mark.parametrize("route", sorted(ROUTES))
def test_map_equals_its_rays(route):
    torch = require_gpu()
    args, n, plane, kw = ROUTES[route]
    po, pl = params_pair(*args, plane=plane, method=irs.IRS_INTERP, **{"n_star": n, **kw})
    qo = oracle.size(po)
    xy, m = lenses_for(qo, n, shape="uniform", seed=7, kappa_star=args[0], plane=plane)
    with irs.Plan(pl) as plan:
        _check(torch, pl, plan, *to_dev(torch, xy, m))


def test_a_block_fuller_than_the_shared_buffer():
    """600 lenses within 0.05 theta_E of each other: their block's lenses are
    read from memory, every other block's from the shared buffer."""
    torch = require_gpu()
    args = (0.3, 0.0, 0.3, (-2.0, 2.0, -2.0, 2.0), 48, 9.0)
    po, pl = params_pair(*args, method=irs.IRS_INTERP, n_star=900)
    qo = oracle.size(po)
    xy, m = lenses_for(qo, 900, shape="equal", seed=3, kappa_star=args[0])
    xy[:600] = 0.02 + np.random.default_rng(1).uniform(-0.025, 0.025, (600, 2))
    with irs.Plan(pl) as plan:
        _check(torch, pl, plan, *to_dev(torch, xy, m))


@pytest.mark.parametrize("variant,n", [(0, 700), (1, 40), (2, 257), (11, 256), (14, 9), (15, 513), (0, 0)])
def test_brute_map_equals_its_rays(variant, n):
    """The brute force: every ray of the lattice (served tile by tile) adds up
    to the map, and a few rays asked for alone (each with its own lenses'
    conversion) come out with the same beta and pixel, whatever rows share
    their reciprocals."""
    torch = require_gpu()
    args = (0.3, 0.1, 0.25, (-2, 3, -2.5, 2.1), (37, 29), 4.0)
    po, pl = params_pair(*args, method=irs.IRS_BRUTE, n_star=n, kernel_variant=variant)
    qo = oracle.size(po)
    xy, m = lenses_for(qo, n, shape="uniform", seed=5, kappa_star=args[0])
    dxy, dm = to_dev(torch, xy, m)
    with irs.Plan(pl) as plan:
        counts, _ = plan.make_map(dxy, dm)
        idx = torch.arange(int(plan.info.n_rays), device="cuda")
        beta, pix = plan.shoot_rays(dxy, dm, idx)
        some = torch.from_numpy(np.random.default_rng(2).integers(0, idx.numel(), 95)).cuda()
        b1, p1 = plan.shoot_rays(dxy, dm, torch.cat([some, torch.tensor([-1, idx.numel()], device="cuda")]))
        plan.sync()
    shape = (pl.npix_y, pl.npix_x)
    assert np.array_equal(counts.cpu().numpy().astype(np.int64), _counts_of(pix.cpu().numpy(), shape))
    assert torch.equal(b1[:95], beta[some]) and torch.equal(p1[:95], pix[some])
    assert torch.isnan(b1[95:]).all() and (p1[95:] == -1).all()


@pytest.mark.parametrize("variant", [0, 2, 11])
def test_brute_bands_equal_their_rays(variant):
    """Bands that start and end inside a tile or inside one warp's rows, down
    to a single row, and the last, ragged tile row: warps without a row of the
    band sum nothing."""
    torch = require_gpu()
    args = (0.3, 0.1, 0.25, (-2, 3, -2.5, 2.1), (37, 29), 4.0)
    po, pl = params_pair(*args, method=irs.IRS_BRUTE, n_star=300, kernel_variant=variant)
    xy, m = lenses_for(oracle.size(po), 300, shape="uniform", seed=5, kappa_star=args[0])
    dxy, dm = to_dev(torch, xy, m)
    with irs.Plan(pl) as plan:
        nrx, nry = int(plan.info.n_rays_x), int(plan.info.n_rays_y)
        counts, _ = plan.make_map(dxy, dm)
        _, pix = plan.shoot_rays(dxy, dm, torch.arange(nrx * nry, device="cuda"))
        plan.sync()
        pix = pix.cpu().numpy()
        for r0, r1 in ((0, 1), (15, 17), (48, 112), (63, 64), (70, 71), (nry - 1, nry), (nry - 70, nry)):
            counts.zero_()
            irs.irs_make_map_rows(plan.handle, dxy, dm, r0, r1, counts)
            plan.sync()
            want = _counts_of(pix[r0 * nrx:r1 * nrx], (pl.npix_y, pl.npix_x))
            assert np.array_equal(counts.cpu().numpy().astype(np.int64), want), (r0, r1)


def test_masses_of_both_signs():
    """Lens masses may have either sign; the bound that leaves units out takes
    their magnitudes."""
    torch = require_gpu()
    args = (0.4, 0.0, 0.2, (-0.8, 0.8, -0.7, 0.7), (48, 42), 9.0)
    po, pl = params_pair(*args, method=irs.IRS_INTERP, n_star=700)
    xy, m = lenses_for(oracle.size(po), 700, shape="salpeter", seed=9, kappa_star=args[0])
    m[::3] *= -1.0
    with irs.Plan(pl) as plan:
        _check(torch, pl, plan, *to_dev(torch, xy, m))
