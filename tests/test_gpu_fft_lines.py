"""The far field's line FFTs at the edges of their launch shapes: lines of a few
elements, many lines per CTA and few, one line per CTA, up to the longest line
(9216 elements, all of a CTA's shared memory) as rows and as columns.  Sampled
deflections against the FP64 oracle, within the deflection bar."""
import pytest

from gpu_common import DEFLECTION_TOL, require_gpu
from test_gpu_interp import sampled_check

pytestmark = pytest.mark.gpu

WIDE = (-10.0, 10.0, -10.0, 10.0)
# (kappa_*, kappa_s, gamma, source, pixels, rays/px), lenses, cell multiplier, cells of the longer side
LINES = {
    "a few cells": ((0.2, 0.0, 0.1, (-0.5, 0.5, -0.4, 0.4), 16, 9.0), 30, 2.0, 2),
    "tens of cells": ((0.3, 0.1, 0.25, (-2.0, 3.0, -2.5, 2.1), (101, 93), 4.0), 900, 0.5, 20),
    "hundreds of cells": ((0.4, 0.0, 0.3, (-5.0, 5.0, -5.0, 5.0), 300, 9.0), 20000, 0.7, 200),
    "the longest rows": ((0.45, 0.0, 0.45, WIDE, 1000, 6.0), 60000, 0.17, 4375),
    "the longest columns": ((0.45, 0.0, -0.45, WIDE, 1000, 6.0), 60000, 0.17, 4375),
}


@pytest.mark.parametrize("lines", sorted(LINES))
def test_sampled_deflections(lines):
    cfg, n, mult, cells = LINES[lines]
    err, far, _, _, info = sampled_check(require_gpu(), cfg, n, "uniform", seed=4, cell_mult=mult)
    assert max(info.ncell_x, info.ncell_y) >= cells
    assert err[far].max() <= DEFLECTION_TOL, f"max deflection error {err[far].max():.3e}"
