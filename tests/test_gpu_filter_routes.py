"""The 3D filter on grids on either side of the lines between its two kernels
(offset list up to 4096, 8192 or 32768 elements, staged layers above), with
extents that are no multiples of the staged kernel's 32 x 4 x 4 tiles and axes
thinner than the filter, against the oracle.  Tolerance: sums of terms of one sign,
1e-12 relative, as in the other filter tests."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from oracle import fe, filters
from workloads import rand_density, small_problem

pytestmark = pytest.mark.gpu

GRIDS = [((32, 16, 8), 3), ((36, 12, 12), 3), ((32, 16, 16), 3), ((36, 16, 16), 3), ((32, 32, 32), 3),
         ((36, 12, 80), 3), ((4, 132, 64), 3), ((132, 4, 64), 3), ((64, 36, 16), 3), ((132, 68, 4), 3)]


@pytest.mark.parametrize("nel,levels", GRIDS)
@pytest.mark.parametrize("rmin", [1.2, 1.5, 2.0, 2.2, 2.3, 2.5, 3.0])
def test_filter(nel, levels, rmin):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("cantilever3d", nelx=nel[0], nely=nel[1], nelz=nel[2], mg_levels=levels, rmin=rmin)
    H, Hs = filters.filter_matrix(fe.Grid.of(p), rmin)
    x = rand_density(p.nel, 3) * 10.0 ** np.random.default_rng(4).integers(-9, 3, p.nel)
    with Ctx(p, precision="mixed") as c:
        out = dev(np.zeros(p.nel))
        B.to_filter(c.ctx, B.TO_FILTER_DENSITY, dev(x), out)
        assert np.max(np.abs(host(out) * Hs / (H @ x) - 1.0)) <= 1e-12
        B.to_filter(c.ctx, B.TO_FILTER_SENS, dev(-x), out)
        assert np.max(np.abs(host(out) / -(H.T @ (x / Hs)) - 1.0)) <= 1e-12
