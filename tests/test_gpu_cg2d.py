"""Mixed MGCG in 2D, whose K p is formed in double-float by a kernel of its own
(with the dot product p . q): solutions on the smallest grid, on grids around
its block size and on a long one, with and without springs, against the
float64 path of the same context data.

Both solve to rtol 1e-8 (the mixed path's pairs hold u to 2^-48, which puts a
floor of some 1e-10 under its true residual on the long grid: K's entries times
2^-48 of displacements 2,000 times the load); they are compared through the
compliance f . u, whose error is second order: 1e-8.  The float32 V-cycle is the float64
one up to rounding, so with an accurate K p the iteration counts stay within
a tenth (and 3) of float64's; a float32 K p takes up to twice as many."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from workloads import rand_density, small_problem

pytestmark = pytest.mark.gpu

GRIDS = [("mbb2d", 2, 2, 2), ("mbb2d", 30, 14, 2), ("cantilever2d", 34, 30, 2),
         ("inverter2d", 48, 24, 3), ("mbb2d", 640, 160, 6)]


@pytest.mark.parametrize("kind,nx,ny,levels", GRIDS)
def test_mixed_solve_2d(kind, nx, ny, levels):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem(kind, nelx=nx, nely=ny, mg_levels=levels)
    # smooth density with holes, as a design in progress has
    x, y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny)
    rho = 0.55 + 0.4 * np.cos(9.0 * x + 2.0) * np.cos(5.0 * y) + rand_density(p.nel, 4, -0.05, 0.05).reshape(ny, nx)
    out = {}
    for precision in ("fp64", "mixed"):
        with Ctx(p, precision=precision) as c:
            if p.springs:
                B.to_mesh_springs(c.ctx, [d for d, _ in p.springs], [k for _, k in p.springs])
            c.set_density(np.clip(rho, 1e-3, 1.0).reshape(-1))
            u = dev(np.zeros(p.ndof))
            it, rel, ok = B.to_mgcg_solve(c.ctx, 1e-8, 400, 0, u)
            assert ok and rel < 1e-8
            out[precision] = it, host(u)
    c64, cm = (p.f @ out[k][1] for k in ("fp64", "mixed"))
    assert abs(cm - c64) <= 1e-8 * abs(c64)
    assert not np.any(out["mixed"][1][p.fixed.astype(bool)])
    assert out["mixed"][0] <= 1.1 * out["fp64"][0] + 3
