"""CG iterations replayed as one captured graph against the same iterations
launched kernel by kernel (which the profiler's timers ask for): same bits,
whatever the iteration limit, the start, the buffer and the density before (the
mixed 3D solves of these gray designs stagnate and escalate on the way)."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from workloads import rand_density, small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,kw,levels", [("mbb2d", dict(nelx=60, nely=20), 3),
                                            ("cantilever3d", dict(nelx=24, nely=8, nelz=16), 3)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_replayed_iterations_give_the_launched_ones(kind, kw, levels, precision):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem(kind, mg_levels=levels, **kw)
    with Ctx(p, precision=precision) as c:
        def solve(maxit, profiled, u0=None):
            u = dev(np.full(p.ndof, np.nan) if u0 is None else u0)
            B.to_profile_enable(c.ctx, profiled)
            it, rel, ok = B.to_mgcg_solve(c.ctx, 1e-8, maxit, 0 if u0 is None else 1, u)
            B.to_profile_enable(c.ctx, False)
            return it, rel, ok, host(u)

        for density in (40, 41, 42):     # the moduli alternate between two buffers
            c.set_density(rand_density(p.nel, density, 0.2, 1.0))
            for maxit in (1, 2, 3, 7, 200):
                a, b = solve(maxit, False), solve(maxit, True)
                assert a[:3] == b[:3] and np.array_equal(a[3], b[3])
            a, b = solve(200, False, 0.9 * a[3]), solve(200, True, 0.9 * a[3])
            assert a[:3] == b[:3] and np.array_equal(a[3], b[3])
