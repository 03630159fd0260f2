"""to_vcycle takes any right-hand side.  What it holds on fixed DOFs reaches no
free DOF (the operators are masked) and is smoothed twice by the identity rows
there, omega (2 - omega) r; repeated calls, and calls with other buffers, give
the same bits (the mixed cycle replays a captured graph)."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,kw,levels", [("mbb2d", dict(nelx=12, nely=4), 2),
                                            ("cantilever3d", dict(nelx=24, nely=8, nelz=16), 3),
                                            ("bridge3d", dict(nelx=32, nely=16, nelz=16), 4)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_fixed_dofs_of_the_input(kind, kw, levels, precision):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem(kind, mg_levels=levels, **kw)
    fixed = p.fixed.astype(bool)
    r = rand_vector(p.ndof, 31)
    assert np.any(r[fixed])
    clean = np.where(fixed, 0.0, r)
    with Ctx(p, precision=precision) as c:
        c.set_density(rand_density(p.nel, 30, 0.05, 1.0))

        def cycle(x):
            z = dev(np.full(p.ndof, np.nan))
            B.to_vcycle(c.ctx, dev(x), z)
            return host(z)

        z, z0, again = cycle(r), cycle(clean), cycle(r)
        poisoned = cycle(np.where(fixed, np.nan, r))
    assert np.array_equal(z, again)
    assert np.array_equal(z[~fixed], z0[~fixed]) and np.array_equal(z[~fixed], poisoned[~fixed])
    assert not np.any(z0[fixed])
    eps = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    assert np.max(np.abs(z[fixed] - 0.6 * 1.4 * r[fixed])) <= 8 * eps * np.max(np.abs(r))
