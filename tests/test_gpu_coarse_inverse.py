"""The coarsest grid's explicit inverse (blocked elimination over all SMs) at
sizes around its block edges: two-level V-cycles against the oracle, whose
coarse solve is a Cholesky factorisation.

Tolerance: an explicit inverse formed from the factor is off by at most a
small multiple of n * unit roundoff * cond_2(A); the rest of the cycle adds a
few roundoffs.  cond_2 is taken from the oracle's matrix."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from oracle import fe, sensitivity, solvers
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu

# kind, grid, coarsest DOFs: below one block, exact blocks, one over, many
GRIDS = [
    ("mbb2d", dict(nelx=2, nely=2), 8),
    ("mbb2d", dict(nelx=6, nely=2), 16),
    ("mbb2d", dict(nelx=2, nely=14), 32),
    ("mbb2d", dict(nelx=32, nely=2), 68),
    ("cantilever3d", dict(nelx=4, nely=2, nelz=2), 36),
    ("cantilever3d", dict(nelx=12, nely=6, nelz=6), 336),
    ("mbb2d", dict(nelx=46, nely=24), 624),
]


@pytest.mark.parametrize("kind,kw,n", GRIDS)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_two_level_vcycle(kind, kw, n, precision):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem(kind, mg_levels=2, **kw)
    g = fe.Grid.of(p)
    rho = rand_density(g.nel, 3, 0.3, 1.0)
    E = sensitivity.simp_modulus(rho, p.E0, p.Emin, p.penal)
    mg = solvers.Multigrid(g, fe.stiffness(g, E, fe.element_stiffness(p.dim, p.nu), p.fixed),
                           p.fixed, 2)
    A = mg.A[-1].toarray()
    assert A.shape[0] == n
    r = rand_vector(g.ndof, 4, fixed=p.fixed)
    ref = mg.vcycle(r)
    with Ctx(p, precision=precision) as c:
        c.set_density(rho)
        z = dev(np.zeros(g.ndof))
        B.to_vcycle(c.ctx, dev(r), z)
        z = host(z)
    eps = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    tol = eps * (100.0 + 4.0 * n * np.linalg.cond(A))
    assert np.linalg.norm(z - ref) <= min(tol, 0.1) * np.linalg.norm(ref)
