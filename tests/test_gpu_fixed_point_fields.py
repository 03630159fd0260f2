"""The float64 finest-grid operator on a field with one component uniform and
the others 1e-8 of it, at Poisson's ratios on either side of the line between
its fixed-point and its float64 kernel.

A uniform component exerts no force, so away from the supports (where masking
breaks the uniformity) the product is that of the other components, to their own
rounding: 1e-13 of the largest entry, as for the other float64 products."""

import numpy as np
import pytest

from gpu_helpers import Ctx, dev, host
from oracle import fe, sensitivity
from workloads import rand_density, rand_vector, small_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nel", [(16, 8, 8), (34, 16, 6)])
@pytest.mark.parametrize("nu", [0.3, 0.45])
@pytest.mark.parametrize("comp", [0, 1, 2])
def test_uniform_component(nel, nu, comp):
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("cantilever3d", nelx=nel[0], nely=nel[1], nelz=nel[2], mg_levels=2, nu=nu)
    rho = rand_density(p.nel, 5, 0.1, 1.0)
    E = sensitivity.simp_modulus(rho, p.E0, p.Emin, p.penal)
    K = fe.stiffness(fe.Grid.of(p), E, fe.element_stiffness(3, nu), p.fixed)
    small = 1e-8 * rand_vector(p.ndof, 6, fixed=p.fixed)
    small[comp::3] = 0.0
    x = small.copy()
    x[comp::3] = 0.7 * (p.fixed[comp::3] == 0)
    nodes = tuple(n + 1 for n in nel[::-1])
    held = p.fixed.reshape(-1, 3).any(1).reshape(nodes)
    near = held.copy()                    # nodes of an element with a held node
    for ax in range(3):
        a = np.moveaxis(near, ax, 0)
        g = a.copy()
        g[1:] |= a[:-1]
        g[:-1] |= a[1:]
        near = np.moveaxis(g, 0, ax)
    away = ~np.repeat(near.ravel(), 3)
    assert away.sum() > p.ndof // 2
    ref = K @ small
    with Ctx(p, precision="fp64") as c:
        c.set_density(rho)
        y = dev(np.zeros(p.ndof))
        B.to_apply(c.ctx, B.TO_OP_K, B.TO_PREC_FP64, dev(x), y)
        y = host(y)
    assert np.max(np.abs(y - ref)[away]) <= 1e-13 * np.max(np.abs(ref))


@pytest.mark.parametrize("nu", [0.3, 0.4, 0.45])
def test_vcycle(nu):
    """Both kernels' residual and smoother epilogues, against the oracle's
    V-cycle (1e-10, as in the parity test)."""
    from oracle import solvers
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("cantilever3d", nelx=24, nely=12, nelz=12, mg_levels=3, nu=nu)
    g = fe.Grid.of(p)
    rho = rand_density(p.nel, 7, 0.2, 1.0)
    E = sensitivity.simp_modulus(rho, p.E0, p.Emin, p.penal)
    K = fe.stiffness(g, E, fe.element_stiffness(3, nu), p.fixed)
    r = rand_vector(p.ndof, 8, fixed=p.fixed)
    ref = solvers.Multigrid(g, K, p.fixed, 3).vcycle(r)
    with Ctx(p, precision="fp64") as c:
        c.set_density(rho)
        z = dev(np.zeros(p.ndof))
        B.to_vcycle(c.ctx, dev(r), z)
        assert np.max(np.abs(host(z) - ref)) <= 1e-10 * np.max(np.abs(ref))


def test_subnormal_results():
    """Results below the normal range keep their bits.  Both sides round every
    product or element force at 2^-1074: 128 units for the oracle's 81 per row."""
    from paper_2205_00385_gb300 import binding as B
    p = small_problem("cantilever3d", nelx=16, nely=8, nelz=8, mg_levels=2)
    rho = rand_density(p.nel, 9, 0.1, 1.0)
    E = sensitivity.simp_modulus(rho, p.E0, p.Emin, p.penal)
    K = fe.stiffness(fe.Grid.of(p), E, fe.element_stiffness(3, p.nu), p.fixed)
    x = 1e-312 * rand_vector(p.ndof, 10, fixed=p.fixed)
    with Ctx(p, precision="fp64") as c:
        c.set_density(rho)
        y = dev(np.zeros(p.ndof))
        B.to_apply(c.ctx, B.TO_OP_K, B.TO_PREC_FP64, dev(x), y)
        y = host(y)
    ref = K @ x
    assert np.max(np.abs(ref)) > 1e-313
    assert np.max(np.abs(y - ref)) <= 128 * 2.0 ** -1074
